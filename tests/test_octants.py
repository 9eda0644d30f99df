"""The octree level translation (csrc/q2x_octants.cu): its table against the
translation matrix written out from the definition (CPU), and its results
against q2x_translate, one translation a child, on the GPU.

Tolerances: a table entry is one or two products of the recursion, at most p
steps of a few roundings of 1.1e-16 each, against the largest entry of its
pair of degrees: 1e-14.  The results are sums of the same terms in another order;
1e-13 in the norm that scales degree n by h^n is the bound of the upward
tests."""
import math

import numpy as np
import pytest


def harmonics(p, t):
    """R_n^m(t) as {(n, m): value} by Eq. (rec2)."""
    x, y, z = t
    R = {(0, 0): 1.0 + 0j}
    for n in range(1, p + 1):
        for m in range(-n, n + 1):
            v = (0.5j * (x + 1j * y) * R.get((n - 1, m - 1), 0) + 0.5j * (x - 1j * y) * R.get((n - 1, m + 1), 0)
                 - z * R.get((n - 1, m), 0))
            R[n, m] = v / n
    return R


def matrix(p, t, norm):
    """The real matrix of the translation by t in packed coefficients."""
    R = harmonics(p, t)
    nc = (p + 1) ** 2
    A = np.zeros((nc, nc))
    for q in range(p + 1):
        for j in range(-q, q + 1):
            F = {(q, abs(j)): 1.0 if j >= 0 else 1j}
            F[q, -abs(j)] = (-1) ** j * np.conj(F[q, abs(j)])
            for n in range(q, p + 1):
                for m in range(n + 1):
                    k = n - q
                    v = sum((R.get((k, m - s), 0) if norm else (-1) ** k * R.get((k, s - m), 0)) * F[q, s]
                            for s in {j, -j})
                    A[n * n + n + m, q * q + q + j] = np.real(v)
                    if m:
                        A[n * n + n - m, q * q + q + j] = np.imag(v)
    return A


def parity(n, m):
    im, am = int(m < 0), abs(m)
    return im | ((am + im) % 2) << 1 | ((n + am) % 2) << 2


def decode(buf, p):
    """The rows of the table's matrix, and the parity index of each term."""
    nc = (p + 1) ** 2
    nt = (nc + 31) // 32 * 32
    head = buf[:16].view(np.int32)
    A, C = np.zeros((nc, nc)), np.full((nc, nc), -1)
    rows = []
    for q in range(head[3]):
        r0, r1, nj, steps, terms, slots, val, code, start, first = buf[16 + 40 * q:56 + 40 * q].view(np.int32)
        rows.append((r0, r1))
        assert slots <= nc + nt
        f = buf[first:first + 2 * (r1 - r0 + 1)].view(np.uint16)
        for run in range(nt):
            n = min(steps, terms - run * steps)
            slot = int(buf[start + 2 * run:start + 2 * run + 2].view(np.uint16)[0])
            for k in range(max(n, 0)):
                a = val + 8 * (k * nt + run)
                b = code + 2 * (k * nt + run)
                cd = int(buf[b:b + 2].view(np.uint16)[0])
                i = r0 + int(np.searchsorted(f, slot, side="right")) - 1
                c, j = divmod(cd & 0xfff, nc)
                assert j < nj and C[i, j] < 0
                A[i, j], C[i, j] = buf[a:a + 8].view(np.float64)[0], c
                slot += cd >> 15
    assert rows[0][0] == 0 and rows[-1][1] == nc and all(a[1] == b[0] for a, b in zip(rows, rows[1:]))
    return A, C


@pytest.mark.parametrize("norm", [0, 1])
@pytest.mark.parametrize("p,n_dst", [(0, 1), (1, 7), (2, 1000), (4, 1), (7, 3), (9, 100), (12, 1), (12, 5000)])
def test_table(p, n_dst, norm):
    from paper_2107_10942_gb300.q2x import octant_table_host
    h = 0.37
    A, C = decode(octant_table_host(p, norm, h, n_dst).numpy(), p)
    want = matrix(p, (h, h, h), norm)
    n = np.array([k for k in range(p + 1) for _ in range(2 * k + 1)])
    big = np.array([h ** k / math.factorial(k) for k in range(p + 1)])
    d = np.maximum(n[:, None] - n[None, :], 0)
    assert np.all(np.abs(A - want) <= 1e-14 * big[d])
    chi = np.array([parity(k, m) for k in range(p + 1) for m in range(-k, k + 1)])
    has = C >= 0
    assert np.all(C[has] == (chi[:, None] ^ chi[None, :])[has]) and has.diagonal().all()
    for o in range(8):  # the mirrored shifts by signs
        s = np.array([(-1) ** bin(c & o).count("1") for c in chi])
        t = [-h if o >> b & 1 else h for b in range(3)]
        assert np.all(np.abs(s[:, None] * A * s[None, :] - matrix(p, t, norm)) <= 1e-14 * big[d])


@pytest.mark.gpu
@pytest.mark.parametrize("norm", ["coeff", "moment"])
@pytest.mark.parametrize("p,n_dst", [(0, 3), (1, 40), (3, 1), (5, 1000), (12, 1), (12, 40), (12, 700), (20, 2), (20, 300)])
def test_against_translate(p, n_dst, norm):
    """Full, partly filled and empty parents, octants in any order and twice,
    adding to what is there, and an octant that does not exist."""
    import torch

    import paper_2107_10942_gb300 as q2x
    rng = np.random.default_rng(p * 1000 + n_dst)
    h, nc = 0.21, (p + 1) ** 2
    octs = [rng.permutation(8)[:rng.integers(0, 9)] for _ in range(n_dst)]
    octs[0], octs[-1] = np.array([5, 5, 0, 7]), np.arange(8)
    oct_ = np.concatenate(octs).astype(np.int32)
    off = np.concatenate([[0], np.cumsum([len(o) for o in octs])]).astype(np.int64)
    dst_c = rng.integers(-8, 8, (3, n_dst)) * 0.5
    t = np.where((oct_[None, :] >> np.arange(3)[:, None]) & 1, -h, h)
    src_c = np.repeat(dst_c, np.diff(off), axis=1) + t
    n = np.array([k for k in range(p + 1) for _ in range(2 * k + 1)])
    scale = h ** n / np.array([float(math.factorial(k)) for k in n])
    src = rng.standard_normal((len(oct_), nc)) * scale
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    plan = q2x.Plan(p, norm=norm)
    table = plan.octant_table(h, n_dst)
    want = plan.translate(dev(src), dev(src_c), dev(off), dev(dst_c))
    got = plan.translate_octants(dev(src), table, dev(oct_), dev(off))
    again = plan.translate_octants(dev(src), table, dev(oct_), dev(off), dst_coef=got.clone(), accumulate=True)
    assert plan.device_errors() == 0
    err = ((got - want).cpu().numpy() / scale).reshape(n_dst, -1)
    top = np.abs(want.cpu().numpy() / scale).max(axis=1, keepdims=True)
    assert np.all(np.abs(err) <= 1e-13 * np.where(top > 0, top, 1.0))
    assert torch.equal(again, 2 * got)
    bad = oct_.copy()
    bad[1] = 8
    less = np.delete(np.arange(len(oct_)), 1)
    off2 = np.maximum(off - (off > 1), 0)
    got = plan.translate_octants(dev(src), table, dev(bad), dev(off))
    assert plan.device_errors() & 1
    want = plan.translate_octants(dev(src[less]), table, dev(oct_[less]), dev(off2))
    assert torch.equal(got, want)
    with pytest.raises(ValueError):
        plan.translate_octants(dev(src), plan.octant_table(h, n_dst + 1), dev(oct_), dev(off))


@pytest.mark.gpu
@pytest.mark.parametrize("norm", ["coeff", "moment"])
@pytest.mark.parametrize("p", [0, 1, 2, 12, 20])
def test_rounded_centres(p, norm):
    """Shifts that differ from +-h by up to 1e-10 h: as accurate as with their
    own shifts (the second order, 190 x 1e-20, is far below the tolerance), and
    1e-10 n off, so beyond it, without the rest."""
    import torch

    import paper_2107_10942_gb300 as q2x
    rng = np.random.default_rng(p)
    h, nc, n_dst = 0.21, (p + 1) ** 2, 30
    oct_ = np.tile(np.arange(8), n_dst).astype(np.int32)
    off = np.arange(0, 8 * n_dst + 1, 8).astype(np.int64)
    sign = np.where((oct_[None, :] >> np.arange(3)[:, None]) & 1, -h, h)
    delta = h * 1e-10 * rng.uniform(-1, 1, sign.shape)
    src_c = sign + delta
    delta = src_c - sign
    n = np.array([k for k in range(p + 1) for _ in range(2 * k + 1)])
    scale = h ** n / np.array([float(math.factorial(k)) for k in n])
    src = rng.standard_normal((len(oct_), nc)) * scale
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    plan = q2x.Plan(p, norm=norm)
    table = plan.octant_table(h, n_dst)
    want = plan.translate(dev(src), dev(src_c), dev(off), dev(np.zeros((3, n_dst)))).cpu().numpy()
    top = np.abs(want / scale).max(axis=1, keepdims=True)
    for rest in (dev(delta), None):
        got = plan.translate_octants(dev(src), table, dev(oct_), dev(off), delta=rest).cpu().numpy()
        ok = np.abs(got - want) / scale <= 1e-13 * top
        assert ok.all() if rest is not None or p == 0 else not ok.all()
    assert plan.device_errors() == 0


@pytest.mark.gpu
def test_upward_in_any_cube():
    """A cube whose centres are rounded: the pass as with each child's own shift."""
    import torch

    import paper_2107_10942_gb300 as q2x
    from paper_2107_10942_gb300.upward import Upward
    p, depth, lo, size = 8, 6, -1.1, 2.3
    rng = np.random.default_rng(2)
    ijk = np.unique(rng.integers(0, 1 << depth, (500, 3)), axis=0)
    leaf_c = (lo + (ijk.T + 0.5) * (size / (1 << depth)))
    n = np.array([k for k in range(p + 1) for _ in range(2 * k + 1)])
    h = size / (2 << depth)
    coef = torch.from_numpy(rng.standard_normal((len(ijk), (p + 1) ** 2)) * h ** n).cuda()
    up = Upward(q2x.Plan(p), leaf_c, lo, size, depth, device="cuda")
    assert any(o is not None and o[2] is not None for o in up.octants)
    one = [x.clone() for x in up.run(coef, precomputed_shifts=False)]
    for k, (a, b) in enumerate(zip(up.run(coef), one)):
        s = (h * 2.0 ** (k + 1)) ** n
        assert float(((a - b).cpu().abs() / torch.from_numpy(s)).max()) <= 1e-13 * float((b.cpu().abs() / torch.from_numpy(s)).max())
