// q2x_plan.h -- the plan object behind q2x_plan_t (internal to the library).
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <memory>
#include <string>
#include <utility>
#include <vector>

#include "q2x.h"

// A far-field call's scratch that a captured graph owns: `dropped` is set when
// the graph and its instances are gone (q2x_plan_scratch), and the plan frees
// or reuses the memory then.
struct q2x_graph_scratch {
    void* p = nullptr;
    size_t bytes = 0;
    std::shared_ptr<std::atomic<bool>> dropped;
};

struct q2x_plan_s {
    int p_max = 0;
    int norm = 0;
    int prec = 0;  // 0 FP64, 1 FP32-mixed
    cudaStream_t stream = nullptr;
    int device = 0;
    int num_sms = 0;
    unsigned* d_err = nullptr;
    unsigned* h_err = nullptr;  // pinned
    void* ws = nullptr;
    size_t ws_bytes = 0;
    bool ws_captured = false;     // a captured graph uses ws: it is kept when a larger one takes its place
    std::vector<std::pair<void*, size_t>> ws_kept;
    // far-field scratch (q2x_plan_scratch)
    void* far = nullptr;
    size_t far_bytes = 0;
    cudaStream_t far_stream = nullptr;  // of the last call that used it
    cudaEvent_t far_left = nullptr;     // recorded when the plan leaves that stream
    std::vector<q2x_graph_scratch> far_graphs;
    int occ_cache[2][9][5] = {};  // [precision][element combo][capacity bin]
    int tile_occ[4][5] = {};  // resident CTAs per SM of the FP32 leaf-tile kernels [combo][bin]
    int dir_occ[9][11] = {};  // resident CTAs per SM of the FP64 direction kernels [warps per CTA][combo]
    int timing = 0;
    std::vector<cudaEvent_t> ev_pool;                            // idle events
    std::vector<std::pair<cudaEvent_t, cudaEvent_t>> ev_pending;  // recorded pairs
    int64_t launches = 0;
    std::string last_error;
};

// While memory is given back: the thread may be capturing a graph on a stream
// of its own (a garbage collector runs when it likes), and neither a wait on the
// legacy stream nor cudaFree may end that capture.  Waits for the plan's stream
// where that can be waited for; freeing waits by itself.
struct q2x_release {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    explicit q2x_release(cudaStream_t st)
    {
        cudaThreadExchangeStreamCaptureMode(&mode);
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(st, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone)
            cudaStreamSynchronize(st);
        else
            cudaGetLastError();
    }
    ~q2x_release() { cudaThreadExchangeStreamCaptureMode(&mode); }
    q2x_release(const q2x_release&) = delete;
    q2x_release& operator=(const q2x_release&) = delete;
};

// status helpers shared by the library's translation units
q2x_status q2x_fail(q2x_plan_t plan, q2x_status st, const char* fmt, ...);
q2x_status q2x_cuda_fail(q2x_plan_t plan, cudaError_t e, const char* what);
// grow the plan's device workspace to at least `bytes` (synchronises the
// plan's stream when it has to reallocate; a workspace that a captured graph
// uses is kept until the plan goes)
q2x_status q2x_plan_workspace(q2x_plan_t plan, size_t bytes);
// Scratch of one call on the plan's stream that no other call shares while it
// runs: calls on one stream follow one another in the plan's buffer, a call on
// another stream waits for them, and a captured call has a buffer of its own
// that lives as long as its graph.  *out NULL (and Q2X_OK) where there is none
// to be had.
q2x_status q2x_plan_scratch(q2x_plan_t plan, size_t bytes, void** out);
// Receiver-side integration by the direction kernels (q2x_api.cu): *taken
// false where the call has to take the row kernel (its tile list would not fit).
q2x_status q2x_galerkin_directions(q2x_plan_t plan, int64_t n_elem, int64_t n_vert, const double* vxyz,
                                   const int32_t* idx, const double* sigma, int64_t n_leaves, const int64_t* leaf_off,
                                   const double* leaf_c, int layer, const double* w, double* out, bool* taken);
