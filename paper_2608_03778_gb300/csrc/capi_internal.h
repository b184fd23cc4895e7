// Internal state of the C-ABI objects, shared by the translation units that
// implement the entry points (capi.cu: single scenario; capi_batch.cu:
// batched scenarios, power-virus evaluation).
#pragma once
#include <cstdint>
#include <string>
#include <vector>

#include "diffpower.h"
#include "kernels.h"

struct dp_ctx {
    int device = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    int sm_count = 0;
    int clock_khz = 0;
    int *d_err = nullptr;   // device error word: a bounded wait gave up
    bool switched = false;  // the calls have been on more than one stream
    std::string err;
};

// Buffers of the batched path (S scenarios, scenario innermost).  They are
// sized for `cap` scenarios and reallocated only when a larger S arrives.
struct dp_batch {
    int64_t S = 0;                 // scenarios of the staged inputs
    int64_t cap = 0;               // scenarios the buffers hold
    dp::BatchBufs b{};
    double *weights = nullptr;     // [cap] staging of host weights
    float *stage = nullptr;        // [max(n_nets, n_cells) * cap] staging of host outputs (lazy)
    std::vector<void *> allocs;    // freed together on reallocation
    size_t bytes = 0;
    bool fwd_valid = false;
    int fwd_tr_mode = -1;
    dp::BatchShape fwd_shape{128, 1}, bwd_shape{128, 1};
    dp::GroupShape fwd_group, bwd_group;   // group passes that were faster than the level launches at tuned_S
    int fwd_flow = 0, bwd_flow = 0;        // scenarios per thread of the dataflow passes, where faster than both (0: not)
    bool flow_refused = false;     // the runtime refused a dataflow pass's cooperative launch: the others run
    int flow_sms = 0;              // > 0: a self-test's SM count for its grid
    int groups_fit = -1;           // the device has room for the groups' clusters of 16 blocks (-1: not asked yet)
    bool shape_from_env = false;   // DP_BATCH_SHAPE fixed the level launches
    int64_t tuned_S = 0;           // S the shapes were tuned for (0: not tuned)
    bool shapes_locked = false;    // keep the shapes whatever S comes (a server fixes them once)
    float tune_ms[2] = {0.f, 0.f}; // best forward / backward time of the level launches seen by the tuner
    float pass_ms[2] = {0.f, 0.f}; // ... of all passes: the ones in use (0: not timed)
    // power-virus evaluation (Eq. 3): words [n_nets * 2 ceil(S/64)], partials, sums, staging
    int64_t vcap = 0;
    uint64_t *vwords = nullptr;
    double *vpart = nullptr, *vout = nullptr;
    float *vsp = nullptr;
    uint8_t *vv0 = nullptr;
    std::vector<void *> vallocs;
    size_t vbytes = 0;
};

struct dp_design {
    dp_ctx *ctx = nullptr;
    dp::DevDesign d{};
    dp::OpTable ops{}, cell_ops{};   // the function table; the same with the functions' classes, for the batched passes
    std::vector<int32_t> lvl_ptr;
    int64_t n_edges = 0;
    int32_t n_ops = 0;
    std::vector<void *> allocs;
    size_t bytes = 0;
    int words_T = 0;
    // output staging for host outputs
    float *st_gsp = nullptr, *st_gtr = nullptr, *st_gpin = nullptr, *st_gcl = nullptr;
    // state
    bool inputs_set = false;
    bool batched = false;          // the staged inputs are a batch (dp_set_inputs_batch)
    bool fwd_valid = false;
    int fwd_tr_mode = -1;
    bool sim_valid = false;
    bool bwd_valid = false;        // gnet holds the adjoint of the current state
    int bwd_grad_mode = -1;
    // staging of host sizing deltas (dp_set_pincap): grown on demand, never shrunk; pc_done is
    // recorded after the kernels that read it, so a later call waits for them on any stream
    int32_t *pc_cells = nullptr;
    float *pc_caps = nullptr;
    int64_t pc_cap = 0;
    cudaEvent_t pc_done = nullptr;
    // sizing-score scratch (lazy): scores [n_cells], candidates [n_cells], selection state, and for the ordering
    // the candidates' keys and the ordered cells and scores
    float *sc_scores = nullptr;
    int32_t *sc_idx = nullptr;
    unsigned *sc_state = nullptr;
    unsigned long long *sc_keys = nullptr;
    int32_t *sc_top = nullptr;
    float *sc_tops = nullptr;
    dp_batch batch;
    // graph of the whole step for one config
    cudaGraphExec_t graph = nullptr;
    dp_config graph_cfg{};
    cudaStream_t cap_stream = nullptr, cap_stream2 = nullptr;
    cudaEvent_t fork = nullptr, join = nullptr;
    // the step's output copies: a side stream that starts them when the gradient branch of
    // the step graph is done (ev_grads, recorded by the graph), and their completion
    cudaStream_t out_stream = nullptr;
    cudaEvent_t ev_grads = nullptr, ev_copies = nullptr;
    // a dp_simulate that directly follows a dp_propagate may start beside it, at ev[0]: nothing queued on the stream
    // since writes what it reads or uses what it writes.  Not once any call on the design has been captured: a replay
    // of the user's graph queues that call's work without the library knowing
    bool sim_ahead = false;
    bool captured = false;
    int grid[4] = {0, 0, 0, 0};   // persistent grids: forward, simulation, backward, wide simulation
    int flow_grid[3] = {0, 0, 0};  // dataflow grids: forward, simulation, reverse
    int block_threads = 0;         // > 0: the design fits the single-block passes, with this many threads
    dp::SlicePlan sl;              // the sliced simulation (sl.slots > 0: the design uses it)
    dp::ClusterMap cl;             // the single-cluster passes (cl.threads > 0: the design uses them)
    int64_t graph_kernels = 0;
    int64_t step_kernels = 0;
    // phase boundaries: start, forward, simulation levels, hybrid + power, backward, outputs
    cudaEvent_t ev[6] = {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
    bool ev_valid[6] = {false, false, false, false, false, false};
};

namespace dpi {

struct DeviceGuard {
    int prev = -1;
    explicit DeviceGuard(int dev) {
        if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
        if (prev != dev) cudaSetDevice(dev);
    }
    ~DeviceGuard() {
        int cur = -1;
        if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
    }
};

dp_status set_err(dp_ctx *c, dp_status s, const std::string &m);
dp_status cuda_err(dp_ctx *c, cudaError_t e, const char *where);
dp_status launch_check(dp_ctx *c, const char *where);
// Reads and clears the device error word (synchronises the stream).
dp_status check_device_error(dp_ctx *c);
// cudaMalloc of `bytes` with the DP_FAULT=alloc:N injection; the pointer is
// appended to *list and its size added to *total.
dp_status alloc_into(dp_ctx *c, void **p, size_t bytes, std::vector<void *> *list, size_t *total);
double power_K(const dp_config &c);
dp_status check_cfg(dp_ctx *ctx, const dp_config *c);
// true when the stream is being captured into a CUDA graph
bool capturing(cudaStream_t s);
// dp_design_upload; simulates: with the tables of the sliced simulation (a server's designs do without)
dp_status upload_design(dp_ctx *ctx, const dp_compiled *cp, bool simulates, dp_design **out);
// notes a call on the design that is being captured (every entry point that queues work on its single-scenario state)
inline void note_capture(dp_design *D) { D->captured = D->captured || capturing(D->ctx->stream); }
// frees the batched buffers (the caller has synchronised)
void free_batch(dp_design *D);
// batched halves of dp_propagate, dp_get_power and dp_get_nets (capi_batch.cu)
dp_status batch_propagate(dp_design *D, const dp_config &c);
// the forward and the reverse pass of the staged batch (B.S scenarios), by groups or by levels
cudaError_t batch_forward(dp_design *D, int tr_mode, cudaStream_t s);
cudaError_t batch_reverse(dp_design *D, int tr_mode, cudaStream_t s);
dp_status batch_get_power(dp_design *D, int hybrid, double *watts, int on_device);
dp_status batch_get_nets(dp_design *D, float *sp, float *tr, int on_device);
// batch buffers for S scenarios plus the host-output staging (synchronises; not under capture)
dp_status batch_reserve(dp_design *D, int64_t S);
// runs the launch-shape tuner on the staged batch of B.S scenarios, then locks the shapes
dp_status batch_tune_and_lock(dp_design *D);

template <class T>
dp_status dalloc(dp_design *D, T **p, size_t count) {
    void *v = nullptr;
    dp_status s = alloc_into(D->ctx, &v, sizeof(T) * (count ? count : 1), &D->allocs, &D->bytes);
    *p = static_cast<T *>(v);
    return s;
}

}  // namespace dpi
