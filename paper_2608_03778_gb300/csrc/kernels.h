// Launch wrappers for the GPU kernels (implemented in kern_*.cu).
#pragma once
#include <cstdint>

#include <cuda_runtime.h>

namespace dp {

// The functions whose truth tables are compiled into the batched passes (kern_cells.cuh): class, inputs, table.
// Any other function of k inputs: class 18 + k.
#define DP_CELL_CLASSES(X)                                                                                     \
    X(1, 1, 0x1u) X(2, 1, 0x2u)                                                           /* INV BUF */         \
    X(3, 2, 0x8u) X(4, 2, 0x7u) X(5, 2, 0xEu) X(6, 2, 0x1u) X(7, 2, 0x6u) X(8, 2, 0x9u)   /* AND..XNOR, 2 */    \
    X(9, 3, 0x80u) X(10, 3, 0x7Fu) X(11, 3, 0xFEu) X(12, 3, 0x01u)                        /* AND..NOR, 3 */     \
    X(13, 3, 0x07u) X(14, 3, 0xF8u) X(15, 3, 0x1Fu) X(16, 3, 0xE0u) X(17, 3, 0xE2u)       /* AOI21 AO21 OAI21 OA21 MUX2 */
inline uint32_t cell_class(uint32_t k, uint32_t tt) {
#define DP_CELL(I, K, TT) if (k == K && tt == TT) return I;
    DP_CELL_CLASSES(DP_CELL)
#undef DP_CELL
    return 18 + k;
}

// Per-design function table passed by value to kernels (lives in the
// constant bank): entry = truth table (bits 0..15) | arity << 16 | (batched passes only) class << 19 |
// (for arity <= 3) the 8-bit LOP3 table of the function << 24, whose entry
// 4 x2 + 2 x1 + x0 is f(x0, x1, x2) (inputs beyond the arity ignored).
struct OpTable {
    uint32_t e[256];
};

constexpr int kPersistThreads = 512;
// the persistent forward pass runs beside the startpoint generator: a smaller block leaves
// the generator more registers on every SM (one block of 256 threads per SM still gives one
// thread per cell of a 38,912-cell level)
constexpr int kFwdThreads = 256;
constexpr int kSimThreads = 512;
// the single-block passes of small designs: at most kBlockMaxWidth cells per level
// (one per thread) and state within kBlockSmemMax bytes of shared memory
constexpr int kBlockThreads = 1024;
constexpr int kBlockMaxWidth = kBlockThreads;
constexpr int kBlockSmemMax = 224 * 1024;   // dynamic; the 227 KiB a block may hold less room for static arrays
// bounded waits give up after this many SM cycles (about 2 s at 2 GHz)
constexpr long long kWaitLimitCycles = 4000000000LL;

// Device-resident design state; every pointer is device memory.
struct DevDesign {
    int64_t n_nets, n_start, n_cells;
    int32_t n_levels;
    const uint4 *fanin;        // [n_cells]: 4 internal net ids, logic id in bits 24..31 of .x
    const int32_t *fout_ptr;   // [n_nets+1]
    const int32_t *fout_edge;  // [n_edges]: 4*cell + slot
    const int32_t *edge_fpos;  // [4*n_cells]: position of edge (cell, slot) in the fanout CSR, -1 unused
    const int32_t *lvl;        // [n_levels+1] level boundaries over internal cells
    const int32_t *net_of_user;
    const int32_t *cell_of_user;
    const float *base_cap;     // wire + DFF D pin caps
    float *pincap;             // [n_cells]
    float *cload;              // [n_nets]
    float *sp_in, *tr_in;      // [n_start] staged inputs
    float4 *pq;                // [n_nets] (P(net=1), P(net=0)) as float-float pairs (P.hi, P.lo, Q.hi, Q.lo)
    float *tr;                 // [n_nets] TR_model (startpoints: input TR in tr_mode 0)
    float *beta, *trh;         // [n_nets] beta and hybrid TR
    uint32_t *toggles, *ones;  // [n_nets]
    float *gnet;               // [n_nets] SP adjoint per net
    float *gfo;                // [n_edges] adjoint contribution of each edge, in fanout-CSR order
    unsigned long long *edges; // [n_edges] the dataflow reverse pass's edges, in fanout-CSR order: partial
                               // derivative, sink cell << 32
    uint64_t *words;           // [n_nets * T]
    double *partials;          // [2 * power_blocks]
    double *power;             // [4]: model, hybrid
    unsigned *bar;             // level-barrier arrival counters of the persistent passes (128-byte lines)
    unsigned long long *gcell; // [n_cells] the dataflow reverse pass's cell adjoints: value, pass number << 32
    uint32_t *epoch;           // [8] pass counters: [0] forward (its parity tags the stored pairs), [1] dataflow
                               // simulation, [2] dataflow reverse; [4], [5] blocks done of [0], [2] and [3] a wait
                               // of [0] gave up (0 at rest)
    const int32_t *pair_ptr;   // [n_levels+1] level-aligned cell pairs: pairs of level l are [pair_ptr[l-1], pair_ptr[l])
    unsigned *simdone;         // [n_cells] pass number of the simulation pass that last wrote the cell's words
    const int32_t *dead_ptr;   // [n_levels+2] nets by death level d (the highest level reading the net, else
    const int32_t *dead_net;   // [n_nets]      its own): dead_net[dead_ptr[d] .. dead_ptr[d+1])
    int *err;                  // device error word of the context (bounded wait gave up)
};

constexpr int kPowerBlocks = 304;   // fixed grid of the power reduction -> deterministic order
constexpr int kPowerThreads = 256;

// forward (kern_fwd.cu)
void launch_init_start(const DevDesign &d, int tr_mode, cudaStream_t s);
void launch_fwd_level(const DevDesign &d, const OpTable &ops, int32_t c0, int32_t c1, cudaStream_t s);
void launch_cload(const DevDesign &d, cudaStream_t s);
void launch_set_pincap(const DevDesign &d, const int32_t *cells, const float *caps, int32_t n, cudaStream_t s);
// power: sum_n alpha_n C_n (alpha = tr, or beta*tr when hybrid), times K, into d.power[slot]
// (and, after a forward pass in which a wait gave up, the pairs' tags)
void launch_power(const DevDesign &d, bool hybrid, double K, int slot, cudaStream_t s);
// outputs in user order: grad_cload (K alpha), grad_pincap (K sum fanin alpha), grad_tr_in (K beta C or 0)
void launch_cap_grads(const DevDesign &d, const OpTable &ops, bool hybrid, int tr_mode, double K, float *grad_cload,
                      float *grad_pincap, float *grad_tr_in, cudaStream_t s);
// per-net results of the single-scenario passes in user order (NULL: not wanted)
struct NetOutputs {
    float *sp, *tr, *beta, *trh;
    uint32_t *toggles, *ones;
};
void launch_nets_user(const DevDesign &d, const NetOutputs &o, cudaStream_t s);

// backward (kern_bwd.cu)
void launch_bwd_level(const DevDesign &d, const OpTable &ops, int32_t c0, int32_t c1, int grad_mode, float K,
                      cudaStream_t s);
void launch_bwd_start(const DevDesign &d, int grad_mode, int tr_mode, float K, float *grad_sp_in, cudaStream_t s);

// pass counters and the dataflow schedule (kern_flow.cu); the passes advance their own counters
void launch_bump(uint32_t *counter, cudaStream_t s);
int flow_grid(int which, int sm_count);   // which: 0 forward, 1 simulation, 2 reverse; 0 = unavailable
cudaError_t launch_fwd_flow(const DevDesign &d, const OpTable &ops, int tr_mode, int grid, cudaStream_t s);
// the reverse pass in two kernels: the partial derivatives and local terms, which need the forward pass
// only (so they can run beside the simulation), then the levels.  cells: the partial derivatives by cell
// (the cluster's pass); NULL: by fanout edge, with the sink cell, into d.edges
void launch_bwd_coef(const DevDesign &d, const OpTable &ops, int tr_mode, float K, float *cells, cudaStream_t s);
cudaError_t launch_bwd_flow(const DevDesign &d, int grad_mode, float *out_gsp, int grid, cudaStream_t s);
// simulation levels without barriers (T % 4 == 0), bumps epoch[1] first
cudaError_t launch_sim_flow(const DevDesign &d, const OpTable &ops, int T, int grid, cudaStream_t s);

// persistent schedule (kern_persist.cu): one cooperative launch per pass
int persist_grid(int which, int sm_count);   // which: 0 forward, 1 simulation, 2 backward, 3 wide simulation
bool wide_ok(int T);                         // the wide simulation handles this word count
cudaError_t launch_sim_wide(const DevDesign &d, const OpTable &ops, int T, int grid, cudaStream_t s);
size_t persist_bar_words(int n_levels);      // counters needed by the three passes
// the forward and the reverse pass of a mid-size design in one cluster of kClusterBlocks blocks
// (kern_cluster.cu): every level cut into one contiguous chunk per block, each net kept in the
// shared memory of the block that computes it; no barrier between levels, a cell waits for its own inputs.
constexpr int kClusterBlocks = 16;
constexpr int kClusterMaxThreads = 512;
struct ClusterMap {
    int threads = 0;                    // threads per block (0: the design does not use the cluster)
    int64_t slots = 0;                  // the most nets one block holds
    int64_t edges = 0;                  // the most edge adjoints one block holds
    const int32_t *chunk = nullptr;     // [L+1] cells of level l per block (level 0: the startpoints)
    const int32_t *base = nullptr;      // [C][L+1] first slot of block b's chunk of level l
    const int32_t *floc = nullptr;      // [4 nc] location of each input net: owner block << 24 | slot
    const int32_t *range = nullptr;     // [2 nn] net n's fanout range in its owner's copy: first, count
    const int32_t *push = nullptr;      // [4 nc] each input edge's place: owner block << 24 | position, -1 unused
    float *coef = nullptr;              // [4 nc] the reverse pass's partial derivatives
};
// cluster_smem: dynamic shared memory per block (0 forward, 1 reverse, 2 the state of both passes,
// which decides whether a design takes the cluster); cluster_fits:
// whether one such cluster can run on this device (also sets the kernels' shared-memory and
// cluster-size attributes)
size_t cluster_smem(int which, int64_t slots, int64_t n_edges_local, int n_levels);
bool cluster_fits(int threads, size_t smem_fwd, size_t smem_bwd);
cudaError_t launch_fwd_cluster(const DevDesign &d, const OpTable &ops, const ClusterMap &m, int tr_mode,
                               cudaStream_t s);
cudaError_t launch_bwd_cluster(const DevDesign &d, const ClusterMap &m, int grad_mode, float *out_gsp,
                               cudaStream_t s);   // after launch_bwd_coef with m.coef

// the forward and the reverse pass of a small design in one block (kern_persist.cu);
// block_smem(0 forward, 1 reverse, ...): the dynamic shared memory each needs;
// block_smem_init: raises the kernels' shared-memory limit to kBlockSmemMax (once)
size_t block_smem(int which, int64_t n_nets, int64_t n_edges, int n_levels);
bool block_smem_init();
// (the forward kernel also advances the pass counter)
cudaError_t launch_fwd_block(const DevDesign &d, const OpTable &ops, int tr_mode, int threads, cudaStream_t s);
cudaError_t launch_bwd_block(const DevDesign &d, const OpTable &ops, int grad_mode, int tr_mode, float K,
                             float *out_gsp, int64_t n_edges, int threads, cudaStream_t s);
// ready (may be null) is recorded on s just before the kernel: a branch forked there becomes
// ready with it rather than ahead of it
cudaError_t launch_fwd_persist(const DevDesign &d, const OpTable &ops, int tr_mode, int grid, cudaStream_t s,
                               cudaEvent_t ready = nullptr);
cudaError_t launch_sim_persist(const DevDesign &d, const OpTable &ops, int T, int grid, cudaStream_t s);
// pre: the form that loads each level's static part a level ahead (about 120 registers: no
// other kernel fits beside it on an SM); otherwise the 64-register form
cudaError_t launch_bwd_persist(const DevDesign &d, const OpTable &ops, int grad_mode, int tr_mode, float K,
                               float *out_gsp, int grid, bool pre, cudaStream_t s);
cudaError_t launch_wait_selftest(unsigned *bar, int *err, long long limit, cudaStream_t s);
// latency probes (buffers owned by the caller; bar zeroed by the caller, 32 words per level)
cudaError_t launch_probe_levels(float *buf, int levels, int gather, int grid, int threads, unsigned *bar, int *err,
                                cudaStream_t s);
cudaError_t launch_probe_chase(const uint32_t *next, int hops, uint32_t *sink, cudaStream_t s);

// Batched scenarios (kern_batch.cu): S scenarios of one design, every per-net
// value stored scenario-innermost (value[n * S + s]).
struct BatchBufs {
    int64_t S;
    float *sp_in, *tr_in;   // [n_start * S] staged inputs
    float2 *pq;             // [n_nets * S] float-float P(net=1) (hi, lo; bit 30 of lo: tag); P(net=0) = 1 - P re-derived
    float *gfo;             // [n_edges * S] edge adjoints in fanout-CSR order
    float *gsp;             // [n_start * S] SP adjoint of the startpoints
    double *partials;       // [kBatchPowerChunks * S]
    double *power;          // [S] model power per scenario
    float *ks;              // [S] per-scenario seed of the backward (K * weight), binary32
    const float *dcl;       // [n_nets * S] per-scenario change of C_load (sizing deltas), or NULL
    uint32_t *state;        // [8] the dataflow passes' (0 at rest): [0] columns of pq if such a pass wrote it, else 0;
                            // [1] forward passes; [2] 1: every word of gfo is at rest; [3], [4] blocks done; [5] as [2], of gfo2;
                            // [6], [7] a wait of the pass that runs gave up (forward, reverse)
    // lag-one mode (tr_mode 2) only, else NULL:
    float *tq;              // [n_nets * S] TR of every net
    float2 *gfo2;           // [n_edges * S] edge adjoints of (P, TR)
    float *gtr;             // [n_start * S] TR adjoint of the startpoints
};
constexpr int kBatchPowerChunks = 1024;   // fixed split of the nets -> deterministic FP64 sums

struct BatchShape {
    int bx, by;   // threads over scenarios x cells per block
    int v = 1;    // scenarios per thread in the forward and reverse cell levels (1, 2 or 4; 1 unless S is a multiple)
};

void launch_fwdb(const DevDesign &d, const BatchBufs &b, const OpTable &ops, const int32_t *lvl_host, int tr_mode,
                 BatchShape sh, cudaStream_t s);
// lag-one mode (kern_lag1.cu): forward of (P, TR) and reverse pass of both adjoints
void launch_fwdl(const DevDesign &d, const BatchBufs &b, const OpTable &ops, const int32_t *lvl_host, BatchShape sh,
                 cudaStream_t s);
void launch_bwdl(const DevDesign &d, const BatchBufs &b, const OpTable &ops, const int32_t *lvl_host, BatchShape sh,
                 cudaStream_t s);
// the same passes by scenario groups, one launch each (kern_group.cu): groups of lanes x v scenarios, each on a
// cluster of `blocks` blocks of `threads` threads (v = 0: not used; S a multiple of v)
struct GroupShape {
    int lanes = 0, v = 0, blocks = 0, threads = 0;
};
// a block is whole rows of lanes threads, at least one (a stride of no rows would never end), in whole warps
inline bool group_ok(const GroupShape &g) {
    return (g.v == 1 || g.v == 2 || g.v == 4) && g.blocks >= 1 && g.blocks <= 16 && (g.blocks & (g.blocks - 1)) == 0 &&
           g.threads >= 32 && g.threads <= 512 && (g.threads & 31) == 0 && g.lanes >= 1 && g.lanes <= g.threads &&
           g.threads % g.lanes == 0;
}
// the shape as a pass runs it: the lag-one state takes two scenarios' registers, in twice the lanes where they still
// make whole rows
inline GroupShape group_for(GroupShape g, int tr_mode) {
    if (tr_mode == 2 && g.v == 4) {
        g.v = 2;
        if (g.threads % (2 * g.lanes) == 0) g.lanes *= 2;
    }
    return g;
}
// whether clusters of `blocks` full blocks can run on this device, in every mode with one or two scenarios per thread
bool group_fits(int blocks);
cudaError_t launch_fwdb_group(const DevDesign &d, const BatchBufs &b, const OpTable &ops, int tr_mode, GroupShape sh,
                              cudaStream_t s);
cudaError_t launch_bwdb_group(const DevDesign &d, const BatchBufs &b, const OpTable &ops, int tr_mode, GroupShape sh,
                              cudaStream_t s);
// the same passes in one launch each without barriers between levels (kern_flowb.cu): v scenarios
// per thread (S a multiple of v; in the lag-one mode at most 2); edges: the elements of gfo.  At most kFlowbLevels
// levels (their bounds are in shared memory) and 2^28 scenarios (a row's bytes are counted in 32 bits).
constexpr int kFlowbLevels = 8192;
cudaError_t launch_fwdb_flow(const DevDesign &d, const BatchBufs &b, const OpTable &ops, int tr_mode, int v, int sms,
                             cudaStream_t s);
cudaError_t launch_bwdb_flow(const DevDesign &d, const BatchBufs &b, const OpTable &ops, int tr_mode, int v,
                             int64_t edges, int sms, cudaStream_t s);
void launch_powerb(const DevDesign &d, const BatchBufs &b, int tr_mode, double K, cudaStream_t s);
// ks[s] = K * weights[s] (weights NULL: K)
void launch_seedb(const BatchBufs &b, double K, const double *weights, cudaStream_t s);
void launch_bwdb(const DevDesign &d, const BatchBufs &b, const OpTable &ops, const int32_t *lvl_host, int tr_mode,
                 BatchShape sh, cudaStream_t s);
// per-scenario gradient outputs ([x][S], user order), or summed over scenarios in FP64 ([x]) when reduce
void launch_gradb(const DevDesign &d, const BatchBufs &b, const OpTable &ops, int tr_mode, bool reduce, float *gtr,
                  float *gpin, float *gcl, cudaStream_t s);
void launch_netb_user(const DevDesign &d, const BatchBufs &b, int tr_mode, float *sp, float *tr, cudaStream_t s);
// Sizing deltas of a served batch (kern_serve.cu): per-scenario changes of cell
// pin caps turned into per-scenario C_load changes, deterministically.
constexpr int kMaxFanin = 4;
struct SizingDeltas {
    const int32_t *cell;        // [ne] cell-line index of each entry
    const float *cap;           // [ne] its new input pin cap, fF
    const int32_t *off;         // [n_req + 1] entries of request (scenario) s: [off[s], off[s+1]); an entry's
    int32_t n_req;              //   position within its request (the last one counts) is its index - off[s]
    int *win;                   // [n_cells * S] -1 at rest
    float *dpin;                // [n_cells * S] 0 at rest
    unsigned *flag;             // [n_nets * S] 0 at rest
    int64_t *list;              // [kMaxFanin * ne] claimed (net, scenario) slots
    unsigned long long *count;  // entries of list
};
// fills dcl[n * S + s] for every net loaded by a changed cell
void launch_sizing_deltas(const DevDesign &d, const OpTable &ops, const SizingDeltas &z, int64_t ne, int64_t S,
                          float *dcl, cudaStream_t s);
// A request's host buffers, as the device reads and writes them (sp, tr NULL: the reference inputs; nd resized cells
// from entry off of the batch's on; a gradient NULL: not wanted)
struct ServeIo {
    const float *sp, *tr;
    const int32_t *cells;
    const float *caps;
    float *gsp, *gtr, *gpin;
    int32_t nd, off;
};
// the inputs (in_sp NULL: not needed) and resized cells (off NULL: none) of the batch's S requests into its buffers
void launch_serve_in(const ServeIo *io, int64_t S, int64_t ns, int64_t most_nd, const float *ref_sp, const float *ref_tr,
                     float *in_sp, float *in_tr, int32_t *cell, float *cap, int32_t *off, cudaStream_t s);
// its gradients, request-major, into the requests' buffers
void launch_serve_out(const ServeIo *io, int64_t S, int64_t ns, int64_t nc, const float *sp, const float *tr,
                      const float *pin, cudaStream_t s);
// the reference inputs' forward state (P of every net, TR of every startpoint) into every
// scenario column of a batch: a batch of requests on the reference inputs skips the forward pass (state: BatchBufs')
void launch_bcast_ref(const float2 *ref_pq, const float *ref_tr, float2 *pq, float *tr_in, int64_t nn, int64_t ns,
                      int64_t S, uint32_t *state, cudaStream_t s);
// returns win, dpin, flag and dcl to rest after the batch
void launch_sizing_clear(const DevDesign &d, const SizingDeltas &z, int64_t ne, int64_t S, float *dcl,
                         cudaStream_t s);
// out[c][r] = in[r][c] (row-major R x C in, C x R out)
void launch_transpose(const float *in, float *out, int64_t R, int64_t C, cudaStream_t s);
// x <- clip(x + eta g, 0, 1) (Algorithm 4 ascent step with projection)
void launch_ascent(float *x, const float *g, int64_t n, float eta, cudaStream_t s);
// Eq. 3: threshold SP at 0.5 into v0 (v1 = not v0), two bitwise forwards, sum of C over nets whose values differ
void launch_virus(const DevDesign &d, const OpTable &ops, const int32_t *lvl_host, const float *sp, int64_t S,
                  uint64_t *words, uint8_t *v0, double *partials, double *out, cudaStream_t s);

// sizing score (kern_size.cu): Eq. 8 per cell line, and the radix select of its top k.  state: kSelectWords words;
// [kSelectWords - 1] the number of candidates (at or above the k-th score) once launch_select has run, in idx in
// no order; where they are at most kSelectMax, top and top_scores (may be NULL) hold the k best in order
constexpr int kSelectWords = 1031;
constexpr int kSelectMax = 8192;
cudaError_t launch_scores(const DevDesign &d, bool hybrid, float K, int mode, float *out, unsigned *state, int64_t k,
                          cudaStream_t s);
cudaError_t launch_select(const float *scores, int64_t n, int64_t k, unsigned *state, int32_t *idx,
                          unsigned long long *keys, int32_t *top, float *top_scores, cudaStream_t s);

// simulation by slices of lanes and cycles, the live nets in shared memory (kern_slice.cu)
struct SlicePlan {
    int64_t slots = 0;                    // live nets at most (0: the design does not use it)
    int threads = 0;                      // threads per block: cells per round
    const uint32_t *rec = nullptr;        // [4 x threads x rounds] the cells' records, levels padded to whole rounds
    const int32_t *round_ptr = nullptr;   // [L+1] first round of level l + 1
    const uint16_t *fourth = nullptr;     // [nc] 4-input cells: fourth input slot
    const int32_t *start_slot = nullptr;  // [ns] slot of each startpoint, -1 if nothing reads it
};
struct SliceShape {
    int nv, lanes;   // 32-bit words per net and block; lanes per block (8, 16 or 32)
};
constexpr int64_t kSliceMaxSlots = 224 * 1024 / 4;   // one 32-bit word per net
bool slice_fits(int64_t slots);   // also raises the kernels' shared-memory limit
// the fastest shape for T words; nv = 0 where the wide simulation is faster
SliceShape slice_shape(const SlicePlan &p, int64_t n_cells, int n_levels, int T, int sm_count);
cudaError_t launch_sim_slice(const DevDesign &d, const SlicePlan &p, int T, SliceShape sh, cudaStream_t s);

// simulation (kern_sim.cu)
void launch_sim_start(const DevDesign &d, int T, uint64_t seed, cudaStream_t s);
void launch_sim_level(const DevDesign &d, const OpTable &ops, int32_t c0, int32_t c1, int T, cudaStream_t s);
void launch_hybrid(const DevDesign &d, int T, int tr_mode, float beta_min, float beta_max, cudaStream_t s);

}  // namespace dp
