// Dataflow passes: no barriers between levels.  One cooperative launch per pass, one block
// per SM; the cells of a level are dealt out in chunks of 32 (one cell per lane), chunk i to
// block i mod G, and every warp walks the levels in order.  A cell waits only for its own
// inputs, and the data is its own ready flag: a (P, Q) pair carries the parity of the forward
// pass that wrote it, an edge adjoint the number of its reverse pass, in the same single-copy
// atomic word, so there is no fence and no flag.  A level then costs a store, the load that
// sees it and the cell's arithmetic.
//
// What bounds a level is the way from one SM to another through L2: 500 cycles when both SMs and
// the line's home are on one die, 870 to 1,040 otherwise (a ping-pong of relaxed stores and loads);
// leaving out the cell's arithmetic changes nothing.  A level-synchronous pass pays a grid barrier
// (1.26 us) on top.  Forward pass with the model power, barrier against this: 300,000 cells / 54
// levels 122 -> 72 us, 652,000 / 104 220 -> 134, 2,000,000 / 80 196 -> 167.  A warp holds at most one chunk of a level at a time
// and polls only for that, so few warps poll (a schedule whose warps took chunks far ahead of
// the level being computed was slower than the barrier: thousands of lanes polled).
//
// Progress: a chunk depends only on lower levels (reverse pass: higher), every warp takes its
// chunks in that order, and the cooperative launch keeps all warps resident, so the lowest
// unfinished chunk can always proceed.  Every wait is bounded by a clock limit; a lane that
// gives up records the context's error word, and the others stop at their next wait.
#include "kern_common.cuh"

namespace dp {
namespace {

constexpr int kFlowThreads = 256;

__global__ void k_bump(uint32_t *counter) { *counter += 1u; }

__device__ __forceinline__ int ld_err(const int *err) {
    int v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(err) : "memory");
    return v;
}
__device__ __forceinline__ void prefetch_l2(const void *p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// Every wait is a loop of the whole warp: the lanes that have their inputs go round with those
// that have not.  With a loop per lane, lanes left the wait at different times, a lane ahead
// could spin on what a lane behind it in the same warp had yet to write, and a level took the
// 5.6 us after which the hardware switches between a warp's divergent paths.

// true when a wait that began at t0 has to give up (looked at every 64th spin)
__device__ __forceinline__ bool gives_up(unsigned &spins, long long t0, int *err, long long limit) {
    if ((++spins & 63u) != 0) return false;
    if (ld_err(err) != 0) return true;
    if (clock64() - t0 <= limit) return false;
    atomicExch(err, 1);
    return true;
}

// Reads a stored pair as two single-copy-atomic 8-byte halves, through L2.
__device__ __forceinline__ void ld_pair_halves(const float4 *src, unsigned long long &h0, unsigned long long &h1) {
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(h0), "=l"(h1) : "l"(src) : "memory");
}

// A cell's input pairs on their way: the loads of all its inputs are issued together.  (Issued
// before the warp fetches what later levels need, most came back too early, and a second round
// trip followed the one just missed: 140 us against 133 us on 652,000 cells.)
struct PairWait {
    uint32_t n[4];
    unsigned long long h0[4], h1[4];
};
__device__ __forceinline__ void issue_pairs(PairWait &w, const float4 *pq, const uint4 &r, int k, uint32_t par) {
    w.n[0] = r.x & kMask24, w.n[1] = r.y, w.n[2] = r.z, w.n[3] = r.w;
    const unsigned long long want = (unsigned long long)par << 31;
#pragma unroll
    for (int j = 0; j < 4; j++) {
        w.h0[j] = want;
        w.h1[j] = want | (0x3F800000ull);   // an unused slot: P = 0, Q = 1
        if (j < k) ld_pair_halves(pq + w.n[j], w.h0[j], w.h1[j]);
    }
}
// Waits until they carry this pass's parity in both halves; false, in every lane, when the
// wait gave up.
__device__ __forceinline__ bool wait_pairs(PairWait &w, const float4 *pq, uint32_t par, int *err, long long limit,
                                           pair_ff (&x)[4]) {
    const uint32_t want = par << 31;
    auto late = [&](int j) { return (((uint32_t)w.h0[j] ^ want) | ((uint32_t)w.h1[j] ^ want)) & 0x80000000u; };
    bool ok = true;
    if (__any_sync(0xFFFFFFFFu, (late(0) | late(1) | late(2) | late(3)) != 0)) {
        const long long t0 = clock64();
        unsigned spins = 0;
        do {
#pragma unroll
            for (int j = 0; j < 4; j++)
                if (late(j)) ld_pair_halves(pq + w.n[j], w.h0[j], w.h1[j]);
            if (gives_up(spins, t0, err, limit)) ok = false;
        } while (__any_sync(0xFFFFFFFFu, (late(0) | late(1) | late(2) | late(3)) != 0) &&
                 __all_sync(0xFFFFFFFFu, ok));
    }
#pragma unroll
    for (int j = 0; j < 4; j++) {
        x[j].p = ff{__uint_as_float((uint32_t)w.h0[j] & 0x7FFFFFFFu), __uint_as_float((uint32_t)(w.h0[j] >> 32))};
        x[j].q = ff{__uint_as_float((uint32_t)w.h1[j] & 0x7FFFFFFFu), __uint_as_float((uint32_t)(w.h1[j] >> 32))};
    }
    return __all_sync(0xFFFFFFFFu, ok);
}

// The last block to finish a pass stores the pass number it ran as (every block read the
// counter before it got here) and returns the arrival counter to zero.
__device__ __forceinline__ void end_pass(uint32_t *counter, uint32_t *arrived, uint32_t pass) {
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(arrived, 1u) == gridDim.x - 1) {
        *arrived = 0u;
        *counter = pass;
    }
}

// this thread's place in a level: chunk i of 32 cells to block i mod gridDim.x
__device__ __forceinline__ int64_t spread_tid() {
    return ((int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32 + (threadIdx.x & 31);
}

__global__ void __launch_bounds__(kFlowThreads) k_fwd_flow(const uint4 *__restrict__ fanin, float4 *pq, float *tr,
                                                           const float *__restrict__ sp_in,
                                                           const float *__restrict__ tr_in,
                                                           const int32_t *__restrict__ lvl, int L, int64_t ns,
                                                           int tr_mode, OpTable ops, uint32_t *epoch, int *err,
                                                           long long limit) {
    const int64_t tid = spread_tid(), T = (int64_t)gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31;
    const uint32_t pass = *reinterpret_cast<volatile uint32_t *>(epoch) + 1u, par = pass & 1u;
    auto rec = [&](int l) {   // the fanin record of this thread's cell on level l (if any)
        if (l > L) return make_uint4(0, 0, 0, 0);
        const int64_t c = lvl[l - 1] + tid;
        return c < lvl[l] ? fanin[c] : make_uint4(0, 0, 0, 0);
    };
    uint4 r0 = rec(1), r1 = rec(2);
    for (int64_t k = tid; k < ns; k += T) {
        const pair_ff a = pair_of(sp_in[k]);
        pair_put(pq + k, a, par);
        tr[k] = tr_mode ? pair_tr(a) : tr_in[k];
    }
    bool ok = true;
    for (int l = 1; l <= L && ok; l++) {
        const int64_t c0 = lvl[l - 1] + tid, c1 = lvl[l];
        const uint4 r2 = rec(l + 2);   // records two levels ahead, their lines in L2 five ahead
        if (l + 5 <= L) {
            const int64_t cp = lvl[l + 4] + tid;
            if (cp < lvl[l + 5]) prefetch_l2(fanin + cp);
        }
        for (int64_t c = c0; c - lane < c1; c += T) {   // the whole warp, as long as it has a cell
            if (c != c0) r0 = c < c1 ? fanin[c] : make_uint4(0, 0, 0, 0);
            const int k = c < c1 ? op_arity(ops, r0.x >> 24) : 0;
            PairWait w;
            issue_pairs(w, pq, r0, k, par);
            pair_ff x[4];
            ok = wait_pairs(w, pq, par, err, limit, x);
            if (!ok) {
                epoch[3] = 1u;   // pairs of two parities: the power pass puts the tags right
                break;
            }
            if (c < c1) {
                const pair_ff o = cell_pair(k, op_tt(ops, r0.x >> 24), x);
                pair_put(pq + ns + c, o, par);
                tr[ns + c] = pair_tr(o);
            }
            __syncwarp();
        }
        r0 = r1;
        r1 = r2;
    }
    end_pass(epoch, epoch + 4, pass);
}

// ---------------------------------------------------------------- reverse
// Two kernels.  k_bwd_coef forms, with the whole grid and without any order, everything that
// does not depend on an adjoint: every edge's partial derivative dP_sink/dP_net in fanout-CSR
// order, and every net's local term (left in gnet until its adjoint replaces it).  k_bwd_flow
// then walks the levels down: a net pulls the adjoints of its sink cells, g_n = sum_e g_sink(e)
// coef_e + local.  What it waits on is one 8-byte word per cell, written coalesced by the warp
// that owns 32 consecutive cells.  (Pushing contributions, one word per edge scattered over the
// fanout CSR, made every line of it a target of sixteen partial writes while other SMs polled
// it: 164 us against 147 us for both kernels here on 652,000 cells and 104 levels, 225 against
// 180 us on 2,000,000 cells and 80 levels; with the grid barrier 203 and 196 us.)
__device__ __forceinline__ unsigned long long ld_tagged(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void put_tagged(unsigned long long *p, float g, uint32_t pass) {
    const unsigned long long v = (unsigned long long)__float_as_uint(g) | ((unsigned long long)pass << 32);
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__global__ void __launch_bounds__(256) k_bwd_coef(const uint4 *__restrict__ fanin, const int4 *__restrict__ efpos,
                                                  const float4 *__restrict__ pq, const float *__restrict__ cload,
                                                  float4 *cells, unsigned long long *edges, float *gnet, int64_t nn,
                                                  int64_t ns, int tr_mode, float K, OpTable ops) {
    const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= nn) return;
    if (n < ns) {
        gnet[n] = tr_mode ? adj_local(K, cload[n], pair_qmp(pq[n])) : 0.f;
        return;
    }
    const int64_t c = n - ns;
    const uint4 r = fanin[c];
    gnet[n] = adj_local(K, cload[n], pair_qmp(pq[n]));
    const uint32_t op = r.x >> 24;
    const int k = op_arity(ops, op);
    float p[4], q[4], d[4];
    gather_pairs(pq, r, k, p, q);
    cell_partials(k, op_tt(ops, op), p, q, d);
    if (cells) {
        cells[c] = make_float4(d[0], d[1], d[2], d[3]);
        return;
    }
    const int4 ep = efpos[c];
    const int at[4] = {ep.x, ep.y, ep.z, ep.w};
#pragma unroll
    for (int j = 0; j < 4; j++)
        if (j < k) edges[at[j]] = (unsigned long long)__float_as_uint(d[j]) | ((unsigned long long)c << 32);
}

// a net's first kFlowEdges fanout edges (sink net, coefficient) and its local term and beta,
// loaded a level before they are used: nets with more are few, and read the rest in place
constexpr int kFlowEdges = 8;
struct FlowPre {
    int32_t e0, e1;
    unsigned long long edge[kFlowEdges];
    float local, b;
};
__device__ __forceinline__ void flow_edges(const unsigned long long *edges, int32_t e0, int32_t e1,
                                           unsigned long long (&edge)[kFlowEdges]) {
#pragma unroll
    for (int i = 0; i < kFlowEdges; i++) edge[i] = e0 + i < e1 ? edges[e0 + i] : 0ull;
}

__device__ __forceinline__ void issue_sinks(unsigned long long (&v)[kFlowEdges], const unsigned long long *gcell,
                                            const unsigned long long (&edge)[kFlowEdges], int32_t cnt, uint32_t pass) {
#pragma unroll
    for (int i = 0; i < kFlowEdges; i++)
        v[i] = i < cnt ? ld_tagged(gcell + (edge[i] >> 32)) : (unsigned long long)pass << 32;
}

// The sum over a net's fanout edges, in index order, of the sink cell's adjoint times the edge's
// coefficient, once all of them are from this pass (v: the first loads, already issued); false,
// in every lane, when the wait gave up.  The product and the sum are rounded each on its own, as
// where the cell writes the product and the net adds it.
__device__ __forceinline__ bool wait_sum(FlowPre &w, unsigned long long (&v)[kFlowEdges],
                                         const unsigned long long *gcell, const unsigned long long *edges,
                                         uint32_t pass, int *err, long long limit, float &acc) {
    acc = 0.f;
    bool ok = true;
    for (int32_t e = w.e0;;) {
        auto late = [&] {
            bool any = false;
#pragma unroll
            for (int i = 0; i < kFlowEdges; i++) any |= (uint32_t)(v[i] >> 32) != pass;
            return any;
        };
        if (__any_sync(0xFFFFFFFFu, late())) {
            const long long t0 = clock64();
            unsigned spins = 0;
            do {
#pragma unroll
                for (int i = 0; i < kFlowEdges; i++)
                    if ((uint32_t)(v[i] >> 32) != pass) v[i] = ld_tagged(gcell + (w.edge[i] >> 32));
                if (gives_up(spins, t0, err, limit)) ok = false;
            } while (__any_sync(0xFFFFFFFFu, late()) && __all_sync(0xFFFFFFFFu, ok));
            if (!__all_sync(0xFFFFFFFFu, ok)) return false;
        }
#pragma unroll
        for (int i = 0; i < kFlowEdges; i++)
            if (e + i < w.e1) acc = __fadd_rn(acc, __fmul_rn(__uint_as_float((uint32_t)v[i]), __uint_as_float((uint32_t)w.edge[i])));
        e += kFlowEdges;
        if (!__any_sync(0xFFFFFFFFu, e < w.e1)) return true;
        flow_edges(edges, e, w.e1, w.edge);
        issue_sinks(v, gcell, w.edge, w.e1 - e, pass);
    }
}

__global__ void __launch_bounds__(kFlowThreads) k_bwd_flow(const int32_t *__restrict__ fptr,
                                                           const unsigned long long *__restrict__ edges,
                                                           const float *__restrict__ beta, float *gnet,
                                                           unsigned long long *gcell, const int32_t *__restrict__ lvl,
                                                           int L, int64_t ns, int grad_mode, float *out_gsp,
                                                           uint32_t *epoch, int *err, long long limit) {
    const int64_t tid = spread_tid(), T = (int64_t)gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31;
    const uint32_t pass = *reinterpret_cast<volatile uint32_t *>(epoch + 2) + 1u;
    auto on = [&](int l) { return l >= 1 && lvl[l - 1] + tid < lvl[l]; };
    auto range = [&](int l) {   // the fanout range of this thread's cell on level l (empty if none)
        if (!on(l)) return make_int2(0, 0);
        const int64_t n = ns + lvl[l - 1] + tid;
        return make_int2(fptr[n], fptr[n + 1]);
    };
    auto fill = [&](FlowPre &w, const int2 &r, int64_t n) {
        w.e0 = r.x;
        w.e1 = r.y;
        flow_edges(edges, r.x, r.y, w.edge);
        w.local = gnet[n];
        w.b = grad_mode ? beta[n] : 1.f;
    };
    FlowPre w{};
    if (on(L)) fill(w, range(L), ns + lvl[L - 1] + tid);
    int2 r1 = range(L - 1), r2 = range(L - 2);
    bool ok = true;
    for (int l = L; l >= 1 && ok; l--) {
        const int64_t c0 = lvl[l - 1] + tid, c1 = lvl[l];
        FlowPre cur = w;
        // the next level's edges into registers, the lines of those of the one after it into L2,
        // the fanout ranges three levels ahead (their lines six ahead)
        w.e0 = w.e1 = 0;
        if (on(l - 1)) fill(w, r1, ns + lvl[l - 2] + tid);
        if (r2.x < r2.y) prefetch_l2(edges + r2.x);
        const int2 r3 = range(l - 3);
        if (on(l - 6)) {
            const int64_t n = ns + lvl[l - 7] + tid;
            prefetch_l2(fptr + n);
            prefetch_l2(gnet + n);
            if (grad_mode) prefetch_l2(beta + n);
        }
        for (int64_t c = c0; c - lane < c1; c += T) {   // the whole warp, as long as it has a cell
            const bool mine = c < c1;
            if (c != c0) {
                cur.e0 = cur.e1 = 0;
                if (mine) fill(cur, make_int2(fptr[ns + c], fptr[ns + c + 1]), ns + c);
            }
            unsigned long long v[kFlowEdges];
            issue_sinks(v, gcell, cur.edge, cur.e1 - cur.e0, pass);
            float acc;
            ok = wait_sum(cur, v, gcell, edges, pass, err, limit, acc);
            if (!ok) break;
            if (mine) {
                const float g = adj_combine(grad_mode, acc, cur.local, cur.b);
                put_tagged(gcell + c, g, pass);
                gnet[ns + c] = g;
            }
            __syncwarp();
        }
        r1 = r2;
        r2 = r3;
    }
    for (int64_t k = tid; k - lane < ns && ok; k += T) {
        w.e0 = w.e1 = 0;
        if (k < ns) fill(w, make_int2(fptr[k], fptr[k + 1]), k);
        unsigned long long v[kFlowEdges];
        issue_sinks(v, gcell, w.edge, w.e1 - w.e0, pass);
        float acc;
        ok = wait_sum(w, v, gcell, edges, pass, err, limit, acc);
        if (!ok || k >= ns) break;
        const float g = adj_combine(grad_mode, acc, w.local, w.b);
        gnet[k] = g;
        if (out_gsp) out_gsp[k] = g;
    }
    end_pass(epoch + 2, epoch + 5, pass);
}

// ------------------------------------------------------ simulation, dataflow
// The wide simulation (16 lanes per cell, two cells of one level per warp)
// without level barriers.  Cells are grouped in level-aligned pairs; warp w
// takes pairs w, w + W, w + 2W, ... in increasing order, and lane h < k of a
// half-warp waits only for the flag of fanin h when that fanin is a cell.  A
// cell publishes its words by storing the pass number into its flag with
// release semantics after a warp barrier that orders the sixteen lanes'
// stores; the waiting lane reads the flag with acquire semantics and a warp
// barrier orders that before the other lanes' word loads.  Flags need no
// clearing: each pass has its own number.  A pair depends only on pairs of
// lower levels, which come earlier in the order, so (all warps co-resident)
// the lowest unfinished pair can always proceed.
__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned *p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release_u32(unsigned *p, unsigned v) {
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// true once the flag holds this pass's number; false when the wait gave up
__device__ __forceinline__ bool wait_done(const unsigned *f, unsigned ep, const int *err, long long limit) {
    if (ld_acquire_u32(f) == ep) return true;
    const long long t0 = clock64();
    for (;;) {
        __nanosleep(32);
        if (ld_acquire_u32(f) == ep) return true;
        if (clock64() - t0 > limit || ld_err(err) != 0) return false;
    }
}

// cell index of pair p (from level lv on, updated) and half h; -1 past the end
__device__ __forceinline__ int64_t pair_cell(int64_t p, int &lv, int L, const int32_t *lvl, const int32_t *pair_ptr,
                                             int h) {
    while (lv <= L && p >= pair_ptr[lv]) lv++;
    if (lv > L) return -1;
    const int64_t c = lvl[lv - 1] + 2 * (p - pair_ptr[lv - 1]) + h;
    return c < lvl[lv] ? c : -1;
}

__global__ void __launch_bounds__(kSimThreads, 2) k_sim_flow(const uint4 *__restrict__ fanin, uint64_t *words,
                                                            uint32_t *toggles, uint32_t *ones, unsigned *done,
                                                            const int32_t *__restrict__ lvl,
                                                            const int32_t *__restrict__ pair_ptr, int L, int64_t ns,
                                                            int T, OpTable ops, const uint32_t *epoch, int *err,
                                                            long long limit) {
    const unsigned ep = epoch[1];
    const int lane = threadIdx.x & 31, half = lane >> 4, hl = lane & 15;
    const int64_t W = (int64_t)gridDim.x * (blockDim.x >> 5);
    const int64_t npairs = pair_ptr[L];
    int lv = 1, lvn = 1;
    int64_t p = (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    int64_t cn = p < npairs ? pair_cell(p, lvn, L, lvl, pair_ptr, half) : -1;
    uint4 rn = cn >= 0 ? fanin[cn] : make_uint4(0, 0, 0, 0);
    for (; p < npairs; p += W) {   // warp-uniform
        const int64_t c = cn;
        const uint4 r = rn;
        lv = lvn;
        // the next pair's record, ahead of its use
        cn = p + W < npairs ? pair_cell(p + W, lvn, L, lvl, pair_ptr, half) : -1;
        rn = cn >= 0 ? fanin[cn] : make_uint4(0, 0, 0, 0);
        const bool valid = c >= 0;
        const uint32_t op = r.x >> 24;
        const int k = valid ? op_arity(ops, op) : 0;
        const uint32_t tt = op_tt(ops, op), lut = op_lut(ops, op);
        const uint32_t nid[4] = {r.x & kMask24, r.y, r.z, r.w};
        bool ok = true;
        if (hl < k) {
            const uint32_t n = hl == 0 ? nid[0] : hl == 1 ? nid[1] : hl == 2 ? nid[2] : nid[3];
            if (n >= ns) ok = wait_done(done + (n - ns), ep, err, limit);
        }
        if (!__all_sync(0xFFFFFFFFu, ok)) {
            if (!ok) atomicExch(err, 1);
            return;
        }
        __syncwarp();   // the flags' acquire before every lane's word loads
        uint64_t *out = words + (size_t)(ns + (valid ? c : 0)) * T;
        uint32_t tg = 0, on = 0;
        uint64_t carry = 0;
        for (int base = 0; base < T; base += 64) {
            const int t = base + 4 * hl;
            const bool act = valid && t < T;
            uint64_t w[4];
            if (k <= 3) {
                uint64_t x[3][4];
#pragma unroll
                for (int j = 0; j < 3; j++) {
                    x[j][0] = x[j][1] = x[j][2] = x[j][3] = 0;
                    if (act && j < k) {
                        const uint64_t *src = words + (size_t)nid[j] * T + t;
                        const ulonglong2 a = __ldcg(reinterpret_cast<const ulonglong2 *>(src));
                        const ulonglong2 b = __ldcg(reinterpret_cast<const ulonglong2 *>(src + 2));
                        x[j][0] = a.x;
                        x[j][1] = a.y;
                        x[j][2] = b.x;
                        x[j][3] = b.y;
                    }
                }
                const uint64_t a0[4] = {x[0][0], x[1][0], x[2][0], 0}, a1[4] = {x[0][1], x[1][1], x[2][1], 0};
                const uint64_t b0[4] = {x[0][2], x[1][2], x[2][2], 0}, b1[4] = {x[0][3], x[1][3], x[2][3], 0};
                cell_bits_lop3(lut, a0, a1, w[0], w[1]);
                cell_bits_lop3(lut, b0, b1, w[2], w[3]);
            } else {
#pragma unroll
                for (int h2 = 0; h2 < 2; h2++) {
                    uint64_t x0[4] = {0, 0, 0, 0}, x1[4] = {0, 0, 0, 0};
                    if (act)
#pragma unroll
                        for (int j = 0; j < 4; j++) {
                            const ulonglong2 a = __ldcg(
                                reinterpret_cast<const ulonglong2 *>(words + (size_t)nid[j] * T + t + 2 * h2));
                            x0[j] = a.x;
                            x1[j] = a.y;
                        }
                    w[2 * h2] = bits_eval<4>(tt, x0);
                    w[2 * h2 + 1] = bits_eval<4>(tt, x1);
                }
            }
            const uint64_t prev = __shfl_up_sync(0xFFFFFFFFu, w[3], 1, 16);
            const uint64_t last = __shfl_sync(0xFFFFFFFFu, w[3], 15, 16);
            if (act) {
                *reinterpret_cast<ulonglong2 *>(out + t) = make_ulonglong2(w[0], w[1]);
                *reinterpret_cast<ulonglong2 *>(out + t + 2) = make_ulonglong2(w[2], w[3]);
                on += __popcll(w[0]) + __popcll(w[1]) + __popcll(w[2]) + __popcll(w[3]);
                tg += __popcll(w[1] ^ w[0]) + __popcll(w[2] ^ w[1]) + __popcll(w[3] ^ w[2]);
                if (t > 0) tg += __popcll(w[0] ^ (hl > 0 ? prev : carry));
            }
            carry = last;
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) {
            tg += __shfl_xor_sync(0xFFFFFFFFu, tg, o);
            on += __shfl_xor_sync(0xFFFFFFFFu, on, o);
        }
        __syncwarp();   // every lane's word stores before the flag's release
        if (valid && hl == 0) {
            toggles[ns + c] = tg;
            ones[ns + c] = on;
            st_release_u32(done + c, ep);
        }
    }
}

}  // namespace

void launch_bump(uint32_t *counter, cudaStream_t s) { k_bump<<<1, 1, 0, s>>>(counter); }

int flow_grid(int which, int sm_count) {
    int per = 0;
    const cudaError_t e =
        which == 1   ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_sim_flow, kSimThreads, 0)
        : which == 2 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_bwd_flow, kFlowThreads, 0)
                     : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_fwd_flow, kFlowThreads, 0);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    const int cap = which == 1 ? 2 : 1;
    return sm_count * (per < cap ? per : cap);
}

namespace {
// all warps co-resident: needed for progress
template <class... Args>
cudaError_t launch_coop(void (*kern)(Args...), int grid, int block, cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}
}  // namespace

cudaError_t launch_fwd_flow(const DevDesign &d, const OpTable &ops, int tr_mode, int grid, cudaStream_t s) {
    return launch_coop(k_fwd_flow, grid, kFlowThreads, s, d.fanin, d.pq, d.tr, (const float *)d.sp_in,
                       (const float *)d.tr_in, d.lvl, d.n_levels, d.n_start, tr_mode, ops, d.epoch, d.err,
                       kWaitLimitCycles);
}

void launch_bwd_coef(const DevDesign &d, const OpTable &ops, int tr_mode, float K, float *cells, cudaStream_t s) {
    if (d.n_nets == 0) return;
    k_bwd_coef<<<(unsigned)((d.n_nets + 255) / 256), 256, 0, s>>>(d.fanin, (const int4 *)d.edge_fpos, d.pq, d.cload,
                                                                  (float4 *)cells, d.edges, d.gnet, d.n_nets,
                                                                  d.n_start, tr_mode, K, ops);
}

cudaError_t launch_bwd_flow(const DevDesign &d, int grad_mode, float *out_gsp, int grid, cudaStream_t s) {
    return launch_coop(k_bwd_flow, grid, kFlowThreads, s, d.fout_ptr, (const unsigned long long *)d.edges,
                       (const float *)d.beta, d.gnet, d.gcell, d.lvl, d.n_levels, d.n_start, grad_mode, out_gsp,
                       d.epoch, d.err, kWaitLimitCycles);
}

cudaError_t launch_sim_flow(const DevDesign &d, const OpTable &ops, int T, int grid, cudaStream_t s) {
    launch_bump(d.epoch + 1, s);   // a new pass number for the flags
    return launch_coop(k_sim_flow, grid, kSimThreads, s, d.fanin, d.words, d.toggles, d.ones, d.simdone, d.lvl,
                       d.pair_ptr, d.n_levels, d.n_start, T, ops, (const uint32_t *)d.epoch, d.err, kWaitLimitCycles);
}

}  // namespace dp
