// Batched passes without barriers between levels: one cooperative launch per pass, every warp of the
// grid walks the (cell, 32 x V scenarios) items of all levels in order, dealt out in turn, and an
// item waits only for its own inputs.  The data is its own ready flag.
//
// Forward: the low part of a stored P never has bit 30 set (|lo| < 2 for |P| < 2^25), so the bit carries the
// parity of the pass that wrote it, in the same single-copy atomic word; everything that reads a
// stored P drops it (pair_get).  Reverse: an edge's contribution is written once and read once, and its
// reader leaves kNotYet behind for the next pass.  launch_flowb_prep brings both to rest where another pass wrote
// the arrays in between.
//
// What bounds it: the level launches end a grid and start the next per level, about 3 us, with 58 instructions per
// (cell, scenario) to do in between (30 % of the issue slots used, 38 % of the warps active).  Without them a pass
// runs into the L2: 50,000 cells / 44 levels x 256 scenarios forward 81 us with 29 M sectors, 120,000 / 48 x 512 217 us.
// Four scenarios per thread spread the item's address and record work; 24 warps per SM forward, 20 reverse, where the
// registers end without spills to speak of (a reverse pass whose 80 registers spilled wrote three times the
// sectors).  Fetching the next item's record ahead cost more registers than it hid.  The reverse pass computes the
// partial derivatives before it waits for the fanout, so only sums and products are on the way from level to level.
// Forward with the model power + reverse, level launches against this: 120,000 x 512 404 + 575 us -> 366 + 435;
// 50,000 x 256 172 + 220 -> 124 + 137; 50,000 x 128 145 + 189 -> 104 + 103; 20,000 / 38 x 37 84 + 105 -> 66 + 68; 2,000 /
// 24 x 512 67 + 83 -> 50 + 50 (the power pass's own gain, 16 us at 50,000 x 256, included).
//
// Progress: an item depends on lower levels only (reverse: higher), every warp takes its items in that
// order and the cooperative launch keeps all warps resident, so the lowest unfinished item can always
// proceed.  Every wait is a loop of the whole warp, bounded by a clock limit; a warp that gives
// up records the context's error word, and the others stop at their next wait.
//
// Every (cell, scenario) is computed by the same code as in the other batched passes: same bits.
#include "kern_cells.cuh"

namespace dp {
namespace {

constexpr unsigned kAll = 0xFFFFFFFFu;
constexpr uint32_t kNotYet = 0xFFFFFFFFu;   // arithmetic gives the NaN 0x7FFFFFFF only

__device__ __forceinline__ uint32_t ld_word(const void *p) {
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// rows of single-copy atomic elements, read through L2 at the point of the call
template <int V>
__device__ __forceinline__ Row2<V> ld_row(const float2 *p) {
    Row2<V> r;
    if constexpr (V == 1)
        asm volatile("ld.relaxed.gpu.global.v2.f32 {%0,%1}, [%2];" : "=f"(r.v[0].x), "=f"(r.v[0].y) : "l"(p) : "memory");
    else if constexpr (V == 2)
        asm volatile("ld.relaxed.gpu.global.v4.f32 {%0,%1,%2,%3}, [%4];"
                     : "=f"(r.v[0].x), "=f"(r.v[0].y), "=f"(r.v[1].x), "=f"(r.v[1].y)
                     : "l"(p)
                     : "memory");
    else
        asm volatile("ld.relaxed.gpu.global.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=f"(r.v[0].x), "=f"(r.v[0].y), "=f"(r.v[1].x), "=f"(r.v[1].y), "=f"(r.v[2].x), "=f"(r.v[2].y),
                       "=f"(r.v[3].x), "=f"(r.v[3].y)
                     : "l"(p)
                     : "memory");
    return r;
}
template <int V>
__device__ __forceinline__ Row1<V> ld_row(const float *p) {
    Row1<V> r;
    if constexpr (V == 1)
        asm volatile("ld.relaxed.gpu.global.f32 %0, [%1];" : "=f"(r.v[0]) : "l"(p) : "memory");
    else if constexpr (V == 2)
        asm volatile("ld.relaxed.gpu.global.v2.f32 {%0,%1}, [%2];" : "=f"(r.v[0]), "=f"(r.v[1]) : "l"(p) : "memory");
    else
        asm volatile("ld.relaxed.gpu.global.v4.f32 {%0,%1,%2,%3}, [%4];"
                     : "=f"(r.v[0]), "=f"(r.v[1]), "=f"(r.v[2]), "=f"(r.v[3])
                     : "l"(p)
                     : "memory");
    return r;
}

// true (in every lane) when a wait that began at t0 has to give up
__device__ __forceinline__ bool gives_up(unsigned &spins, long long t0, int *err, long long limit) {
    if ((++spins & 63u) != 0) return false;
    bool lost = ld_word(err) != 0;
    if (clock64() - t0 > limit) {
        atomicExch(err, 1);
        lost = true;
    }
    return __any_sync(kAll, lost);
}

// A warp's walk through the items: a net of the level and one of m chunks of 32 V scenarios.
struct Walk {
    const int *first;   // level l's nets are first[l] .. first[l + 1] (level 0: the startpoints)
    int L, m, drow, dq;
    bool down;
    int l, rows, n;     // the level (from the far end in the reverse pass), its first net and nets; done: l > L
    int i, q;
    __device__ __forceinline__ void enter() {
        const int ll = down ? L - l : l;
        rows = first[ll];
        n = first[ll + 1] - rows;
    }
    __device__ __forceinline__ void settle() {
        while (i >= n) {
            i -= n;
            if (++l > L) break;
            enter();
        }
    }
    __device__ __forceinline__ void begin(const int *bounds, int levels, int chunks, bool rev, int w, int W) {
        first = bounds;
        L = levels;
        m = chunks;
        down = rev;
        drow = W / m;
        dq = W % m;
        l = 0;
        i = w / m;
        q = w % m;
        enter();
        settle();
    }
    __device__ __forceinline__ void next() {
        i += drow;
        q += dq;
        if (q >= m) q -= m, i++;
        settle();
    }
    __device__ __forceinline__ bool more() const { return l <= L; }
    __device__ __forceinline__ uint32_t row() const { return (uint32_t)(rows + i); }
};

__device__ __forceinline__ void level_bounds(int *bounds, const int32_t *lvl, int L, uint32_t ns) {
    for (int k = threadIdx.x; k <= L + 1; k += blockDim.x) bounds[k] = k == 0 ? 0 : (int)ns + lvl[k - 1];
    __syncthreads();
}

// true in one thread of the last block to get here (a block that gave up has recorded it before); done is 0 again
__device__ __forceinline__ bool last_block(uint32_t *done) {
    __syncthreads();
    if (threadIdx.x != 0) return false;
    __threadfence();
    if (atomicAdd(done, 1u) != gridDim.x - 1) return false;
    *done = 0u;
    return true;
}

template <int V, int THREADS, int BLOCKS>
__global__ void __launch_bounds__(THREADS, BLOCKS)
    k_fwdb_flow(const uint4 *__restrict__ fanin, float2 *pq, const float *__restrict__ sp_in,
                const int32_t *__restrict__ lvl, int L, uint32_t ns, uint32_t S, uint32_t *state, OpTable ops, int *err,
                long long limit) {
    extern __shared__ int bounds[];
    level_bounds(bounds, lvl, L, ns);
    const int lane = threadIdx.x & 31;
    const uint32_t pass = ld_word(state + 1) + 1u, tag = (pass & 1u) << 30;
    Walk at;
    at.begin(bounds, L, (int)((S + 32 * V - 1) / (32 * V)), false,
             (int)blockIdx.x * (THREADS / 32) + (int)(threadIdx.x >> 5), (THREADS / 32) * (int)gridDim.x);
    uint32_t row = 0, s = 0, f = 0;
    uint4 r = make_uint4(0, 0, 0, 0);
    auto record = [&] {
        if (!at.more()) return;
        row = at.row();
        s = ((uint32_t)at.q * 32u + (uint32_t)lane) * V;
        if (row >= ns) r = fanin[row - ns], f = ops.e[r.x >> 24];
    };
    bool ok = true;
    while (at.more() && ok) {
        record();
        const uint32_t c = row, e = f;
        const uint32_t n[4] = {r.x & kMask24, r.y, r.z, r.w};
        const bool on = s < S;
        const uint32_t sc = on ? s : 0;   // a lane past the batch goes along with the first columns
        float2 *const pqs = pq + sc;
        at.next();
        Row2<V> o;
        if (c < ns) {
            const Row1<V> a = ld1<V>(row_at(sp_in + sc, c, S));
#pragma unroll
            for (int i = 0; i < V; i++) o.v[i] = make_float2(a.v[i], 0.f);
        } else {
            const int k = (int)((e >> 16) & 7u);
            Row2<V> x[4];
            bool late[4];
            auto look = [&](int j) {
                x[j] = ld_row<V>(row_at(pqs, n[j], S));
            };
            auto check = [&](int j) {
                uint32_t bad = 0;
#pragma unroll
                for (int i = 0; i < V; i++) bad |= __float_as_uint(x[j].v[i].y) ^ tag;
                return (bad & kTagBit) != 0;
            };
#pragma unroll
            for (int j = 0; j < 4; j++)
                if (j < k) look(j);
#pragma unroll
            for (int j = 0; j < 4; j++) late[j] = j < k && check(j);
            if (__any_sync(kAll, late[0] || late[1] || late[2] || late[3])) {
                const long long t0 = clock64();
                unsigned spins = 0;
                do {
#pragma unroll
                    for (int j = 0; j < 4; j++) {
                        if (late[j]) look(j);
                    }
#pragma unroll
                    for (int j = 0; j < 4; j++) late[j] = late[j] && check(j);
                    if (gives_up(spins, t0, err, limit)) ok = false;
                } while (ok && __any_sync(kAll, late[0] || late[1] || late[2] || late[3]));
            }
            Row1<V> none;
            cell_value<V, false>(
                e, [&](int j, Row2<V> &xj, Row1<V> &) { xj = x[j]; }, o, none);
        }
        if (on) {
#pragma unroll
            for (int i = 0; i < V; i++)
                o.v[i].y = __uint_as_float((__float_as_uint(o.v[i].y) & ~kTagBit) | tag);
            st2<V>(row_at(pqs, c, S), o);
        }
    }
    if (last_block(state + 3)) {
        state[0] = ld_word(err) ? 0u : S;
        state[1] = pass;
    }
}

template <int V, int THREADS, int BLOCKS>
__global__ void __launch_bounds__(THREADS, BLOCKS)
    k_bwdb_flow(const uint4 *__restrict__ fanin, const int32_t *__restrict__ fptr, const int4 *__restrict__ efpos,
                const float2 *__restrict__ pq, const float *__restrict__ cload, const float *__restrict__ dcl,
                const float *__restrict__ ks, float *gfo, float *gsp, const int32_t *__restrict__ lvl, int L,
                uint32_t ns, uint32_t S, int tr_mode, uint32_t *state, OpTable ops, int *err, long long limit) {
    extern __shared__ int bounds[];
    level_bounds(bounds, lvl, L, ns);
    const int lane = threadIdx.x & 31;
    Walk at;
    at.begin(bounds, L, (int)((S + 32 * V - 1) / (32 * V)), true,
             (int)blockIdx.x * (THREADS / 32) + (int)(threadIdx.x >> 5), (THREADS / 32) * (int)gridDim.x);
    uint32_t row = 0, s = 0, f = 0;
    uint4 r = make_uint4(0, 0, 0, 0);
    int4 ep = make_int4(0, 0, 0, 0);
    int32_t e0 = 0, e1 = 0;
    auto record = [&] {
        if (!at.more()) return;
        row = at.row();
        s = ((uint32_t)at.q * 32u + (uint32_t)lane) * V;
        e0 = fptr[row];
        e1 = fptr[row + 1];
        if (row >= ns) r = fanin[row - ns], ep = efpos[row - ns], f = ops.e[r.x >> 24];
    };
    bool ok = true;
    while (at.more() && ok) {
        record();
        const uint32_t c = row, e = f;
        const uint32_t n[4] = {r.x & kMask24, r.y, r.z, r.w};
        const uint32_t pos[4] = {(uint32_t)ep.x, (uint32_t)ep.y, (uint32_t)ep.z, (uint32_t)ep.w};
        const int32_t f0 = e0, f1 = e1;
        const bool on = s < S;
        const uint32_t sc = on ? s : 0;
        at.next();
        const float2 *const pqs = pq + sc;
        float *const gs = gfo + sc;
        const int k = c < ns ? 0 : (int)((e >> 16) & 7u);
        // what does not wait for the fanout: the partial derivatives, and the local term's factors (bwdb_adjoint)
        Row1<V> two_kc = ld1<V>(ks + sc), qmp, d[4];
        {
            Row1<V> dc;
            if (dcl) dc = ld1<V>(row_at(dcl + sc, c, S));
            const float cl = cload[c];
            const Row2<V> self = ld2<V>(row_at(pqs, c, S));
            if (c >= ns) cell_partials<V>(e, [&](int j) { return ld2<V>(row_at(pqs, n[j], S)); }, d);
#pragma unroll
            for (int i = 0; i < V; i++) {
                two_kc.v[i] = __fmul_rn(__fmul_rn(2.f, two_kc.v[i]), dcl ? cl + dc.v[i] : cl);
                qmp.v[i] = qmp32(self.v[i]);
            }
        }
        // the fanout sum in index order, F edges in flight
        constexpr int F = V == 4 ? 2 : 4;
        Row1<V> a;
#pragma unroll
        for (int i = 0; i < V; i++) a.v[i] = 0.f;
        for (int32_t p = f0; p < f1 && ok; p += F) {
            Row1<V> u[F];
            bool late[F];
            auto look = [&](int j) { u[j] = ld_row<V>(row_at((const float *)gs, (uint32_t)(p + j), S)); };
            auto check = [&](int j) {
                bool b = false;
#pragma unroll
                for (int i = 0; i < V; i++) b = b || __float_as_uint(u[j].v[i]) == kNotYet;
                return b && on;
            };
#pragma unroll
            for (int j = 0; j < F; j++)
                if (p + j < f1) look(j);
#pragma unroll
            for (int j = 0; j < F; j++) late[j] = p + j < f1 && check(j);
            auto any = [&] {
                bool b = false;
#pragma unroll
                for (int j = 0; j < F; j++) b = b || late[j];
                return __any_sync(kAll, b) != 0;
            };
            if (any()) {
                const long long t0 = clock64();
                unsigned spins = 0;
                do {
#pragma unroll
                    for (int j = 0; j < F; j++)
                        if (late[j]) look(j);
#pragma unroll
                    for (int j = 0; j < F; j++) late[j] = late[j] && check(j);
                    if (gives_up(spins, t0, err, limit)) ok = false;
                } while (ok && any());
            }
            Row1<V> rest;
#pragma unroll
            for (int i = 0; i < V; i++) rest.v[i] = __uint_as_float(kNotYet);
#pragma unroll
            for (int j = 0; j < F; j++)
                if (p + j < f1) {
#pragma unroll
                    for (int i = 0; i < V; i++) a.v[i] += u[j].v[i];
                    if (on) st1<V>(row_at(gs, (uint32_t)(p + j), S), rest);
                }
        }
        if (!on) continue;
        if (c >= ns || tr_mode) {
#pragma unroll
            for (int i = 0; i < V; i++) a.v[i] = fmaf(two_kc.v[i], qmp.v[i], a.v[i]);
        }
        if (c < ns) {
            st1<V>(row_at(gsp + sc, c, S), a);
            continue;
        }
#pragma unroll
        for (int j = 0; j < 4; j++)
            if (j < k) {
#pragma unroll
                for (int i = 0; i < V; i++) d[j].v[i] = __fmul_rn(a.v[i], d[j].v[i]);
                st1<V>(row_at(gs, pos[j], S), d[j]);
            }
    }
    if (last_block(state + 4)) state[2] = ld_word(err) ? 0u : 1u;
}

// The arrays of a pass (0 forward: the pairs of the batch; 1 reverse: all edges) as the pass expects them, where the
// last to write them was not a dataflow pass (forward: of the same S).
__global__ void k_flowb_prep(int which, float2 *pq, int64_t n, uint32_t S, float *gfo, int64_t m,
                             const uint32_t *state) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, T = (int64_t)gridDim.x * blockDim.x;
    if (which == 0) {
        if (state[0] == S) return;
        const float2 v = make_float2(0.f, __uint_as_float((state[1] & 1u) << 30));
        for (int64_t i = t; i < n; i += T) pq[i] = v;
    } else {
        if (state[2] == 1u) return;
        for (int64_t i = t; i < m; i += T) gfo[i] = __uint_as_float(kNotYet);
    }
}

// threads per block and blocks per SM by scenarios per thread (see above; 50,000 x 256 reverse, v = 4: 512 threads per
// SM 137 us, 640 137, 768 150; 120,000 x 512 485, 441, 467)
template <int V>
struct Cfg {
    static constexpr int fthreads = V == 4 ? 384 : 512, fblocks = 2;
    static constexpr int bthreads = V == 4 ? 320 : 448, bblocks = 2;
};

template <class... KArgs, class... Args>
cudaError_t launch_flowb(void (*kern)(KArgs...), int threads, int blocks, int L, cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = sizeof(int) * (size_t)(L + 2);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}

}  // namespace

cudaError_t launch_fwdb_flow(const DevDesign &d, const BatchBufs &b, const OpTable &ops, int v, int sms,
                             cudaStream_t s) {
    k_flowb_prep<<<(unsigned)(sms * 4), 512, 0, s>>>(0, b.pq, d.n_nets * b.S, (uint32_t)b.S, b.gfo, 0, b.state);
    auto go = [&](auto kern, int threads, int blocks) {
        return launch_flowb(kern, threads, blocks * sms, d.n_levels, s, d.fanin, b.pq, b.sp_in, d.lvl, d.n_levels,
                            d.n_start, b.S, b.state, ops, d.err, kWaitLimitCycles);
    };
#define GO(V) go(k_fwdb_flow<V, Cfg<V>::fthreads, Cfg<V>::fblocks>, Cfg<V>::fthreads, Cfg<V>::fblocks)
    return v == 4 ? GO(4) : v == 2 ? GO(2) : GO(1);
#undef GO
}

cudaError_t launch_bwdb_flow(const DevDesign &d, const BatchBufs &b, const OpTable &ops, int tr_mode, int v,
                             int64_t edges, int sms, cudaStream_t s) {
    k_flowb_prep<<<(unsigned)(sms * 4), 512, 0, s>>>(1, b.pq, 0, (uint32_t)b.S, b.gfo, edges, b.state);
    auto go = [&](auto kern, int threads, int blocks) {
        return launch_flowb(kern, threads, blocks * sms, d.n_levels, s, d.fanin, d.fout_ptr, (const int4 *)d.edge_fpos,
                            b.pq, d.cload, b.dcl, b.ks, b.gfo, b.gsp, d.lvl, d.n_levels, d.n_start, b.S, tr_mode,
                            b.state, ops, d.err, kWaitLimitCycles);
    };
#define GO(V) go(k_bwdb_flow<V, Cfg<V>::bthreads, Cfg<V>::bblocks>, Cfg<V>::bthreads, Cfg<V>::bblocks)
    return v == 4 ? GO(4) : v == 2 ? GO(2) : GO(1);
#undef GO
}

}  // namespace dp
