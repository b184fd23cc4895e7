// Batched passes without barriers between levels: one cooperative launch per pass, every warp of the
// grid walks the (cell, 32 x V scenarios) items of all levels in order, dealt out in turn, and an
// item waits only for its own inputs.  The data is its own ready flag.
//
// Forward: the low part of a stored P never has bit 30 set (|lo| < 2 for |P| < 2^25), so the bit carries the
// parity of the pass that wrote it; a stored P (hi, lo) is written and read as one 64-bit element, so the bit speaks
// for both halves.  Everything that reads a stored P drops it (pair_get).  Reverse: an edge's contribution is written once and read once, and its
// reader leaves kNotYet behind for the next pass.  k_flowb_prep brings both to rest where another pass wrote
// the arrays in between.  Lag-one mode: a net's T has no bit to spare; it starts as kNotYet in every pass (27 MB, 6 us
// at 50,000 x 128).
//
// What bounds it: the level launches end a grid and start the next per level, about 3 us, with 58 instructions per
// (cell, scenario) to do in between (30 % of the issue slots used, 38 % of the warps active).  Without them a pass
// runs into the L2: 120,000 cells / 48 levels x 512 scenarios forward 217 us at 7.7 TB/s, reverse 385 us at 8.5 (reads
// alone reach 8.1 to 8.7 on this part); 50,000 / 44 x 256 forward 81 us, more than half of its load sectors polls.
// Four scenarios per thread spread the item's address and record work; 24 warps per SM forward, 20 reverse, where the
// registers end without spills to speak of (a reverse pass whose 80 registers spilled wrote three times the
// sectors).  Fetching the next item's record ahead cost more registers than it hid.  The reverse pass computes the
// partial derivatives before it waits for the fanout, so only sums and products are on the way from level to level.
// Forward with the model power + reverse, level launches against this: 120,000 x 512 404 + 575 us -> 366 + 435;
// 50,000 x 256 172 + 220 -> 124 + 137; 50,000 x 128 145 + 189 -> 104 + 103; 20,000 / 38 x 37 84 + 105 -> 66 + 68; 2,000 /
// 24 x 512 67 + 83 -> 50 + 50 (the power pass's own gain, 16 us at 50,000 x 256, included).  Lag-one mode: 50,000 x
// 128 142 + 257 -> 115 + 135, 120,000 x 256 555 + 1197 (level launches, general cell functions) -> 304 + 448.
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
// Rows between warps of the grid, through L2, by relaxed accesses whose elements are single-copy atomic: a (hi, lo) or
// (P, T) pair is one 64-bit element, so a reader that sees the tag in one half has the other half of the same store.
// (The elements of a vector access are accesses of their own: four-byte elements would let a new lo come with an old hi.)
__device__ __forceinline__ uint64_t pair_bits(const float2 &v) {
    return (uint64_t)__float_as_uint(v.x) | (uint64_t)__float_as_uint(v.y) << 32;
}
__device__ __forceinline__ float2 bits_pair(uint64_t b) {
    return make_float2(__uint_as_float((uint32_t)b), __uint_as_float((uint32_t)(b >> 32)));
}
template <int V>
__device__ __forceinline__ Row2<V> ld_row(const float2 *p) {
    uint64_t b[V];
    if constexpr (V == 1)
        asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(b[0]) : "l"(p) : "memory");
    else if constexpr (V == 2)
        asm volatile("ld.relaxed.gpu.global.v2.u64 {%0,%1}, [%2];" : "=l"(b[0]), "=l"(b[1]) : "l"(p) : "memory");
    else
        asm volatile("ld.relaxed.gpu.global.v4.u64 {%0,%1,%2,%3}, [%4];"
                     : "=l"(b[0]), "=l"(b[1]), "=l"(b[2]), "=l"(b[3])
                     : "l"(p)
                     : "memory");
    Row2<V> r;
#pragma unroll
    for (int i = 0; i < V; i++) r.v[i] = bits_pair(b[i]);
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
template <int V>
__device__ __forceinline__ void put_row(float2 *p, const Row2<V> &r) {
    if constexpr (V == 1)
        asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(pair_bits(r.v[0])) : "memory");
    else if constexpr (V == 2)
        asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1,%2};" ::"l"(p), "l"(pair_bits(r.v[0])), "l"(pair_bits(r.v[1]))
                     : "memory");
    else
        asm volatile("st.relaxed.gpu.global.v4.u64 [%0], {%1,%2,%3,%4};" ::"l"(p), "l"(pair_bits(r.v[0])),
                     "l"(pair_bits(r.v[1])), "l"(pair_bits(r.v[2])), "l"(pair_bits(r.v[3]))
                     : "memory");
}
template <int V>
__device__ __forceinline__ void put_row(float *p, const Row1<V> &r) {
    if constexpr (V == 1)
        asm volatile("st.relaxed.gpu.global.f32 [%0], %1;" ::"l"(p), "f"(r.v[0]) : "memory");
    else if constexpr (V == 2)
        asm volatile("st.relaxed.gpu.global.v2.f32 [%0], {%1,%2};" ::"l"(p), "f"(r.v[0]), "f"(r.v[1]) : "memory");
    else
        asm volatile("st.relaxed.gpu.global.v4.f32 [%0], {%1,%2,%3,%4};" ::"l"(p), "f"(r.v[0]), "f"(r.v[1]), "f"(r.v[2]),
                     "f"(r.v[3])
                     : "memory");
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

// an edge's adjoint: of P, in the lag-one mode of P and T
template <bool LAG>
struct Edge {
    using T = float;
    template <int V>
    using Row = Row1<V>;
    __device__ __forceinline__ static float rest() { return __uint_as_float(kNotYet); }
};
template <>
struct Edge<true> {
    using T = float2;
    template <int V>
    using Row = Row2<V>;
    __device__ __forceinline__ static float2 rest() {
        return make_float2(__uint_as_float(kNotYet), __uint_as_float(kNotYet));
    }
};
__device__ __forceinline__ bool waits(float v) { return __float_as_uint(v) == kNotYet; }
__device__ __forceinline__ bool waits(const float2 &v) { return waits(v.x) || waits(v.y); }

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

// true in one thread of the last block to get here (a block that gave up has recorded it before, in a word of the pass's
// own: the context's error word may be read and cleared by a call on another stream); done is 0 again
__device__ __forceinline__ bool last_block(uint32_t *done) {
    __syncthreads();
    if (threadIdx.x != 0) return false;
    __threadfence();
    if (atomicAdd(done, 1u) != gridDim.x - 1) return false;
    __threadfence();
    *done = 0u;
    return true;
}

template <int V, bool LAG, int THREADS, int BLOCKS>
__global__ void __launch_bounds__(THREADS, BLOCKS)
    k_fwdb_flow(const uint4 *__restrict__ fanin, float2 *pq, float *tq, const float *__restrict__ sp_in,
                const float *__restrict__ tr_in, const int32_t *__restrict__ lvl, int L, uint32_t ns, uint32_t S, uint32_t *state, OpTable ops, int *err,
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
        float *const tqs = LAG ? tq + sc : nullptr;
        at.next();
        Row2<V> o;
        Row1<V> ot;
        if (c < ns) {
            const Row1<V> a = ld1<V>(row_at(sp_in + sc, c, S));
#pragma unroll
            for (int i = 0; i < V; i++) o.v[i] = make_float2(a.v[i], 0.f);
            if (LAG) {
                ot = ld1<V>(row_at(tr_in + sc, c, S));
#pragma unroll
                for (int i = 0; i < V; i++)   // a caller's NaN of these bits is stored as another
                    if (__float_as_uint(ot.v[i]) == kNotYet) ot.v[i] = __uint_as_float(0x7FFFFFFFu);
            }
        } else {
            const int k = (int)((e >> 16) & 7u);
            Row2<V> x[4];
            Row1<V> t[4];
            bool late[4];
            auto look = [&](int j) {
                x[j] = ld_row<V>(row_at((const float2 *)pqs, n[j], S));
                if (LAG) t[j] = ld_row<V>(row_at((const float *)tqs, n[j], S));
            };
            auto check = [&](int j) {
                uint32_t bad = 0;
#pragma unroll
                for (int i = 0; i < V; i++) bad |= __float_as_uint(x[j].v[i].y) ^ tag;
                bool b = (bad & kTagBit) != 0;
                if (LAG)
#pragma unroll
                    for (int i = 0; i < V; i++) b = b || __float_as_uint(t[j].v[i]) == kNotYet;
                return b;
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
            cell_value<V, LAG>(
                e,
                [&](int j, Row2<V> &xj, Row1<V> &tj) {
                    xj = x[j];
                    if (LAG) tj = t[j];
                },
                o, ot);
        }
        if (on) {
#pragma unroll
            for (int i = 0; i < V; i++)
                o.v[i].y = __uint_as_float((__float_as_uint(o.v[i].y) & ~kTagBit) | tag);
            put_row<V>(row_at(pqs, c, S), o);
            if (LAG) put_row<V>(row_at(tqs, c, S), ot);
        }
    }
    if (!ok) state[6] = 1u;   // before the block's arrival
    if (last_block(state + 3)) {
        state[0] = ld_word(state + 6) ? 0u : S;
        state[1] = pass;
        state[6] = 0u;
    }
}

template <int V, bool LAG, int THREADS, int BLOCKS>
__global__ void __launch_bounds__(THREADS, BLOCKS)
    k_bwdb_flow(const uint4 *__restrict__ fanin, const int32_t *__restrict__ fptr, const int4 *__restrict__ efpos,
                const float2 *__restrict__ pq, const float *__restrict__ tq, const float *__restrict__ cload, const float *__restrict__ dcl,
                const float *__restrict__ ks, typename Edge<LAG>::T *gfo, float *gsp, float *gtr,
                const int32_t *__restrict__ lvl, int L,
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
        typename Edge<LAG>::T *const gs = gfo + sc;
        const int k = c < ns ? 0 : (int)((e >> 16) & 7u);
        // what does not wait for the fanout: the partial derivatives, the load, the local term's factor (bwdb_adjoint)
        const Row1<V> Ks = ld1<V>(ks + sc);
        Row1<V> cl, qmp, d[4], dp[4], dt[4];
        {
            if (dcl) cl = ld1<V>(row_at(dcl + sc, c, S));
            const float c0 = cload[c];
            Row2<V> self;
            if (!LAG) self = ld2<V>(row_at(pqs, c, S));
            if (c >= ns)
                cell_partials<V, LAG>(
                    e,
                    [&](int j, Row2<V> &x, Row1<V> &t) {
                        x = ld2<V>(row_at(pqs, n[j], S));
                        if (LAG) t = ld1<V>(row_at(tq + sc, n[j], S));
                    },
                    d, dp, dt);
#pragma unroll
            for (int i = 0; i < V; i++) {
                cl.v[i] = dcl ? c0 + cl.v[i] : c0;
                if (!LAG) {
                    cl.v[i] = __fmul_rn(__fmul_rn(2.f, Ks.v[i]), cl.v[i]);
                    qmp.v[i] = qmp32(self.v[i]);
                }
            }
        }
        // the fanout sum in index order, F edges in flight
        constexpr int F = V == 4 || (LAG && V == 2) ? 2 : 4;
        Row1<V> a, b;
#pragma unroll
        for (int i = 0; i < V; i++) a.v[i] = b.v[i] = 0.f;
        for (int32_t p = f0; p < f1 && ok; p += F) {
            using R = typename Edge<LAG>::template Row<V>;
            R u[F];
            bool late[F];
            auto look = [&](int j) {
                u[j] = ld_row<V>(row_at((const typename Edge<LAG>::T *)gs, (uint32_t)(p + j), S));
            };
            auto check = [&](int j) {
                bool w = false;
#pragma unroll
                for (int i = 0; i < V; i++) w = w || waits(u[j].v[i]);
                return w && on;
            };
#pragma unroll
            for (int j = 0; j < F; j++)
                if (p + j < f1) look(j);
#pragma unroll
            for (int j = 0; j < F; j++) late[j] = p + j < f1 && check(j);
            auto any = [&] {
                bool w = false;
#pragma unroll
                for (int j = 0; j < F; j++) w = w || late[j];
                return __any_sync(kAll, w) != 0;
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
            R rest;
#pragma unroll
            for (int i = 0; i < V; i++) rest.v[i] = Edge<LAG>::rest();
#pragma unroll
            for (int j = 0; j < F; j++)
                if (p + j < f1) {
#pragma unroll
                    for (int i = 0; i < V; i++) {
                        if constexpr (LAG) a.v[i] += u[j].v[i].x, b.v[i] += u[j].v[i].y;
                        else a.v[i] += u[j].v[i];
                    }
                    if (on) put_row(row_at(gs, (uint32_t)(p + j), S), rest);
                }
        }
        if (!on) continue;
        if (LAG) {
#pragma unroll
            for (int i = 0; i < V; i++) b.v[i] = fmaf(Ks.v[i], cl.v[i], b.v[i]);
        } else if (c >= ns || tr_mode) {
#pragma unroll
            for (int i = 0; i < V; i++) a.v[i] = fmaf(cl.v[i], qmp.v[i], a.v[i]);
        }
        if (c < ns) {
            st1<V>(row_at(gsp + sc, c, S), a);
            if (LAG) st1<V>(row_at(gtr + sc, c, S), b);
            continue;
        }
#pragma unroll
        for (int j = 0; j < 4; j++)
            if (j < k) {
                typename Edge<LAG>::template Row<V> g;
#pragma unroll
                for (int i = 0; i < V; i++) {
                    if constexpr (LAG)
                        g.v[i] = make_float2(fmaf(a.v[i], d[j].v[i], __fmul_rn(b.v[i], dp[j].v[i])),
                                             __fmul_rn(b.v[i], dt[j].v[i]));
                    else g.v[i] = __fmul_rn(a.v[i], d[j].v[i]);
                }
                put_row(row_at(gs, pos[j], S), g);
            }
    }
    if (!ok) state[7] = 1u;
    if (last_block(state + 4)) {
        state[LAG ? 5 : 2] = ld_word(state + 7) ? 0u : 1u;
        state[7] = 0u;
    }
}

// The arrays of a pass as it expects them: which 0, the forward pass's pairs, where the last to write them was not a
// dataflow pass of the same S (and tq, n words, always); 1, the reverse pass's edges, m words, where the last was not one
// (clean: its mark)
__global__ void k_flowb_prep(int which, float2 *pq, float *tq, int64_t n, uint32_t S, float *gfo, int64_t m,
                             const uint32_t *state, const uint32_t *clean) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, T = (int64_t)gridDim.x * blockDim.x;
    if (which == 0) {
        if (tq)
            for (int64_t i = t; i < n; i += T) tq[i] = __uint_as_float(kNotYet);
        if (state[0] == S) return;
        const float2 v = make_float2(0.f, __uint_as_float((state[1] & 1u) << 30));
        for (int64_t i = t; i < n; i += T) pq[i] = v;
    } else {
        if (*clean == 1u) return;
        for (int64_t i = t; i < m; i += T) gfo[i] = __uint_as_float(kNotYet);
    }
}

// threads per block and blocks per SM by scenarios per thread (see above; 50,000 x 256 reverse, v = 4: 512 threads per
// SM 137 us, 640 137, 768 150; 120,000 x 512 485, 441, 467)
template <int V, bool LAG>
struct Cfg {
    static constexpr int fthreads = V == 4 || LAG ? 384 : 512, fblocks = 2;
    static constexpr int bthreads = V == 4 ? 320 : LAG ? 256 : 448, bblocks = 2;
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

template <int V, bool LAG>
cudaError_t fwd(const DevDesign &d, const BatchBufs &b, const OpTable &ops, int sms, cudaStream_t s) {
    using C = Cfg<V, LAG>;
    k_flowb_prep<<<(unsigned)(sms * 4), 512, 0, s>>>(0, b.pq, LAG ? b.tq : nullptr, d.n_nets * b.S, (uint32_t)b.S,
                                                     nullptr, 0, b.state, nullptr);
    return launch_flowb(k_fwdb_flow<V, LAG, C::fthreads, C::fblocks>, C::fthreads, C::fblocks * sms, d.n_levels, s,
                        d.fanin, b.pq, b.tq, b.sp_in, b.tr_in, d.lvl, d.n_levels, d.n_start, b.S, b.state, ops, d.err,
                        kWaitLimitCycles);
}
template <int V, bool LAG>
cudaError_t bwd(const DevDesign &d, const BatchBufs &b, const OpTable &ops, int tr_mode, int64_t edges, int sms,
                cudaStream_t s) {
    using C = Cfg<V, LAG>;
    typename Edge<LAG>::T *gfo;
    if constexpr (LAG) gfo = b.gfo2;
    else gfo = b.gfo;
    k_flowb_prep<<<(unsigned)(sms * 4), 512, 0, s>>>(1, nullptr, nullptr, 0, (uint32_t)b.S, (float *)gfo,
                                                     edges * (LAG ? 2 : 1), b.state, b.state + (LAG ? 5 : 2));
    return launch_flowb(k_bwdb_flow<V, LAG, C::bthreads, C::bblocks>, C::bthreads, C::bblocks * sms, d.n_levels, s,
                        d.fanin, d.fout_ptr, (const int4 *)d.edge_fpos, b.pq, b.tq, d.cload, b.dcl, b.ks, gfo, b.gsp,
                        b.gtr, d.lvl, d.n_levels, d.n_start, b.S, tr_mode, b.state, ops, d.err, kWaitLimitCycles);
}

}  // namespace

cudaError_t launch_fwdb_flow(const DevDesign &d, const BatchBufs &b, const OpTable &ops, int tr_mode, int v, int sms,
                             cudaStream_t s) {
    if (tr_mode == 2) return v == 1 ? fwd<1, true>(d, b, ops, sms, s) : fwd<2, true>(d, b, ops, sms, s);
    if (v == 4) return fwd<4, false>(d, b, ops, sms, s);
    return v == 2 ? fwd<2, false>(d, b, ops, sms, s) : fwd<1, false>(d, b, ops, sms, s);
}

cudaError_t launch_bwdb_flow(const DevDesign &d, const BatchBufs &b, const OpTable &ops, int tr_mode, int v,
                             int64_t edges, int sms, cudaStream_t s) {
    if (tr_mode == 2)
        return v == 1 ? bwd<1, true>(d, b, ops, tr_mode, edges, sms, s) : bwd<2, true>(d, b, ops, tr_mode, edges, sms, s);
    if (v == 4) return bwd<4, false>(d, b, ops, tr_mode, edges, sms, s);
    return v == 2 ? bwd<2, false>(d, b, ops, tr_mode, edges, sms, s) : bwd<1, false>(d, b, ops, tr_mode, edges, sms, s);
}

}  // namespace dp
