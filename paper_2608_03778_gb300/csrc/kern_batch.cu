// Batched scenarios: S input-activity scenarios of one design per launch.
// Every per-net value is stored scenario-innermost (value[n * S + s]), so the
// S values of one fanin are contiguous: a warp covering 32 scenarios of one
// cell reads each fanin as 256 consecutive bytes.  A block is bx scenarios x
// by cells; blockIdx.y walks the cells of a level.  Each thread computes one
// (cell, scenario) independently of the block shape, so every shape gives
// bitwise identical results and the shape is free for the autotuner.
//
// Each cell evaluates P(out = 1) as the multilinear extension of its truth
// table in float-float (the same reading of Eq. 2 as the single-scenario
// path), and only P is stored, as a float-float value (8 bytes per net and
// scenario): Q is re-derived as 1 - P in float-float, exact to about 1e-14
// absolute, wherever it is read.  That loses Q's relative accuracy only for nets within about 1e-9
// of 1, which matters for the hybrid beta (Eq. 5, single-scenario only) and
// not for the model power, SP, TR or gradients at their tolerances; it halves
// the bytes every gather moves.  The gradient is the model gradient (Sec. III-E,
// Eq. 7) in binary32, scaled per scenario by a seed K * w_s so that a caller
// can back-propagate any weighted sum of the scenario powers.
#include "kern_cells.cuh"

namespace dp {
namespace {

__host__ __device__ inline int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }

__global__ void k_fwdb_start(const float *__restrict__ sp_in, float2 *pq, int64_t n, uint32_t *state) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) state[0] = 0u;   // no dataflow pass wrote these
    if (i >= n) return;
    pq[i] = make_float2(sp_in[i], 0.f);
}

// the same, four values per thread (n a multiple of 4): one 16-byte load, two 16-byte stores
__global__ void k_fwdb_start4(const float *__restrict__ sp_in, float2 *pq, int64_t n, uint32_t *state) {
    const int64_t i = 4 * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x);
    if (i == 0) state[0] = 0u;
    if (i >= n) return;
    const float4 a = *reinterpret_cast<const float4 *>(sp_in + i);
    reinterpret_cast<float4 *>(pq + i)[0] = make_float4(a.x, 0.f, a.y, 0.f);
    reinterpret_cast<float4 *>(pq + i)[1] = make_float4(a.z, 0.f, a.w, 0.f);
}

// V consecutive values of a row in 8- or 16-byte accesses
template <int V>
__device__ __forceinline__ void row_load(const float2 *src, float2 (&v)[V]) {
    if constexpr (V == 1) {
        v[0] = *src;
    } else {
#pragma unroll
        for (int h = 0; h < V / 2; h++) {
            const float4 t = reinterpret_cast<const float4 *>(src)[h];
            v[2 * h] = make_float2(t.x, t.y);
            v[2 * h + 1] = make_float2(t.z, t.w);
        }
    }
}
template <int V>
__device__ __forceinline__ void row_store(float2 *dst, const float2 (&v)[V]) {
    if constexpr (V == 1) {
        *dst = v[0];
    } else {
#pragma unroll
        for (int h = 0; h < V / 2; h++)
            reinterpret_cast<float4 *>(dst)[h] = make_float4(v[2 * h].x, v[2 * h].y, v[2 * h + 1].x, v[2 * h + 1].y);
    }
}
template <int V>
__device__ __forceinline__ void row_add(const float *src, float (&acc)[V]) {
    if constexpr (V == 1) {
        acc[0] += *src;
    } else if constexpr (V == 2) {
        const float2 t = *reinterpret_cast<const float2 *>(src);
        acc[0] += t.x, acc[1] += t.y;
    } else {
        const float4 t = *reinterpret_cast<const float4 *>(src);
        acc[0] += t.x, acc[1] += t.y, acc[2] += t.z, acc[3] += t.w;
    }
}
template <int V>
__device__ __forceinline__ void row_store(float *dst, const float (&v)[V]) {
    if constexpr (V == 1) *dst = v[0];
    else if constexpr (V == 2) *reinterpret_cast<float2 *>(dst) = make_float2(v[0], v[1]);
    else *reinterpret_cast<float4 *>(dst) = make_float4(v[0], v[1], v[2], v[3]);
}

// One level, V consecutive scenarios per thread (1, or 2 or 4 with S a multiple of V): each fanin
// gather is V / 2 16-byte loads of those scenarios' P, so a warp keeps V times the bytes in flight.
template <int V>
__global__ void k_fwdb_level(const uint4 *__restrict__ fanin, float2 *pq, int32_t c0, int32_t c1, int64_t ns,
                             int64_t S, OpTable ops) {
    const int64_t s = V * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x);
    pdl_trigger();
    if (s >= S) return;
    const int64_t step = (int64_t)gridDim.y * blockDim.y;
    const int64_t cf = c0 + (int64_t)blockIdx.y * blockDim.y + threadIdx.y;
    uint4 r = cf < c1 ? fanin[cf] : make_uint4(0, 0, 0, 0);   // static: before the wait
    pdl_wait();
    for (int64_t c = cf; c < c1; c += step) {
        if (c != cf) r = fanin[c];
        const uint32_t op = r.x >> 24;
        const uint32_t n[4] = {r.x & kMask24, r.y, r.z, r.w};
        with_cell(ops.e[op], [&](const auto f) {
            constexpr int K = decltype(f)::k;
            float2 x[K ? K : 1][V], out[V];
#pragma unroll
            for (int j = 0; j < K; j++) row_load(pq + (int64_t)n[j] * S + s, x[j]);
#pragma unroll
            for (int i = 0; i < V; i++) {
                pair_ff a[4];
#pragma unroll
                for (int j = 0; j < K; j++) a[j] = pair_get(x[j][i]);
                const ff p = f.prob(a);
                out[i] = make_float2(p.hi, p.lo);
            }
            row_store(pq + (ns + c) * S + s, out);
        });
    }
}

// Eq. 1 per scenario: chunk b of the nets -> partials[s * nchunks + b], then
// the chunks of each scenario summed in FP64 in a fixed order (reproducible).
// Within a chunk a thread forms each term alpha * C in binary32 (TR = 2 P Q
// with Q from the float-float pair, so it keeps its relative accuracy near
// P = 1; about 1e-7 relative per term) and adds it with TwoSum into a
// float-float sum (about 48 significant bits), so the FP64 pipe, slow on this
// part, sees one conversion per chunk instead of several operations per term.
// V consecutive scenarios per thread (S a multiple of V), kPowerNets nets' loads in flight before their terms are
// added in net order.
template <class R, class T>
__device__ __forceinline__ R read_row(const T *p) {   // through L1: a few scenarios' rows share its lines
    R r;
    constexpr int n = sizeof(R) / sizeof(float);
    float *const o = reinterpret_cast<float *>(&r);
    const float *const a = reinterpret_cast<const float *>(p);
    if constexpr (n == 1) {
        o[0] = a[0];
    } else if constexpr (n == 2) {
        const float2 t = *reinterpret_cast<const float2 *>(a);
        o[0] = t.x, o[1] = t.y;
    } else {
#pragma unroll
        for (int i = 0; i < n; i += 4) {
            const float4 t = *reinterpret_cast<const float4 *>(a + i);
            o[i] = t.x, o[i + 1] = t.y, o[i + 2] = t.z, o[i + 3] = t.w;
        }
    }
    return r;
}
template <int V>
__global__ void k_powerb_partials(const float2 *__restrict__ pq, const float *__restrict__ tr_in,
                                  const float *__restrict__ cload, const float *__restrict__ dcl, double *partials,
                                  int64_t nn, int64_t ns, int64_t S, int64_t chunk, int nchunks, int tr_mode) {
    const int64_t s = V * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x);
    const int64_t b = (int64_t)blockIdx.y * blockDim.y + threadIdx.y;
    if (s >= S || b >= nchunks) return;
    constexpr int kPowerNets = V == 1 ? 8 : 4;
    const int64_t n0 = b * chunk, n1 = n0 + chunk < nn ? n0 + chunk : nn;
    ff acc[V];
#pragma unroll
    for (int v = 0; v < V; v++) acc[v] = ff_make(0.f);
    auto stored = [&](int64_t m) { return tr_mode == 2 || (m < ns && tr_mode == 0); };   // its TR, not its P
    for (int64_t n = n0; n < n1; n += kPowerNets) {
        Row2<V> w[kPowerNets];
        Row1<V> t[kPowerNets], d[kPowerNets];
        float c[kPowerNets];
#pragma unroll
        for (int i = 0; i < kPowerNets; i++) {
            const int64_t m = n + i;
            if (m >= n1) continue;
            if (stored(m)) t[i] = read_row<Row1<V>>(tr_in + m * S + s);
            else w[i] = read_row<Row2<V>>(pq + m * S + s);
            if (dcl) d[i] = read_row<Row1<V>>(dcl + m * S + s);
            c[i] = cload[m];
        }
#pragma unroll
        for (int i = 0; i < kPowerNets; i++) {
            if (n + i >= n1) continue;
            const bool st = stored(n + i);
#pragma unroll
            for (int v = 0; v < V; v++) {
                float a;
                if (st) {
                    a = t[i].v[v];
                } else {
                    const pair_ff pr = pair_get(w[i].v[v]);
                    a = 2.f * (pr.p.hi + pr.p.lo) * (pr.q.hi + pr.q.lo);
                }
                const ff u = two_sum(acc[v].hi, a * (dcl ? c[i] + d[i].v[v] : c[i]));
                acc[v] = fast_two_sum(u.hi, u.lo + acc[v].lo);
            }
        }
    }
#pragma unroll
    for (int v = 0; v < V; v++) partials[(s + v) * nchunks + b] = (double)acc[v].hi + (double)acc[v].lo;
}

// one warp per scenario: lane l sums chunks l, l + 32, ... in order, then a fixed shuffle tree
__global__ void k_sumb_final(const double *__restrict__ partials, int nchunks, int64_t S, double K, double *out) {
    const int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (s >= S) return;
    double acc = 0.0;
    for (int b0 = lane; b0 < nchunks; b0 += 32 * 16) {   // sixteen loads in flight, added in order
        double v[16];
#pragma unroll
        for (int i = 0; i < 16; i++) v[i] = b0 + 32 * i < nchunks ? partials[s * nchunks + b0 + 32 * i] : 0.0;
#pragma unroll
        for (int i = 0; i < 16; i++)
            if (b0 + 32 * i < nchunks) acc += v[i];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) out[s] = K * acc;
}

__global__ void k_seedb(float *ks, const double *__restrict__ w, double K, int64_t S) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s < S) ks[s] = (float)(w ? K * w[s] : K);
}

// reverse level: each net's adjoint is its fanout range summed in index order
// plus its local term d(K_s C 2PQ)/dP = 2 K_s C (Q - P); the cell then writes
// one contribution per input edge (no atomics).  V consecutive scenarios per thread as in the forward level.
template <int V>
__global__ void k_bwdb_level(const uint4 *__restrict__ fanin, const int32_t *__restrict__ fptr,
                             const int4 *__restrict__ efpos, const float2 *__restrict__ pq,
                             const float *__restrict__ cload, const float *__restrict__ dcl,
                             const float *__restrict__ ks, float *gfo, int32_t c0, int32_t c1, int64_t ns, int64_t S,
                             OpTable ops) {
    const int64_t s = V * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x);
    pdl_trigger();
    if (s >= S) return;
    const int64_t step = (int64_t)gridDim.y * blockDim.y;
    const int64_t cf = c0 + (int64_t)blockIdx.y * blockDim.y + threadIdx.y;
    uint4 rf = cf < c1 ? fanin[cf] : make_uint4(0, 0, 0, 0);   // static: before the wait
    pdl_wait();
    float Ks[V];
#pragma unroll
    for (int i = 0; i < V; i++) Ks[i] = ks[s + i];
    for (int64_t c = cf; c < c1; c += step) {
        const int64_t n = ns + c;
        // everything that does not depend on the fanout sum goes out first, so its loads
        // overlap the fanout range's
        const uint4 r = c == cf ? rf : fanin[c];
        const int4 ep = efpos[c];
        const int32_t e0 = fptr[n], e1 = fptr[n + 1];
        float2 self[V];
        row_load(pq + n * S + s, self);
        float cl[V];
#pragma unroll
        for (int i = 0; i < V; i++) cl[i] = cl_of(cload, dcl, n, S, s + i);
        const uint32_t op = r.x >> 24;
        const uint32_t nid[4] = {r.x & kMask24, r.y, r.z, r.w};
        const int pos[4] = {ep.x, ep.y, ep.z, ep.w};
        with_cell(ops.e[op], [&](const auto f) {
            constexpr int K = decltype(f)::k;
            float2 x[K ? K : 1][V];
#pragma unroll
            for (int j = 0; j < K; j++) row_load(pq + (int64_t)nid[j] * S + s, x[j]);
            float acc[V];
#pragma unroll
            for (int i = 0; i < V; i++) acc[i] = 0.f;
            for (int32_t e = e0; e < e1; e++) row_add(gfo + (int64_t)e * S + s, acc);
            float g[K ? K : 1][V];
#pragma unroll
            for (int i = 0; i < V; i++) {
                float p[4], q[4], d[4];
#pragma unroll
                for (int j = 0; j < K; j++) {
                    const pair_ff a = pair_get(x[j][i]);
                    p[j] = a.p.hi + a.p.lo;
                    q[j] = a.q.hi + a.q.lo;
                }
                f.partials(p, q, d);
                const float gn = bwdb_adjoint(acc[i], Ks[i], cl[i], self[i]);
#pragma unroll
                for (int j = 0; j < K; j++) g[j][i] = __fmul_rn(gn, d[j]);
            }
#pragma unroll
            for (int j = 0; j < K; j++) row_store(gfo + (int64_t)pos[j] * S + s, g[j]);
        });
    }
}

// startpoints: fanout sum, plus the local term when their TR derives from their SP (tr_mode 1)
__global__ void k_bwdb_start(const int32_t *__restrict__ fptr, const float2 *__restrict__ pq,
                             const float *__restrict__ cload, const float *__restrict__ dcl,
                             const float *__restrict__ ks,
                             const float *__restrict__ gfo, float *gsp, int64_t ns, int64_t S, int tr_mode,
                             uint32_t *state) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    pdl_trigger();
    if (s >= S) return;
    pdl_wait();
    if (s == 0 && blockIdx.y == 0 && threadIdx.y == 0) state[2] = 0u;   // gfo holds values
    const float Ks = ks[s];
    const int64_t step = (int64_t)gridDim.y * blockDim.y;
    for (int64_t k = (int64_t)blockIdx.y * blockDim.y + threadIdx.y; k < ns; k += step) {
        const int32_t e0 = fptr[k], e1 = fptr[k + 1];
        float acc = 0.f;
        for (int32_t e = e0; e < e1; e++) acc += gfo[(int64_t)e * S + s];
        gsp[k * S + s] = tr_mode ? bwdb_adjoint(acc, Ks, cl_of(cload, dcl, k, S, s), pq[k * S + s]) : acc;
    }
}

// The same with four consecutive scenarios per thread (S a multiple of 4): 16-byte
// loads of the edge adjoints, eight edges' loads in flight before they are added in
// index order (the same order as above, so bitwise the same).
__global__ void k_bwdb_start4(const int32_t *__restrict__ fptr, const float2 *__restrict__ pq,
                              const float *__restrict__ cload, const float *__restrict__ dcl,
                              const float *__restrict__ ks, const float *__restrict__ gfo, float *gsp, int64_t ns,
                              int64_t S, int tr_mode, uint32_t *state) {
    const int64_t s = 4 * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x);
    pdl_trigger();
    if (s >= S) return;
    pdl_wait();
    if (s == 0 && blockIdx.y == 0 && threadIdx.y == 0) state[2] = 0u;
    const float4 Ks = *reinterpret_cast<const float4 *>(ks + s);
    const int64_t step = (int64_t)gridDim.y * blockDim.y;
    for (int64_t k = (int64_t)blockIdx.y * blockDim.y + threadIdx.y; k < ns; k += step) {
        const int32_t e0 = fptr[k], e1 = fptr[k + 1];
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int32_t e = e0; e < e1; e += 8) {
            float4 t[8];
#pragma unroll
            for (int i = 0; i < 8; i++)
                t[i] = e + i < e1 ? *reinterpret_cast<const float4 *>(gfo + (int64_t)(e + i) * S + s)
                                  : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int i = 0; i < 8; i++)
                if (e + i < e1) {
                    acc.x += t[i].x;
                    acc.y += t[i].y;
                    acc.z += t[i].z;
                    acc.w += t[i].w;
                }
        }
        float g[4] = {acc.x, acc.y, acc.z, acc.w};
        if (tr_mode) {
            const float ksv[4] = {Ks.x, Ks.y, Ks.z, Ks.w};
            const float4 u0 = reinterpret_cast<const float4 *>(pq + k * S + s)[0];
            const float4 u1 = reinterpret_cast<const float4 *>(pq + k * S + s)[1];
            const float2 w[4] = {make_float2(u0.x, u0.y), make_float2(u0.z, u0.w), make_float2(u1.x, u1.y),
                                 make_float2(u1.z, u1.w)};
#pragma unroll
            for (int v = 0; v < 4; v++) g[v] = bwdb_adjoint(g[v], ksv[v], cl_of(cload, dcl, k, S, s + v), w[v]);
        }
        *reinterpret_cast<float4 *>(gsp + k * S + s) = make_float4(g[0], g[1], g[2], g[3]);
    }
}

// dP_s/dC_n = K_s alpha_n(s); dP_s/dpincap_c = K_s sum_j alpha_{fanin j}(s)
// (one pin cap per cell, loading each of its fanin nets); dP_s/dTR_k = K_s C_k
// at a startpoint in tr_mode 0, else 0
__global__ void k_gradb_rows(const uint4 *__restrict__ fanin, const float2 *__restrict__ pq,
                             const float *__restrict__ tr_in, const float *__restrict__ cload,
                             const float *__restrict__ dcl,
                             const int32_t *__restrict__ net_of_user, const int32_t *__restrict__ cell_of_user,
                             const float *__restrict__ ks, const float *__restrict__ gtr_lag1, float *gcl,
                             float *gpin, float *gtr, int64_t nn, int64_t nc, int64_t ns, int64_t S, int tr_mode,
                             OpTable ops) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= S) return;
    const float Ks = ks[s];
    const int64_t rows = (gcl ? nn : 0) + (gpin ? nc : 0) + (gtr ? ns : 0);
    const int64_t step = (int64_t)gridDim.y * blockDim.y;
    for (int64_t r = (int64_t)blockIdx.y * blockDim.y + threadIdx.y; r < rows; r += step) {
        int64_t u = r;
        if (gcl) {
            if (u < nn) {
                gcl[u * S + s] = Ks * alpha32(pq, tr_in, net_of_user[u], ns, S, s, tr_mode);
                continue;
            }
            u -= nn;
        }
        if (gpin) {
            if (u < nc) {
                const uint4 f = fanin[cell_of_user[u]];
                const int k = op_arity(ops, f.x >> 24);
                const uint32_t n[4] = {f.x & kMask24, f.y, f.z, f.w};
                float a = 0.f;
#pragma unroll
                for (int j = 0; j < 4; j++)
                    if (j < k) a += alpha32(pq, tr_in, n[j], ns, S, s, tr_mode);
                gpin[u * S + s] = Ks * a;
                continue;
            }
            u -= nc;
        }
        gtr[u * S + s] = tr_mode == 2 ? gtr_lag1[u * S + s] : (tr_mode ? 0.f : Ks * cl_of(cload, dcl, u, S, s));
    }
}

// Cap gradients summed over the scenarios in FP64: one warp per row, lane l
// takes scenarios l, l + 32, ... in order, then a fixed shuffle tree.
__global__ void k_gradb_reduce(const uint4 *__restrict__ fanin, const float2 *__restrict__ pq,
                               const float *__restrict__ tr_in, const int32_t *__restrict__ net_of_user,
                               const int32_t *__restrict__ cell_of_user, const float *__restrict__ ks, float *gcl,
                               float *gpin, int64_t nn, int64_t nc, int64_t ns, int64_t S, int tr_mode, OpTable ops) {
    const int lane = threadIdx.x & 31;
    const int64_t rows = (gcl ? nn : 0) + (gpin ? nc : 0);
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t W = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t r = w0; r < rows; r += W) {
        int64_t u = r;
        const bool is_cl = gcl && u < nn;
        if (gcl && !is_cl) u -= nn;
        uint32_t n[4] = {0, 0, 0, 0};
        int k = 1;
        if (is_cl) {
            n[0] = (uint32_t)net_of_user[u];
        } else {
            const uint4 f = fanin[cell_of_user[u]];
            k = op_arity(ops, f.x >> 24);
            n[0] = f.x & kMask24;
            n[1] = f.y;
            n[2] = f.z;
            n[3] = f.w;
        }
        double acc = 0.0;
        for (int64_t s = lane; s < S; s += 32) {
            float a = 0.f;
#pragma unroll
            for (int j = 0; j < 4; j++)
                if (j < k) a += alpha32(pq, tr_in, n[j], ns, S, s, tr_mode);
            acc += (double)(ks[s] * a);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0) {
            if (is_cl) gcl[u] = (float)acc;
            else gpin[u] = (float)acc;
        }
    }
}

__global__ void k_netb_user(const float2 *__restrict__ pq, const float *__restrict__ tr_in,
                            const int32_t *__restrict__ net_of_user, float *sp_out, float *tr_out, int64_t nn,
                            int64_t ns, int64_t S, int tr_mode) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= S) return;
    const int64_t step = (int64_t)gridDim.y * blockDim.y;
    for (int64_t u = (int64_t)blockIdx.y * blockDim.y + threadIdx.y; u < nn; u += step) {
        const int64_t n = net_of_user[u];
        if (sp_out) {
            const float2 v = untag(pq[n * S + s]);
            sp_out[u * S + s] = v.x + v.y;
        }
        if (tr_out) tr_out[u * S + s] = alpha32(pq, tr_in, n, ns, S, s, tr_mode);
    }
}

__global__ void k_ascent(float *x, const float *__restrict__ g, int64_t n, float eta) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float v = __fadd_rn(x[i], __fmul_rn(eta, g[i]));
    x[i] = fminf(fmaxf(v, 0.f), 1.f);
}

// ---- Eq. 3: P_virus of the thresholded vectors ----
// words of net n: [2W] with W = ceil(S / 64); word w < W holds v0 of scenarios
// 64 w .. 64 w + 63, word W + w holds v1 = not v0 of the same scenarios
__global__ void k_virus_start(const float *__restrict__ sp, uint64_t *words, uint8_t *v0, int64_t ns, int64_t S,
                              int64_t W) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= ns * W) return;
    const int64_t k = i / W, w = i - k * W;
    uint64_t b0 = 0, valid = 0;
    for (int b = 0; b < 64; b++) {
        const int64_t s = w * 64 + b;
        if (s >= S) break;
        const bool one = sp[k * S + s] >= 0.5f;
        if (v0) v0[k * S + s] = one ? 1 : 0;
        b0 |= (uint64_t)one << b;
        valid |= 1ull << b;
    }
    words[k * 2 * W + w] = b0;
    words[k * 2 * W + W + w] = ~b0 & valid;
}

__global__ void k_virus_level(const uint4 *__restrict__ fanin, uint64_t *words, int32_t c0, int32_t c1, int64_t ns,
                              int64_t W2, OpTable ops) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)(c1 - c0) * W2) return;
    const int64_t c = c0 + i / W2, w = i % W2;
    const uint4 r = fanin[c];
    const uint32_t op = r.x >> 24;
    const int k = op_arity(ops, op);
    const uint32_t n[4] = {r.x & kMask24, r.y, r.z, r.w};
    uint64_t x[4];
#pragma unroll
    for (int j = 0; j < 4; j++) x[j] = j < k ? words[(int64_t)n[j] * W2 + w] : 0ull;
    words[(ns + c) * W2 + w] = cell_bits(k, op_tt(ops, op), x);
}

__global__ void k_virus_partials(const uint64_t *__restrict__ words, const float *__restrict__ cload,
                                 double *partials, int64_t nn, int64_t S, int64_t W, int64_t chunk, int nchunks) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= S) return;
    const int64_t w = s >> 6;
    const int b = (int)(s & 63);
    const int64_t n0 = (int64_t)blockIdx.y * chunk, n1 = n0 + chunk < nn ? n0 + chunk : nn;
    double acc = 0.0;
    for (int64_t n = n0; n < n1; n++) {
        const uint64_t d = words[n * 2 * W + w] ^ words[n * 2 * W + W + w];
        if ((d >> b) & 1ull) acc += (double)cload[n];
    }
    partials[s * nchunks + blockIdx.y] = acc;
}

// out[c * ldo + r] = in[r * C + c] for an R x C block, through 32 x 32 tiles in shared memory
__global__ void k_transpose(const float *__restrict__ in, float *out, int64_t R, int64_t C, int64_t ldo) {
    __shared__ float t[32][33];
    const int64_t r0 = (int64_t)blockIdx.y * 32, c0 = (int64_t)blockIdx.x * 32;
    for (int i = threadIdx.y; i < 32; i += blockDim.y) {
        const int64_t r = r0 + i, c = c0 + threadIdx.x;
        if (r < R && c < C) t[i][threadIdx.x] = in[r * C + c];
    }
    __syncthreads();
    for (int i = threadIdx.y; i < 32; i += blockDim.y) {
        const int64_t c = c0 + i, r = r0 + threadIdx.x;
        if (r < R && c < C) out[c * ldo + r] = t[threadIdx.x][i];
    }
}


int nchunks_of(int64_t nn, int64_t *chunk) {
    const int64_t m = nn > 0 ? nn : 1;
    *chunk = cdiv(m, kBatchPowerChunks);
    return (int)cdiv(m, *chunk);
}

}  // namespace

void launch_fwdb(const DevDesign &d, const BatchBufs &b, const OpTable &ops, const int32_t *lvl, int tr_mode,
                 BatchShape sh, cudaStream_t s) {
    if (tr_mode == 2) {
        launch_fwdl(d, b, ops, lvl, sh, s);
        return;
    }
    const int64_t S = b.S;
    if (d.n_start && (d.n_start * S) % 4 == 0)
        k_fwdb_start4<<<(unsigned)cdiv(d.n_start * S / 4, 256), 256, 0, s>>>(b.sp_in, b.pq, d.n_start * S, b.state);
    else if (d.n_start)
        k_fwdb_start<<<(unsigned)cdiv(d.n_start * S, 256), 256, 0, s>>>(b.sp_in, b.pq, d.n_start * S, b.state);
    const int v = scen_per_thread(sh, S);
    sh = fit_shape(sh, S / v);
    const dim3 blk((unsigned)sh.bx, (unsigned)sh.by);
    for (int l = 1; l <= d.n_levels; l++) {
        const int32_t c0 = lvl[l - 1], c1 = lvl[l];
        if (c1 <= c0) continue;
        const dim3 g = bgrid(S / v, sh, c1 - c0);
        if (v == 4) launch_pdl(k_fwdb_level<4>, g, blk, s, d.fanin, b.pq, c0, c1, d.n_start, S, ops);
        else if (v == 2) launch_pdl(k_fwdb_level<2>, g, blk, s, d.fanin, b.pq, c0, c1, d.n_start, S, ops);
        else launch_pdl(k_fwdb_level<1>, g, blk, s, d.fanin, b.pq, c0, c1, d.n_start, S, ops);
    }
}

void launch_powerb(const DevDesign &d, const BatchBufs &b, int tr_mode, double K, cudaStream_t s) {
    const int64_t S = b.S;
    int64_t chunk = 0;
    const int nch = nchunks_of(d.n_nets, &chunk);
    const int v = S % 4 == 0 && S >= 256 ? 4 : S % 2 == 0 && S >= 128 ? 2 : 1;
    // 65,536 threads and more take two or four scenarios each (forward with power, us, v = 1 / 2 / 4: 50,000 cells x 256
    // 226 / 218 / 207, 120,000 x 64 155 / 166 / 177), and fewer go into smaller blocks, for every SM to have some
    // (2,000,000 x 2: 587 with blocks of 128, 484 so)
    int width = 1, bx = 1;
    while (width < 128 && (int64_t)width * 608 < nch * (S / v)) width <<= 1;
    while (bx < width && bx * v < S) bx <<= 1;
    const int by = width / bx;
    const dim3 g((unsigned)cdiv(S / v, bx), (unsigned)cdiv(nch, by)), blk((unsigned)bx, (unsigned)by);
    const float *act = tr_mode == 2 ? b.tq : b.tr_in;
    auto go = [&](auto kern) {
        kern<<<g, blk, 0, s>>>(b.pq, act, d.cload, b.dcl, b.partials, d.n_nets, d.n_start, S, chunk, nch, tr_mode);
    };
    if (v == 4) go(k_powerb_partials<4>);
    else if (v == 2) go(k_powerb_partials<2>);
    else go(k_powerb_partials<1>);
    k_sumb_final<<<(unsigned)cdiv(S * 32, 256), 256, 0, s>>>(b.partials, nch, S, K, b.power);
}

void launch_seedb(const BatchBufs &b, double K, const double *weights, cudaStream_t s) {
    k_seedb<<<(unsigned)cdiv(b.S, 128), 128, 0, s>>>(b.ks, weights, K, b.S);
}

void launch_bwdb(const DevDesign &d, const BatchBufs &b, const OpTable &ops, const int32_t *lvl, int tr_mode,
                 BatchShape sh, cudaStream_t s) {
    if (tr_mode == 2) {
        launch_bwdl(d, b, ops, lvl, sh, s);
        return;
    }
    const int64_t S = b.S;
    const int v = scen_per_thread(sh, S);   // scenarios per thread in the cell levels
    const BatchShape sh1 = fit_shape(sh, S);
    sh = fit_shape(sh, S / v);
    const dim3 blk((unsigned)sh.bx, (unsigned)sh.by);
    for (int l = d.n_levels; l >= 1; l--) {
        const int32_t c0 = lvl[l - 1], c1 = lvl[l];
        if (c1 <= c0) continue;
        const dim3 g = bgrid(S / v, sh, c1 - c0);
        if (v == 4)
            launch_pdl(k_bwdb_level<4>, g, blk, s, d.fanin, d.fout_ptr, (const int4 *)d.edge_fpos, b.pq, d.cload,
                       b.dcl, b.ks, b.gfo, c0, c1, d.n_start, S, ops);
        else if (v == 2)
            launch_pdl(k_bwdb_level<2>, g, blk, s, d.fanin, d.fout_ptr, (const int4 *)d.edge_fpos, b.pq, d.cload,
                       b.dcl, b.ks, b.gfo, c0, c1, d.n_start, S, ops);
        else
            launch_pdl(k_bwdb_level<1>, g, blk, s, d.fanin, d.fout_ptr, (const int4 *)d.edge_fpos, b.pq, d.cload,
                       b.dcl, b.ks, b.gfo, c0, c1, d.n_start, S, ops);
    }
    if (d.n_start && S % 4 == 0) {
        const BatchShape s4 = fit_shape(BatchShape{128, 1, 4}, S / 4);
        launch_pdl(k_bwdb_start4, bgrid(S / 4, s4, d.n_start), dim3((unsigned)s4.bx, (unsigned)s4.by), s, d.fout_ptr,
                   b.pq, d.cload, b.dcl, b.ks, b.gfo, b.gsp, d.n_start, S, tr_mode, b.state);
    } else if (d.n_start) {
        launch_pdl(k_bwdb_start, bgrid(S, sh1, d.n_start), dim3((unsigned)sh1.bx, (unsigned)sh1.by), s, d.fout_ptr,
                   b.pq, d.cload, b.dcl, b.ks, b.gfo, b.gsp, d.n_start, S, tr_mode, b.state);
    }
}

void launch_gradb(const DevDesign &d, const BatchBufs &b, const OpTable &ops, int tr_mode, bool reduce, float *gtr,
                  float *gpin, float *gcl, cudaStream_t s) {
    const int64_t S = b.S;
    if (reduce) {
        const int64_t rows = (gcl ? d.n_nets : 0) + (gpin ? d.n_cells : 0);
        if (rows) {
            const int64_t blocks = cdiv(rows, 8);
            k_gradb_reduce<<<(unsigned)(blocks < 152 * 16 ? blocks : 152 * 16), 256, 0, s>>>(
                d.fanin, b.pq, tr_mode == 2 ? b.tq : b.tr_in, d.net_of_user, d.cell_of_user, b.ks, gcl, gpin,
                d.n_nets, d.n_cells, d.n_start, S, tr_mode, ops);
        }
        gcl = gpin = nullptr;
    }
    const int64_t rows = (gcl ? d.n_nets : 0) + (gpin ? d.n_cells : 0) + (gtr ? d.n_start : 0);
    if (rows == 0) return;
    const BatchShape sh = fit_shape(BatchShape{S >= 128 ? 128 : 32, S >= 128 ? 1 : 4}, S);
    k_gradb_rows<<<bgrid(S, sh, rows), dim3((unsigned)sh.bx, (unsigned)sh.by), 0, s>>>(
        d.fanin, b.pq, tr_mode == 2 ? b.tq : b.tr_in, d.cload, b.dcl, d.net_of_user, d.cell_of_user, b.ks,
        b.gtr, gcl, gpin, gtr, d.n_nets, d.n_cells, d.n_start, S, tr_mode, ops);
}

void launch_netb_user(const DevDesign &d, const BatchBufs &b, int tr_mode, float *sp, float *tr, cudaStream_t s) {
    if (!d.n_nets || (!sp && !tr)) return;
    const BatchShape sh = fit_shape(BatchShape{b.S >= 128 ? 128 : 32, b.S >= 128 ? 1 : 4}, b.S);
    k_netb_user<<<bgrid(b.S, sh, d.n_nets), dim3((unsigned)sh.bx, (unsigned)sh.by), 0, s>>>(
        b.pq, tr_mode == 2 ? b.tq : b.tr_in, d.net_of_user, sp, tr, d.n_nets, d.n_start, b.S, tr_mode);
}

void launch_transpose(const float *in, float *out, int64_t R, int64_t C, cudaStream_t s) {
    if (R <= 0 || C <= 0) return;
    const int64_t gy = cdiv(R, 32);
    for (int64_t y0 = 0; y0 < gy; y0 += 65535) {   // grid.y limit: the rows go in slabs
        const int64_t rows = (gy - y0 < 65535 ? gy - y0 : 65535) * 32;
        const int64_t rr = R - y0 * 32 < rows ? R - y0 * 32 : rows;
        k_transpose<<<dim3((unsigned)cdiv(C, 32), (unsigned)cdiv(rr, 32)), dim3(32, 8), 0, s>>>(
            in + y0 * 32 * C, out + y0 * 32, rr, C, R);
    }
}

void launch_ascent(float *x, const float *g, int64_t n, float eta, cudaStream_t s) {
    if (n) k_ascent<<<(unsigned)cdiv(n, 256), 256, 0, s>>>(x, g, n, eta);
}

void launch_virus(const DevDesign &d, const OpTable &ops, const int32_t *lvl, const float *sp, int64_t S,
                  uint64_t *words, uint8_t *v0, double *partials, double *out, cudaStream_t s) {
    const int64_t W = cdiv(S, 64), W2 = 2 * W;
    if (d.n_start)
        k_virus_start<<<(unsigned)cdiv(d.n_start * W, 128), 128, 0, s>>>(sp, words, v0, d.n_start, S, W);
    for (int l = 1; l <= d.n_levels; l++) {
        const int64_t m = (int64_t)(lvl[l] - lvl[l - 1]) * W2;
        if (m)
            k_virus_level<<<(unsigned)cdiv(m, 256), 256, 0, s>>>(d.fanin, words, lvl[l - 1], lvl[l], d.n_start, W2,
                                                                 ops);
    }
    int64_t chunk = 0;
    const int nch = nchunks_of(d.n_nets, &chunk);
    k_virus_partials<<<dim3((unsigned)cdiv(S, 128), (unsigned)nch), 128, 0, s>>>(words, d.cload, partials, d.n_nets,
                                                                                S, W, chunk, nch);
    k_sumb_final<<<(unsigned)cdiv(S * 32, 256), 256, 0, s>>>(partials, nch, S, 1.0, out);
}

}  // namespace dp
