// Lag-one mode of the batched path (tr_mode 2): every net carries SP and
// T = P(x_t != x_{t+1}) of a stationary two-state process, so two consecutive
// values follow q(a, b) with q(1,1) = P - T/2, q(0,0) = P(net=0) - T/2,
// q(0,1) = q(1,0) = T/2.  Under spatial independence a cell's output toggles
// with probability
//     T_y = sum over input pairs (a, b) of prod_i q_i(a_i, b_i) [f(a) != f(b)],
// its exact toggle probability on fanout-free circuits (an extension of Eq. 2,
// which it equals when every startpoint has T = 2P(1-P)).  SP is the
// multilinear pair of the other modes.  The power is K sum_n T_n C_n (Eq. 1).
//
// T_y is a fold over the 4^k joint input states, input 0 innermost: leaf m
// (digit i of m in base 4 = 2 a_i + b_i) holds [f(a) != f(b)], and each input
// folds four sub-results with its weights q_i.  Its derivatives are the same
// fold with one input's weights replaced by dq/dP = (-1, 0, 0, 1) or
// dq/dT = (-1/2, 1/2, 1/2, -1/2).  The reverse pass carries two adjoints per
// net (of P and of T); edge contributions are float2 in fanout-CSR order, so a
// net sums one contiguous range, without atomics, as in the other modes.
#include "kern_cells.cuh"

namespace dp {
namespace {

__global__ void k_fwdl_start(const float *__restrict__ sp_in, const float *__restrict__ tr_in, float2 *pq, float *tq,
                             int64_t n, uint32_t *state) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) state[0] = 0u;   // no dataflow pass wrote these
    if (i >= n) return;
    pq[i] = make_float2(sp_in[i], 0.f);
    tq[i] = tr_in[i];
}

__global__ void k_fwdl_level(const uint4 *__restrict__ fanin, float2 *pq, float *tq, int32_t c0, int32_t c1,
                             int64_t ns, int64_t S, OpTable ops) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    pdl_trigger();
    if (s >= S) return;
    const int64_t step = (int64_t)gridDim.y * blockDim.y;
    const int64_t cf = c0 + (int64_t)blockIdx.y * blockDim.y + threadIdx.y;
    const uint4 rf = cf < c1 ? fanin[cf] : make_uint4(0, 0, 0, 0);   // static: before the wait
    pdl_wait();
    for (int64_t c = cf; c < c1; c += step) {
        const uint4 r = c == cf ? rf : fanin[c];
        const uint32_t op = r.x >> 24;
        const uint32_t n[4] = {r.x & kMask24, r.y, r.z, r.w};
        with_cell(ops.e[op], [&](const auto f) {
            constexpr int K = decltype(f)::k;
            pair_ff x[4];
            float w[4][4];
#pragma unroll
            for (int j = 0; j < K; j++) {
                x[j] = pair_get(pq[(int64_t)n[j] * S + s]);
                lag1_weights(x[j], tq[(int64_t)n[j] * S + s], w[j]);
            }
            const ff p = f.prob(x);
            pq[(ns + c) * S + s] = make_float2(p.hi, p.lo);
            tq[(ns + c) * S + s] = f.toggle(w);
        });
    }
}

// reverse level: the net's adjoints (gP from its fanout range, gT from its range
// plus the direct term K_s C), then per input edge the contributions
// (gP dP/dP_j + gT dT/dP_j, gT dT/dT_j)
__global__ void k_bwdl_level(const uint4 *__restrict__ fanin, const int32_t *__restrict__ fptr,
                             const int4 *__restrict__ efpos, const float2 *__restrict__ pq,
                             const float *__restrict__ tq, const float *__restrict__ cload,
                             const float *__restrict__ dcl, const float *__restrict__ ks, float2 *gfo2, int32_t c0,
                             int32_t c1, int64_t ns, int64_t S, OpTable ops) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    pdl_trigger();
    if (s >= S) return;
    pdl_wait();
    const float Ks = ks[s];
    const int64_t step = (int64_t)gridDim.y * blockDim.y;
    for (int64_t c = c0 + (int64_t)blockIdx.y * blockDim.y + threadIdx.y; c < c1; c += step) {
        const int64_t n = ns + c;
        float gp = 0.f, gt = 0.f;
        for (int32_t e = fptr[n]; e < fptr[n + 1]; e++) {
            const float2 g = gfo2[(int64_t)e * S + s];
            gp += g.x;
            gt += g.y;
        }
        gt = fmaf(Ks, cl_of(cload, dcl, n, S, s), gt);
        const uint4 r = fanin[c];
        const uint32_t op = r.x >> 24;
        const uint32_t nid[4] = {r.x & kMask24, r.y, r.z, r.w};
        const int4 ep = efpos[c];
        const int pos[4] = {ep.x, ep.y, ep.z, ep.w};
        with_cell(ops.e[op], [&](const auto f) {
            constexpr int K = decltype(f)::k;
            float w[4][4], p[4], q[4], d[4], dp[4], dt[4];
#pragma unroll
            for (int j = 0; j < K; j++) {
                const pair_ff v = pair_get(pq[(int64_t)nid[j] * S + s]);
                lag1_weights(v, tq[(int64_t)nid[j] * S + s], w[j]);
                p[j] = v.p.hi + v.p.lo;
                q[j] = v.q.hi + v.q.lo;
            }
            f.partials(p, q, d);
            f.toggle_partials(w, dp, dt);
#pragma unroll
            for (int j = 0; j < K; j++)
                gfo2[(int64_t)pos[j] * S + s] = make_float2(fmaf(gp, d[j], __fmul_rn(gt, dp[j])), __fmul_rn(gt, dt[j]));
        });
    }
}

__global__ void k_bwdl_start(const int32_t *__restrict__ fptr, const float *__restrict__ cload,
                             const float *__restrict__ dcl, const float *__restrict__ ks,
                             const float2 *__restrict__ gfo2, float *gsp, float *gtr, int64_t ns, int64_t S,
                             uint32_t *state) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    pdl_trigger();
    if (s >= S) return;
    pdl_wait();
    if (s == 0 && blockIdx.y == 0 && threadIdx.y == 0) state[5] = 0u;   // gfo2 holds values
    const float Ks = ks[s];
    const int64_t step = (int64_t)gridDim.y * blockDim.y;
    for (int64_t k = (int64_t)blockIdx.y * blockDim.y + threadIdx.y; k < ns; k += step) {
        float gp = 0.f, gt = 0.f;
        for (int32_t e = fptr[k]; e < fptr[k + 1]; e++) {
            const float2 g = gfo2[(int64_t)e * S + s];
            gp += g.x;
            gt += g.y;
        }
        gsp[k * S + s] = gp;
        gtr[k * S + s] = fmaf(Ks, cl_of(cload, dcl, k, S, s), gt);
    }
}

}  // namespace

void launch_fwdl(const DevDesign &d, const BatchBufs &b, const OpTable &ops, const int32_t *lvl, BatchShape sh,
                 cudaStream_t s) {
    const int64_t S = b.S;
    if (d.n_start)
        k_fwdl_start<<<(unsigned)bcdiv(d.n_start * S, 256), 256, 0, s>>>(b.sp_in, b.tr_in, b.pq, b.tq, d.n_start * S, b.state);
    sh = fit_shape(sh, S);
    const dim3 blk((unsigned)sh.bx, (unsigned)sh.by);
    for (int l = 1; l <= d.n_levels; l++) {
        const int32_t c0 = lvl[l - 1], c1 = lvl[l];
        if (c1 > c0)
            launch_pdl(k_fwdl_level, bgrid(S, sh, c1 - c0), blk, s, d.fanin, b.pq, b.tq, c0, c1, d.n_start, S, ops);
    }
}

void launch_bwdl(const DevDesign &d, const BatchBufs &b, const OpTable &ops, const int32_t *lvl, BatchShape sh,
                 cudaStream_t s) {
    const int64_t S = b.S;
    sh = fit_shape(sh, S);
    const dim3 blk((unsigned)sh.bx, (unsigned)sh.by);
    for (int l = d.n_levels; l >= 1; l--) {
        const int32_t c0 = lvl[l - 1], c1 = lvl[l];
        if (c1 > c0)
            launch_pdl(k_bwdl_level, bgrid(S, sh, c1 - c0), blk, s, d.fanin, d.fout_ptr, (const int4 *)d.edge_fpos,
                       b.pq, b.tq, d.cload, b.dcl, b.ks, b.gfo2, c0, c1, d.n_start, S, ops);
    }
    if (d.n_start)
        launch_pdl(k_bwdl_start, bgrid(S, sh, d.n_start), blk, s, d.fout_ptr, d.cload, b.dcl, b.ks, b.gfo2, b.gsp,
                   b.gtr, d.n_start, S, b.state);
}

}  // namespace dp
