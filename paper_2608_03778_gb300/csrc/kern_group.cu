// Batched passes by scenario groups: one launch per pass.  Scenarios do not depend on each other,
// so a group of them (lanes x V consecutive ones) is walked through all levels by one thread-block
// cluster (1 to 16 blocks; 1: a single block), with the cluster's barrier between levels, and the
// groups never wait for each other.  The level launches (kern_batch.cu, kern_lag1.cu) spread every
// level of all scenarios over the whole grid instead and pay a launch and a drained grid per level.
//
// A block is lanes x rows threads: a thread takes V consecutive scenarios of one cell (loads of up
// to 32 bytes), the lanes of a row the group's scenarios, the rows of all blocks of the cluster
// consecutive cells of the level.  What other blocks write is read through L2; the static records of
// a level are loaded between the arrival at the barrier before it and the wait.
//
// Every (cell, scenario) is computed by the same code as in the level launches, so the results are
// bitwise the same in any shape.
#include <cooperative_groups.h>

#include "kern_cells.cuh"

namespace cg = cooperative_groups;

namespace dp {
namespace {

constexpr int kGroupThreads = 512;

// this thread's place: scenario, first cell of a level, distance to its next one
struct Place {
    int64_t s;
    int first, stride, C;
    __device__ __forceinline__ Place(int lanes, int V) {
        const cg::cluster_group cl = cg::this_cluster();
        C = (int)cl.num_blocks();
        const int rows = (int)blockDim.x / lanes, row = (int)threadIdx.x / lanes;
        s = ((int64_t)((int)blockIdx.x / C) * lanes + (int)threadIdx.x % lanes) * V;
        first = (int)cl.block_rank() * rows + row;
        stride = C * rows;
    }
    __device__ __forceinline__ void arrive() const {
        __syncwarp();
        if (C > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    }
    __device__ __forceinline__ void wait() const {
        __syncwarp();
        if (C > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        else __syncthreads();
    }
};

template <int V, bool LAG>
__global__ void __launch_bounds__(kGroupThreads) k_fwdb_group(const uint4 *__restrict__ fanin, float2 *pq, float *tq,
                                                             const float *__restrict__ sp_in,
                                                             const float *__restrict__ tr_in,
                                                             const int32_t *__restrict__ lvl, int L, int64_t ns,
                                                             int64_t S, int lanes, OpTable ops, uint32_t *state) {
    const Place at(lanes, V);
    if (blockIdx.x == 0 && threadIdx.x == 0) state[0] = 0u;   // no dataflow pass wrote these
    const bool on = at.s < S;
    pq += at.s;
    if (LAG) tq += at.s;
    if (on)
        for (int64_t k = at.first; k < ns; k += at.stride) {
            const Row1<V> a = ld1<V>(sp_in + k * S + at.s);
            Row2<V> o;
#pragma unroll
            for (int i = 0; i < V; i++) o.v[i] = make_float2(a.v[i], 0.f);
            st2<V>(pq + k * S, o);
            if (LAG) st1<V>(tq + k * S, ld1<V>(tr_in + k * S + at.s));
        }
    int32_t c1 = lvl[0];
    for (int l = 1; l <= L; l++) {
        int32_t c = c1 + at.first;
        c1 = lvl[l];
        at.arrive();
        uint4 r = on && c < c1 ? fanin[c] : make_uint4(0, 0, 0, 0);
        at.wait();
        if (!on) continue;
        while (c < c1) {
            const uint4 cur = r;
            float2 *const out = pq + (ns + c) * S;
            float *const out_t = LAG ? tq + (ns + c) * S : nullptr;
            c += at.stride;
            if (c < c1) r = fanin[c];
            const uint32_t op = cur.x >> 24;
            const uint32_t n[4] = {cur.x & kMask24, cur.y, cur.z, cur.w};
            const int k = (int)((ops.e[op] >> 16) & 7u);
            Row2<V> x[4], o;
            Row1<V> t[4], ot;
#pragma unroll
            for (int j = 0; j < 4; j++)
                if (j < k) {
                    x[j] = ld2<V>(pq + (int64_t)n[j] * S);
                    if (LAG) t[j] = ld1<V>(tq + (int64_t)n[j] * S);
                }
            cell_value<V, LAG>(
                ops.e[op], [&](int j, Row2<V> &xj, Row1<V> &tj) { xj = x[j], tj = t[j]; }, o, ot);
            st2<V>(out, o);
            if (LAG) st1<V>(out_t, ot);
        }
    }
}

template <int V, bool LAG>
__global__ void __launch_bounds__(kGroupThreads) k_bwdb_group(
    const uint4 *__restrict__ fanin, const int32_t *__restrict__ fptr, const int4 *__restrict__ efpos,
    const float2 *pq, const float *tq, const float *__restrict__ cload, const float *__restrict__ dcl,
    const float *__restrict__ ks, float *gfo, float2 *gfo2, float *gsp, float *gtr, const int32_t *__restrict__ lvl,
    int L, int64_t ns, int64_t S, int lanes, int tr_mode, OpTable ops, uint32_t *state) {
    const Place at(lanes, V);
    if (blockIdx.x == 0 && threadIdx.x == 0) state[LAG ? 5 : 2] = 0u;   // the edges will hold values
    const bool on = at.s < S;
    pq += at.s;
    gsp += at.s;
    if (dcl) dcl += at.s;
    if (LAG) tq += at.s, gfo2 += at.s, gtr += at.s;
    else gfo += at.s;
    Row1<V> Ks;
#pragma unroll
    for (int i = 0; i < V; i++) Ks.v[i] = on ? ks[at.s + i] : 0.f;
    auto load_of = [&](int64_t n) {
        Row1<V> c;
#pragma unroll
        for (int i = 0; i < V; i++) c.v[i] = dcl ? cload[n] + dcl[n * S + i] : cload[n];
        return c;
    };
    for (int l = L; l >= 1; l--) {
        const int32_t c0 = lvl[l - 1], c1 = lvl[l];
        int32_t c = c0 + at.first;
        if (l < L) at.arrive();
        uint4 r = make_uint4(0, 0, 0, 0);
        int4 ep = make_int4(0, 0, 0, 0);
        int32_t e0 = 0, e1 = 0;
        auto record = [&] {
            if (!on || c >= c1) return;
            r = fanin[c];
            ep = efpos[c];
            e0 = fptr[ns + c];
            e1 = fptr[ns + c + 1];
        };
        record();
        if (l < L) at.wait();
        if (!on) continue;
        while (c < c1) {
            const uint4 cur = r;
            const int4 pos4 = ep;
            const int32_t f0 = e0, f1 = e1;
            const int64_t n = ns + c;
            c += at.stride;
            record();
            const uint32_t op = cur.x >> 24;
            const uint32_t nid[4] = {cur.x & kMask24, cur.y, cur.z, cur.w};
            const int pos[4] = {pos4.x, pos4.y, pos4.z, pos4.w};
            const int k = (int)((ops.e[op] >> 16) & 7u);
            Row2<V> x[4], self;
            Row1<V> t[4], a, b;
#pragma unroll
            for (int j = 0; j < 4; j++)
                if (j < k) {
                    x[j] = ld2<V>(pq + (int64_t)nid[j] * S);
                    if (LAG) t[j] = ld1<V>(tq + (int64_t)nid[j] * S);
                }
            if (!LAG) self = ld2<V>(pq + n * S);
            const Row1<V> cl = load_of(n);
            fanout_sum<V, LAG>(gfo, gfo2, f0, f1, (uint32_t)S, a, b);
            Row1<V> g[4];
            Row2<V> g2[4];
            cell_adjoints<V, LAG>(ops.e[op], x, t, self, Ks, cl, a, b, g, g2);
#pragma unroll
            for (int j = 0; j < 4; j++)
                if (j < k) {
                    if constexpr (LAG) st2<V>(gfo2 + (int64_t)pos[j] * S, g2[j]);
                    else st1<V>(gfo + (int64_t)pos[j] * S, g[j]);
                }
        }
    }
    at.arrive();
    at.wait();
    if (!on) return;
    for (int64_t k = at.first; k < ns; k += at.stride) {
        Row1<V> a, b;
        fanout_sum<V, LAG>(gfo, gfo2, fptr[k], fptr[k + 1], (uint32_t)S, a, b);
        if (LAG || tr_mode) {
            const Row1<V> cl = load_of(k);
            Row2<V> self;
            if (!LAG) self = ld2<V>(pq + k * S);
#pragma unroll
            for (int i = 0; i < V; i++) {
                if constexpr (LAG) b.v[i] = fmaf(Ks.v[i], cl.v[i], b.v[i]);
                else a.v[i] = bwdb_adjoint(a.v[i], Ks.v[i], cl.v[i], self.v[i]);
            }
        }
        st1<V>(gsp + k * S, a);
        if (LAG) st1<V>(gtr + k * S, b);
    }
}

template <class... KArgs, class... Args>
cudaError_t launch_group(void (*kern)(KArgs...), GroupShape sh, int64_t S, cudaStream_t s, Args... args) {
    if (!group_ok(sh) || S % sh.v != 0) return cudaErrorInvalidConfiguration;
    cudaError_t e = cudaSuccess;
    if (sh.blocks > 8) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    const int64_t per = (int64_t)sh.lanes * sh.v;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((S + per - 1) / per * sh.blocks));
    cfg.blockDim = dim3((unsigned)sh.threads);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)sh.blocks;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}

template <class K>
bool fits(K kern, int blocks) {
    if (blocks > 8 && cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return false;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3((unsigned)kGroupThreads);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)blocks;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    return cudaOccupancyMaxActiveClusters(&n, kern, &cfg) == cudaSuccess && n > 0;
}

}  // namespace

bool group_fits(int blocks) {
    const bool ok = fits(k_fwdb_group<1, false>, blocks) && fits(k_fwdb_group<2, false>, blocks) &&
                    fits(k_fwdb_group<1, true>, blocks) && fits(k_fwdb_group<2, true>, blocks) &&
                    fits(k_bwdb_group<1, false>, blocks) && fits(k_bwdb_group<2, false>, blocks) &&
                    fits(k_bwdb_group<1, true>, blocks) && fits(k_bwdb_group<2, true>, blocks);
    cudaGetLastError();
    return ok;
}

cudaError_t launch_fwdb_group(const DevDesign &d, const BatchBufs &b, const OpTable &ops, int tr_mode, GroupShape sh,
                              cudaStream_t s) {
    sh = group_for(sh, tr_mode);
    auto go = [&](auto kern) {
        return launch_group(kern, sh, b.S, s, d.fanin, b.pq, b.tq, b.sp_in, b.tr_in, d.lvl, d.n_levels, d.n_start, b.S,
                            sh.lanes, ops, b.state);
    };
    if (tr_mode == 2) return sh.v >= 2 ? go(k_fwdb_group<2, true>) : go(k_fwdb_group<1, true>);
    return sh.v == 4 ? go(k_fwdb_group<4, false>) : sh.v == 2 ? go(k_fwdb_group<2, false>) : go(k_fwdb_group<1, false>);
}

cudaError_t launch_bwdb_group(const DevDesign &d, const BatchBufs &b, const OpTable &ops, int tr_mode, GroupShape sh,
                              cudaStream_t s) {
    sh = group_for(sh, tr_mode);
    auto go = [&](auto kern) {
        return launch_group(kern, sh, b.S, s, d.fanin, d.fout_ptr, (const int4 *)d.edge_fpos, b.pq, b.tq, d.cload, b.dcl,
                            b.ks, b.gfo, b.gfo2, b.gsp, b.gtr, d.lvl, d.n_levels, d.n_start, b.S, sh.lanes, tr_mode,
                            ops, b.state);
    };
    if (tr_mode == 2) return sh.v >= 2 ? go(k_bwdb_group<2, true>) : go(k_bwdb_group<1, true>);
    return sh.v == 4 ? go(k_bwdb_group<4, false>) : sh.v == 2 ? go(k_bwdb_group<2, false>) : go(k_bwdb_group<1, false>);
}

}  // namespace dp
