// Forward and reverse passes of a mid-size design in one thread-block cluster.
//
// A design too large for one block's shared memory but whose per-block share fits (up to
// about 130,000 nets on a 16-block cluster) runs each pass on one cluster of kClusterBlocks
// blocks.  Every level (the startpoints are level 0) is cut into C contiguous chunks, block b
// taking chunk b: consecutive cells of a level share their function (levels are sorted by logic
// id), so a warp's cells mostly take the same branch.  A net lives in the shared memory of the
// block that computes it, at a slot that the host assigns level by level (loc = block << 24 |
// slot): its (P, Q) pair in the forward pass, the edge adjoints of its fanout range in the
// reverse pass.
//
// There is no barrier between levels: a value is its own ready flag.  Forward: a cell polls its
// fanins' pairs in their owners' shared memory (distributed shared memory) until both halves
// carry the ready tag in their sign bits.  Reverse: a cell's contributions are stored straight
// into the owners of its fanin nets, and a net polls its own block's shared memory until none of
// its edges holds the sentinel (a NaN pattern that no arithmetic produces).  What bounds a level
// is then one hop between two blocks of the cluster plus the cell's arithmetic; with the hardware
// cluster barrier between levels it was the barrier (450 to 930 cycles) and a burst of gathers on
// top.  Against the dataflow passes over the whole grid (kern_flow.cu) a hop costs 200 to 300
// cycles instead of 500 (both blocks and the line on one die) to 1,000 (otherwise).  Forward pass
// with the model power and whole reverse pass, cluster barrier -> this: 13,000 cells / 70 levels
// 99 -> 77 and 117 -> 58 us (over the whole grid 85 and 82), 120,000 / 48 98 -> 72 and 98 -> 51 us
// (over the whole grid 68 and 68).
//
// Progress: every warp takes the levels in order and a cell waits for lower levels only
// (reverse: higher), and the blocks of a cluster are resident together.  Every wait is bounded by
// a clock limit; all blocks meet at a final cluster barrier, so none leaves while another may
// still read or write its shared memory.
//
// Each value is computed by the same code in the same order as in the grid-wide passes (a
// net's fanout range keeps its order in its owner's copy), so the results are bitwise the same.
#include <cooperative_groups.h>

#include "kern_common.cuh"

namespace cg = cooperative_groups;

namespace dp {
namespace {

constexpr uint32_t kSlotMask = 0xFFFFFFu;

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// block r of C prefetches its share of the 128-byte lines of bytes [p, p + n) into L2
__device__ __forceinline__ void prefetch_share_l2(const void *p, int64_t n, int r, int C) {
    const char *c = static_cast<const char *>(p);
    for (int64_t i = ((int64_t)r * blockDim.x + threadIdx.x) * 128; i < n; i += (int64_t)C * blockDim.x * 128)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(c + i));
}

__device__ __forceinline__ int ld_err(const int *err) {
    int v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(err) : "memory");
    return v;
}
// true when a wait that began at t0 has to give up (looked at every 256th spin); waits are loops
// of the whole warp, as in kern_flow.cu
__device__ __forceinline__ bool gives_up(unsigned &spins, long long t0, int *err, long long limit) {
    if ((++spins & 255u) != 0) return false;
    if (ld_err(err) != 0) return true;
    if (clock64() - t0 <= limit) return false;
    atomicExch(err, 1);
    return true;
}

// the address of this block's shared location `local` in block `rank` of the cluster
__device__ __forceinline__ uint32_t dsm_addr(uint32_t local, uint32_t rank) {
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(local), "r"(rank));
    return a;
}
__device__ __forceinline__ void dsm_ld_pair(uint32_t a, unsigned long long &h0, unsigned long long &h1) {
    asm volatile("ld.relaxed.cluster.shared::cluster.v2.u64 {%0, %1}, [%2];" : "=l"(h0), "=l"(h1) : "r"(a) : "memory");
}
// a pair with the ready tag, as two single-copy-atomic halves, into this block's shared memory
__device__ __forceinline__ void sh_put_pair(uint32_t a, const pair_ff &v) {
    const float4 t = pair_store(v, 1u);
    const unsigned long long h0 = (unsigned long long)__float_as_uint(t.x) | ((unsigned long long)__float_as_uint(t.y) << 32);
    const unsigned long long h1 = (unsigned long long)__float_as_uint(t.z) | ((unsigned long long)__float_as_uint(t.w) << 32);
    asm volatile("st.relaxed.cluster.shared::cta.v2.u64 [%0], {%1, %2};" ::"r"(a), "l"(h0), "l"(h1) : "memory");
}
__device__ __forceinline__ uint32_t sh_ld(uint32_t a) {
    uint32_t v;
    asm volatile("ld.relaxed.cluster.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void dsm_st(uint32_t a, float v) {
    asm volatile("st.relaxed.cluster.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
constexpr uint32_t kNotYet = 0xFFFFDEADu;   // an edge adjoint that has not arrived

// the block's tables in shared memory: level bounds (cells), chunk length per level, and the
// first slot of the block's chunk of each level
struct Tables {
    int *lvl, *chunk, *base;
};
__device__ __forceinline__ void load_tables(const Tables &s, const int32_t *lvl, const int32_t *chunk,
                                            const int32_t *base, int L, int r) {
    for (int i = threadIdx.x; i <= L; i += blockDim.x) {
        s.lvl[i] = lvl[i];
        s.chunk[i] = chunk[i];
        s.base[i] = base[(int64_t)r * (L + 1) + i];
    }
}

// this thread's cell on level l >= 1 (if any): its internal cell index and own slot
__device__ __forceinline__ bool cell_at(const Tables &s, int l, int L, int r, int t, int64_t &c, int &slot) {
    if (l < 1 || l > L) return false;
    const int chunk = s.chunk[l];
    c = s.lvl[l - 1] + (int64_t)r * chunk + t;
    slot = s.base[l] + t;
    return t < chunk && c < s.lvl[l];
}

// Shared memory: the block's slots of (P, Q) pairs, then its tables.
__global__ void __launch_bounds__(kClusterMaxThreads) k_fwd_cluster(
    const uint4 *__restrict__ fanin, const uint4 *__restrict__ floc, float4 *pq, float *tr,
    const float *__restrict__ sp_in, const float *__restrict__ tr_in, const int32_t *__restrict__ lvl,
    const int32_t *__restrict__ chunk, const int32_t *__restrict__ base, int L, int64_t ns, int64_t nn,
    int64_t slots, int tr_mode, OpTable ops, uint32_t *epoch, int *err, long long limit) {
    extern __shared__ float4 spq[];
    const cg::cluster_group cl = cg::this_cluster();
    const int C = (int)cl.num_blocks(), rk = (int)cl.block_rank();
    int *tab = reinterpret_cast<int *>(spq + slots);
    const Tables s{tab, tab + (L + 1), tab + 2 * (L + 1)};
    const int t = threadIdx.x, B = blockDim.x;
    const uint32_t spq0 = (uint32_t)__cvta_generic_to_shared(spq);
    const uint32_t pass = *reinterpret_cast<volatile uint32_t *>(epoch) + 1u, par = pass & 1u;   // before the barrier
    prefetch_share_l2(fanin, (nn - ns) * (int64_t)sizeof(uint4), rk, C);
    prefetch_share_l2(floc, (nn - ns) * (int64_t)sizeof(uint4), rk, C);
    load_tables(s, lvl, chunk, base, L, rk);
    for (int64_t i = t; i < slots; i += B) spq[i] = make_float4(0.f, 0.f, 0.f, 0.f);   // no ready tag
    __syncthreads();
    cluster_arrive();
    // this thread's cells, two levels ahead: record and fanin locations
    int64_t c = 0, c1 = 0;
    int slot = 0, slot1 = 0;
    uint4 r = make_uint4(0, 0, 0, 0), f = r, r1 = r, f1 = r;
    bool on = cell_at(s, 1, L, rk, t, c, slot), on1 = cell_at(s, 2, L, rk, t, c1, slot1);
    if (on) r = fanin[c], f = floc[c];
    if (on1) r1 = fanin[c1], f1 = floc[c1];
    cluster_wait();   // every block's slots are clear
    for (int p = t; p < s.chunk[0]; p += B) {   // the block's startpoints
        const int64_t n = (int64_t)rk * s.chunk[0] + p;
        if (n >= ns) break;
        const pair_ff a = pair_of(sp_in[n]);
        sh_put_pair(spq0 + 16u * (uint32_t)(s.base[0] + p), a);
        pq[n] = pair_store(a, par);
        tr[n] = tr_mode ? pair_tr(a) : tr_in[n];
    }
    __syncwarp();
    bool ok = true;
    for (int l = 1; l <= L; l++) {
        if (__any_sync(0xFFFFFFFFu, on)) {
            const uint32_t op = r.x >> 24;
            const int k = on ? op_arity(ops, op) : 0;
            const uint32_t fl[4] = {f.x, f.y, f.z, f.w};
            uint32_t at[4];
            unsigned long long h0[4], h1[4];
#pragma unroll
            for (int j = 0; j < 4; j++) {
                at[j] = dsm_addr(spq0 + 16u * (fl[j] & kSlotMask), j < k ? fl[j] >> 24 : 0u);
                h0[j] = 0x80000000ull;
                h1[j] = 0xBF800000ull;   // an unused slot: P = 0, Q = 1
                if (j < k) dsm_ld_pair(at[j], h0[j], h1[j]);
            }
            auto late = [&](int j) { return (~(uint32_t)h0[j] | ~(uint32_t)h1[j]) & 0x80000000u; };
            if (__any_sync(0xFFFFFFFFu, (late(0) | late(1) | late(2) | late(3)) != 0)) {
                const long long t0 = clock64();
                unsigned spins = 0;
                do {
#pragma unroll
                    for (int j = 0; j < 4; j++)
                        if (late(j)) dsm_ld_pair(at[j], h0[j], h1[j]);
                    if (gives_up(spins, t0, err, limit)) ok = false;
                } while (__any_sync(0xFFFFFFFFu, (late(0) | late(1) | late(2) | late(3)) != 0) &&
                         __all_sync(0xFFFFFFFFu, ok));
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
            }
            if (on) {
                pair_ff x[4];
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    x[j].p = ff{__uint_as_float((uint32_t)h0[j] & 0x7FFFFFFFu), __uint_as_float((uint32_t)(h0[j] >> 32))};
                    x[j].q = ff{__uint_as_float((uint32_t)h1[j] & 0x7FFFFFFFu), __uint_as_float((uint32_t)(h1[j] >> 32))};
                }
                const pair_ff o = cell_pair(k, op_tt(ops, op), x);
                sh_put_pair(spq0 + 16u * (uint32_t)slot, o);
                pq[ns + c] = pair_store(o, par);
                tr[ns + c] = pair_tr(o);
            }
            __syncwarp();
        }
        c = c1, slot = slot1, r = r1, f = f1, on = on1;   // the next level's cell; the one after it now
        on1 = cell_at(s, l + 2, L, rk, t, c1, slot1);
        if (on1) r1 = fanin[c1], f1 = floc[c1];
    }
    if (!ok) epoch[3] = 1u;   // pairs of two parities: the power pass puts the tags right
    cluster_arrive();
    cluster_wait();   // nothing remote after this
    if (rk == 0 && t == 0) epoch[0] = pass;
}

// the static data of one cell for the reverse pass
struct ClPre {
    int4 push;    // its input edges' places: owner block << 24 | position in its copy, -1 unused
    float4 d;     // their partial derivatives
    int2 range;   // its own fanout edges in this block's copy: first, count
    float local, b;
};
__device__ __forceinline__ void cl_pre(ClPre &w, const int4 *push, const float4 *coef, const int2 *range,
                                       const float *gnet, const float *beta, int64_t c, int64_t ns, int grad_mode) {
    w.push = push[c];
    w.d = coef[c];
    w.range = range[ns + c];
    w.local = gnet[ns + c];
    w.b = grad_mode ? beta[ns + c] : 1.f;
}

// The sum of edges [first, first + cnt) of this block's copy in index order, once all have
// arrived; false, in every lane, when the wait gave up.
__device__ __forceinline__ bool cl_sum(uint32_t sgfo0, int first, int cnt, int *err, long long limit, float &acc) {
    acc = 0.f;
    bool ok = true;
    for (int i = 0; __any_sync(0xFFFFFFFFu, i < cnt); i += 4) {
        uint32_t v[4];
#pragma unroll
        for (int j = 0; j < 4; j++) v[j] = i + j < cnt ? sh_ld(sgfo0 + 4u * (uint32_t)(first + i + j)) : 0u;
        auto late = [&] { return v[0] == kNotYet || v[1] == kNotYet || v[2] == kNotYet || v[3] == kNotYet; };
        if (__any_sync(0xFFFFFFFFu, late())) {
            const long long t0 = clock64();
            unsigned spins = 0;
            do {
#pragma unroll
                for (int j = 0; j < 4; j++)
                    if (v[j] == kNotYet) v[j] = sh_ld(sgfo0 + 4u * (uint32_t)(first + i + j));
                if (gives_up(spins, t0, err, limit)) ok = false;
            } while (__any_sync(0xFFFFFFFFu, late()) && __all_sync(0xFFFFFFFFu, ok));
            if (!__all_sync(0xFFFFFFFFu, ok)) return false;
        }
#pragma unroll
        for (int j = 0; j < 4; j++)
            if (i + j < cnt) acc += __uint_as_float(v[j]);
    }
    return true;
}

// The partial derivatives (coef) and local terms (in gnet) come from k_bwd_coef.  Shared memory:
// the edge adjoints of the block's nets, then its tables.
__global__ void __launch_bounds__(kClusterMaxThreads) k_bwd_cluster(
    const int4 *__restrict__ push, const float4 *__restrict__ coef, const int2 *__restrict__ range,
    const float *__restrict__ beta, float *gnet, const int32_t *__restrict__ lvl, const int32_t *__restrict__ chunk,
    const int32_t *__restrict__ base, int L, int64_t ns, int64_t nn, int64_t ne_local, int grad_mode, float *out_gsp,
    int *err, long long limit) {
    extern __shared__ uint32_t sgfo[];
    const cg::cluster_group cl = cg::this_cluster();
    const int C = (int)cl.num_blocks(), rk = (int)cl.block_rank();
    int *tab = reinterpret_cast<int *>(sgfo + ne_local);
    const Tables s{tab, tab + (L + 1), tab + 2 * (L + 1)};
    const int t = threadIdx.x, B = blockDim.x;
    const int64_t nc = nn - ns;
    const uint32_t sgfo0 = (uint32_t)__cvta_generic_to_shared(sgfo);
    prefetch_share_l2(push, nc * (int64_t)sizeof(int4), rk, C);
    prefetch_share_l2(range, nn * (int64_t)sizeof(int2), rk, C);
    if (grad_mode) prefetch_share_l2(beta, nn * (int64_t)sizeof(float), rk, C);
    load_tables(s, lvl, chunk, base, L, rk);
    for (int64_t i = t; i < ne_local; i += B) sgfo[i] = kNotYet;
    __syncthreads();
    cluster_arrive();
    // this thread's cells, three levels ahead (a level takes less than a load from L2)
    int64_t c[3];
    bool on[3];
    ClPre w[3];
    auto load = [&](int i, int l) {
        int slot;
        on[i] = cell_at(s, l, L, rk, t, c[i], slot);
        w[i].range = make_int2(0, 0);
        if (on[i]) cl_pre(w[i], push, coef, range, gnet, beta, c[i], ns, grad_mode);
    };
#pragma unroll
    for (int i = 0; i < 3; i++) load(i, L - i);
    cluster_wait();   // every block's edges are clear
    bool ok = true;
    for (int l = L; l >= 1 && ok; l -= 3) {
#pragma unroll
        for (int i = 0; i < 3; i++) {
            if (l - i < 1 || !ok) break;
            if (__any_sync(0xFFFFFFFFu, on[i])) {
                float acc;
                ok = cl_sum(sgfo0, w[i].range.x, w[i].range.y, err, limit, acc);
                if (!ok) break;
                if (on[i]) {
                    const float g = adj_combine(grad_mode, acc, w[i].local, w[i].b);
                    const int at[4] = {w[i].push.x, w[i].push.y, w[i].push.z, w[i].push.w};
                    const float d[4] = {w[i].d.x, w[i].d.y, w[i].d.z, w[i].d.w};
#pragma unroll
                    for (int j = 0; j < 4; j++)
                        if (at[j] >= 0)
                            dsm_st(dsm_addr(sgfo0 + 4u * ((uint32_t)at[j] & kSlotMask), (uint32_t)at[j] >> 24),
                                   __fmul_rn(g, d[j]));
                    gnet[ns + c[i]] = g;
                }
                __syncwarp();
            }
            load(i, l - i - 3);
        }
    }
    for (int p = t; p - (t & 31) < s.chunk[0] && ok; p += B) {   // the block's startpoints
        const int64_t n = (int64_t)rk * s.chunk[0] + p;
        const bool mine = p < s.chunk[0] && n < ns;
        const int2 rg = mine ? range[n] : make_int2(0, 0);
        float acc;
        ok = cl_sum(sgfo0, rg.x, rg.y, err, limit, acc);
        if (!ok) break;
        if (mine) {
            const float g = adj_combine(grad_mode, acc, gnet[n], grad_mode ? beta[n] : 1.f);
            gnet[n] = g;
            if (out_gsp) out_gsp[n] = g;
        }
        __syncwarp();
    }
    cluster_arrive();
    cluster_wait();   // nothing remote after this
}

template <class... KArgs, class... Args>
cudaError_t launch_cluster(void (*kern)(KArgs...), int threads, size_t smem, cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)kClusterBlocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)kClusterBlocks;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}

}  // namespace

size_t cluster_smem(int which, int64_t slots, int64_t n_edges_local, int n_levels) {
    const size_t tables = 3 * (size_t)(n_levels + 1) * sizeof(int);
    if (which == 0) return (size_t)slots * sizeof(float4) + tables;
    if (which == 1) return (size_t)n_edges_local * sizeof(float) + tables;
    return (size_t)slots * sizeof(float4) + (size_t)n_edges_local * sizeof(float) + tables;   // both, in one block
}

bool cluster_fits(int threads, size_t smem_fwd, size_t smem_bwd) {
    const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
    if (cudaFuncSetAttribute(k_fwd_cluster, a, kBlockSmemMax) != cudaSuccess ||
        cudaFuncSetAttribute(k_bwd_cluster, a, kBlockSmemMax) != cudaSuccess ||
        cudaFuncSetAttribute(k_fwd_cluster, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaFuncSetAttribute(k_bwd_cluster, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    for (int w = 0; w < 2; w++) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)kClusterBlocks);
        cfg.blockDim = dim3((unsigned)threads);
        cfg.dynamicSmemBytes = w ? smem_bwd : smem_fwd;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = (unsigned)kClusterBlocks;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int n = 0;
        const cudaError_t e = w ? cudaOccupancyMaxActiveClusters(&n, k_bwd_cluster, &cfg)
                                : cudaOccupancyMaxActiveClusters(&n, k_fwd_cluster, &cfg);
        if (e != cudaSuccess || n < 1) {
            cudaGetLastError();
            return false;
        }
    }
    return true;
}

cudaError_t launch_fwd_cluster(const DevDesign &d, const OpTable &ops, const ClusterMap &m, int tr_mode,
                               cudaStream_t s) {
    return launch_cluster(k_fwd_cluster, m.threads, cluster_smem(0, m.slots, 0, d.n_levels), s, d.fanin,
                          (const uint4 *)m.floc, d.pq, d.tr, (const float *)d.sp_in, (const float *)d.tr_in, d.lvl,
                          (const int32_t *)m.chunk, (const int32_t *)m.base, d.n_levels, d.n_start, d.n_nets,
                          m.slots, tr_mode, ops, d.epoch, d.err, kWaitLimitCycles);
}

cudaError_t launch_bwd_cluster(const DevDesign &d, const ClusterMap &m, int grad_mode, float *out_gsp,
                               cudaStream_t s) {
    return launch_cluster(k_bwd_cluster, m.threads, cluster_smem(1, 0, m.edges, d.n_levels), s,
                          (const int4 *)m.push, (const float4 *)m.coef, (const int2 *)m.range, (const float *)d.beta,
                          d.gnet, d.lvl, (const int32_t *)m.chunk, (const int32_t *)m.base, d.n_levels, d.n_start,
                          d.n_nets, m.edges, grad_mode, out_gsp, d.err, kWaitLimitCycles);
}

}  // namespace dp
