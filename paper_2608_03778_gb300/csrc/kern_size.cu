// Gradient-weighted sizing score (Eq. 8) and its top-k ranking.
//
// For cell line u with output net y:  S_u = |dP/dP_sw| * P_sw,
//   P_sw = K * alpha_y * C_load,y   (alpha: TR_model, or the hybrid TR after a hybrid reverse pass)
//   mode 0: dP/dP_sw read as the SP adjoint of y (the global sensitivity the reverse pass leaves);
//   mode 1: the chain rule through Eq. 2, adjoint / (2 - 4 SP_y), |2 - 4 SP_y| floored at 1e-6.
// Scores are non-negative floats, so their bit patterns order like unsigned
// integers: the k-th largest is found by a radix select over 8-bit digits,
// most significant first (integer histograms, so the counts and the threshold
// are exact).  The scores' kernel counts the first digit, and the last block of
// each pass picks the digit and hands the next pass its prefix, so the host does
// not wait between them; the cells at or above the threshold are ordered by one
// block (score descending, ties by cell) when they fit its shared memory.  With
// a wait per digit, every score copied back and the candidates sorted on the host
// the selection of 1,000 of 300,000 cells took 311 us of host time.
#include "kern_common.cuh"

namespace dp {
namespace {

__host__ __device__ inline int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }

// state of a selection (SelectState): per pass 256 counts; then
constexpr int kPrefix = 1024, kLeft = 1025, kDone = 1026, kCount = 1030;

// The last block to have added its counts to hist: picks the largest digit whose cells and those of
// the digits above it still hold `left` cells.  All threads of the block (256) call it.
__device__ void pick_digit(unsigned *state, int pass, unsigned left) {
    __shared__ bool last;
    __shared__ unsigned sum[256];
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(state + kDone + pass, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    const int t = threadIdx.x;
    const unsigned mine = __ldcg(state + 256 * pass + t);
    sum[t] = mine;
    __syncthreads();
    for (int o = 1; o < 256; o <<= 1) {   // sum[t] = cells of digits t and above
        const unsigned add = t + o < 256 ? sum[t + o] : 0u;
        __syncthreads();
        sum[t] += add;
        __syncthreads();
    }
    const bool here = (sum[t] >= left || t == 0) && (t == 255 || sum[t + 1] < left);
    if (here) {
        state[kPrefix] = (pass ? state[kPrefix] : 0u) | (unsigned)t << (24 - 8 * pass);
        state[kLeft] = left - (sum[t] - mine);
    }
}

__device__ __forceinline__ void count_digit(unsigned *h, uint32_t bits, int pass) {
    atomicAdd(h + ((bits >> (24 - 8 * pass)) & 255u), 1u);
}
__device__ __forceinline__ void flush_counts(const unsigned *h, unsigned *hist) {
    __syncthreads();
    if (h[threadIdx.x]) atomicAdd(hist + threadIdx.x, h[threadIdx.x]);
}

// the scores and, for a selection of the k best (k > 0), their first digits
__global__ void __launch_bounds__(256) k_scores(const int32_t *__restrict__ cell_of_user,
                                                const float4 *__restrict__ pq, const float *__restrict__ alpha,
                                                const float *__restrict__ gnet, const float *__restrict__ cload,
                                                int64_t ns, int64_t nc, float K, int mode, float *out, unsigned *state,
                                                unsigned k) {
    __shared__ unsigned h[256];
    h[threadIdx.x] = 0u;
    __syncthreads();
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < nc; u += (int64_t)gridDim.x * blockDim.x) {
        const int64_t y = ns + cell_of_user[u];
        const float psw = K * alpha[y] * cload[y];
        float sens = fabsf(gnet[y]);
        if (mode == 1) {
            // 2 - 4 SP = 2 (P(net=0) - P): from the float-float pair, without the cancellation
            // of forming 2 - 4 SP from a rounded SP near SP = 0.5
            float d = 2.f * pair_qmp(pq[y]);
            if (fabsf(d) < 1e-6f) d = d < 0.f ? -1e-6f : 1e-6f;
            sens = fabsf(gnet[y] / d);
        }
        const float s = sens * psw;
        const float v = s > 0.f ? s : 0.f;   // +0 for zero, negative zero or NaN: the bits then order like the values
        out[u] = v;
        if (k) count_digit(h, __float_as_uint(v), 0);
    }
    if (!k) return;
    flush_counts(h, state);
    pick_digit(state, 0, k);
}

__global__ void __launch_bounds__(256) k_radix_hist(const float *__restrict__ s, int64_t n, int pass,
                                                    unsigned *state) {
    __shared__ unsigned h[256];
    const uint32_t prefix = state[kPrefix], mask = 0xFFFFFFFFu << (32 - 8 * pass);
    const unsigned left = state[kLeft];
    h[threadIdx.x] = 0u;
    __syncthreads();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t b = __float_as_uint(s[i]);
        if ((b & mask) == prefix) count_digit(h, b, pass);
    }
    flush_counts(h, state + 256 * pass);
    pick_digit(state, pass, left);
}

// the cells at or above the threshold, and the order they belong in as a key: score descending, then cell
__global__ void k_radix_collect(const float *__restrict__ s, int64_t n, unsigned *state, int32_t *idx,
                                unsigned long long *keys) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint32_t b = __float_as_uint(s[i]);
    if (b < state[kPrefix]) return;
    const unsigned at = atomicAdd(state + kCount, 1u);
    idx[at] = (int32_t)i;   // at most n of them
    if (at < (unsigned)kSelectMax) keys[at] = (unsigned long long)~b << 32 | (unsigned long long)(uint32_t)i;
}

// bitonic sort of the keys in one block's shared memory; nothing when there are more than it holds
__global__ void __launch_bounds__(1024) k_sort_top(const unsigned long long *__restrict__ keys, const unsigned *state,
                                                   int k, int32_t *top, float *top_scores) {
    extern __shared__ unsigned long long sk[];
    const int count = (int)state[kCount];
    if (count > kSelectMax) return;
    int n = 2;
    while (n < count) n <<= 1;
    for (int i = threadIdx.x; i < n; i += blockDim.x) sk[i] = i < count ? keys[i] : ~0ull;
    __syncthreads();
    for (int size = 2; size <= n; size <<= 1)
        for (int d = size >> 1; d > 0; d >>= 1) {
            for (int i = threadIdx.x; i < n / 2; i += blockDim.x) {
                const int a = 2 * i - (i & (d - 1)), b = a + d;
                const bool up = (a & size) == 0;
                const unsigned long long x = sk[a], y = sk[b];
                if ((x > y) == up) sk[a] = y, sk[b] = x;
            }
            __syncthreads();
        }
    for (int i = threadIdx.x; i < k && i < count; i += blockDim.x) {
        top[i] = (int32_t)(uint32_t)sk[i];
        if (top_scores) top_scores[i] = __uint_as_float(~(uint32_t)(sk[i] >> 32));
    }
}

}  // namespace

cudaError_t launch_scores(const DevDesign &d, bool hybrid, float K, int mode, float *out, unsigned *state, int64_t k,
                          cudaStream_t s) {
    if (d.n_cells == 0) return cudaSuccess;
    if (k > 0) {
        const cudaError_t e = cudaMemsetAsync(state, 0, sizeof(unsigned) * kSelectWords, s);
        if (e != cudaSuccess) return e;
    }
    const int64_t blocks = cdiv(d.n_cells, 256);
    k_scores<<<(unsigned)(blocks < 1216 ? blocks : 1216), 256, 0, s>>>(d.cell_of_user, d.pq, hybrid ? d.trh : d.tr,
                                                                      d.gnet, d.cload, d.n_start, d.n_cells, K, mode,
                                                                      out, state, (unsigned)k);
    return cudaGetLastError();
}

cudaError_t launch_select(const float *scores, int64_t n, int64_t k, unsigned *state, int32_t *idx,
                          unsigned long long *keys, int32_t *top, float *top_scores, cudaStream_t s) {
    const int64_t blocks = cdiv(n, 256);
    for (int pass = 1; pass < 4; pass++)
        k_radix_hist<<<(unsigned)(blocks < 608 ? blocks : 608), 256, 0, s>>>(scores, n, pass, state);
    k_radix_collect<<<(unsigned)blocks, 256, 0, s>>>(scores, n, state, idx, keys);
    cudaError_t e = cudaFuncSetAttribute(k_sort_top, cudaFuncAttributeMaxDynamicSharedMemorySize, kSelectMax * 8);
    if (e != cudaSuccess) return e;
    k_sort_top<<<1, 1024, kSelectMax * 8, s>>>(keys, state, (int)k, top, top_scores);
    return cudaGetLastError();
}

}  // namespace dp
