// Bit-parallel simulation cut by lanes and time instead of by cells: a block simulates the whole
// netlist, but only a slice of `lanes` of the 64 chains over a run of consecutive cycles.
//
// The chains are independent and a cycle's words depend on that cycle's startpoint words only, so
// the blocks never talk to each other: levels are separated by a block barrier, and a net's value
// sits in shared memory from the level that computes it to the last level that reads it.  The
// host assigns the slots by those lifetimes (a tenth of the nets are alive at a time in the
// generator's netlists), so a design of up to about 550,000 nets fits.
//
// A net's value in a block is a bit string of NV 32-bit words, cycle-major: cycle i of the run in
// bits [i lanes, (i + 1) lanes).  Its toggles are popc(x ^ (x << lanes)), so a run starts with the
// last cycle of the run before it.  Each block adds its counts to the design's with one reduction
// per cell.
//
// What bounds it: instructions and bank conflicts of the gathers (16-byte loads at random slots: 8.3
// wavefronts instead of 4; the LSU 45 % and the issue slots 41 % busy on 117,000 cells and 256
// words), then the level's barrier and shared-memory round trip.  Leaving out the reductions, the
// population counts or the function changes 10 % at most.  Spreading cells over the grid instead
// costs a grid barrier and a dependent round trip through L2 per level and per 64 words
// (kern_persist.cu).
#include "kern_common.cuh"

namespace dp {
namespace {

constexpr int kSliceSmem = 224 * 1024;

// f(x0, x1, x2) of an 8-entry table on 32 lanes: a multiplexer tree, the table's entries as masks
// (the same instructions for every function, so a warp of mixed cells does not diverge)
__device__ __forceinline__ uint32_t mux(uint32_t s, uint32_t a1, uint32_t a0) { return (s & a1) | (~s & a0); }
__device__ __forceinline__ uint32_t eval8(const uint32_t (&m)[8], uint32_t x0, uint32_t x1, uint32_t x2) {
    const uint32_t a = mux(x0, m[1], m[0]), b = mux(x0, m[3], m[2]), c = mux(x0, m[5], m[4]), d = mux(x0, m[7], m[6]);
    return mux(x2, mux(x1, d, c), mux(x1, b, a));
}

template <int NV>
struct Bits {
    uint32_t v[NV];
};
template <int NV>
__device__ __forceinline__ Bits<NV> slot_get(const uint32_t *sh, uint32_t slot) {
    Bits<NV> b;
    const uint32_t *p = sh + (size_t)slot * NV;
    if (NV == 1) {
        b.v[0] = p[0];
    } else if (NV == 2) {
        const uint2 t = *reinterpret_cast<const uint2 *>(p);
        b.v[0] = t.x, b.v[1 % NV] = t.y;
    } else {
#pragma unroll
        for (int i = 0; i < NV / 4; i++) {
            const uint4 t = reinterpret_cast<const uint4 *>(p)[i];
            b.v[(4 * i) % NV] = t.x, b.v[(4 * i + 1) % NV] = t.y, b.v[(4 * i + 2) % NV] = t.z, b.v[(4 * i + 3) % NV] = t.w;
        }
    }
    return b;
}
template <int NV>
__device__ __forceinline__ void slot_put(uint32_t *sh, uint32_t slot, const Bits<NV> &b) {
    uint32_t *p = sh + (size_t)slot * NV;
    if (NV == 1) {
        p[0] = b.v[0];
    } else if (NV == 2) {
        *reinterpret_cast<uint2 *>(p) = make_uint2(b.v[0], b.v[1 % NV]);
    } else {
#pragma unroll
        for (int i = 0; i < NV / 4; i++)
            reinterpret_cast<uint4 *>(p)[i] =
                make_uint4(b.v[(4 * i) % NV], b.v[(4 * i + 1) % NV], b.v[(4 * i + 2) % NV], b.v[(4 * i + 3) % NV]);
    }
}

// the eight entries of a table as masks: entry i moved to the top of byte i, then that sign bit
// spread over the word (one PRMT each)
__device__ __forceinline__ uint32_t spread_sign(uint32_t v, uint32_t sel) {   // selectors with the sign bit set
    uint32_t d;
    asm("prmt.b32 %0, %1, 0, %2;" : "=r"(d) : "r"(v), "r"(sel));
    return d;
}
__device__ __forceinline__ void table_masks(uint32_t tt, uint32_t (&m)[8]) {
    const uint32_t lo = (tt & 15u) * 0x10204080u, hi = ((tt >> 4) & 15u) * 0x10204080u;
#pragma unroll
    for (int i = 0; i < 4; i++) {
        m[i] = spread_sign(lo, 0x8888u + 0x1111u * i);
        m[4 + i] = spread_sign(hi, 0x8888u + 0x1111u * i);
    }
}

// Block (q, r): lanes [q LANES, (q + 1) LANES), cycles r N .. (r + 1) N with N = 32 NV / LANES - 1.
// The cells come in rounds of blockDim.x records (levels padded to whole rounds; round_ptr[l] the
// first round of level l + 1), so a thread's records lie blockDim.x apart whatever the level: what
// bounds a wide level is the number of instructions per cell, not the accesses, and one 16-byte
// load with a constant stride replaces the level's bounds.  Two records are held ahead.
// A record: x, y three input slots and the output slot (0xFFFF: nobody reads it) of 16 bits (unused
// inputs: slot 0, and a table that ignores them), z the table of at most 3 inputs | 4-input flag <<
// 8 | upper half of a 4-input table << 16, w the cell (-1: padding).
template <int NV, int LANES>
__global__ void __launch_bounds__(NV > 4 ? 512 : 1024, 1) k_sim_slice(
    const uint4 *__restrict__ rec, const int32_t *__restrict__ round_ptr, const uint16_t *__restrict__ fourth,
    const int32_t *__restrict__ start_slot, const uint64_t *__restrict__ words, int L, int64_t ns, int T,
    uint32_t *toggles, uint32_t *ones) {
    extern __shared__ uint4 sh4[];
    uint32_t *sh = reinterpret_cast<uint32_t *>(sh4);
    constexpr int kSlices = 64 / LANES, kPer = 32 / LANES, kSteps = NV * kPer;
    constexpr uint32_t kLane = LANES == 32 ? 0xFFFFFFFFu : (1u << LANES % 32) - 1u;
    const int q = (int)blockIdx.x % kSlices, run = (int)blockIdx.x / kSlices;
    const int t0 = run * (kSteps - 1);
    const int have = T - t0 < kSteps ? T - t0 : kSteps;   // cycles of the run that exist
    const int rounds = round_ptr[L];
    const uint4 *next = rec + threadIdx.x;
    const uint4 none = make_uint4(0u, 0xFFFF0000u, 0u, 0xFFFFFFFFu);
    uint4 r0 = rounds > 0 ? next[0] : none, r1 = rounds > 1 ? next[blockDim.x] : none;
    next += 2 * blockDim.x;
    for (int64_t k = threadIdx.x; k < ns; k += blockDim.x) {
        const int slot = start_slot[k];
        const uint64_t *w = words + (size_t)k * T + t0;
        uint32_t v[kSteps];   // all of the startpoint's loads in flight together
#pragma unroll
        for (int i = 0; i < kSteps; i++) v[i] = i < have ? (uint32_t)(w[i] >> (q * LANES)) & kLane : 0u;
        Bits<NV> b;
#pragma unroll
        for (int i = 0; i < NV; i++) {
            b.v[i] = 0u;
#pragma unroll
            for (int j = 0; j < kPer; j++) b.v[i] |= v[i * kPer + j] << (j * LANES);
        }
        if (slot >= 0) slot_put<NV>(sh, (uint32_t)slot, b);
    }
    // counted: the cycles after the first (it belongs to the run before), and in the first run all
    uint32_t mt[NV];
    auto below = [&](int bits) { return bits >= 32 ? 0xFFFFFFFFu : bits <= 0 ? 0u : (1u << bits) - 1u; };
#pragma unroll
    for (int i = 0; i < NV; i++) mt[i] = below(have * LANES - 32 * i) & ~(i ? 0u : kLane);
    const uint32_t mo0 = run ? mt[0] : below(have * LANES);
    int left = rounds;
    for (int l = 1; l <= L; l++) {
        int n = round_ptr[l] - round_ptr[l - 1];
        __syncthreads();   // the levels below are in shared memory, and the slots of the nets that died are free
        for (; n > 0; n--) {
            const uint4 cur = r0;
            r0 = r1;
            if (--left > 1) r1 = *next;
            next += blockDim.x;
            if ((int32_t)cur.w < 0) continue;
            const Bits<NV> x0 = slot_get<NV>(sh, cur.x & 0xFFFFu), x1 = slot_get<NV>(sh, cur.x >> 16);
            const Bits<NV> x2 = slot_get<NV>(sh, cur.y & 0xFFFFu);
            Bits<NV> o;
            uint32_t m[8];
            table_masks(cur.z, m);
#pragma unroll
            for (int i = 0; i < NV; i++) o.v[i] = eval8(m, x0.v[i], x1.v[i], x2.v[i]);
            if (cur.z & 0x100u) {   // that was the cofactor of x3 = 0: the one of x3 = 1, then a select
                const Bits<NV> x3 = slot_get<NV>(sh, fourth[cur.w]);
                table_masks(cur.z >> 16, m);
#pragma unroll
                for (int i = 0; i < NV; i++) o.v[i] = mux(x3.v[i], eval8(m, x0.v[i], x1.v[i], x2.v[i]), o.v[i]);
            }
            if ((cur.y >> 16) != 0xFFFFu) slot_put<NV>(sh, cur.y >> 16, o);
            uint32_t tg = 0, on = 0;
#pragma unroll
            for (int i = 0; i < NV; i++) {
                on += __popc(o.v[i] & (i ? mt[i] : mo0));
                tg += __popc((o.v[i] ^ __funnelshift_lc(i ? o.v[i > 0 ? i - 1 : 0] : 0u, o.v[i], LANES)) & mt[i]);
            }
            atomicAdd(toggles + cur.w, tg);   // the results are not used: reductions
            atomicAdd(ones + cur.w, on);
        }
    }
}

template <int NV, int LANES>
cudaError_t launch(const DevDesign &d, const SlicePlan &p, int T, cudaStream_t s) {
    constexpr int n = 32 * NV / LANES - 1;
    k_sim_slice<NV, LANES><<<(unsigned)((T - 1 + n - 1) / n * (64 / LANES)), p.threads, (size_t)p.slots * NV * 4, s>>>(
        (const uint4 *)p.rec, p.round_ptr, p.fourth, p.start_slot, d.words, d.n_levels, d.n_start, T,
        d.toggles + d.n_start, d.ones + d.n_start);
    return cudaGetLastError();
}
template <int NV>
cudaError_t launch(const DevDesign &d, const SlicePlan &p, int T, int lanes, cudaStream_t s) {
    if (lanes == 8) return launch<NV, 8>(d, p, T, s);
    if (lanes == 16) return launch<NV, 16>(d, p, T, s);
    return launch<(NV > 1 ? NV : 2), 32>(d, p, T, s);   // one 32-lane cycle is no run: never asked for
}
template <int NV>
bool raise_smem() {
    const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
    return cudaFuncSetAttribute(k_sim_slice<NV, 8>, a, kSliceSmem) == cudaSuccess &&
           cudaFuncSetAttribute(k_sim_slice<NV, 16>, a, kSliceSmem) == cudaSuccess &&
           cudaFuncSetAttribute(k_sim_slice<(NV > 1 ? NV : 2), 32>, a, kSliceSmem) == cudaSuccess;
}

}  // namespace

bool slice_fits(int64_t slots) {
    return slots <= kSliceMaxSlots && raise_smem<1>() && raise_smem<2>() && raise_smem<4>() &&
           raise_smem<8>();
}

// A block takes about 0.35 + 0.12 NV ns per cell and 0.35 us per level, and the blocks go over the
// SMs in waves; of two equal shapes the wider slice (a startpoint word is then read by fewer blocks).
// The wide simulation takes about 2.3 us per level and its words' way through L2 (three gathers and a
// store of 8 T bytes per cell at 4.8 TB/s).  Measured, this against that, with the generator (a third slower then):
// 13,000 cells / 70 levels 64 words 45 / 193 us, 250 words 70 / 355; 117,000 / 84 64 words 122 / 262, 250
// words 213 / 568; 120,000 / 48 120 / 181 and 276 / 385; 300,000 / 54 33 words 205 / 288, but 64 words
// (two waves) 364 / 272, where the rule takes the wide one.
SliceShape slice_shape(const SlicePlan &p, int64_t n_cells, int n_levels, int T, int sm_count) {
    SliceShape best{0, 0};
    double cost = 2.3 * n_levels + 5.3e-6 * (double)n_cells * T;
    for (int nv = 1; nv <= 8; nv *= 2) {
        if (p.slots * nv * 4 > kSliceSmem || (nv > 4 && p.threads > 512)) break;
        for (int lanes = 32; lanes >= 8; lanes /= 2) {
            const int n = 32 * nv / lanes - 1;
            if (n < 1) continue;
            const int64_t blocks = (int64_t)((T - 1 + n - 1) / n) * (64 / lanes);
            const double c = (double)((blocks + sm_count - 1) / sm_count) *
                             ((double)n_cells * (0.35 + 0.12 * nv) * 1e-3 + 0.35 * n_levels);
            if (c < cost) best = SliceShape{nv, lanes}, cost = c;
        }
    }
    return best;
}

cudaError_t launch_sim_slice(const DevDesign &d, const SlicePlan &p, int T, SliceShape sh, cudaStream_t s) {
    cudaError_t e = cudaSuccess;
    if (d.n_cells) {
        e = cudaMemsetAsync(d.toggles + d.n_start, 0, sizeof(uint32_t) * (size_t)d.n_cells, s);
        if (e == cudaSuccess) e = cudaMemsetAsync(d.ones + d.n_start, 0, sizeof(uint32_t) * (size_t)d.n_cells, s);
    }
    if (e != cudaSuccess) return e;
    switch (sh.nv) {
        case 1: return launch<1>(d, p, T, sh.lanes, s);
        case 2: return launch<2>(d, p, T, sh.lanes, s);
        case 4: return launch<4>(d, p, T, sh.lanes, s);
        default: return launch<8>(d, p, T, sh.lanes, s);
    }
}

}  // namespace dp
