// Cell evaluation of the batched passes by function: the truth tables of the common gates are
// template arguments, so the leaves of the multilinear fold, the entries of the difference tables
// and the toggle table of the lag-one fold are known when the kernel is compiled, and the terms
// they make 0 or 1 are never formed.  A NAND2 costs 14 operations instead of 41, an AOI21 about 40
// instead of 105 (its partial derivatives 8 instead of 90).  Any other function takes the same folds
// over its table at run time.
//
// The value of a cell is a function of its inputs and table alone, whatever the launch shape.
#pragma once
#include "kern_batch.cuh"

namespace dp {

// ---- P(out = 1) in float-float: a fold whose operands may be known to be 0 or 1
enum Known { kZero, kOne, kAny };

// Q a + P b: fold_pq without the operations that a known operand makes exact, and the others in its order, so the
// result is fold_pq's to the last bit
template <int A, int B>
__device__ __forceinline__ ff fold_known(const pair_ff &x, const ff &a, const ff &b) {
    if (A == kZero && B == kZero) return ff_make(0.f);
    if (A == kZero && B == kOne) return x.p;
    if (A == kOne && B == kZero) return x.q;
    if (A == kAny && B == kAny) return fold_pq(x, a, b);
    if (A == kZero) return ff_mul(x.p, b);
    if (B == kZero) return ff_mul(x.q, a);
    if (A == kOne && B == kOne) {   // Q + P, 1 to about 4e-15
        const ff u = two_sum(x.q.hi, x.p.hi);
        return fast_two_sum(u.hi, __fadd_rn(__fadd_rn(u.lo, x.q.lo), x.p.lo));
    }
    const ff &s = A == kOne ? x.q : x.p, &f = A == kOne ? x.p : x.q, &g = A == kOne ? b : a;   // s + f g
    const float t = __fmul_rn(f.hi, g.hi);
    const ff u = two_sum(s.hi, t);
    float lo = __fadd_rn(u.lo, fmaf(f.hi, g.hi, -t));
    if (A == kOne) lo = __fadd_rn(lo, s.lo);
    lo = fmaf(f.hi, g.lo, lo);
    lo = fmaf(f.lo, g.hi, lo);
    if (B == kOne) lo = __fadd_rn(lo, s.lo);
    return fast_two_sum(u.hi, lo);
}

template <uint32_t TT, int I, int M>
struct ProbNode {   // inputs 0 .. I folded, entry M of what is left
    using A = ProbNode<TT, I - 1, 2 * M>;
    using B = ProbNode<TT, I - 1, 2 * M + 1>;
    static constexpr int kind = A::kind == kZero && B::kind == kZero ? kZero : kAny;
    __device__ __forceinline__ static ff val(const pair_ff (&x)[4]) {
        return fold_known<A::kind, B::kind>(x[I], A::val(x), B::val(x));
    }
};
template <uint32_t TT, int M>
struct ProbNode<TT, 0, M> {
    static constexpr bool a = (TT >> (2 * M)) & 1u, b = (TT >> (2 * M + 1)) & 1u;
    static constexpr int kind = a == b ? (a ? kOne : kZero) : kAny;
    __device__ __forceinline__ static ff val(const pair_ff (&x)[4]) {
        return a == b ? ff_make(a ? 1.f : 0.f) : a ? x[0].q : x[0].p;
    }
};

// ---- dP / dP_J in binary32: the difference table's entries are -1, 0 or 1
template <uint32_t TT, int J, int F, int M>
struct DiffNode {   // F inputs other than J folded
    using A = DiffNode<TT, J, F - 1, 2 * M>;
    using B = DiffNode<TT, J, F - 1, 2 * M + 1>;
    static constexpr bool known = A::known && B::known && A::value == 0 && B::value == 0;
    static constexpr int value = 0;
    __device__ __forceinline__ static float val(const float (&p)[4], const float (&q)[4]) {
        constexpr int i = F - 1 < J ? F - 1 : F;
        if (known) return 0.f;
        if (A::known && A::value == 0) {   // P b
            if (B::known) return B::value > 0 ? p[i] : -p[i];
            return __fmul_rn(p[i], B::val(p, q));
        }
        const float t = A::known ? (A::value > 0 ? q[i] : -q[i]) : __fmul_rn(q[i], A::val(p, q));   // Q a
        if (B::known && B::value == 0) return t;
        if (B::known) return B::value > 0 ? __fadd_rn(p[i], t) : __fsub_rn(t, p[i]);
        return fmaf(p[i], B::val(p, q), t);
    }
};
template <uint32_t TT, int J, int M>
struct DiffNode<TT, J, 0, M> {
    static constexpr int m0 = ((M >> J) << (J + 1)) | (M & ((1 << J) - 1)), m1 = m0 | (1 << J);
    static constexpr bool known = true;
    static constexpr int value = (int)((TT >> m1) & 1u) - (int)((TT >> m0) & 1u);
    __device__ __forceinline__ static float val(const float (&)[4], const float (&)[4]) { return (float)value; }
};

// ---- the lag-one toggle probability: the sum over joint input states (a, b) of prod_i w_i(a_i, b_i)
// [f(a) != f(b)], input 0 innermost; SUB >= 0 replaces input SUB's weights by their derivative with respect to
// its P (D = 0: -1, 0, 0, 1) or T (D = 1: -1/2, 1/2, 1/2, -1/2)
template <int SUB, int D, int I>
__device__ __forceinline__ float lag_term(const float (&w)[4][4], int d, float v) {
    if (SUB != I) return __fmul_rn(w[I][d], v);
    return D == 0 ? (d == 0 ? -v : v) : __fmul_rn(d == 0 || d == 3 ? -0.5f : 0.5f, v);
}
template <int SUB, int D, int I>
__device__ __forceinline__ float lag_add(const float (&w)[4][4], int d, float v, float acc) {
    if (SUB != I) return fmaf(w[I][d], v, acc);
    return D == 0 ? __fadd_rn(acc, d == 0 ? -v : v) : fmaf(d == 0 || d == 3 ? -0.5f : 0.5f, v, acc);
}
template <uint32_t TT, int K, int SUB, int D, int I, int M>
struct LagNode {   // inputs 0 .. I folded, entry M (base 4) of what is left
    template <int E>
    using C = LagNode<TT, K, SUB, D, I - 1, 4 * M + E>;
    static constexpr bool skip(int e) { return SUB == I && D == 0 && (e == 1 || e == 2); }
    static constexpr bool on0 = C<0>::on, on1 = C<1>::on && !skip(1), on2 = C<2>::on && !skip(2), on3 = C<3>::on;
    static constexpr bool on = on0 || on1 || on2 || on3;
    __device__ __forceinline__ static float val(const float (&w)[4][4]) {
        float acc = 0.f;
        if (on0) acc = lag_term<SUB, D, I>(w, 0, C<0>::val(w));
        if (on1) acc = on0 ? lag_add<SUB, D, I>(w, 1, C<1>::val(w), acc) : lag_term<SUB, D, I>(w, 1, C<1>::val(w));
        if (on2)
            acc = on0 || on1 ? lag_add<SUB, D, I>(w, 2, C<2>::val(w), acc) : lag_term<SUB, D, I>(w, 2, C<2>::val(w));
        if (on3)
            acc = on0 || on1 || on2 ? lag_add<SUB, D, I>(w, 3, C<3>::val(w), acc)
                                    : lag_term<SUB, D, I>(w, 3, C<3>::val(w));
        return acc;
    }
};
template <uint32_t TT, int K, int SUB, int D, int M>
struct LagNode<TT, K, SUB, D, -1, M> {   // a joint state: does the output differ between its two halves?
    static constexpr uint32_t half(int h) {
        uint32_t a = 0;
        for (int i = 0; i < K; i++) a |= (uint32_t)((M >> (2 * i + h)) & 1) << i;
        return a;
    }
    static constexpr bool on = (((TT >> half(1)) ^ (TT >> half(0))) & 1u) != 0;
    __device__ __forceinline__ static float val(const float (&)[4][4]) { return 1.f; }
};

// a cell of K inputs whose table is known when the kernel is compiled
template <int K, uint32_t TT>
struct CellFn {
    static constexpr int k = K;
    __device__ __forceinline__ ff prob(const pair_ff (&x)[4]) const { return ProbNode<TT, K - 1, 0>::val(x); }
    __device__ __forceinline__ void partials(const float (&p)[4], const float (&q)[4], float (&d)[4]) const {
        d[0] = DiffNode<TT, 0, K - 1, 0>::val(p, q);
        if (K > 1) d[1] = DiffNode<TT, (K > 1 ? 1 : 0), K - 1, 0>::val(p, q);
        if (K > 2) d[2] = DiffNode<TT, (K > 2 ? 2 : 0), K - 1, 0>::val(p, q);
    }
    __device__ __forceinline__ float toggle(const float (&w)[4][4]) const {
        return LagNode<TT, K, -1, 0, K - 1, 0>::val(w);
    }
    __device__ __forceinline__ void toggle_partials(const float (&w)[4][4], float (&dp)[4], float (&dt)[4]) const {
        dp[0] = LagNode<TT, K, 0, 0, K - 1, 0>::val(w);
        dt[0] = LagNode<TT, K, 0, 1, K - 1, 0>::val(w);
        if (K > 1) {
            dp[1] = LagNode<TT, K, (K > 1 ? 1 : 0), 0, K - 1, 0>::val(w);
            dt[1] = LagNode<TT, K, (K > 1 ? 1 : 0), 1, K - 1, 0>::val(w);
        }
        if (K > 2) {
            dp[2] = LagNode<TT, K, (K > 2 ? 2 : 0), 0, K - 1, 0>::val(w);
            dt[2] = LagNode<TT, K, (K > 2 ? 2 : 0), 1, K - 1, 0>::val(w);
        }
    }
};

// the lag-one fold over a table known at run time (kern_batch's general form of the above)
template <int K>
__device__ __forceinline__ float lag1_fold(uint32_t tt, const float (&w)[4][4], int sub, const float (&dv)[4]) {
    constexpr int M = 1 << (2 * K);
    float v[M];
#pragma unroll
    for (int m = 0; m < M; m++) {
        int a = 0, b = 0;
#pragma unroll
        for (int i = 0; i < K; i++) {
            const int dgt = (m >> (2 * i)) & 3;
            a |= (dgt >> 1) << i;
            b |= (dgt & 1) << i;
        }
        v[m] = (((tt >> a) ^ (tt >> b)) & 1u) ? 1.f : 0.f;
    }
#pragma unroll
    for (int i = 0; i < K; i++) {
        float c[4];
#pragma unroll
        for (int d = 0; d < 4; d++) c[d] = i == sub ? dv[d] : w[i][d];
#pragma unroll
        for (int m = 0; m < (M >> (2 * (i + 1))); m++)
            v[m] = fmaf(c[3], v[4 * m + 3], fmaf(c[2], v[4 * m + 2], fmaf(c[1], v[4 * m + 1], c[0] * v[4 * m])));
    }
    return v[0];
}

// four inputs have 256 joint states: kept out of line, once per kernel
static __device__ __noinline__ float lag1_fold4(uint32_t tt, const float (&w)[4][4], int sub, const float (&dv)[4]) {
    return lag1_fold<4>(tt, w, sub, dv);
}
template <int K>
__device__ __forceinline__ float lag1_fold_any(uint32_t tt, const float (&w)[4][4], int sub, const float (&dv)[4]) {
    if constexpr (K == 4) return lag1_fold4(tt, w, sub, dv);
    else return lag1_fold<K>(tt, w, sub, dv);
}

// any other cell of K inputs (0 to 4)
template <int K>
struct CellAny {
    static constexpr int k = K;
    uint32_t tt;
    __device__ __forceinline__ ff prob(const pair_ff (&x)[4]) const {
        if constexpr (K == 0) return ff_make((tt & 1u) ? 1.f : 0.f);
        else return ml_p<K>(tt, x);
    }
    __device__ __forceinline__ void partials(const float (&p)[4], const float (&q)[4], float (&d)[4]) const {
        cell_partials(K, tt, p, q, d);
    }
    __device__ __forceinline__ float toggle(const float (&w)[4][4]) const {
        const float none[4] = {0.f, 0.f, 0.f, 0.f};
        if constexpr (K == 0) return 0.f;   // a constant never toggles
        else return lag1_fold_any<K>(tt, w, -1, none);
    }
    __device__ __forceinline__ void toggle_partials(const float (&w)[4][4], float (&dp)[4], float (&dt)[4]) const {
        const float dP[4] = {-1.f, 0.f, 0.f, 1.f}, dT[4] = {-0.5f, 0.5f, 0.5f, -0.5f};
        if constexpr (K > 0) {
#pragma unroll
            for (int j = 0; j < K; j++) {
                dp[j] = lag1_fold_any<K>(tt, w, j, dP);
                dt[j] = lag1_fold_any<K>(tt, w, j, dT);
            }
        }
    }
};

// Calls f with the cell's function; consecutive cells of a level mostly share theirs, so a warp takes one
// branch.  f is inlined 22 times: it computes, and loads and stores stay outside.
template <class F>
__device__ __forceinline__ void with_cell(uint32_t e, const F &f) {
    switch ((e >> 19) & 31u) {
#define DP_CELL(I, K, TT) case I: return f(CellFn<K, TT>{});
        DP_CELL_CLASSES(DP_CELL)
#undef DP_CELL
        case 18: return f(CellAny<0>{e & 0xFFFFu});
        case 19: return f(CellAny<1>{e & 0xFFFFu});
        case 20: return f(CellAny<2>{e & 0xFFFFu});
        case 21: return f(CellAny<3>{e & 0xFFFFu});
        default: return f(CellAny<4>{e & 0xFFFFu});
    }
}

// ---- rows of V consecutive scenarios

// row n of an array of S columns: one multiply-add
template <class T>
__device__ __forceinline__ T *row_at(T *base, uint32_t n, uint32_t S) {
    return reinterpret_cast<T *>(reinterpret_cast<uint64_t>(base) + (uint64_t)n * (uint64_t)(S * (uint32_t)sizeof(T)));
}

// V consecutive float2 or float values of a row, through L2
template <int V>
struct Row2 {
    float2 v[V];
};
template <int V>
struct Row1 {
    float v[V];
};
template <int V>
__device__ __forceinline__ Row2<V> ld2(const float2 *p) {
    Row2<V> r;
    if constexpr (V == 1) {
        r.v[0] = __ldcg(p);
    } else if constexpr (V == 2) {
        const float4 t = __ldcg(reinterpret_cast<const float4 *>(p));
        r.v[0] = make_float2(t.x, t.y), r.v[1] = make_float2(t.z, t.w);
    } else {
        asm volatile("ld.global.cg.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=f"(r.v[0].x), "=f"(r.v[0].y), "=f"(r.v[1].x), "=f"(r.v[1].y), "=f"(r.v[2].x), "=f"(r.v[2].y),
                       "=f"(r.v[3].x), "=f"(r.v[3].y)
                     : "l"(p)
                     : "memory");
    }
    return r;
}
template <int V>
__device__ __forceinline__ void st2(float2 *p, const Row2<V> &r) {
    if constexpr (V == 1) {
        *p = r.v[0];
    } else if constexpr (V == 2) {
        *reinterpret_cast<float4 *>(p) = make_float4(r.v[0].x, r.v[0].y, r.v[1].x, r.v[1].y);
    } else {
        asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "f"(r.v[0].x), "f"(r.v[0].y),
                     "f"(r.v[1].x), "f"(r.v[1].y), "f"(r.v[2].x), "f"(r.v[2].y), "f"(r.v[3].x), "f"(r.v[3].y)
                     : "memory");
    }
}
template <int V>
__device__ __forceinline__ Row1<V> ld1(const float *p) {
    Row1<V> r;
    if constexpr (V == 1) {
        r.v[0] = __ldcg(p);
    } else if constexpr (V == 2) {
        const float2 t = __ldcg(reinterpret_cast<const float2 *>(p));
        r.v[0] = t.x, r.v[1] = t.y;
    } else {
        const float4 t = __ldcg(reinterpret_cast<const float4 *>(p));
        r.v[0] = t.x, r.v[1] = t.y, r.v[2] = t.z, r.v[3] = t.w;
    }
    return r;
}
template <int V>
__device__ __forceinline__ void st1(float *p, const Row1<V> &r) {
    if constexpr (V == 1) *p = r.v[0];
    else if constexpr (V == 2) *reinterpret_cast<float2 *>(p) = make_float2(r.v[0], r.v[1]);
    else *reinterpret_cast<float4 *>(p) = make_float4(r.v[0], r.v[1], r.v[2], r.v[3]);
}

// P (LAG: and T) of a cell of table entry e from its inputs' rows; get(j, x, t) reads input j's
template <int V, bool LAG, class G>
__device__ __forceinline__ void cell_value(uint32_t e, const G &get, Row2<V> &o, Row1<V> &ot) {
    with_cell(e, [&](const auto f) {
        constexpr int K = decltype(f)::k;
        Row2<V> x[4];
        Row1<V> t[4];
#pragma unroll
        for (int j = 0; j < K; j++) get(j, x[j], t[j]);
#pragma unroll
        for (int i = 0; i < V; i++) {
            pair_ff a[4];
            float w[4][4];
#pragma unroll
            for (int j = 0; j < K; j++) {
                a[j] = pair_get(x[j].v[i]);
                if (LAG) lag1_weights(a[j], t[j].v[i], w[j]);
            }
            const ff p = f.prob(a);
            o.v[i] = make_float2(p.hi, p.lo);
            if (LAG) ot.v[i] = f.toggle(w);
        }
    });
}

// What a cell adds to its inputs' adjoints, from the fanout sums a (LAG: and b, of T) of its net: g, LAG: (of P, of T)
// in g2.  self: the net's own P, cl: its load.
template <int V, bool LAG>
__device__ __forceinline__ void cell_adjoints(uint32_t e, const Row2<V> (&x)[4],
                                              const Row1<V> (&t)[4], const Row2<V> &self, const Row1<V> &Ks,
                                              const Row1<V> &cl, const Row1<V> &a, const Row1<V> &b, Row1<V> (&g)[4],
                                              Row2<V> (&g2)[4]) {
    with_cell(e, [&](const auto f) {
        constexpr int K = decltype(f)::k;
#pragma unroll
        for (int i = 0; i < V; i++) {
            float p[4], q[4], d[4], w[4][4];
#pragma unroll
            for (int j = 0; j < K; j++) {
                const pair_ff v = pair_get(x[j].v[i]);
                p[j] = v.p.hi + v.p.lo;
                q[j] = v.q.hi + v.q.lo;
                if (LAG) lag1_weights(v, t[j].v[i], w[j]);
            }
            f.partials(p, q, d);
            if constexpr (LAG) {
                float dp[4], dt[4];
                f.toggle_partials(w, dp, dt);
                const float gt = fmaf(Ks.v[i], cl.v[i], b.v[i]);
#pragma unroll
                for (int j = 0; j < K; j++)
                    g2[j].v[i] = make_float2(fmaf(a.v[i], d[j], __fmul_rn(gt, dp[j])), __fmul_rn(gt, dt[j]));
            } else {
#pragma unroll
                for (int j = 0; j < K; j++) g[j].v[i] = d[j];
            }
        }
    });
    if (!LAG)
#pragma unroll
        for (int i = 0; i < V; i++) {
            const float gn = bwdb_adjoint(a.v[i], Ks.v[i], cl.v[i], self.v[i]);
#pragma unroll
            for (int j = 0; j < 4; j++) g[j].v[i] = __fmul_rn(gn, g[j].v[i]);
        }
}

// the partial derivatives of a cell with respect to its inputs (get(j, x, t) reads input j): of P by P in d, LAG: of T by
// P and by T in dp and dt
template <int V, bool LAG, class G>
__device__ __forceinline__ void cell_partials(uint32_t e, const G &get, Row1<V> (&d)[4], Row1<V> (&dp)[4],
                                              Row1<V> (&dt)[4]) {
    with_cell(e, [&](const auto f) {
        constexpr int K = decltype(f)::k;
        Row2<V> x[4];
        Row1<V> t[4];
#pragma unroll
        for (int j = 0; j < K; j++) get(j, x[j], t[j]);
#pragma unroll
        for (int i = 0; i < V; i++) {
            float p[4], q[4], g[4], w[4][4];
#pragma unroll
            for (int j = 0; j < K; j++) {
                const pair_ff v = pair_get(x[j].v[i]);
                p[j] = v.p.hi + v.p.lo;
                q[j] = v.q.hi + v.q.lo;
                if (LAG) lag1_weights(v, t[j].v[i], w[j]);
            }
            f.partials(p, q, g);
#pragma unroll
            for (int j = 0; j < K; j++) d[j].v[i] = g[j];
            if constexpr (LAG) {
                float gp[4], gt[4];
                f.toggle_partials(w, gp, gt);
#pragma unroll
                for (int j = 0; j < K; j++) dp[j].v[i] = gp[j], dt[j].v[i] = gt[j];
            }
        }
    });
}

// the sums over a net's fanout range [e0, e1) in index order, four edges' loads in flight: the adjoints of P in a, LAG:
// of T in b
template <int V, bool LAG>
__device__ __forceinline__ void fanout_sum(const float *gfo, const float2 *gfo2, int32_t e0, int32_t e1, uint32_t S,
                                           Row1<V> &a, Row1<V> &b) {
#pragma unroll
    for (int i = 0; i < V; i++) a.v[i] = b.v[i] = 0.f;
    for (int32_t e = e0; e < e1; e += 4) {
        Row1<V> u[4];
        Row2<V> u2[4];
#pragma unroll
        for (int k = 0; k < 4; k++)
            if (e + k < e1) {
                if constexpr (LAG) u2[k] = ld2<V>(row_at(gfo2, (uint32_t)(e + k), S));
                else u[k] = ld1<V>(row_at(gfo, (uint32_t)(e + k), S));
            }
#pragma unroll
        for (int k = 0; k < 4; k++)
            if (e + k < e1)
#pragma unroll
                for (int i = 0; i < V; i++) {
                    if constexpr (LAG) a.v[i] += u2[k].v[i].x, b.v[i] += u2[k].v[i].y;
                    else a.v[i] += u[k].v[i];
                }
    }
}

}  // namespace dp
