// k_edge.cuh -- fused pass over the stored entries: LS target, one-point
// least-squares fit for every stored off-diagonal, row-relative threshold
// and strength flags.
//
// For row i and its stored entries p = (i, j):
//   1. y_i = x_i - (1/a_ii) sum_p a(i,col_p) x(col_p)     (Eqs. (3.2), (4.1):
//      the residual-corrected target, one local Jacobi step; same rounding
//      as the relaxation sweep with omega = 1), or y_i = x_i (Eq. (3.1)).
//   2. for every off-diagonal (§4.1, Eq. (4.3)):
//        S_xx = sum_k w_k x_jk^2, S_yx = sum_k w_k y_ik x_jk
//        a_ij = S_yx / S_xx (0 if S_xx = 0)
//        LS_ij = sum_k w_k (y_ik - a_ij x_jk)^2   (second pass over the K
//        components, each residual one fused multiply-add: no cancellation
//        of S_yy - a S_yx; an error in a_ij enters LS only to second order)
//      A residual-target row with one off-diagonal has y_i proportional to
//      x_j exactly: a = -a_ij/a_ii, LS = 0.
//      Mixed precisions (FP32 arithmetic on FP32/BF16 vectors): the three
//      sums are compensated (AMGD_SUM_COMPENSATED, below) or plain FMA
//      chains; a row with an edge of LS < 1e-4 S_yy is recomputed in FP64
//      (k_edge_fixup), with y_i rebuilt from the FP64 values of A, so
//      cancellation never decides a distance.
//   3. m_i = min_p LS_ip; slot p is strong iff LS_p = 0 or theta LS_p < m_i
//      (§4.2, Eq. (4.4), r = 1/LS); per-row strong count.
// Outputs are in the caller's numbering.  The vectors are read in the
// sweeps' row order in place (renumbered column indices) for search depth 1,
// from a caller-order copy otherwise.
//
// Two kernels.  S_xx depends on the neighbour alone, so k_norms forms it once
// per row instead of once per entry; k_edge_fit does the rest with a few
// lanes per row.
#pragma once
#include <type_traits>

#include "amgd_internal.cuh"
#include "rowops.cuh"
#include "staging.cuh"

namespace amgd {
namespace edge_impl {

constexpr int kFitThreads = 128;

template <int G, class T>
__device__ __forceinline__ T group_sum(T v, unsigned mask)
{
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o, G);
    return v;
}

// the mixed path's coefficient only needs FP32 relative accuracy (its error
// enters LS at second order): the fast division is enough
__device__ __forceinline__ float divide(float a, float b) { return __fdividef(a, b); }

// ---------------------------------------------------------------------------
// Order of the K-term sums.  A row is P pieces of V components (16 bytes).
// Every piece has its own partial sum, in component order, and the pieces are
// joined by the binary tree that adds piece q and piece q + P/2, then q and
// q + P/4, ... (the order of a shuffle butterfly over P lanes that hold one
// piece each, which is how k_norms forms S_xx).  tree_sum walks that tree
// depth first, so that at most log2(P) partial sums are live.
// ---------------------------------------------------------------------------
template <int L, int H, int END, class Leaf, class Join>
__device__ __forceinline__ auto tree_sum(Leaf &leaf, Join &join)
{
    if constexpr (H == END) {
        return leaf(L);
    } else {
        const auto a = tree_sum<L, 2 * H, END>(leaf, join);
        const auto b = tree_sum<L + H, 2 * H, END>(leaf, join);
        return join(a, b);
    }
}

// ---------------------------------------------------------------------------
// Compensated FP32 sums (mixed paths, AMGD_SUM_COMPENSATED).  Each sum is two
// FP32 words: a running sum and the exact rounding error of every addition,
// taken by TwoSum (six IEEE additions, no fusion) -- the Kahan-Babuska-
// Neumaier scheme; two partial sums are joined by TwoSum again, adding the
// error words, and the two words are added once at the end.  Two independent
// chains share the FP32x2 instructions: two pieces of S_yx, the even and odd
// components of an LS piece.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float2 sub2(float2 a, float2 b)
{
    return __ffma2_rn(b, make_float2(-1.f, -1.f), a);     // a - b, one rounding
}
// s + e == a + b exactly (Knuth's TwoSum, both halves of the pair)
__device__ __forceinline__ void two_sum2(float2 a, float2 b, float2 &s, float2 &e)
{
    s = __fadd2_rn(a, b);
    const float2 bp = sub2(s, a);
    const float2 ap = sub2(s, bp);
    e = __fadd2_rn(sub2(a, ap), sub2(b, bp));
}
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    const float bp = __fsub_rn(s, a);
    const float ap = __fsub_rn(s, bp);
    e = __fadd_rn(__fsub_rn(a, ap), __fsub_rn(b, bp));
}
struct Comp {
    float s, c;
};
// two sums side by side
struct Comp2 {
    float2 s, c;
};
__device__ __forceinline__ Comp2 comp2_join(const Comp2 &a, const Comp2 &b)
{
    Comp2 r;
    float2 e;
    two_sum2(a.s, b.s, r.s, e);
    r.c = __fadd2_rn(__fadd2_rn(a.c, b.c), e);
    return r;
}
// the chain t(0), t(1), ..., t(N - 1): the first term is exact
template <int N, class Term>
__device__ __forceinline__ Comp2 comp2_chain(const Term &t)
{
    Comp2 r{t(0), make_float2(0.f, 0.f)};
#pragma unroll
    for (int k = 1; k < N; ++k) {
        float2 sn, e;
        two_sum2(r.s, t(k), sn, e);
        r.s = sn;
        r.c = k == 1 ? e : __fadd2_rn(r.c, e);
    }
    return r;
}
struct CompJoin {
    __device__ __forceinline__ Comp operator()(const Comp &a, const Comp &b) const
    {
        Comp r;
        float e;
        two_sum(a.s, b.s, r.s, e);
        r.c = __fadd_rn(__fadd_rn(a.c, b.c), e);
        return r;
    }
};

// ---------------------------------------------------------------------------
// S_xx of every vector row: on the mixed paths FP32 sums in the order above
// (P lanes per row, one piece each); FP64 with its reciprocal, so that a fit
// needs no FP64 division (nine operations of the FP64 pipe, which retires two
// per clock and SM), one thread per row (K + 10 operations; P lanes would run
// the division P times: 25 against 6 us at 111k rows, K = 13).  The reciprocal
// is NaN where S_xx or 1/S_xx leaves the range in which the quotient's
// correction is exact: those fits divide.  Bound: one read of the vectors,
// most of it from the L2 that the last sweep left them in.
// ---------------------------------------------------------------------------
constexpr int kNormThreads = 256;

// Chains of an FP64 sum (even and odd components of every M-th piece) joined.  Chains of
// a few terms, for the rounding errors: with two over a lane's 16 components and two over
// a whole row here, a was off by 1.13 (K = 16) to 1.40 (K = 64) units of its last place
// (rms, against 80-bit sums of uniform vectors), by 1.03 as it is, as with a tree over
// all pieces.
template <int M>
__device__ __forceinline__ double join_chains(const double (&c0)[M], const double (&c1)[M])
{
    double s[M];
#pragma unroll
    for (int m = 0; m < M; ++m) s[m] = c0[m] + c1[m];
#pragma unroll
    for (int h = M / 2; h > 0; h /= 2)
#pragma unroll
        for (int m = 0; m < h; ++m) s[m] += s[m + h];
    return s[0];
}

template <class TS, int P, bool UW, bool COMP>
__global__ void __launch_bounds__(kNormThreads) k_norms(const TS *X, const void *wv, int32_t n,
                                                        void *out)
{
    using S = Store<TS>;
    using C = typename S::C;
    constexpr int V = S::V;
    if constexpr (std::is_same<C, double>::value) {
        const int64_t r = (int64_t)blockIdx.x * kNormThreads + threadIdx.x;
        chain_wait();
        chain_release();
        if (r >= n) return;
        constexpr int M = P < 4 ? 1 : P <= 8 ? 2 : P / 4;          // piece q belongs to chain q mod M
        double c0[M] = {}, c1[M] = {};
#pragma unroll 4
        for (int q0 = 0; q0 < P; q0 += M)
#pragma unroll
            for (int m = 0; m < M; ++m) {
                const int q = q0 + m;
                double x[V];
                S::unpack(ld16(X + (r * P + q) * V), x);
                const double2 w = UW ? make_double2(1.0, 1.0) : ld_plain((const double2 *)wv + q);
                c0[m] = fma(UW ? x[0] : w.x * x[0], x[0], c0[m]);
                c1[m] = fma(UW ? x[1] : w.y * x[1], x[1], c1[m]);
            }
        const double s = join_chains(c0, c1);
        ((double2 *)out)[r] = make_double2(s, s > 1e-290 && s < 1e290 ? 1.0 / s : NAN);
    } else {
        const int lane = threadIdx.x % P;
        const int64_t r0 = (int64_t)blockIdx.x * (kNormThreads / P) + threadIdx.x / P;
        const int64_t r = r0 < n ? r0 : n - 1;          // every lane takes part in the shuffles
        chain_wait();
        chain_release();
        C x[V];
        S::unpack(ld16(X + (r * P + lane) * V), x);
        float wx[V];
#pragma unroll
        for (int e = 0; e < V; ++e) wx[e] = UW ? x[e] : ((const float *)wv)[lane * V + e] * x[e];
        float total;
        if constexpr (COMP) {
            Comp v{__fmul_rn(wx[0], x[0]), 0.f};
            CompJoin join;
#pragma unroll
            for (int e = 1; e < V; ++e) {
                float s, err;
                two_sum(v.s, __fmul_rn(wx[e], x[e]), s, err);
                v.s = s;
                v.c = __fadd_rn(v.c, err);
            }
#pragma unroll
            for (int o = P / 2; o > 0; o >>= 1) {
                const Comp other{__shfl_xor_sync(0xffffffffu, v.s, o, P), __shfl_xor_sync(0xffffffffu, v.c, o, P)};
                v = join(v, other);
            }
            total = v.s + v.c;
        } else {
            float2 s = make_float2(0.f, 0.f);
#pragma unroll
            for (int e = 0; e < V; e += 2)
                s = __ffma2_rn(make_float2(wx[e], wx[e + 1]), make_float2(x[e], x[e + 1]), s);
            total = group_sum<P>(s.x + s.y, 0xffffffffu);
        }
        if (r0 < n && lane == 0) ((float *)out)[r] = total;
    }
}

// ---------------------------------------------------------------------------
// G lanes share a row.  A lane holds NP = P / G of its pieces: the pairs
// (2m, 2m + 1) with m = t G + lane, t = 0 .. NP/2 - 1, so that each of its
// 32-byte loads lies beside its neighbours' (P = 1: the one piece).  The two
// pieces of a pair run side by side in the FP32x2 instructions, through the
// levels of the tree inside the lane (over t), then across the lanes, and are
// joined last.
// ---------------------------------------------------------------------------
template <int G, int NP>
__device__ __forceinline__ int fit_piece(int lane, int q)
{
    return NP == 1 ? q : 2 * ((q / 2) * G + lane) + (q & 1);
}

template <int G>
__device__ __forceinline__ float comp_total(Comp2 v, unsigned mask)
{
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
        Comp2 w;
        w.s.x = __shfl_xor_sync(mask, v.s.x, o, G);
        w.s.y = __shfl_xor_sync(mask, v.s.y, o, G);
        w.c.x = __shfl_xor_sync(mask, v.c.x, o, G);
        w.c.y = __shfl_xor_sync(mask, v.c.y, o, G);
        v = comp2_join(v, w);
    }
    float s, e;
    two_sum(v.s.x, v.s.y, s, e);
    return s + __fadd_rn(__fadd_rn(v.c.x, v.c.y), e);
}
template <int G>
__device__ __forceinline__ float plain_total(float2 v, unsigned mask)
{
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1)
        v = __fadd2_rn(v, make_float2(__shfl_xor_sync(mask, v.x, o, G), __shfl_xor_sync(mask, v.y, o, G)));
    return v.x + v.y;
}

// S_xx (FP32) or S_xx and its reciprocal (FP64) as k_norms left them
template <class C> struct Norm { using T = float; };
template <> struct Norm<double> { using T = double2; };

// One fit: S_yx, a_ij and LS_ij from the lane's pieces of x_j (as stored), of
// the target and of the weights (w, UW: unused), the first np of them not all
// padding; every lane of the row ends with the result.  OWN: S_xx is formed here,
// in k_norms' order (plain sums; nr is not read).
template <class TS, int G, int NP, bool UW, bool COMP, bool OWN, class W>
__device__ __forceinline__ void fit_entry(const uint4 (&raw)[NP],
                                          const typename Store<TS>::C (&y)[NP][Store<TS>::V], const W &w,
                                          const typename Norm<typename Store<TS>::C>::T &nr, int np, unsigned mask,
                                          typename Store<TS>::C &a_, typename Store<TS>::C &ls_)
{
    using S = Store<TS>;
    using C = typename S::C;
    constexpr int V = S::V;
    if constexpr (std::is_same<C, double>::value) {
        // chains of at most four terms, joined once
        constexpr int M = NP > 4 ? 2 : 1;
        double s0[M] = {}, s1[M] = {};
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            if (q >= np) break;
            C x[V];
            S::unpack(raw[q], x);
            s0[q % M] = fma(UW ? x[0] : w(q, 0) * x[0], y[q][0], s0[q % M]);
            s1[q % M] = fma(UW ? x[1] : w(q, 1) * x[1], y[q][1], s1[q % M]);
        }
        const double syx = group_sum<G>(join_chains(s0, s1), mask);
        // a = S_yx / S_xx: the product with the reciprocal, corrected by its
        // exact remainder (Markstein's division step); operands outside its
        // range divide
        a_ = syx * nr.y;
        if ((__double2hiint(a_) & 0x7fffffff) < 0x7f000000) a_ = fma(fma(-a_, nr.x, syx), nr.y, a_);
        else a_ = nr.x == 0.0 ? 0.0 : syx / nr.x;
        double r0[M] = {}, r1[M] = {};
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            if (q >= np) break;
            C x[V];
            S::unpack(raw[q], x);
            const double d0 = fma(-a_, x[0], y[q][0]), d1 = fma(-a_, x[1], y[q][1]);
            r0[q % M] = fma(UW ? d0 : w(q, 0) * d0, d0, r0[q % M]);
            r1[q % M] = fma(UW ? d1 : w(q, 1) * d1, d1, r1[q % M]);
        }
        ls_ = group_sum<G>(join_chains(r0, r1), mask);
    } else if constexpr (NP == 1) {
        C x[V];
        S::unpack(raw[0], x);
        float sxx = nr;
        auto wx = [&](int e) { return UW ? x[e] : w(0, e) * x[e]; };
        float syx;
        if constexpr (COMP) {
            Comp v{__fmul_rn(wx(0), y[0][0]), 0.f};
#pragma unroll
            for (int e = 1; e < V; ++e) {
                float s, err;
                two_sum(v.s, __fmul_rn(wx(e), y[0][e]), s, err);
                v.s = s;
                v.c = __fadd_rn(v.c, err);
            }
            syx = v.s + v.c;
        } else {
            float2 s = make_float2(0.f, 0.f);
#pragma unroll
            for (int e = 0; e < V; e += 2)
                s = __ffma2_rn(make_float2(wx(e), wx(e + 1)), make_float2(y[0][e], y[0][e + 1]), s);
            syx = s.x + s.y;
            if constexpr (OWN) {
                float2 n2 = make_float2(0.f, 0.f);
#pragma unroll
                for (int e = 0; e < V; e += 2)
                    n2 = __ffma2_rn(make_float2(wx(e), wx(e + 1)), make_float2(x[e], x[e + 1]), n2);
                sxx = n2.x + n2.y;
            }
        }
        a_ = (sxx == 0.f) ? 0.f : divide(syx, sxx);
        auto d2 = [&](int e) { return make_float2(fmaf(-a_, x[e], y[0][e]), fmaf(-a_, x[e + 1], y[0][e + 1])); };
        auto wd2 = [&](int e, float2 d) { return UW ? d : make_float2(w(0, e) * d.x, w(0, e + 1) * d.y); };
        if constexpr (COMP) {
            const Comp2 v = comp2_chain<V / 2>([&](int k) {
                const float2 d = d2(2 * k);
                return __fmul2_rn(wd2(2 * k, d), d);
            });
            ls_ = comp_total<1>(v, mask);
        } else {
            const float2 na = make_float2(-a_, -a_);
            float2 s = make_float2(0.f, 0.f);
#pragma unroll
            for (int e = 0; e < V; e += 2) {
                const float2 d = __ffma2_rn(na, make_float2(x[e], x[e + 1]), make_float2(y[0][e], y[0][e + 1]));
                s = __ffma2_rn(wd2(e, d), d, s);
            }
            ls_ = s.x + s.y;
        }
    } else {
        float syx, sxx = nr;
        // products w x y of component e of the pair's two pieces
        auto xy = [&](const C (&x0)[V], const C (&x1)[V], int q, int e) {
            return make_float2(__fmul_rn(UW ? x0[e] : w(q, e) * x0[e], y[q][e]),
                               __fmul_rn(UW ? x1[e] : w(q + 1, e) * x1[e], y[q + 1][e]));
        };
        if constexpr (COMP) {
            auto leaf = [&](int t) {
                C x0[V], x1[V];
                S::unpack(raw[2 * t], x0);
                S::unpack(raw[2 * t + 1], x1);
                return comp2_chain<V>([&](int e) { return xy(x0, x1, 2 * t, e); });
            };
            auto join = [](const Comp2 &a, const Comp2 &b) { return comp2_join(a, b); };
            syx = comp_total<G>(tree_sum<0, 1, NP / 2>(leaf, join), mask);
        } else {
            // piece q's part of S_yx, or of S_xx
            auto piece = [&](int q, bool norm) {
                C x[V];
                S::unpack(raw[q], x);
                float2 s = make_float2(0.f, 0.f);
#pragma unroll
                for (int e = 0; e < V; e += 2)
                    s = __ffma2_rn(UW ? make_float2(x[e], x[e + 1]) : make_float2(w(q, e) * x[e], w(q, e + 1) * x[e + 1]),
                                   norm ? make_float2(x[e], x[e + 1]) : make_float2(y[q][e], y[q][e + 1]), s);
                return s.x + s.y;
            };
            auto join = [](float2 a, float2 b) { return __fadd2_rn(a, b); };
            auto leaf = [&](int t) { return make_float2(piece(2 * t, false), piece(2 * t + 1, false)); };
            syx = plain_total<G>(tree_sum<0, 1, NP / 2>(leaf, join), mask);
            if constexpr (OWN) {
                auto nleaf = [&](int t) { return make_float2(piece(2 * t, true), piece(2 * t + 1, true)); };
                sxx = plain_total<G>(tree_sum<0, 1, NP / 2>(nleaf, join), mask);
            }
        }
        a_ = (sxx == 0.f) ? 0.f : divide(syx, sxx);
        // residuals of component e of a pair's two pieces, times the weights
        auto terms = [&](int t, float2 (&d)[V], float2 (&wd)[V]) {
            C x0[V], x1[V];
            S::unpack(raw[2 * t], x0);
            S::unpack(raw[2 * t + 1], x1);
#pragma unroll
            for (int e = 0; e < V; ++e) {
                d[e] = make_float2(fmaf(-a_, x0[e], y[2 * t][e]), fmaf(-a_, x1[e], y[2 * t + 1][e]));
                wd[e] = UW ? d[e] : make_float2(w(2 * t, e) * d[e].x, w(2 * t + 1, e) * d[e].y);
            }
        };
        if constexpr (COMP) {
            // even and odd components of a piece are separate chains
            auto leaf = [&](int t) {
                float2 d[V], wd[V];
                terms(t, d, wd);
                const Comp2 even = comp2_chain<V / 2>([&](int k) { return __fmul2_rn(wd[2 * k], d[2 * k]); });
                const Comp2 odd = comp2_chain<V / 2>([&](int k) { return __fmul2_rn(wd[2 * k + 1], d[2 * k + 1]); });
                return comp2_join(even, odd);
            };
            auto join = [](const Comp2 &a, const Comp2 &b) { return comp2_join(a, b); };
            ls_ = comp_total<G>(tree_sum<0, 1, NP / 2>(leaf, join), mask);
        } else {
            const float2 na = make_float2(-a_, -a_);
            auto piece = [&](int q) {
                C x[V];
                S::unpack(raw[q], x);
                float2 s = make_float2(0.f, 0.f);
#pragma unroll
                for (int e = 0; e < V; e += 2) {
                    const float2 d = __ffma2_rn(na, make_float2(x[e], x[e + 1]), make_float2(y[q][e], y[q][e + 1]));
                    s = __ffma2_rn(UW ? d : make_float2(w(q, e) * d.x, w(q, e + 1) * d.y), d, s);
                }
                return s.x + s.y;
            };
            auto leaf = [&](int t) { return make_float2(piece(2 * t), piece(2 * t + 1)); };
            auto join = [](float2 a, float2 b) { return __fadd2_rn(a, b); };
            ls_ = plain_total<G>(tree_sum<0, 1, NP / 2>(leaf, join), mask);
        }
    }
}

// ---------------------------------------------------------------------------
// G lanes per row, a block per run of consecutive rows.  The block's stored
// entries are one contiguous run of slots: their gather indices and values
// come into shared memory with coalesced loads, the fits replace them there
// (a over the values; LS over the indices where the sizes agree), and a, LS
// and the flags leave with coalesced stores.  A block whose run exceeds `cap`
// slots works on global memory directly.  The neighbour row of the next entry
// is in flight while an entry is fitted.
//
// Bound: the FP32 pipe on the compensated mixed paths (8 FP32 operations per
// component for S_yx and 9 for LS), the FP64 pipe on FP64 (3K + 7 operations
// per entry at two per clock and SM).  Few lanes per row keep y_i in registers
// for all its entries and spend little on reductions; a lane per entry (y_i
// from shared memory, row minima by shuffles) issued twice the instructions.
//
// Lanes per row, entries in flight and resident blocks (measured, us per pass,
// K = 16 FP32 9-point 1024^2 / K = 32 FP32 7-point 128^3): a share of 16
// components per lane 174 / 623, of 8 281 / 897 (the joins across lanes), of 32
// - / 699 (a 32-byte load of a lane is an L1 wavefront of its own unless its
// neighbours read the same 128-byte line).  One entry at a time with seven
// resident blocks beats two with five (193 / 689) and a double-buffered one
// with four (204 / 784): warps hide the gathers better than registers do.
// BF16 rows of 64 bytes and more keep 32 components per lane (7-point 96^3,
// K = 32: 231 against 268).  FP64 is at 70-80 % of its pipe whatever the shape.
// Before (G = P lanes per row, S_xx per entry) the two workloads took 193 (with
// the best shape) and 1331 us (752 with the best), K = 13 FP64 7-point 333^2
// 385 (150 now), 25 entries per row of BF16 K = 16 (512^2) 236 (92 now).
//
// Plain sums are half the arithmetic and bound by the gathers: they form S_xx from the
// row at hand rather than read the vectors once more for it and gather the norms, and
// run in more and smaller blocks.  us, in the compensated sums' layout -> in this one /
// in the former row kernel's tuned shapes: 9-point 1024^2 K = 16 FP32 169 -> 147 / 149,
// BF16 143 -> 117 / 120, K = 32 FP32 313 -> 287 / 268; 7-point 128^3 K = 32 FP32
// 575 -> 484 / 460, K = 16 298 -> 249 / 234; 300k-row graph K = 16 FP32 187 -> 148 / 172.
// Two entries at a time lose as above (152 -> 170).
// ---------------------------------------------------------------------------
template <class TS, int P, bool COMP>
struct FitLayout {
    using C = typename Store<TS>::C;
    static constexpr int V = Store<TS>::V, KP = P * V;
    static constexpr int CL = sizeof(TS) == 2 ? 32 : 16;               // components per lane
    static constexpr int G = KP <= CL ? 1 : KP / CL;
    static constexpr int NP = P / G;
    static constexpr int U = sizeof(TS) == 8 && NP <= 4 ? 4 : 1;      // entries gathered at a time
    // plain FP32 sums form S_xx with the fit, in blocks of 64 threads (not with 32
    // components a lane: BF16 K = 32, 2M-row graph 1212 us with the norms pass, 1417
    // without; 9-point 1024^2 192 / 199, 7-point 128^3 372 / 370)
    static constexpr bool OWN = !COMP && sizeof(TS) < 8 && NP * V <= 16;
    static constexpr int THREADS = OWN ? 64 : kFitThreads;
    // uneven rows may be taken by length (go_fit; FP32 of K = 16 has the form for its shared
    // memory alone: without those 384 bytes a 2M-row graph took 1356 us instead of 1212)
    static constexpr bool SORTS = sizeof(TS) == 8 || KP >= 16;
    // resident blocks (of kFitThreads); as many as spill nothing, and leave the gathers
    // some L1 beside the slots (plain sums with 8 for K = 16 FP32: 2M-row graph 967 ->
    // 1783 us)
    static constexpr int MINB = sizeof(TS) == 8 ? 4
                              : OWN ? (NP == 1 ? 8 : 7)
                              : sizeof(TS) == 4 ? 7 : NP * V <= 16 ? 6 : 5;
    static constexpr int WB = KP * (int)sizeof(C);                    // weights of the block
    static constexpr bool LS_OVER = sizeof(C) == 4;                    // LS replaces the gather index
    static constexpr int SLOT = 4 + (LS_OVER ? 1 : 2) * (int)sizeof(C) + 1;
    static constexpr int UT = NP <= 2 || (sizeof(TS) == 8 && NP <= 4) ? 4 : (NP <= 4 ? 2 : 1);   // and in the target
    static int bytes(int cap, bool unit_w, int shared_rows)           // of a block (shared_rows: with several shares)
    {
        return (unit_w ? 0 : WB) + shared_rows * KP * (int)sizeof(C) + cap * SLOT;
    }
    static_assert(NP == 1 ? G == 1 : NP % 2 == 0, "pairs of pieces");
};

// SHARED: several shares per row (el of them; else one).  Every lane of the row then
// forms the target of pieces of its own, and y_i reaches the others by shared memory
// (20000 rows of 70 entries, K = 16 FP64, four shares: 215 us, 420 with the whole
// target in each).
template <class TS, int P, bool UW, bool PX, bool COMP, bool SHARED>
__global__ void __launch_bounds__(kFitThreads, FitLayout<TS, P, COMP>::MINB) k_edge_fit(EdgeArgs A, int cap, int shares)
{
    using S = Store<TS>;
    using C = typename S::C;
    using AV = typename S::A;
    using L = FitLayout<TS, P, COMP>;
    constexpr int V = S::V, KP = L::KP, G = L::G, NP = L::NP, UT = L::UT, U = L::U;
    constexpr bool kMixed = !std::is_same<C, double>::value;
    extern __shared__ __align__(16) unsigned char esm[];
    const int T = blockDim.x, tid = threadIdx.x;
    // el shares of a row's entries, G lanes each; gmask: the lanes of a share,
    // rmask: of the row
    const int el = SHARED ? shares : 1;
    const int gl = tid % G, sub = tid / G % el, width = G * el;
    const unsigned gmask = G == 1 ? 1u << (tid % 32) : ((1u << G) - 1u) << ((tid % 32) / G * G);
    const unsigned rmask = width == 32 ? 0xffffffffu : ((1u << width) - 1u) << ((tid % 32) / width * width);
    const int rows = T / width;
    C *ws = reinterpret_cast<C *>(esm);                              // weights (UW: none)
    C *ys = reinterpret_cast<C *>(esm + (UW ? 0 : L::WB));            // targets (SHARED)
    C *a_s = ys + (SHARED ? rows * KP : 0);                          // values, then a
    C *lsep = a_s + cap;                                             // LS where it has its own place
    int32_t *x_s = reinterpret_cast<int32_t *>(L::LS_OVER ? lsep : lsep + cap);   // gather indices
    C *ls_s = L::LS_OVER ? reinterpret_cast<C *>(x_s) : lsep;
    uint8_t *fl_s = reinterpret_cast<uint8_t *>(x_s + cap);

    const int np = G == 1 ? (A.K + V - 1) / V : NP;                   // pieces that are not all padding
    const int64_t R0 = (int64_t)blockIdx.x * rows;
    const int nr = (int)min((int64_t)rows, A.n - R0);
    const int S0 = __ldg(A.prp + R0), S1 = __ldg(A.prp + R0 + nr);
    const bool staged = S1 - S0 <= cap;
    const int32_t *__restrict__ xcol = PX ? A.xcol : A.col;          // gather index of A's slots
    const int32_t *__restrict__ fcol = PX ? A.xcol : A.pcol;         // and of the fits' slots
    const AV *val = (const AV *)A.val;
    const TS *X = (const TS *)A.x;
    C *a_out = (C *)A.a_out;
    C *ls_out = (C *)A.ls_out;
    if (staged)
        for (int q = tid; q < S1 - S0; q += T) x_s[q] = __ldg(fcol + S0 + q);
    chain_wait();
    chain_release();
    if constexpr (!UW)
        for (int k = tid; k < KP; k += T) ws[k] = ((const C *)A.w)[k];
    if (PX && staged)                                                // d = 1: the fits' slots are A's
        for (int q = tid; q < S1 - S0; q += T) a_s[q] = (C)ld_plain(val + S0 + q);
    __syncthreads();

    // uneven rows in the order of their lengths, so that the rows of a warp take as
    // long (launch: A.uneven)
    int place = min(tid / width, nr - 1);
    if (L::SORTS && A.uneven) {
        __shared__ int bin[64];
        __shared__ uint8_t order[kFitThreads];
        for (int b = tid; b < 64; b += T) bin[b] = 0;
        __syncthreads();
        const bool one = tid < nr;                                    // (a block has at most T rows)
        int key = 0, at = 0;
        if (one) {
            key = 63 - min(63, __ldg(A.prp + R0 + tid + 1) - __ldg(A.prp + R0 + tid));
            at = atomicAdd(&bin[key], 1);
        }
        __syncthreads();
        if (tid < 32) {
            const int b0 = bin[2 * tid], b1 = bin[2 * tid + 1];
            int s = b0 + b1;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, s, o);
                if (tid >= o) s += v;
            }
            bin[2 * tid] = s - b0 - b1;
            bin[2 * tid + 1] = s - b1;
        }
        __syncthreads();
        if (one) order[bin[key] + at] = (uint8_t)tid;
        __syncthreads();
        place = order[place];
    }
    if (tid / width < nr) {
        const int64_t r = R0 + place;
        const int q0 = __ldg(A.prp + r);
        int q1 = __ldg(A.prp + r + 1);
        const int p0 = PX ? q0 : __ldg(A.rp + r);
        int p1 = PX ? q1 : __ldg(A.rp + r + 1);
        // k_edge_long fits the longer rows.  (No branch: what follows is requested without
        // waiting for the row pointers; 7-point 128^3, K = 4 FP32 195 -> 170 us.)
        if (q1 - q0 > A.long_len) {
            q1 = q0;
            p1 = p0;
        }
        const int64_t xr = (PX && A.xrow) ? checked_row(__ldg(A.xrow + r), A.n, A.status) : r;
        const C diag = (C)ld_plain((const AV *)A.diag + r);
        auto gather = [&](int64_t j, uint4 (&raw)[NP]) {
            const TS *src = X + checked_row(j, A.n, A.status) * KP;
            if constexpr (NP == 1) {
                raw[0] = ld16(src);
            } else {
#pragma unroll
                for (int q = 0; q < NP; q += 2) ld32(src + fit_piece<G, NP>(gl, q) * V, raw[q], raw[q + 1]);
            }
        };
        auto w = [&](int q, int e) { return UW ? C(1) : ws[fit_piece<G, NP>(gl, q) * V + e]; };

        // ---- 1. target ------------------------------------------------------------
        C y[NP][V];
        float syy = 0.f;
        int j1 = -1;                 // exact rule: the row's one off-diagonal (gather index)
        C a1 = C(0);
        if constexpr (SHARED) {
            constexpr int US = 5;                                    // entries in flight
            C *yr = ys + tid / width * KP;
            const C d = C(1) / diag;
            for (int t = tid % width; t < (G == 1 ? np : P); t += width) {
                Acc<C, V> acc;
                acc.zero();
                if (A.target == 0) {
                    for (int pb = p0; pb < p1; pb += US) {
                        uint4 raw[US];
                        C vv[US];
#pragma unroll
                        for (int u = 0; u < US; ++u) {
                            const int p = pb + u;
                            if (p >= p1) break;
                            const int64_t j = PX && staged ? x_s[p - S0] : __ldg(xcol + p);
                            vv[u] = PX && staged ? a_s[p - S0] : (C)ld_plain(val + p);
                            raw[u] = ld16(X + checked_row(j, A.n, A.status) * KP + t * V);
                        }
#pragma unroll
                        for (int u = 0; u < US; ++u) {
                            if (pb + u >= p1) break;
                            C x[V];
                            S::unpack(raw[u], x);
                            acc.fma_piece(vv[u], x);
                        }
                    }
                }
                C xi[V];
                S::unpack(ld16(X + xr * KP + t * V), xi);
#pragma unroll
                for (int e = 0; e < V; ++e) yr[t * V + e] = A.target == 0 ? fma(-d, acc.get(e), xi[e]) : xi[e];
            }
            __syncwarp(rmask);
#pragma unroll
            for (int q = 0; q < NP; ++q)
#pragma unroll
                for (int e = 0; e < V; ++e) y[q][e] = yr[fit_piece<G, NP>(gl, q) * V + e];
        } else {
            Acc<C, V> acc[NP];
#pragma unroll
            for (int t = 0; t < NP; ++t) acc[t].zero();
            if (A.target == 0) {
                for (int pb = p0; pb < p1; pb += UT) {
                    int jj[UT];
                    C vv[UT];
#pragma unroll
                    for (int u = 0; u < UT; ++u) {
                        const int p = pb + u;
                        const bool ok = p < p1;
                        if (PX && staged) {
                            jj[u] = ok ? x_s[p - S0] : -1;
                            vv[u] = ok ? a_s[p - S0] : C(0);
                        } else {
                            jj[u] = ok ? __ldg(xcol + p) : -1;
                            vv[u] = ok ? (C)ld_plain(val + p) : C(0);
                        }
                    }
                    uint4 raw[UT][NP];
#pragma unroll
                    for (int u = 0; u < UT; ++u)
                        if (jj[u] >= 0) gather(jj[u], raw[u]);
#pragma unroll
                    for (int u = 0; u < UT; ++u) {
                        if (jj[u] < 0) break;
#pragma unroll
                        for (int t = 0; t < NP; ++t) {
                            if (sizeof(C) == 8 && t >= np) break;
                            C x[V];
                            S::unpack(raw[u][t], x);
                            acc[t].fma_piece(vv[u], x);
                        }
                    }
                }
            }
            uint4 own[NP];
            gather(xr, own);
            const C d = C(1) / diag;
#pragma unroll
            for (int t = 0; t < NP; ++t) {
                S::unpack(own[t], y[t]);
                if (A.target == 0) {
#pragma unroll
                    for (int e = 0; e < V; ++e) y[t][e] = fma(-d, acc[t].get(e), y[t][e]);
                }
            }
        }
        {
            if constexpr (kMixed) {
                // S_yy, in the order of the other sums
                auto piece = [&](int q) {
                    float s = 0.f;
#pragma unroll
                    for (int e = 0; e < V; ++e) s = fmaf(UW ? y[q][e] : w(q, e) * y[q][e], y[q][e], s);
                    return s;
                };
                if constexpr (NP == 1) {
                    syy = piece(0);
                } else {
                    auto leaf = [&](int t) { return make_float2(piece(2 * t), piece(2 * t + 1)); };
                    auto join = [](float2 a, float2 b) { return __fadd2_rn(a, b); };
                    syy = plain_total<G>(tree_sum<0, 1, NP / 2>(leaf, join), gmask);
                }
            }
            if (A.target == 0 && p1 - p0 == 2) {
                // one off-diagonal j1: y_i is exactly -(a_ij1 / a_ii) x_j1
                const int pj = __ldg(xcol + p0) == xr ? p0 + 1 : p0;
                j1 = __ldg(xcol + pj);
                a1 = -(C)ld_plain(val + pj) / diag;
            }
        }
        if constexpr (G > 1 || SHARED) __syncwarp(rmask);   // the row's values and indices are read out

        // ---- 2. one-point fits ------------------------------------------------------
        C m = C(INFINITY);
        bool defer = false;          // a fit of this row cancelled in FP32: redo the row in FP64
        for (int pb = q0 + sub; pb < q1; pb += U * el) {
            int jj[U];
            uint4 raw[U][NP];
            typename Norm<C>::T nr_j[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int p = pb + u * el;
                jj[u] = p < q1 ? (staged ? x_s[p - S0] : __ldg(fcol + p)) : -1;
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (jj[u] < 0 || jj[u] == xr) continue;
                if constexpr (!L::OWN) nr_j[u] = ld_plain((const typename Norm<C>::T *)A.norms + checked_row(jj[u], A.n, A.status));
                gather(jj[u], raw[u]);
            }
            if constexpr (G > 1) __syncwarp(gmask);      // every lane has read these entries' indices
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (jj[u] < 0) break;
                const int p = pb + u * el;
                C a_ = C(0), ls_ = C(NAN);
                if (jj[u] == xr) {
                } else if (jj[u] == j1) {
                    a_ = a1;
                    ls_ = C(0);
                    m = fmin(m, ls_);
                } else {
                    fit_entry<TS, G, NP, UW, COMP, L::OWN>(raw[u], y, w, nr_j[u], np, gmask, a_, ls_);
                    m = fmin(m, ls_);
                    if constexpr (kMixed) defer = defer || ls_ < C(1e-4) * syy;
                }
                if (gl == 0) {
                    if (staged) { a_s[p - S0] = a_; ls_s[p - S0] = ls_; }
                    else { a_out[p] = a_; ls_out[p] = ls_; }
                }
            }
        }
        // the shares' minima and marks joined; every lane's stores are visible to the row's
        if constexpr (G > 1 || SHARED) __syncwarp(rmask);
        if constexpr (SHARED) {
            for (int o = G; o < width; o <<= 1) m = fmin(m, __shfl_xor_sync(rmask, m, o));
            if constexpr (kMixed) defer = __any_sync(rmask, defer);
        }

        // ---- 3. strength flags (Eq. (4.4) in LS form) and counts --------------------
        const C theta = (C)A.theta;
        int cnt = 0;
        for (int p = q0 + tid % width; p < q1; p += width) {
            const C l = staged ? ls_s[p - S0] : ls_out[p];            // NaN on the diagonal
            const bool strong = l == C(0) || theta * l < m;
            if (staged) fl_s[p - S0] = (uint8_t)strong;
            else A.flag_out[p] = (uint8_t)strong;
            cnt += strong;
        }
        for (int o = 1; o < width; o <<= 1) cnt += __shfl_xor_sync(rmask, cnt, o);
        if (tid % width == 0) {
            A.count_out[r] = cnt;
            if (kMixed && defer) A.defer_list[atomicAdd(A.defer_count, 1u)] = (int32_t)r;
        }
    }
    if (staged) {
        __syncthreads();
        for (int q = tid; q < S1 - S0; q += T) {
            a_out[S0 + q] = a_s[q];
            ls_out[S0 + q] = ls_s[q];
            A.flag_out[S0 + q] = fl_s[q];
        }
    }
}

// ---------------------------------------------------------------------------
// Rows of more than A.long_len entries, one block each; same fits, same order
// of every sum as k_edge_fit.  The target is a chain over the row's entries per
// component (the sweeps' rounding): tiles of neighbour rows land in shared
// memory with cp.async, one ahead, and one thread per component walks them.
// Then every G lanes fit entries of their own.  Bound: latency, of a tile per 1 us for
// the target and of a gather per 256 / G entries for the fits (a graph of 200k rows,
// K = 16, with one row of 30000: FP32 418 us, 20302 with that row in one lane;
// FP64 2524 / 78537).
// ---------------------------------------------------------------------------
constexpr int kLongThreads = 256;

template <class TS, int P>
struct LongLayout {
    static constexpr int V = Store<TS>::V, KP = P * V;
    static constexpr int TILE = P <= 2 ? 512 : 1024 / P;             // neighbour rows per tile
    static constexpr int PPT = TILE * P / kLongThreads;               // 16-byte pieces per thread and tile
    static_assert(TILE * P % kLongThreads == 0, "whole pieces per thread");
};

// component k of a stored row
template <class TS>
__device__ __forceinline__ typename Store<TS>::C component(const TS *x, int k)
{
    if constexpr (std::is_same<TS, __nv_bfloat16>::value) return __bfloat162float(x[k]);
    else return x[k];
}

template <class TS, int P, bool UW, bool PX, bool COMP>
__global__ void __launch_bounds__(kLongThreads) k_edge_long(EdgeArgs A)
{
    using S = Store<TS>;
    using C = typename S::C;
    using AV = typename S::A;
    using L = FitLayout<TS, P, COMP>;
    using LL = LongLayout<TS, P>;
    constexpr int V = S::V, KP = L::KP, G = L::G, NP = L::NP, TILE = LL::TILE, PPT = LL::PPT, W = kLongThreads / 32;
    constexpr bool kMixed = !std::is_same<C, double>::value;
    __shared__ __align__(16) uint4 xs[2][TILE * P];                   // neighbour rows
    __shared__ C vs[2][TILE];                                         // and the row's values
    __shared__ C ys[KP], wsm[UW ? 1 : KP];
    __shared__ C msm[W];
    __shared__ int csm[W];
    const int tid = threadIdx.x, gl = tid % G;
    const unsigned gmask = G == 1 ? 1u << (tid % 32) : ((1u << G) - 1u) << ((tid % 32) / G * G);
    const int np = G == 1 ? (A.K + V - 1) / V : NP;
    const int32_t *__restrict__ xcol = PX ? A.xcol : A.col;
    const int32_t *__restrict__ fcol = PX ? A.xcol : A.pcol;
    const AV *val = (const AV *)A.val;
    const TS *X = (const TS *)A.x;
    C *a_out = (C *)A.a_out;
    C *ls_out = (C *)A.ls_out;
    chain_wait();
    chain_release();
    if constexpr (!UW)
        for (int k = tid; k < KP; k += kLongThreads) wsm[k] = ((const C *)A.w)[k];
    for (int li = blockIdx.x; li < A.n_long; li += gridDim.x) {
        const int64_t r = A.long_rows[li];
        const int q0 = __ldg(A.prp + r), q1 = __ldg(A.prp + r + 1);
        const int p0 = PX ? q0 : __ldg(A.rp + r), p1 = PX ? q1 : __ldg(A.rp + r + 1);
        const int64_t xr = (PX && A.xrow) ? checked_row(__ldg(A.xrow + r), A.n, A.status) : r;
        const C diag = (C)ld_plain((const AV *)A.diag + r);

        // ---- 1. target ------------------------------------------------------------
        C acc = C(0);
        if (A.target == 0) {
            int jj[PPT];                                              // rows of this thread's pieces of a tile
            auto indices = [&](int pb) {
#pragma unroll
                for (int u = 0; u < PPT; ++u) {
                    const int p = pb + (tid + u * kLongThreads) / P;
                    jj[u] = p < p1 ? __ldg(xcol + p) : -1;
                }
            };
            auto copy = [&](int pb, int b) {
#pragma unroll
                for (int u = 0; u < PPT; ++u) {
                    const int q = tid + u * kLongThreads;
                    if (jj[u] >= 0) cp_async16(&xs[b][q], X + checked_row(jj[u], A.n, A.status) * KP + q % P * V);
                }
                cp_async_commit();
                for (int q = tid; q < TILE && pb + q < p1; q += kLongThreads) vs[b][q] = (C)ld_plain(val + pb + q);
            };
            indices(p0);
            copy(p0, 0);
            indices(p0 + TILE);
            for (int pb = p0, b = 0; pb < p1; pb += TILE, b ^= 1) {
                if (pb + TILE < p1) {
                    copy(pb + TILE, b ^ 1);
                    indices(pb + 2 * TILE);
                    cp_async_wait<1>();
                } else {
                    cp_async_wait<0>();
                }
                __syncthreads();                                      // the tile is in place
                if (tid < KP) {
                    const TS *x = (const TS *)xs[b] + tid;
                    const int m = min(TILE, p1 - pb);
#pragma unroll 8
                    for (int q = 0; q < m; ++q) acc = fma(vs[b][q], component<TS>(x, q * KP), acc);
                }
                __syncthreads();                                      // and read out
            }
        }
        const C d = C(1) / diag;
        if (tid < KP) {
            const C xi = component<TS>(X + xr * KP, tid);
            ys[tid] = A.target == 0 ? fma(-d, acc, xi) : xi;
        }
        int j1 = -1;                                                  // (search depth > 1: a short row of A)
        C a1 = C(0);
        if (A.target == 0 && p1 - p0 == 2) {
            const int pj = __ldg(xcol + p0) == xr ? p0 + 1 : p0;
            j1 = __ldg(xcol + pj);
            a1 = -(C)ld_plain(val + pj) / diag;
        }
        __syncthreads();
        C y[NP][V];
        auto w = [&](int q, int e) { return UW ? C(1) : wsm[fit_piece<G, NP>(gl, q) * V + e]; };
#pragma unroll
        for (int q = 0; q < NP; ++q)
#pragma unroll
            for (int e = 0; e < V; ++e) y[q][e] = ys[fit_piece<G, NP>(gl, q) * V + e];
        float syy = 0.f;
        if constexpr (kMixed) {
            auto piece = [&](int q) {
                float s = 0.f;
#pragma unroll
                for (int e = 0; e < V; ++e) s = fmaf(UW ? y[q][e] : w(q, e) * y[q][e], y[q][e], s);
                return s;
            };
            if constexpr (NP == 1) {
                syy = piece(0);
            } else {
                auto leaf = [&](int t) { return make_float2(piece(2 * t), piece(2 * t + 1)); };
                auto join = [](float2 a, float2 b) { return __fadd2_rn(a, b); };
                syy = plain_total<G>(tree_sum<0, 1, NP / 2>(leaf, join), gmask);
            }
        }

        // ---- 2. one-point fits, G lanes per entry ------------------------------------
        C m = C(INFINITY);
        bool defer = false;
        int j = q0 + tid / G < q1 ? __ldg(fcol + q0 + tid / G) : -1;
        for (int p = q0 + tid / G; p < q1; p += kLongThreads / G) {
            const int jn = p + kLongThreads / G < q1 ? __ldg(fcol + p + kLongThreads / G) : -1;
            C a_ = C(0), ls_ = C(NAN);
            if (j == xr) {
            } else if (j == j1) {
                a_ = a1;
                ls_ = C(0);
                m = fmin(m, ls_);
            } else {
                const int64_t row = checked_row(j, A.n, A.status);
                typename Norm<C>::T nr = {};
                if constexpr (!L::OWN) nr = ld_plain((const typename Norm<C>::T *)A.norms + row);
                uint4 raw[NP];
                if constexpr (NP == 1) {
                    raw[0] = ld16(X + row * KP);
                } else {
#pragma unroll
                    for (int q = 0; q < NP; q += 2) ld32(X + row * KP + fit_piece<G, NP>(gl, q) * V, raw[q], raw[q + 1]);
                }
                fit_entry<TS, G, NP, UW, COMP, L::OWN>(raw, y, w, nr, np, gmask, a_, ls_);
                m = fmin(m, ls_);
                if constexpr (kMixed) defer = defer || ls_ < C(1e-4) * syy;
            }
            if (gl == 0) { a_out[p] = a_; ls_out[p] = ls_; }
            j = jn;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = fmin(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (tid % 32 == 0) msm[tid / 32] = m;
        if constexpr (kMixed) defer = __syncthreads_or(defer);
        else __syncthreads();
#pragma unroll
        for (int k = 0; k < W; ++k) m = fmin(m, msm[k]);

        // ---- 3. strength flags and counts --------------------------------------------
        const C theta = (C)A.theta;
        int cnt = 0;
        for (int p = q0 + tid; p < q1; p += kLongThreads) {
            const C l = ls_out[p];                                    // NaN on the diagonal
            const bool strong = l == C(0) || theta * l < m;
            A.flag_out[p] = (uint8_t)strong;
            cnt += strong;
        }
        cnt = __reduce_add_sync(0xffffffffu, cnt);
        if (tid % 32 == 0) csm[tid / 32] = cnt;
        __syncthreads();
        if (tid == 0) {
            int total = 0;
            for (int k = 0; k < W; ++k) total += csm[k];
            A.count_out[r] = total;
            if (kMixed && defer) A.defer_list[atomicAdd(A.defer_count, 1u)] = (int32_t)r;
        }
    }
}

// Mixed paths: rows listed by k_edge_fit (a fit cancelled in FP32, LS < 1e-4
// S_yy) are recomputed here entirely in FP64 from the stored vectors (widened
// exactly) and the FP64 values of A: target with the FP64 path's rounding,
// every one-point fit, the row minimum, flags and count.  One warp per row:
// lanes over the components for the target (two per lane for K > 32), then one
// stored entry per lane for the fits, the K-term sums in the order of a
// butterfly over 32 lanes that hold a component each.  Bound: the FP64 pipe
// (a fit in one lane is 7K FP64 operations; the lanes of a butterfly would
// repeat every addition).
template <class TS>
__device__ __forceinline__ double elem64(const TS *p)
{
    if constexpr (std::is_same<TS, __nv_bfloat16>::value)
        return (double)__bfloat162float(*p);
    else
        return (double)*p;
}

constexpr int kFixThreads = 256;

template <class TS, int P, bool PX>
__global__ void __launch_bounds__(kFixThreads) k_edge_fixup(EdgeArgs A)
{
    using C = typename Store<TS>::C;
    constexpr int KP = P * Store<TS>::V;
    constexpr int LEAVES = KP < 32 ? KP : 32;
    __shared__ double ysm[kFixThreads / 32][KP], wsm[KP];
    chain_wait();
    chain_release();
    const unsigned count = *A.defer_count;
    const int lane = threadIdx.x % 32;
    double *ys = ysm[threadIdx.x / 32];
    const TS *X = (const TS *)A.x;
    if ((unsigned)blockIdx.x * (kFixThreads / 32) >= count) return;
    for (int k = threadIdx.x; k < KP; k += kFixThreads) wsm[k] = A.w64[k];
    __syncthreads();
    // vector row of caller row i (in place: the sweeps' row order; search
    // depth 1, so the fit slots are A's slots)
    auto xrow = [&](int64_t i) -> int64_t { return (PX && A.xrow) ? checked_row(A.xrow[i], A.n, A.status) : i; };
    const int64_t warps = (int64_t)gridDim.x * (kFixThreads / 32);
    for (int64_t q = (int64_t)blockIdx.x * (kFixThreads / 32) + threadIdx.x / 32; q < count; q += warps) {
        const int64_t r = A.defer_list[q];
        const int p0 = A.rp[r], p1 = A.rp[r + 1];         // row of A: target
        const int q0 = A.prp[r], q1 = A.prp[r + 1];       // entries of the fits
        double diag = 1.0;
        int j1 = -1;
        double v1 = 0.0;
        double acc[2] = {0.0, 0.0};
        for (int pb = p0; pb < p1; pb += 4) {
            // four entries' gathers in flight
            double v[4], x[4][2];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (pb + u >= p1) break;
                const int p = pb + u;
                v[u] = A.val64[p];
                if (A.col[p] == r) diag = v[u];
                else if (A.target == 0 && p1 - p0 == 2) { j1 = A.col[p]; v1 = v[u]; }
                const TS *src = X + checked_row(PX ? A.xcol[p] : A.col[p], A.n, A.status) * KP;
#pragma unroll
                for (int h = 0; h < 2; ++h) x[u][h] = lane + 32 * h < KP ? elem64(src + lane + 32 * h) : 0.0;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (pb + u >= p1) break;
#pragma unroll
                for (int h = 0; h < 2; ++h) acc[h] = fma(v[u], x[u][h], acc[h]);
            }
        }
        const double d = 1.0 / diag;
        __syncwarp();                                     // the last row's targets are read out
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int k = lane + 32 * h;
            if (k >= KP) break;
            const double xi = elem64(X + xrow(r) * KP + k);
            ys[k] = (A.target == 0) ? fma(-d, acc[h], xi) : xi;
        }
        __syncwarp();
        double m = INFINITY;
        C *a_out = (C *)A.a_out;
        C *ls_out = (C *)A.ls_out;
        for (int p = q0 + lane; p < q1; p += 32) {
            const int64_t j = A.pcol[p];
            double a64, ls64;
            if (j == r) {
                a64 = 0.0;
                ls64 = NAN;
            } else if (j == j1) {
                a64 = -v1 / diag;
                ls64 = 0.0;
            } else {
                const TS *xj = X + checked_row(PX ? (int64_t)A.xcol[p] : j, A.n, A.status) * KP;
                auto add = [](double a, double b) { return a + b; };
                // component l of the sum (and l + 32 for K > 32): f(w, x, y)
                auto over = [&](auto f) {
                    auto leaf = [&](int l) {
                        double s = f(0.0, wsm[l], elem64(xj + l), ys[l]);
                        if constexpr (KP > 32) s = f(s, wsm[l + 32], elem64(xj + l + 32), ys[l + 32]);
                        return s;
                    };
                    return tree_sum<0, 1, LEAVES>(leaf, add);
                };
                const double sxx = over([](double s, double w, double x, double) { return fma(w * x, x, s); });
                const double syx = over([](double s, double w, double x, double y) { return fma(w * x, y, s); });
                a64 = (sxx == 0.0) ? 0.0 : syx / sxx;
                ls64 = over([&](double s, double w, double x, double y) {
                    const double e = fma(-a64, x, y);
                    return fma(w * e, e, s);
                });
            }
            if (j != r) m = fmin(m, ls64);
            a_out[p] = (C)a64;
            ls_out[p] = (C)ls64;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = fmin(m, __shfl_xor_sync(0xffffffffu, m, o));
        int cnt = 0;
        for (int p = q0 + lane; p < q1; p += 32) {
            const double l = (double)ls_out[p];
            const int strong = (A.pcol[p] != r) && (l == 0.0 || A.theta * l < m);
            A.flag_out[p] = (uint8_t)strong;
            cnt += strong;
        }
        for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
        if (lane == 0) A.count_out[r] = cnt;
    }
}

// Shares of a row's entries and threads of a block.  A small matrix leaves most
// of the chip idle at one lane group per row, and the pass is then the latency
// of a row's entries one after the other: up to four shares, more for rows of more
// than eight entries a share, while the lanes fit in two warps per scheduler, and
// blocks of down to 32 threads while there are fewer than four per SM (64 x 64
// 5-point, K = 8, FP64: 12.9 us with one share, 8.7 with four; 2000 rows of 200,
// K = 16 FP64: 272 with four, 108 with sixteen).
// Long rows fill the shared memory of an SM with the slots of few threads: as many
// shares as leave a block's slots within its part of it (100k rows of 100 entries,
// K = 16 FP32: 528 us with one share, 264 with four; FP64 1545 / 1338).  Of six or
// more blocks one may be lost rather than go from one share to two (9-point depth 2,
// 25 a row, FP32: 112 / 118) or past a lane per piece of the target (20000 rows of
// 100, FP32: 65 with four shares, 79 with eight); of four blocks it may not (of 70,
// K = 16 FP64: 290 with four, 215 with eight).
template <int P, int G>
inline int fit_shares(int64_t n, int64_t nnz, int slot, int blocks)
{
    const int64_t avg = nnz / n, part = (int64_t)227 * 1024 / blocks;
    int el = 1;
    while (G * el < 32 && n * G * el < (int64_t)152 * 256 && (el < 4 || avg > 8 * el)) el *= 2;
    while (G * el < 32) {
        const int64_t bytes = (kFitThreads / (G * el) * avg * 5 / 4 + 32) * slot;
        const bool lose_one = blocks >= 6 && (el == 1 || G * el >= P);
        if (bytes <= (lose_one ? part * 115 / 100 : part)) break;
        el *= 2;
    }
    return el;
}
inline int fit_threads(int64_t lanes, int most)
{
    int t = most;
    while (t > 32 && lanes < (int64_t)152 * 4 * t) t /= 2;
    return t;
}

template <class TS, int P, bool UW, bool PX, bool COMP>
cudaError_t go_fit(EdgeArgs a, cudaStream_t s)
{
    using L = FitLayout<TS, P, COMP>;
    if (a.Kp != L::KP || !a.norms) return cudaErrorInvalidValue;
    if constexpr (P % 2 == 0)                      // 32-byte row reads
        if (!rows_aligned32(a.x, a.Kp, sizeof(TS))) return cudaErrorMisalignedAddress;
    constexpr int per = sizeof(TS) == 8 ? kNormThreads : kNormThreads / P;    // rows per block
    cudaError_t e = cudaSuccess;
    if constexpr (!L::OWN)
        e = launch_chained(k_norms<TS, P, UW, COMP>, (unsigned)(((int64_t)a.n + per - 1) / per), kNormThreads,
                                   0, s, (const TS *)a.x, a.w, a.n, a.norms);
    if (e != cudaSuccess) return e;
    // slots staged per block: the average rows' entries and a quarter more
    // (a block with longer rows works on global memory), at most 96 KB
    const int el = fit_shares<P, L::G>(a.n, a.nnz_p, L::SLOT, L::MINB);
    const int T = fit_threads((int64_t)a.n * L::G * el, L::THREADS);
    const int rows = T / (L::G * el), yrows = el > 1 ? rows : 0;
    // Rows of a graph differ in length (17 entries on average, the longest of 32 rows
    // 26).  Sorted, us: 400k rows FP64 K = 8 / 16 845 / 1426 -> 716 / 1179, BF16 K = 16 /
    // 32 171 / 297 -> 164 / 289, FP32 K = 32 316 -> 304; FP64 gains with several shares a
    // row, too (20k rows 69 / 148 -> 62 / 133).  Shorter rows wait for their gathers and
    // lose the order of them (2M rows, K = 4 FP32 909 -> 1029, BF16 911 -> 981; 300k rows,
    // K = 16 FP32 166 -> 172).
    a.uneven = a.uneven && L::SORTS && (sizeof(TS) == 8 || (el == 1 && L::KP >= (sizeof(TS) == 2 ? 16 : 32)));
    int64_t cap = (int64_t)((double)a.nnz_p / a.n * rows * 1.25) + 32;
    const int64_t most = (96 * 1024 - L::bytes(0, UW, yrows)) / L::SLOT;
    cap = (cap < most ? cap : most) & ~(int64_t)15;
    const int smem = L::bytes((int)cap, UW, yrows);
    const auto kern = el > 1 ? k_edge_fit<TS, P, UW, PX, COMP, true> : k_edge_fit<TS, P, UW, PX, COMP, false>;
    static PerDevice opted[2];               // shared-memory opt-in made on each device
    const int dev = current_device_index();
    if (opted[el > 1].get(dev) == 0) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
        if (e != cudaSuccess) return e;
        opted[el > 1].set(dev, 1);
    }
    e = launch_chained(kern, (unsigned)(((int64_t)a.n + rows - 1) / rows), T, smem, s, a, (int)cap, el);
    if (e != cudaSuccess) return e;
    if (a.n_long > 0) {
        e = launch_chained(k_edge_long<TS, P, UW, PX, COMP>, (unsigned)(a.n_long < 152 * 4 ? a.n_long : 152 * 4),
                           kLongThreads, 0, s, a);
        if (e != cudaSuccess) return e;
    }
    if constexpr (!std::is_same<TS, double>::value)
        e = launch_chained(k_edge_fixup<TS, P, PX>, 152, kFixThreads, 0, s, a);
    return e;
}

template <class TS, bool COMP, int P>
cudaError_t dispatch_w(bool in_place, bool unit_w, const EdgeArgs &a, cudaStream_t s)
{
    if (in_place) return unit_w ? go_fit<TS, P, true, true, COMP>(a, s) : go_fit<TS, P, false, true, COMP>(a, s);
    return unit_w ? go_fit<TS, P, true, false, COMP>(a, s) : go_fit<TS, P, false, false, COMP>(a, s);
}

// one storage type and summation form per translation unit (parallel
// compilation)
template <class TS, bool COMP>
cudaError_t dispatch(bool in_place, bool unit_w, const EdgeArgs &a, cudaStream_t s)
{
    if (a.n <= 0) return cudaSuccess;
    constexpr int V = Store<TS>::V;
    switch (a.Kp / V) {
    case 1: return dispatch_w<TS, COMP, 1>(in_place, unit_w, a, s);
    case 2: return dispatch_w<TS, COMP, 2>(in_place, unit_w, a, s);
    case 4: return dispatch_w<TS, COMP, 4>(in_place, unit_w, a, s);
    case 8: return dispatch_w<TS, COMP, 8>(in_place, unit_w, a, s);
    case 16: if constexpr (16 * V <= 64) return dispatch_w<TS, COMP, 16>(in_place, unit_w, a, s); break;
    case 32: if constexpr (32 * V <= 64) return dispatch_w<TS, COMP, 32>(in_place, unit_w, a, s); break;
    }
    return cudaErrorInvalidValue;
}

}  // namespace edge_impl
}  // namespace amgd
