// k_init.cu -- test-vector start (counter-based Philox4x64-10), layout and
// precision conversions of the vector block, per-slot output export and the
// permutation of A's values.
#include "amgd_internal.cuh"

namespace amgd {
namespace {

constexpr int kThreads = 256;

// Philox4x64-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds of two
// 64x64->128 multiplies with the published 4x64 multipliers, Weyl key
// schedule with the published increments.
struct U64x4 { uint64_t v[4]; };

__device__ __forceinline__ U64x4 philox4x64_10(uint64_t c0, uint64_t c1, uint64_t c2, uint64_t c3,
                                               uint64_t k0, uint64_t k1)
{
    constexpr uint64_t kMulA = 0xD2E7470EE14C6C93ull, kMulB = 0xCA5A826395121157ull;
    constexpr uint64_t kWeylA = 0x9E3779B97F4A7C15ull, kWeylB = 0xBB67AE8584CAA73Bull;
#pragma unroll
    for (int round = 0; round < 10; ++round) {
        const uint64_t hiA = __umul64hi(kMulA, c0), loA = kMulA * c0;
        const uint64_t hiB = __umul64hi(kMulB, c2), loB = kMulB * c2;
        const uint64_t n0 = hiB ^ c1 ^ k0;
        const uint64_t n2 = hiA ^ c3 ^ k1;
        c0 = n0;
        c1 = loB;
        c2 = n2;
        c3 = loA;
        k0 += kWeylA;
        k1 += kWeylB;
    }
    U64x4 o;
    o.v[0] = c0; o.v[1] = c1; o.v[2] = c2; o.v[3] = c3;
    return o;
}

template <class TS> __device__ __forceinline__ TS from_double(double x);
template <> __device__ __forceinline__ double from_double<double>(double x) { return x; }
template <> __device__ __forceinline__ float from_double<float>(double x) { return (float)x; }
template <> __device__ __forceinline__ __nv_bfloat16 from_double<__nv_bfloat16>(double x)
{
    return __double2bfloat16(x);
}
template <class TS> __device__ __forceinline__ double to_double(TS x) { return (double)x; }
template <> __device__ __forceinline__ double to_double<__nv_bfloat16>(__nv_bfloat16 x)
{
    return (double)__bfloat162float(x);
}

// The start value of a component is x = d * 2^-32 with the odd integer
// d = 2m + 1 - 2^32, m the component's 32-bit random integer.  |d| < 2^32,
// so the magnitude a = |d| fits 32 bits: a = 2(m - 2^31) + 1 for m >= 2^31
// (d > 0), a = 2(2^31 - 1 - m) + 1 otherwise (d < 0).  The FP64 and BF16
// values are built as raw bits with 32-bit integer work (the GPU's FP64 pipe
// is narrow; an FP32 step before BF16 would round twice), the FP32 value by
// the hardware's integer-to-FP32 conversion; either way rounded to nearest
// even exactly once.
__device__ __forceinline__ uint32_t start_magnitude(uint32_t m, bool &neg)
{
    neg = (m & 0x80000000u) == 0u;
    return neg ? (((0x7fffffffu - m) << 1) | 1u) : (((m & 0x7fffffffu) << 1) | 1u);
}

// round the odd integer a (1 <= a < 2^32) to P+1 significant bits (nearest,
// ties to even) and return the IEEE fields of a * 2^-32 for a format with P
// stored mantissa bits and exponent bias B: every value here is normal
template <int P, int B>
__device__ __forceinline__ uint32_t encode_fields(uint32_t a, uint32_t &mant)
{
    int lead = 31 - __clz((int)a);                 // 2^lead <= a < 2^(lead+1)
    uint32_t q;
    if (lead <= P) {
        q = a << (P - lead);                       // exact
    } else {
        const int sh = lead - P;
        q = a >> sh;
        const uint32_t rem = a & ((1u << sh) - 1u), half = 1u << (sh - 1);
        if (rem > half || (rem == half && (q & 1u))) ++q;
        if (q == (2u << P)) { q = 1u << P; ++lead; }   // rounded up to the next power of two
    }
    mant = q - (1u << P);
    return (uint32_t)(lead - 32 + B);             // biased exponent
}

// raw bits of the start value of one component in the storage type
template <class TS> struct StartBits;
template <> struct StartBits<double> {
    using Raw = unsigned long long;
    __device__ __forceinline__ static Raw get(uint32_t m) {
        bool neg;
        const uint32_t a = start_magnitude(m, neg);    // < 2^32: exact in FP64
        const int lead = 31 - __clz((int)a);
        const unsigned long long mant = ((unsigned long long)a << (52 - lead)) & ((1ull << 52) - 1ull);
        const unsigned long long expo = (unsigned long long)(lead - 32 + 1023);
        return (neg ? (1ull << 63) : 0ull) | (expo << 52) | mant;
    }
};
template <> struct StartBits<float> {
    using Raw = uint32_t;
    // the odd integer d = 2m + 1 - 2^32 converted to FP32 by the hardware's
    // correctly rounded (nearest-even) integer conversion, then scaled by
    // 2^-32 exactly (|d| >= 1: every value is normal): the same single
    // rounding as the bit assembly of the other storages, in two instructions
    __device__ __forceinline__ static Raw get(uint32_t m) {
        const long long d = 2ll * (long long)m + 1ll - (1ll << 32);
        return __float_as_uint(__ll2float_rn(d) * 0x1p-32f);
    }
};
template <> struct StartBits<__nv_bfloat16> {
    using Raw = uint32_t;                               // low 16 bits used
    __device__ __forceinline__ static Raw get(uint32_t m) {
        bool neg;
        uint32_t mant;
        const uint32_t e = encode_fields<7, 127>(start_magnitude(m, neg), mant);
        return (neg ? 0x8000u : 0u) | (e << 7) | mant;
    }
};

// one thread per (row, block of 8 components): one Philox4x64-10 call gives
// 4 x 64 bits = 8 components of 32 bits (low half first).  Kp is a power of
// two; lq = log2(max(1, Kp / 8)).  Values are assembled as raw bits with
// integer operations and written with 16-byte stores (or per component for
// rows shorter than 8 components).
template <class TS>
__global__ void __launch_bounds__(kThreads) k_tv_init(InitArgs A, int lq)
{
    using SB = StartBits<TS>;
    const int64_t t = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    const int64_t r = t >> lq;
    if (r >= A.n) {
        chain_wait();
        return;
    }
    const int q = (int)(t & ((1 << lq) - 1));
    const int64_t o = A.perm ? A.perm[r] : r;
    int lo = 0, hi = A.nmat;                 // matrix b with mat_off[b] <= o < mat_off[b+1]
    while (hi - lo > 1) {
        const int mid = (lo + hi) / 2;
        if (A.mat_off[mid] <= o) lo = mid; else hi = mid;
    }
    const uint64_t li = (uint64_t)(o - A.mat_off[lo]);
    const uint64_t key1 = A.mat_id ? (uint64_t)A.mat_id[lo] : (uint64_t)lo;
    const U64x4 u = philox4x64_10(li, (uint64_t)q, 0ull, 0ull, A.seed, key1);
    typename SB::Raw v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const uint32_t m = (k & 1) ? (uint32_t)(u.v[k / 2] >> 32) : (uint32_t)u.v[k / 2];
        v[k] = 8 * q + k < A.K ? SB::get(m) : 0;     // padding: +0
    }
    chain_wait();                  // the vectors may still be in use; the draws did not depend on them
    chain_release();
    TS *x = (TS *)A.x + r * A.Kp + 8 * q;
    if (A.Kp >= 8) {
        uint4 *x4 = reinterpret_cast<uint4 *>(x);
        if constexpr (sizeof(TS) == 2) {
            x4[0] = make_uint4(v[0] | (v[1] << 16), v[2] | (v[3] << 16), v[4] | (v[5] << 16),
                               v[6] | (v[7] << 16));
        } else if constexpr (sizeof(TS) == 4) {
            x4[0] = make_uint4(v[0], v[1], v[2], v[3]);
            x4[1] = make_uint4(v[4], v[5], v[6], v[7]);
        } else {
#pragma unroll
            for (int c = 0; c < 4; ++c)
                x4[c] = make_uint4((uint32_t)v[2 * c], (uint32_t)(v[2 * c] >> 32),
                                   (uint32_t)v[2 * c + 1], (uint32_t)(v[2 * c + 1] >> 32));
        }
    } else {
        typename SB::Raw *xr = reinterpret_cast<typename SB::Raw *>(x);
        if constexpr (sizeof(TS) == 2) {
            uint16_t *x16 = reinterpret_cast<uint16_t *>(x);
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (k < A.Kp) x16[k] = (uint16_t)v[k];
        } else {
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (k < A.Kp) xr[k] = v[k];
        }
    }
}

template <class TS>
__global__ void k_import(const double *__restrict__ src, TS *__restrict__ x,
                         const int32_t *__restrict__ perm, int32_t n, int32_t K, int32_t Kp)
{
    const int64_t t = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (t >= (int64_t)n * Kp) return;
    const int64_t r = t / Kp;
    const int kappa = (int)(t % Kp);
    const int64_t o = perm ? perm[r] : r;
    x[t] = from_double<TS>(kappa < K ? src[o * K + kappa] : 0.0);
}

template <class TS>
__global__ void k_export(const TS *__restrict__ x, double *__restrict__ dst,
                         const int32_t *__restrict__ perm, int32_t n, int32_t K, int32_t Kp)
{
    const int64_t t = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (t >= (int64_t)n * K) return;
    const int64_t r = t / K;
    const int kappa = (int)(t % K);
    const int64_t o = perm ? perm[r] : r;
    dst[o * K + kappa] = to_double<TS>(x[r * Kp + kappa]);
}

// 1 / l of an FP32 number in FP64 by long division in base 2^24: the FP32
// reciprocal q1 is the first digit, the remainders 1 - l q1 and 1 - l (q1 + q2) are
// exact FP32 numbers (one fused multiply-add each), their products with q1 the
// next two digits.  The digits are widened on the integer pipe and added in FP64:
// two FP64 operations against six of a division and one per conversion (the FP64
// pipe retires two per clock and SM).  Exact to 2^-71 before the last addition's
// rounding: over every FP32 number of the range it is the division's result but for
// 1 in 10^6, near-ties whose other neighbour it takes (0.5 ulp as the division).
// Numbers near the ends of the range, zeros, infinities and NaN divide.
__device__ __forceinline__ double reciprocal(float l)
{
    if (l != l) return __longlong_as_double(0x7ff8000000000000ll);      // the diagonal: no division for its warp
    if (!(l > 1e-30f && l < 1e20f)) return 1.0 / (double)l;
    const float q1 = __fdividef(1.0f, l);
    const float r1 = fmaf(-l, q1, 1.0f);
    const float q2 = r1 * q1;
    const float q3 = fmaf(-l, q2, r1) * q1;
    return widen_f32_bits(__float_as_uint(q1)) + (widen_f32_bits(__float_as_uint(q2)) + widen_f32_bits(__float_as_uint(q3)));
}
__device__ __forceinline__ double reciprocal(double l) { return 1.0 / l; }      // +inf for LS = 0, NaN stays NaN
__device__ __forceinline__ double widened(float x) { return widen_f32_bits(__float_as_uint(x)); }
__device__ __forceinline__ double widened(double x) { return x; }

// Bound: HBM (8 bytes in and up to 24 out per slot); the plain division and
// conversions made it the FP64 pipe (distance call of the 9-point 512^2 at depth 2,
// 6.5 M slots, BF16: 247 -> 222 us).
template <class C>
__global__ void __launch_bounds__(kThreads) k_export_slots(const C *a_in, const C *ls_in, double *__restrict__ a,
                                                          double *__restrict__ dist, double *__restrict__ ls,
                                                          int64_t nnz)
{
    constexpr int E = 4;                 // slots of a thread, a block apart
    chain_wait();
    chain_release();
    const int64_t base = (int64_t)blockIdx.x * (E * kThreads) + threadIdx.x;
    C l[E], v[E];
#pragma unroll
    for (int u = 0; u < E; ++u) {
        const int64_t t = base + u * kThreads;
        if (t >= nnz) continue;
        if (dist || ls) l[u] = ld_plain(ls_in + t);
        if (a) v[u] = ld_plain(a_in + t);
    }
#pragma unroll
    for (int u = 0; u < E; ++u) {
        const int64_t t = base + u * kThreads;
        if (t >= nnz) continue;
        if (a) a[t] = widened(v[u]);
        if (ls) ls[t] = widened(l[u]);
        if (dist) dist[t] = reciprocal(l[u]);
    }
}

__global__ void k_unpermute(const uint4 *__restrict__ x, uint4 *__restrict__ xc,
                            const int32_t *__restrict__ perm, int32_t n, int32_t pieces)
{
    const int64_t t = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (t >= (int64_t)n * pieces) return;
    const int64_t r = t / pieces;
    const int q = (int)(t % pieces);
    xc[(int64_t)perm[r] * pieces + q] = x[t];
}

__global__ void k_diagonal(const int32_t *__restrict__ rp, const int32_t *__restrict__ col,
                           const double *__restrict__ v, double *__restrict__ d64,
                           float *__restrict__ d32, int32_t n)
{
    const int64_t r = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (r >= n) return;
    double d = 0.0;
    for (int p = rp[r]; p < rp[r + 1]; ++p)
        if (col[p] == r) d = v[p];
    if (d64) d64[r] = d;
    if (d32) d32[r] = (float)d;
}

__global__ void k_check_values(const double *__restrict__ v, int64_t nnz,
                               const int32_t *__restrict__ diag_slot, int32_t n,
                               uint32_t *__restrict__ err)
{
    const int64_t t = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    uint32_t e = 0;
    if (t < nnz && !isfinite(v[t])) e |= 1u;
    if (t < n && v[diag_slot[t]] == 0.0) e |= 2u;
    e = __reduce_or_sync(0xffffffffu, e);
    if (e && (threadIdx.x % 32) == 0) atomicOr(err, e);
}

// one pass over the stored values in caller order into one other copy (slot p at to[p])
__global__ void k_scatter_values(const double *__restrict__ src, int64_t nnz, const int32_t *__restrict__ to,
                                 double *__restrict__ v64, float *__restrict__ v32)
{
    for (int64_t p = (int64_t)blockIdx.x * kThreads + threadIdx.x; p < nnz; p += (int64_t)gridDim.x * kThreads) {
        const int64_t q = to ? to[p] : p;
        if (v64) v64[q] = src[p];
        else v32[q] = (float)src[p];
    }
}

// diagonals in permuted order (perm[r] = caller row of r)
__global__ void k_diag_values(const double *__restrict__ v, const int32_t *__restrict__ diag_slot,
                              const int32_t *__restrict__ perm, int32_t n, double *__restrict__ d64_p)
{
    const int64_t t = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (t < n) d64_p[t] = v[diag_slot[perm ? perm[t] : t]];
}

// Every copy of the values in one pass over them (launch_values).  A block takes
// kThreads consecutive caller rows: their values come in and the caller-order
// copies go out as one contiguous run, and the run waits in shared memory (in the
// type VS of the sweeps) for the sliced copy, where one thread per row writes
// entry k of consecutive rows side by side -- a scatter slot by slot would write
// each value to a line of its own -- and for the diagonals.  Bound: HBM.
template <class VS>
__global__ void __launch_bounds__(kThreads) k_values(ValueArgs A, int cap)
{
    extern __shared__ __align__(16) unsigned char vsm[];
    VS *sv = reinterpret_cast<VS *>(vsm);
    int32_t *sp = reinterpret_cast<int32_t *>(sv + cap);
    const int64_t R0 = (int64_t)blockIdx.x * kThreads;
    const int nr = (int)min((int64_t)kThreads, A.n - R0), tid = threadIdx.x;
    const int S0 = A.rp[R0], S1 = A.rp[R0 + nr];
    const bool fits = S1 - S0 <= cap;
    VS *sell = (VS *)A.sell;
    if (sell && fits)
        for (int q = tid; q < S1 - S0; q += kThreads) sp[q] = __ldg(A.slot_sell + S0 + q);
    chain_wait();
    bool bad = false;
    for (int64_t p = (int64_t)S0 + tid; p < S1; p += kThreads) {   // 64 bits: the last stride may pass 2^31
        const double x = ld_plain(A.src + p);
        bad = bad || !isfinite(x);
        if (A.val_o) A.val_o[p] = x;
        const VS v = (VS)x;
        if (A.val32_o) A.val32_o[p] = (float)v;
        if (A.perm_val) ((VS *)A.perm_val)[A.slot_perm ? A.slot_perm[p] : p] = v;
        if (sell) {
            if (fits) sv[p - S0] = v;
            else sell[A.slot_sell[p]] = v;
        }
    }
    __syncthreads();
    bool zero = false;
    if (tid < nr) {
        const int64_t o = R0 + tid;
        if (sell && fits) {
            const int q1 = A.rp[o + 1] - S0;
            for (int q = A.rp[o] - S0; q < q1; ++q) sell[sp[q]] = sv[q];
        }
        const double d = ld_plain(A.src + A.diag_slot[o]);
        zero = d == 0.0;
        const int64_t r = A.pinv ? A.pinv[o] : o;
        A.d64_o[o] = d;
        A.d32_o[o] = (float)d;
        if (A.d64_p) A.d64_p[r] = d;
        A.d32_p[r] = (float)d;
    }
    if (A.err) {
        const uint32_t e = (__any_sync(0xffffffffu, bad) ? 1u : 0u) | (__any_sync(0xffffffffu, zero) ? 2u : 0u);
        if (e && tid % 32 == 0) atomicOr(A.err, e);
    }
}

// a row and its length into what the distance pass has to know of them (every thread
// of a block; length 0: no row).  cap: rows that a check refuses are listed too.
__device__ __forceinline__ void note_row(const LongArgs &A, int64_t r, int64_t len)
{
    __shared__ unsigned long long sum;
    if (threadIdx.x == 0) sum = 0;
    __syncthreads();
    if (len > A.long_len) {
        const uint32_t at = atomicAdd(A.count, 1u);
        if (at < A.cap) A.rows[at] = (int32_t)r;
        len = 0;
    }
    const unsigned longest = __reduce_max_sync(0xffffffffu, (unsigned)max(len, (int64_t)0));
    if (threadIdx.x % 32 == 0) atomicAdd(&sum, 32ull * longest);
    __syncthreads();
    if (threadIdx.x == 0) atomicAdd(A.filled, sum);
}

// launch_create: one thread per row.  Rows in ascending order hold no duplicate;
// others are compared entry by entry up to kPairRow entries (the same checks on
// the host took most of the 17 ms of a one-call build of a 150k-row graph).  The
// comparisons of a row grow with its square and run in one thread, so longer
// unordered rows go to the host check.  Creating a handle from unordered rows, us,
// host check / here: 120 entries 2768 / 771, 300 entries 6044 / 3772 (thread per
// row; 6243 by way of the host), 400 entries 2327 / 6627, 1000 entries 5531 / 33613.
constexpr int kPairRow = 128;
__global__ void __launch_bounds__(kThreads) k_create(CreateArgs A)
{
    const int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    const int64_t a = i < A.n ? A.rp[i] : 0, b = i < A.n ? A.rp[i + 1] : 0;
    const bool rows_ok = a >= 0 && b >= a && b <= A.nnz;
    note_row(A.rows, A.row0 + i, rows_ok ? b - a : 0);
    if (i >= A.n) return;
    if (!rows_ok) {
        atomicOr(A.err, 1u);
        return;
    }
    if (i == 0) A.rp_o[A.row0] = (int32_t)A.slot0;
    A.rp_o[A.row0 + i + 1] = (int32_t)(A.slot0 + b);
    int64_t d = -1, prev = -1;
    bool bad = false, ordered = true;
    for (int64_t p = a; p < b; ++p) {
        const int64_t j = A.col[p];
        const double v = A.val[p];
        bad = bad || j < 0 || j >= A.n || !isfinite(v);
        ordered = ordered && j > prev;
        prev = j;
        if (j == i) d = p;
        A.col_o[A.slot0 + p] = (int32_t)(A.row0 + j);
        A.val_o[A.slot0 + p] = v;
    }
    uint32_t err = 0;
    if (!ordered) {
        if (b - a > kPairRow) {
            err = 2u;
        } else {
            for (int64_t p = a; p < b; ++p)
                for (int64_t q = a; q < p; ++q) bad = bad || A.col[q] == A.col[p];
        }
    }
    const double diag = d >= 0 ? A.val[d] : 0.0;
    if (bad || diag == 0.0) err |= 1u;
    if (err) atomicOr(A.err, err);
    const int64_t r = A.row0 + i;
    A.diag_slot[r] = (int32_t)(A.slot0 + (d >= 0 ? d : 0));
    A.d64_p[r] = A.d64_o[r] = diag;
    A.d32_p[r] = A.d32_o[r] = (float)diag;
}

__global__ void __launch_bounds__(kThreads) k_long_rows(const int32_t *__restrict__ rp, int32_t n, LongArgs A)
{
    const int64_t r = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    note_row(A, r, r < n ? rp[r + 1] - rp[r] : 0);
}

inline unsigned blocks(int64_t work) { return (unsigned)((work + kThreads - 1) / kThreads); }

// priority keys of the coarse-point selection: one Philox4x64-10 block per
// point, counter (i, stage, 1, 0) (word 2 = 1 keeps them apart from the
// test-vector draws), key (seed, 0); word 0 is the key
__global__ void k_cr_keys(int32_t n, int32_t stage, uint64_t seed, uint64_t *key)
{
    chain_wait();
    chain_release();
    for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        key[i] = philox4x64_10((uint64_t)i, (uint64_t)stage, 1ull, 0ull, seed, 0ull).v[0];
}

}  // namespace

cudaError_t launch_cr_keys(int32_t n, int32_t stage, uint64_t seed, uint64_t *key, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    return launch_chained(k_cr_keys, blocks(n), kThreads, 0, s, n, stage, seed, key);
}

cudaError_t launch_init(int storage, const InitArgs &a, cudaStream_t s)
{
    if (a.Kp & (a.Kp - 1)) return cudaErrorInvalidValue;     // Kp is a power of two
    int lq = 0;
    while ((8 << lq) < a.Kp) ++lq;
    const int64_t work = (int64_t)a.n << lq;
    if (work == 0) return cudaSuccess;
    switch (storage) {
    case ST_FP64: return launch_chained(k_tv_init<double>, blocks(work), kThreads, 0, s, a, lq);
    case ST_FP32: return launch_chained(k_tv_init<float>, blocks(work), kThreads, 0, s, a, lq);
    case ST_BF16: return launch_chained(k_tv_init<__nv_bfloat16>, blocks(work), kThreads, 0, s, a, lq);
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_import(int storage, const double *src, void *x, const int32_t *perm,
                          int32_t n, int32_t K, int32_t Kp, cudaStream_t s)
{
    const int64_t work = (int64_t)n * Kp;
    if (work == 0) return cudaSuccess;
    switch (storage) {
    case ST_FP64: k_import<<<blocks(work), kThreads, 0, s>>>(src, (double *)x, perm, n, K, Kp); break;
    case ST_FP32: k_import<<<blocks(work), kThreads, 0, s>>>(src, (float *)x, perm, n, K, Kp); break;
    case ST_BF16:
        k_import<<<blocks(work), kThreads, 0, s>>>(src, (__nv_bfloat16 *)x, perm, n, K, Kp);
        break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_export(int storage, const void *x, double *dst, const int32_t *perm,
                          int32_t n, int32_t K, int32_t Kp, cudaStream_t s)
{
    const int64_t work = (int64_t)n * K;
    if (work == 0) return cudaSuccess;
    switch (storage) {
    case ST_FP64:
        k_export<<<blocks(work), kThreads, 0, s>>>((const double *)x, dst, perm, n, K, Kp);
        break;
    case ST_FP32:
        k_export<<<blocks(work), kThreads, 0, s>>>((const float *)x, dst, perm, n, K, Kp);
        break;
    case ST_BF16:
        k_export<<<blocks(work), kThreads, 0, s>>>((const __nv_bfloat16 *)x, dst, perm, n, K, Kp);
        break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_export_slots(int storage, const void *a_in, const void *ls_in, double *a,
                                double *dist, double *ls, int64_t nnz, cudaStream_t s)
{
    if (nnz == 0) return cudaSuccess;
    const unsigned grid = (unsigned)((nnz + 4 * kThreads - 1) / (4 * kThreads));
    if (storage == ST_FP64)
        return launch_chained(k_export_slots<double>, grid, kThreads, 0, s, (const double *)a_in, (const double *)ls_in,
                              a, dist, ls, nnz);
    return launch_chained(k_export_slots<float>, grid, kThreads, 0, s, (const float *)a_in, (const float *)ls_in, a,
                          dist, ls, nnz);
}

cudaError_t launch_unpermute(int storage, const void *x, void *x_caller, const int32_t *perm,
                             int32_t n, int32_t Kp, cudaStream_t s)
{
    const int esz = storage == ST_FP64 ? 8 : (storage == ST_FP32 ? 4 : 2);
    const int32_t pieces = (int32_t)((int64_t)Kp * esz / 16);
    const int64_t work = (int64_t)n * pieces;
    if (work == 0) return cudaSuccess;
    k_unpermute<<<blocks(work), kThreads, 0, s>>>((const uint4 *)x, (uint4 *)x_caller, perm, n, pieces);
    return cudaGetLastError();
}

cudaError_t launch_diagonal(const int32_t *rp_perm, const int32_t *col_perm, const double *vp64,
                            double *d64, float *d32, int32_t n, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    k_diagonal<<<blocks(n), kThreads, 0, s>>>(rp_perm, col_perm, vp64, d64, d32, n);
    return cudaGetLastError();
}

cudaError_t launch_check_values(const double *v, int64_t nnz, const int32_t *diag_slot,
                                int32_t n, uint32_t *err, cudaStream_t s)
{
    const int64_t work = nnz > n ? nnz : n;
    if (work == 0) return cudaSuccess;
    k_check_values<<<blocks(work), kThreads, 0, s>>>(v, nnz, diag_slot, n, err);
    return cudaGetLastError();
}

cudaError_t launch_scatter_values(const double *src, int64_t nnz, const int32_t *to, double *v64, float *v32,
                                  cudaStream_t s)
{
    if (nnz == 0) return cudaSuccess;
    const int64_t want = (nnz + kThreads - 1) / kThreads;
    k_scatter_values<<<(unsigned)(want < 152 * 16 ? want : 152 * 16), kThreads, 0, s>>>(src, nnz, to, v64, v32);
    return cudaGetLastError();
}

cudaError_t launch_create(const CreateArgs &a, cudaStream_t s)
{
    if (a.n == 0) return cudaSuccess;
    k_create<<<blocks(a.n), kThreads, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_long_rows(const int32_t *rp, int32_t n, const LongArgs &a, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    k_long_rows<<<blocks(n), kThreads, 0, s>>>(rp, n, a);
    return cudaGetLastError();
}

cudaError_t launch_values(const ValueArgs &a, bool f64, int64_t nnz, cudaStream_t s)
{
    if (a.n == 0) return cudaSuccess;
    // a block's average run and a quarter more, within the default shared memory
    const int slot = (f64 ? 8 : 4) + 4;
    int64_t cap = (int64_t)((double)nnz / a.n * kThreads * 1.25) + 64;
    if (cap * slot > 48 * 1024) cap = 48 * 1024 / slot;
    cap &= ~(int64_t)3;
    if (f64) return launch_chained(k_values<double>, blocks(a.n), kThreads, (size_t)cap * slot, s, a, (int)cap);
    return launch_chained(k_values<float>, blocks(a.n), kThreads, (size_t)cap * slot, s, a, (int)cap);
}

cudaError_t launch_diag_values(const double *v, const int32_t *diag_slot, const int32_t *perm, int32_t n, double *d64_p,
                               cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    k_diag_values<<<blocks(n), kThreads, 0, s>>>(v, diag_slot, perm, n, d64_p);
    return cudaGetLastError();
}

}  // namespace amgd
