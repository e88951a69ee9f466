// k_sell.cu -- the sliced copy of the row-permuted matrix that the sweeps read
// (k_relax.cu): slices of 32 rows of one color, entries column by column.
// Built on the device once per coloring; values follow through the position
// of every caller slot (launch_scatter_values).
#include "amgd_internal.cuh"

namespace amgd {
namespace {

constexpr int kThreads = 256;

// color of a slice: color_slice[c] <= q < color_slice[c + 1]
__device__ __forceinline__ int color_of(const SellArgs &a, int64_t q)
{
    int lo = 0, hi = a.ncolors;
    while (hi - lo > 1) {
        const int mid = (lo + hi) / 2;
        if (a.color_slice[mid] <= q) lo = mid; else hi = mid;
    }
    return lo;
}

// row of (slice q, place l), -1: past the color's last row
__device__ __forceinline__ int64_t row_at(const SellArgs &a, const int32_t *rowmap, int64_t q, int l)
{
    if (rowmap) return rowmap[q * kSellRows + l];
    const int c = color_of(a, q);
    const int64_t r = a.color_row[c] + (q - a.color_slice[c]) * kSellRows + l;
    return r < a.color_row[c + 1] ? r : -1;
}

// One block per window of kSellWindow rows of a color: every row finds its
// place by counting the rows that go before it (longer ones, then smaller
// indices).  Blocks are numbered by the window's first slice.
__global__ void __launch_bounds__(kSellWindow) k_sell_sort(SellArgs a, int32_t *rowmap)
{
    constexpr int SW = kSellWindow / kSellRows;          // slices of a window
    __shared__ int32_t len[kSellWindow];
    const int64_t q = (int64_t)blockIdx.x;               // candidate first slice
    const int c = color_of(a, q);
    if ((q - a.color_slice[c]) % SW) return;
    const int64_t r0 = a.color_row[c] + (q - a.color_slice[c]) * kSellRows;
    const int rows = (int)min((int64_t)kSellWindow, a.color_row[c + 1] - r0);
    const int t = threadIdx.x;
    const int mine = t < rows ? a.rp[r0 + t + 1] - a.rp[r0 + t] : -1;
    len[t] = mine;
    __syncthreads();
    int place = 0;
    for (int k = 0; k < kSellWindow; ++k) place += len[k] > mine || (len[k] == mine && k < t);
    // places past the color's last slice are padding of the last window
    if (q * kSellRows + place < a.color_slice[c + 1] * kSellRows) rowmap[q * kSellRows + place] = t < rows ? (int32_t)(r0 + t) : -1;
}

// the rows of the slices in order
__global__ void __launch_bounds__(kThreads) k_sell_rows(SellArgs a, int32_t *rowmap)
{
    const int64_t q = ((int64_t)blockIdx.x * kThreads + threadIdx.x) / 32;
    const int l = threadIdx.x % 32;
    if (q < a.nslices) rowmap[q * kSellRows + l] = (int32_t)row_at(a, nullptr, q, l);
}

__global__ void __launch_bounds__(kThreads) k_sell_width(SellArgs a, const int32_t *rowmap, int32_t *width, unsigned long long *measured)
{
    __shared__ int ws[kThreads / 32];
    const int64_t q = ((int64_t)blockIdx.x * kThreads + threadIdx.x) / 32;
    const int l = threadIdx.x % 32;
    const int64_t r = q < a.nslices ? row_at(a, rowmap, q, l) : -1;
    const int len = r >= 0 ? a.rp[r + 1] - a.rp[r] : 0;
    const int w = (int)__reduce_max_sync(0xffffffffu, (unsigned)len);
    if (l == 0) {
        if (q < a.nslices) width[q] = w * kSellRows;   // wraps only where the 64-bit total is refused
        ws[threadIdx.x / 32] = w;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long sum = 0, longest = 0;
        for (int k = 0; k < kThreads / 32; ++k) {
            sum += (unsigned long long)ws[k] * kSellRows;
            longest = max(longest, (unsigned long long)ws[k]);
        }
        atomicAdd(measured, sum);
        atomicMax(measured + 1, longest);
    }
}

__global__ void __launch_bounds__(kThreads)
k_sell_fill(SellArgs a, const int32_t *rowmap, const int64_t *__restrict__ ptr, int32_t *__restrict__ sell_col,
            int32_t *__restrict__ slot)
{
    const int64_t q = ((int64_t)blockIdx.x * kThreads + threadIdx.x) / 32;
    const int l = threadIdx.x % 32;
    if (q >= a.nslices) return;
    const int64_t r = row_at(a, rowmap, q, l);
    const int64_t base = ptr[q] + l;
    const int w = (int)((ptr[q + 1] - ptr[q]) / kSellRows);
    int len = 0;
    int64_t p = 0, o = 0;
    if (r >= 0) {
        p = a.rp[r];
        len = (int)(a.rp[r + 1] - p);
        o = a.rp_o[a.perm ? a.perm[r] : r];
    }
    for (int k = 0; k < w; ++k) {
        sell_col[base + (int64_t)kSellRows * k] = k < len ? a.col[p + k] : -1;
        if (k < len) slot[o + k] = (int32_t)(base + (int64_t)kSellRows * k);
    }
}

inline unsigned slice_blocks(int64_t slices) { return (unsigned)((slices * 32 + kThreads - 1) / kThreads); }

}  // namespace

cudaError_t launch_sell_sort(const SellArgs &a, int32_t *rowmap, cudaStream_t s)
{
    if (a.nslices == 0) return cudaSuccess;
    k_sell_sort<<<(unsigned)a.nslices, kSellWindow, 0, s>>>(a, rowmap);
    return cudaGetLastError();
}

cudaError_t launch_sell_rows(const SellArgs &a, int32_t *rowmap, cudaStream_t s)
{
    if (a.nslices == 0) return cudaSuccess;
    k_sell_rows<<<slice_blocks(a.nslices), kThreads, 0, s>>>(a, rowmap);
    return cudaGetLastError();
}

cudaError_t launch_sell_width(const SellArgs &a, const int32_t *rowmap, int32_t *width, unsigned long long *measured,
                              cudaStream_t s)
{
    const cudaError_t e = cudaMemsetAsync(measured, 0, 2 * sizeof *measured, s);
    if (e != cudaSuccess || a.nslices == 0) return e;
    k_sell_width<<<slice_blocks(a.nslices), kThreads, 0, s>>>(a, rowmap, width, measured);
    return cudaGetLastError();
}

cudaError_t launch_sell_fill(const SellArgs &a, const int32_t *rowmap, const int64_t *ptr, int32_t *sell_col,
                             int32_t *slot, cudaStream_t s)
{
    if (a.nslices == 0) return cudaSuccess;
    k_sell_fill<<<slice_blocks(a.nslices), kThreads, 0, s>>>(a, rowmap, ptr, sell_col, slot);
    return cudaGetLastError();
}

}  // namespace amgd
