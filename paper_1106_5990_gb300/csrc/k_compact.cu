// k_compact.cu -- the strength graph M^1 (§4.2) as CSR from the per-slot
// flags and per-row counts written by the edge pass.
//
// No device-wide waits.  The last of up to three launches has every block write
// s_row_ptr for its rows (block scan of the counts plus the tile's offset) and
// compact the flagged slots of its rows' contiguous slot range into s_col (16
// flag bytes per thread, counted with popc, one block scan per 4096 slots),
// keeping A's row and slot order.  Where a tile's offset comes from depends on
// the size, since each launch before it costs two to three microseconds:
//   n <= kDirectRows: the block sums the counts of all earlier rows itself (at
//     most 128 KB from the L2) over tiles of 256 rows -- one launch;
//   up to kLookTiles tiles of kTileRows rows: tile sums in one launch, each
//     block then adds up the sums before its own -- two launches;
//   beyond: one block scans the tile sums in between -- three launches.
// (64 x 64 5-point: 8.2 us for the three launches, 4.0 for the one.)
#include <type_traits>

#include "amgd_internal.cuh"

namespace amgd {
namespace {

constexpr int kSumThreads = 256;
constexpr int kCompactThreads = 256;
constexpr int kRowsPerThread = kTileRows / kCompactThreads;     // 4
constexpr int kSlotsPerThread = 16;                             // one 16-byte flag load

// exclusive block scan of one int per thread; returns the block total
template <int NT>
__device__ __forceinline__ int block_exclusive_scan(int v, int &total, int *smem_warp)
{
    const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) smem_warp[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        int w = lane < NT / 32 ? smem_warp[lane] : 0;
        int winc = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, winc, o);
            if (lane >= o) winc += t;
        }
        if (lane < NT / 32) smem_warp[lane] = winc - w;   // exclusive warp offsets
        if (lane == NT / 32 - 1) smem_warp[32] = winc;     // block total
    }
    __syncthreads();
    const int out = smem_warp[warp] + inc - v;
    total = smem_warp[32];
    __syncthreads();
    return out;
}

__global__ void __launch_bounds__(kSumThreads)
k_tile_sums(const int32_t *count, int32_t n, int32_t *tile_sum)
{
    __shared__ int sm[33];
    chain_wait();
    chain_release();
    const int64_t r = (int64_t)blockIdx.x * kTileRows + threadIdx.x * 4;
    int s = 0;
    if (r + 3 < n) {
        const int4 c = *reinterpret_cast<const int4 *>(count + r);
        s = c.x + c.y + c.z + c.w;
    } else {
        for (int k = 0; k < 4; ++k) s += (r + k < n) ? count[r + k] : 0;
    }
    int total;
    block_exclusive_scan<kSumThreads>(s, total, sm);
    if (threadIdx.x == 0) tile_sum[blockIdx.x] = total;
}

// in-place exclusive scan of ntiles tile sums by one block
__global__ void __launch_bounds__(1024) k_tile_scan(int32_t *tile_sum, int32_t ntiles)
{
    __shared__ int sm[33];
    chain_wait();
    chain_release();
    int carry = 0;
    for (int base = 0; base < ntiles; base += 1024) {
        const int k = base + threadIdx.x;
        const int v = k < ntiles ? tile_sum[k] : 0;
        int total;
        const int ex = block_exclusive_scan<1024>(v, total, sm);
        if (k < ntiles) tile_sum[k] = carry + ex;
        carry += total;
    }
}

// where a tile's offset comes from
enum Offset { OFF_SCANNED, OFF_TILE_SUMS, OFF_COUNTS };

// kept entries of all rows before the block's tile (same value in every thread)
template <Offset OFF>
__device__ __forceinline__ int64_t tile_offset(const int32_t *count, const int32_t *tile,
                                               int64_t row0, int *sm)
{
    if constexpr (OFF == OFF_SCANNED) {
        return tile[blockIdx.x];
    } else {
        // at most kLookTiles tile sums, or kDirectRows counts (row0 is a
        // multiple of the block's rows, so the 16-byte loads end at it)
        const int32_t *src = OFF == OFF_COUNTS ? count : tile;
        const int64_t len = OFF == OFF_COUNTS ? row0 : (int64_t)blockIdx.x;
        int s = 0;
        const int64_t quads = len / 4;
        for (int64_t q = threadIdx.x; q < quads; q += kCompactThreads) {
            const int4 c = *(reinterpret_cast<const int4 *>(src) + q);
            s += c.x + c.y + c.z + c.w;
        }
        for (int64_t q = 4 * quads + threadIdx.x; q < len; q += kCompactThreads) s += src[q];
        int total;
        block_exclusive_scan<kCompactThreads>(s, total, sm);
        return total;
    }
}

// row pointers of the block's RPT * kCompactThreads rows; returns their total
template <int RPT>
__device__ __forceinline__ int write_row_ptr(const int32_t *count, int32_t n, int64_t row0,
                                             int64_t row_end, int64_t off, int64_t *row_ptr, int *sm)
{
    int c[RPT];
    int mine = 0;
    const int64_t rbase = row0 + (int64_t)threadIdx.x * RPT;
#pragma unroll
    for (int k = 0; k < RPT; ++k) {
        c[k] = (rbase + k < row_end) ? count[rbase + k] : 0;
        mine += c[k];
    }
    int total;
    int run = block_exclusive_scan<kCompactThreads>(mine, total, sm);
#pragma unroll
    for (int k = 0; k < RPT; ++k) {
        if (rbase + k < row_end) row_ptr[rbase + k] = off + run;
        run += c[k];
    }
    if (row_end == n && threadIdx.x == 0) row_ptr[n] = off + total;
    return total;
}

template <int RPT, Offset OFF>
__global__ void __launch_bounds__(kCompactThreads)
k_compact(const int32_t *count, const int32_t *__restrict__ rp,
          const int32_t *__restrict__ col, const uint8_t *flag, int32_t n,
          const int32_t *tile, int64_t *s_row_ptr,
          int32_t *s_col)
{
    __shared__ int sm[33];
    const int64_t row0 = (int64_t)blockIdx.x * (RPT * kCompactThreads);
    const int64_t row_end = min((int64_t)n, row0 + RPT * kCompactThreads);
    const int64_t s0 = rp[row0], s1 = rp[row_end];
    chain_wait();
    chain_release();
    const int64_t off = tile_offset<OFF>(count, tile, row0, sm);
    write_row_ptr<RPT>(count, n, row0, row_end, off, s_row_ptr, sm);

    // kept slots of the tile's slot range [s0, s1), in slot order: every
    // thread takes 16 consecutive flag bytes (one 16-byte load from a
    // 16-byte-aligned base; the flag array is padded by 16 bytes) and, if any
    // is set, their 16 column indices (four 16-byte loads; the column array is
    // padded by 64 bytes).  The kept columns of a chunk are collected in
    // shared memory and written out with coalesced stores.
    __shared__ int32_t kept[kCompactThreads * kSlotsPerThread];
    int64_t out = off;
    for (int64_t base = s0 & ~(int64_t)15; base < s1;
         base += (int64_t)kCompactThreads * kSlotsPerThread) {
        const int64_t first = base + (int64_t)threadIdx.x * kSlotsPerThread;
        uint4 v = make_uint4(0, 0, 0, 0);
        if (first < s1) v = *reinterpret_cast<const uint4 *>(flag + first);
        uint32_t w[4] = {v.x, v.y, v.z, v.w};
        // clear the bytes outside [s0, s1)
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const int64_t slot = first + k;
            if (slot < s0 || slot >= s1) w[k / 4] &= ~(0xffu << (8 * (k % 4)));
        }
        const int cnt = __popc(w[0]) + __popc(w[1]) + __popc(w[2]) + __popc(w[3]);
        int chunk;
        int pos = block_exclusive_scan<kCompactThreads>(cnt, chunk, sm);
        if (cnt) {
            int c16[16];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int4 c4 = __ldg(reinterpret_cast<const int4 *>(col + first) + q);
                c16[4 * q] = c4.x; c16[4 * q + 1] = c4.y; c16[4 * q + 2] = c4.z; c16[4 * q + 3] = c4.w;
            }
#pragma unroll
            for (int k = 0; k < 16; ++k)
                if ((w[k / 4] >> (8 * (k % 4))) & 1u) kept[pos++] = c16[k];
        }
        __syncthreads();
        for (int q = threadIdx.x; q < chunk; q += kCompactThreads) s_col[out + q] = kept[q];
        __syncthreads();
        out += chunk;
    }
}

// row pointers only
template <int RPT, Offset OFF>
__global__ void __launch_bounds__(kCompactThreads)
k_row_ptr(const int32_t *count, int32_t n, const int32_t *tile,
          int64_t *row_ptr)
{
    __shared__ int sm[33];
    const int64_t row0 = (int64_t)blockIdx.x * (RPT * kCompactThreads);
    const int64_t row_end = min((int64_t)n, row0 + RPT * kCompactThreads);
    chain_wait();
    chain_release();
    const int64_t off = tile_offset<OFF>(count, tile, row0, sm);
    write_row_ptr<RPT>(count, n, row0, row_end, off, row_ptr, sm);
}

constexpr int32_t kDirectRows = 32768;
constexpr int kLookTiles = 2048;

// tile sums (and their scan) where the size calls for them, then
// last(rows per thread, offset source, blocks)
template <class Last>
cudaError_t with_offsets(const int32_t *count, int32_t n, int32_t *tile_sum, cudaStream_t s, const Last &last)
{
    if (n <= kDirectRows)
        return last(std::integral_constant<int, 1>(), std::integral_constant<Offset, OFF_COUNTS>(),
                    (unsigned)((n + kCompactThreads - 1) / kCompactThreads));
    const int ntiles = (int)(((int64_t)n + kTileRows - 1) / kTileRows);
    cudaError_t e = launch_chained(k_tile_sums, (unsigned)ntiles, kSumThreads, 0, s, count, n, tile_sum);
    if (e != cudaSuccess) return e;
    if (ntiles <= kLookTiles)
        return last(std::integral_constant<int, kRowsPerThread>(), std::integral_constant<Offset, OFF_TILE_SUMS>(),
                    (unsigned)ntiles);
    e = launch_chained(k_tile_scan, 1u, 1024, 0, s, tile_sum, (int32_t)ntiles);
    if (e != cudaSuccess) return e;
    return last(std::integral_constant<int, kRowsPerThread>(), std::integral_constant<Offset, OFF_SCANNED>(),
                (unsigned)ntiles);
}

}  // namespace

cudaError_t launch_row_ptr(const int32_t *count, int32_t n, int32_t *tile_sum, int64_t *row_ptr,
                           cudaStream_t s)
{
    if (n == 0) {
        cudaError_t e = cudaMemsetAsync(row_ptr, 0, sizeof(int64_t), s);
        return e != cudaSuccess ? e : cudaGetLastError();
    }
    return with_offsets(count, n, tile_sum, s, [&](auto rpt, auto off, unsigned blocks) {
        return launch_chained(k_row_ptr<decltype(rpt)::value, decltype(off)::value>, blocks, kCompactThreads, 0, s,
                              count, n, (const int32_t *)tile_sum, row_ptr);
    });
}

cudaError_t launch_strength(const int32_t *count, const int32_t *rp_orig, const int32_t *col_orig,
                            const uint8_t *flag, int32_t n, int32_t *tile_sum,
                            int64_t *s_row_ptr, int32_t *s_col, cudaStream_t s)
{
    if (n == 0) {
        cudaError_t e = cudaMemsetAsync(s_row_ptr, 0, sizeof(int64_t), s);
        return e != cudaSuccess ? e : cudaGetLastError();
    }
    return with_offsets(count, n, tile_sum, s, [&](auto rpt, auto off, unsigned blocks) {
        return launch_chained(k_compact<decltype(rpt)::value, decltype(off)::value>, blocks, kCompactThreads, 0, s,
                              count, rp_orig, col_orig, flag, n, (const int32_t *)tile_sum, s_row_ptr, s_col);
    });
}

}  // namespace amgd
