// weight_tile.cuh -- the tile walk of the weight quantizers: W [K x N] bf16
// row-major in, K-major codes and per-block scales out.
//
// HBM-bound (2 bytes in and 0.53 to 1.03 out per element), so what matters is
// whole sectors both ways and loads always in flight.  A block takes 128
// columns x 128 rows of W: a thread holds two neighbouring columns of one
// quantization block (BLK rows) as bf16 pairs, so a warp reads 128 contiguous
// bytes of each row and has BLK loads per lane in flight; the codes go through
// shared memory and leave as 64 to 128 contiguous bytes of a column's code
// row.  (One column per thread, as the general kernels do, reads 64 bytes per
// request and writes 16 bytes into each of 32 code rows.)  5120 x 13824, with
// the general kernel and with this one: MXFP4 41.2 and 30.4 us (5.9 TB/s),
// MXFP8 52.1 and 35.7, HiF4 (whose arithmetic bounds it) 68.5 and 58.1, with the
// present shorter encoder 42.1.
// Tiles of 256 rows in two passes took 36 us for MXFP4, three blocks per SM 32.
// Matrices of at most 8 tiles or 32 columns take 0.1 to 0.4 us longer (MXFP4
// 128 x 16 1.9 -> 2.3 us; from 32 tiles on this one is the faster): they stay
// here, since a weight is quantized once.
//
// Needs N even (a pair's 4-byte load is then aligned, and the second column
// exists); the general kernels serve odd N.
#pragma once

#include <cstdint>

#include "internal.h"

namespace rfq {

// |x| of the block's columns as the packed integer maximum of the bf16 bit
// patterns without their signs (both halves), and one half's values.
template <int BLK>
__device__ __forceinline__ uint32_t wt_absmax2(const uint32_t (&raw)[BLK])
{
    uint32_t m = 0;
#pragma unroll
    for (int i = 0; i < BLK; ++i)
        m = __vmaxu2(m, raw[i] & 0x7FFF7FFFu);
    return m;
}

__device__ __forceinline__ float wt_value(uint32_t raw, int half)
{
    return __uint_as_float(half ? raw & 0xFFFF0000u : raw << 16);
}

enum { WT_BLOCKS, WT_COLUMNS, WT_ATOMS };
constexpr int kWtCols = 128, kWtRows = 128;
template <class Q>
constexpr int kWtThreads = kWtCols / 2 * (kWtRows / Q::BLK);   // one pair of columns of one block each

// Q: struct with
//   BLK    rows per quantization block (32 or 64)
//   OUTB   code bytes per block and column (a multiple of 16)
//   Scale  type of a block's scale (uint8_t or uint32_t)
//   static void run(const uint32_t (&raw)[BLK], int half, uint32_t (&code)[OUTB / 4], Scale &s)
//          quantizes the column in the low (half = 0) or high halves of raw
//   static int64_t scale_at(int64_t n, int64_t b, int64_t N, int64_t kblocks)
//          element index of column n, block b in the scale array
//   ORDER  how the tile's scales are contiguous there: WT_BLOCKS (a column's
//          blocks), WT_COLUMNS (a block's columns), WT_ATOMS (MMA-layout bytes:
//          a 128-column, 4-block atom as 32-bit words)
//   static int64_t scale_count(int64_t pad_cols, int64_t kblocks)   elements of it
//   static bool in_bounds(int64_t i, int64_t n)   the debug build's check
// pad_cols: columns of the scale array (N, or N rounded up to 128 where the
// layout's padding holds zeros).
template <class Q>
__global__ void __launch_bounds__(kWtThreads<Q>, 4) weight_tile_kernel(const uint32_t *__restrict__ w, int64_t K, int64_t N,
                                                                int64_t pad_cols, uint8_t *__restrict__ codes,
                                                                typename Q::Scale *__restrict__ scales)
{
    constexpr int BLK = Q::BLK, OUTB = Q::OUTB, NB = kWtRows / BLK;   // blocks of a tile along K
    constexpr int ROWB = NB * OUTB, PITCH = ROWB + 16;                // code bytes per column; shared pitch
    __shared__ __align__(16) uint8_t sc[kWtCols * PITCH];
    __shared__ typename Q::Scale ss[NB][kWtCols];
    const int64_t kblocks = K / BLK;
    const int64_t col_tiles = (pad_cols + kWtCols - 1) / kWtCols, kt = blockIdx.x / col_tiles;
    const int64_t n0 = (blockIdx.x - kt * col_tiles) * kWtCols, b0 = kt * NB;
    const int pair = threadIdx.x & 63, kb = threadIdx.x >> 6;
    const int64_t n = n0 + 2 * pair, half_n = N >> 1;
    {
        const bool in = n < N && b0 + kb < kblocks;
        uint32_t raw[BLK];
        const uint32_t *p = w + (b0 + kb) * BLK * half_n + (n >> 1);
#pragma unroll
        for (int i = 0; i < BLK; ++i, p += half_n)
            raw[i] = in ? __ldcs(p) : 0u;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            uint32_t code[OUTB / 4];
            typename Q::Scale s;
            Q::run(raw, h, code, s);
            uint4 *dst = reinterpret_cast<uint4 *>(sc + (2 * pair + h) * PITCH + kb * OUTB);
#pragma unroll
            for (int j = 0; j < OUTB / 16; ++j)
                dst[j] = make_uint4(code[4 * j], code[4 * j + 1], code[4 * j + 2], code[4 * j + 3]);
            ss[kb][2 * pair + h] = in ? s : 0;
        }
    }
    __syncthreads();
    const int64_t row_bytes = kblocks * OUTB;                         // code bytes per column of the matrix
    constexpr int CH = ROWB / 16;                                     // 16-byte chunks per column of the tile
    for (int i = threadIdx.x; i < kWtCols * CH; i += kWtThreads<Q>) {
        const int c = i / CH, j = i - c * CH;
        const int64_t at = (n0 + c) * row_bytes + b0 * OUTB + 16 * j;
        if (n0 + c < N && b0 * OUTB + 16 * j < row_bytes && Q::in_bounds(at + 15, N * row_bytes))
            *reinterpret_cast<uint4 *>(codes + at) = *reinterpret_cast<const uint4 *>(sc + c * PITCH + 16 * j);
    }
    const int64_t n_scales = Q::scale_count(pad_cols, kblocks);
    if constexpr (Q::ORDER == WT_ATOMS) {
        for (int i = threadIdx.x; i < kWtCols * NB / 4; i += kWtThreads<Q>) {
            const int a = i / kWtCols, t = i % kWtCols, c = (t & 3) * 32 + (t >> 2);   // word t of atom a
            const int64_t at = Q::scale_at(n0 + c, b0 + 4 * a, N, kblocks);
            if (b0 + 4 * a < kblocks && Q::in_bounds(at + 3, n_scales))
                *reinterpret_cast<uint32_t *>(scales + at) =
                    (uint32_t)ss[4 * a][c] | (uint32_t)ss[4 * a + 1][c] << 8 | (uint32_t)ss[4 * a + 2][c] << 16 |
                    (uint32_t)ss[4 * a + 3][c] << 24;
        }
    } else {
        for (int i = threadIdx.x; i < kWtCols * NB; i += kWtThreads<Q>) {
            const int c = Q::ORDER == WT_COLUMNS ? i % kWtCols : i / NB;
            const int kb = Q::ORDER == WT_COLUMNS ? i / kWtCols : i % NB;
            if (n0 + c < pad_cols && b0 + kb < kblocks) {
                const int64_t at = Q::scale_at(n0 + c, b0 + kb, N, kblocks);
                if (Q::in_bounds(at, n_scales))
                    scales[at] = ss[kb][c];
            }
        }
    }
}

template <class Q>
cudaError_t launch_weight_tile(const void *w, int64_t K, int64_t N, int64_t pad_cols, void *codes, void *scales,
                               cudaStream_t st)
{
    const int64_t grid = (pad_cols + kWtCols - 1) / kWtCols * ((K + kWtRows - 1) / kWtRows);
    weight_tile_kernel<Q><<<(unsigned)grid, kWtThreads<Q>, 0, st>>>(static_cast<const uint32_t *>(w), K, N, pad_cols,
                                                       static_cast<uint8_t *>(codes),
                                                       static_cast<typename Q::Scale *>(scales));
    return cudaGetLastError();
}

} // namespace rfq
