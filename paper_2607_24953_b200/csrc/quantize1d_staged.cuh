// 1 x 32-block quantizers, FP4 and MXFP8, along the rows of x and of its transpose, for matrices whose rows start anywhere or that are not made
// of whole 128 x 128 tiles: the 2D quantizer's staged tiles (staged_tile.cuh).
//
// A CTA of four warps owns 128 x 128 elements, a warp 32 rows x 128 columns, a lane 8 rows x 16 columns.  Along the rows a block is two
// lanes' halves of a row (one shuffle a row); along the columns it is one column of the warp's 32 rows, whose maxima four lanes
// reduce and whose codes cross shared memory, as in the kernels for whole tiles.  Bound by instructions: a tile's pass through shared
// memory, and code that runs once on an SM takes about ten cycles an instruction.  So the loop over a lane's rows is not unrolled where a row
// is all that is needed (1999 x 2731 FP4 unrolled 8.2 us, rolled 7.1; reading rows twice to roll the other form's loop loses, 8.3 / 10.4).  us, FP4 /
// MXFP8, element-wise loads before and now: 1999 x 2731 12.1 / 12.1 -> 7.2 / 7.1, 4099 x 5001 38.8 / 38.9 -> 14.9 / 14.8 (8.0 / 9.5 at the measured copy
// bandwidth); transposed 11.3 / 12.9 -> 7.0 / 7.5, 23.4 / 32.4 -> 15.9 / 17.2 (17.9 / 19.0 with every row checked by itself,
// 17.2 / 17.9 with four CTAs an SM instead of five).
#pragma once

#include <cuda_bf16.h>

#include "common.cuh"
#include "quant_device.cuh"
#include "staged_tile.cuh"

namespace fp4q {

struct Staged1dParams {
    const uint16_t *x;
    int64_t rows, cols, ld_x;
    uint8_t *q;
    int64_t ld_q;
    uint8_t *scale;
    int64_t ld_s;
    int64_t grid_x;   // tiles along the columns; set by the launch
};

// Which matrices come here.  The work goes by tiles of 128 x 128, whatever is in them: 5 us and 0.45 a million elements of the tiles.  us, the other
// kernels and this one:
// Rows off 16 bytes, blocks along the rows.  Reading them element by element takes 2.2 us and 2 a million elements of long rows, 1 of rows of a few
// hundred, however few rows there are: 300 x 777 3.4 / 5.1, 1999 x 1003 6.2 / 5.4, 3001 x 3001 18.7 / 8.4; 1 x 2000001 6.2 / 27, 8 x 300001 6.3 / 11.8, 17 x 150001
// 8.3 / 8.7, 20 x 100001 6.2 / 5.6, 28 x 100001 8.4 / 5.9; 60000 x 33 3.9 / 8.9, 20001 x 193 6.5 / 7.4, 10001 x 301 5.2 / 6.2, 10001 x 361 6.6 / 6.3, 30001 x 385
// 19.0 / 13.5 (but 30001 x 301 10.6 / 9.9).
inline bool staged_rows_pay(int64_t rows, int64_t cols) { return rows >= 20 && cols >= 360 && rows * cols >= 3 << 19; }
// The transpose of what is not made of whole tiles, rows on words: a kernel that reads words, FP4 12000 x 6002 46.6 / 50.0, 16000 x 11010 118 / 113, MXFP8
// 5000 x 7002 28.6 / 29.6, 6000 x 6002 32.1 / 30.1, 16000 x 4002 56.1 / 49.5; in tiles that are not nearly full 32 x 300002 6.0 / 19.5, 129 x 60002 5.5 / 10.5.
// Others, element by element or here: 300 x 777 7.7 / 4.7, 3001 x 3001 12.9 / 8.8, 5001 x 31 7.8 / 5.2; 1 x 2000001 34 / 114, 1 x 5001 2.4 / 3.8, 8 x 70001 3.9 / 6.8,
// 16 x 151937 6.6 / 12.9, 20 x 5001 5.5 / 4.6, 33 x 60001 8.3 / 7.5, 600001 x 3 22.6 / 51, 70001 x 3 5.0 / 8.3, 200001 x 17 16.4 / 19.4, 60000 x 33 8.8 / 8.5.
inline bool staged_transpose_pays(int64_t rows, int64_t cols, bool words, bool fp8)
{
    const int64_t elements = rows * cols, tiles = ceil_div(rows, 128) * ceil_div(cols, 128), area = tiles * 128 * 128;
    if (words) return elements >= (fp8 ? 34 << 20 : 96 << 20) && 8 * elements >= 7 * area;
    return rows >= 16 && cols >= 8 && (tiles <= 400 || 17 * elements >= 4 * area);
}

// UE8M0 code of MXFP8's truncation-free scale: the smallest e with 448 * 2^e >= M, from the BF16 magnitude bits of M.
__device__ __forceinline__ int e4m3_scale_code(uint32_t mbits)
{
    const int be = (int)(mbits >> 7), m7 = (int)(mbits & 0x7F);
    const int code = be == 0 ? 0 : be - 8 + (m7 > 0x60 ? 1 : 0);
    return code < 0 ? 0 : code;
}

namespace staged1d {

template <bool FP8>
__device__ __forceinline__ int scale_code(uint32_t mbits) { return FP8 ? e4m3_scale_code(mbits) : scale_code_from_max(mbits); }
// Packed |.| maximum with NaN propagation: a non-finite entry shows in the result.
__device__ __forceinline__ uint32_t max_abs_nan(uint32_t a, uint32_t b)
{
    const __nv_bfloat162 m = __hmax2_nan(*reinterpret_cast<const __nv_bfloat162 *>(&a), __habs2(*reinterpret_cast<const __nv_bfloat162 *>(&b)));
    return *reinterpret_cast<const uint32_t *>(&m);
}
// The same over finite entries.
__device__ __forceinline__ uint32_t max_abs_finite(uint32_t a, uint32_t b)
{
    const uint32_t lo = b & 0x7FFFu, hi = (b >> 16) & 0x7FFFu;
    return max(a & 0xFFFFu, lo < 0x7F80u ? lo : 0u) | max(a >> 16, hi < 0x7F80u ? hi : 0u) << 16;
}
__device__ __forceinline__ uint32_t max_pairs(uint32_t a, uint32_t b) { return max(a & 0xFFFFu, b & 0xFFFFu) | max(a >> 16, b >> 16) << 16; }
__device__ __forceinline__ bool any_nonfinite(uint32_t m) { return (m & 0x7FFFu) >= 0x7F80u || (m >> 16 & 0x7FFFu) >= 0x7F80u; }
// NaN -> +0 (infinities saturate in the conversions).
__device__ __forceinline__ uint32_t without_nan(uint32_t w)
{
    if ((w & 0x7FFFu) > 0x7F80u) w &= 0xFFFF0000u;
    if ((w >> 16 & 0x7FFFu) > 0x7F80u) w &= 0x0000FFFFu;
    return w;
}
__device__ __forceinline__ float low(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float high(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

// Blocks along the rows: two lanes' halves of a row.
template <bool FP8>
__device__ __forceinline__ void quantize_rows(const Staged1dParams &p, int64_t tile_row0, int64_t bx, const uint8_t *rows, int lane)
{
    const int t = lane >> 3, rg = (lane >> 1) & 3, ch = lane & 1;
    const int64_t col0 = bx * 128 + 32 * t + 16 * ch;
#pragma unroll 1
    for (int r = 0; r < 8; r++) {
        const int64_t row = tile_row0 + 8 * rg + r;
        uint32_t v[8], m = 0u;
        read_staged_row(p, tile_row0, bx * 128, rows, lane, r, v);
#pragma unroll
        for (int k = 0; k < 8; k++) m = max_abs_nan(m, v[k]);
        if (__any_sync(0xFFFFFFFFu, any_nonfinite(m))) {
            m = 0u;
#pragma unroll
            for (int k = 0; k < 8; k++) {
                m = max_abs_finite(m, v[k]);
                v[k] = without_nan(v[k]);
            }
        }
        m = max_pairs(m, __shfl_xor_sync(0xFFFFFFFFu, m, 1));
        const int code = scale_code<FP8>(max(m & 0x7FFFu, m >> 16 & 0x7FFFu));
        const uint32_t inv2 = (uint32_t)(254 - code) * 0x00800080u;   // 2^-e, twice as BF16
#pragma unroll
        for (int k = 0; k < 8; k++) v[k] = scale_pair(v[k], inv2);
        if (row < p.rows && col0 - 16 * ch < p.cols) {
            uint8_t *dst = p.q + row * p.ld_q;
            if (FP8) {
                uint32_t out[4];
#pragma unroll
                for (int w = 0; w < 4; w++) out[w] = cvt_rn_e4m3x4(high(v[2 * w + 1]), low(v[2 * w + 1]), high(v[2 * w]), low(v[2 * w]));
                *reinterpret_cast<uint4 *>(dst + col0) = make_uint4(out[0], out[1], out[2], out[3]);
            } else {
                uint32_t out[2];
#pragma unroll
                for (int w = 0; w < 2; w++) {
                    const float f[8] = {low(v[4 * w]), high(v[4 * w]), low(v[4 * w + 1]), high(v[4 * w + 1]), low(v[4 * w + 2]), high(v[4 * w + 2]), low(v[4 * w + 3]), high(v[4 * w + 3])};
                    out[w] = cvt_rn_e2m1x8(f);
                }
                *reinterpret_cast<uint2 *>(dst + (col0 >> 1)) = make_uint2(out[0], out[1]);
            }
            if (ch == 0) p.scale[row * p.ld_s + (col0 >> 5)] = (uint8_t)code;
        }
        __syncwarp();
    }
}

template <bool FP8>
__global__ void __launch_bounds__(128) quantize1d_staged_kernel(const __grid_constant__ Staged1dParams p)
{
    __shared__ __align__(16) uint8_t rows[4 * kStageWarpBytes];
    wait_for_predecessor();
    admit_successor();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t by = (int64_t)blockIdx.x / p.grid_x, bx = (int64_t)blockIdx.x - by * p.grid_x, tile_row0 = by * 128 + 32 * warp;
    if (tile_row0 >= p.rows) return;   // 33 x 200001 11.3 -> 9.5 us
    stage_tile_rows(p, tile_row0, bx * 128, rows + warp * kStageWarpBytes, lane);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
    quantize_rows<FP8>(p, tile_row0, bx, rows + warp * kStageWarpBytes, lane);
}

// Blocks along the columns: one column of the warp's 32 rows, which four lanes hold.
template <bool FP8>
__global__ void __launch_bounds__(128, 5) quantize1d_t_staged_kernel(const __grid_constant__ Staged1dParams p)
{
    __shared__ __align__(16) uint8_t stage[4 * kStageWarpBytes];   // the rows, then the codes of 128 columns
    __shared__ uint32_t sc_stage[128];                             // a column's four scale codes
    static_assert(4 * kStageWarpBytes >= 128 * 128, "the codes fit in the rows");
    wait_for_predecessor();
    admit_successor();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, t = lane >> 3, rg = (lane >> 1) & 3, ch = lane & 1;
    const int64_t by = (int64_t)blockIdx.x / p.grid_x, bx = (int64_t)blockIdx.x - by * p.grid_x, tile_row0 = by * 128 + 32 * warp;
    uint32_t raw[8][8], m[8];
    stage_tile_rows(p, tile_row0, bx * 128, stage + warp * kStageWarpBytes, lane);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
#pragma unroll
    for (int r = 0; r < 8; r++) read_staged_row_uncut(p, tile_row0, bx * 128, stage + warp * kStageWarpBytes, lane, r, raw[r]);
    cut_staged_rows(raw, (int)max((int64_t)0, min((int64_t)8, p.rows - tile_row0 - 8 * rg)), (int)max((int64_t)0, min((int64_t)16, p.cols - bx * 128 - 32 * t - 16 * ch)));
    bool nonfinite = false;
#pragma unroll
    for (int k = 0; k < 8; k++) {
        m[k] = 0u;
#pragma unroll
        for (int r = 0; r < 8; r++) m[k] = max_abs_nan(m[k], raw[r][k]);
        nonfinite |= any_nonfinite(m[k]);
    }
    if (__any_sync(0xFFFFFFFFu, nonfinite)) {
#pragma unroll
        for (int k = 0; k < 8; k++) {
            m[k] = 0u;
#pragma unroll
            for (int r = 0; r < 8; r++) {
                m[k] = max_abs_finite(m[k], raw[r][k]);
                raw[r][k] = without_nan(raw[r][k]);
            }
        }
    }
#pragma unroll
    for (int k = 0; k < 8; k++) {
#pragma unroll
        for (int s = 2; s <= 4; s <<= 1) m[k] = max_abs_nan(m[k], __shfl_xor_sync(0xFFFFFFFFu, m[k], s));   // all finite
        const int c0 = scale_code<FP8>(m[k] & 0x7FFFu), c1 = scale_code<FP8>(m[k] >> 16 & 0x7FFFu);
        const uint32_t inv2 = (uint32_t)(254 - c0) << 7 | (uint32_t)(254 - c1) << 23;
#pragma unroll
        for (int r = 0; r < 8; r++) raw[r][k] = scale_pair(raw[r][k], inv2);
        if (rg == 0) {
            uint8_t *sc = reinterpret_cast<uint8_t *>(sc_stage) + (32 * t + 16 * ch + 2 * k) * 4 + warp;
            sc[0] = (uint8_t)c0;
            sc[4] = (uint8_t)c1;
        }
    }
    __syncthreads();   // every warp has read its rows
    // A column's codes are 64 or 128 bytes of staging, in 16-byte chunks XORed by
    // the column's group so that a warp's stores spread over the banks.
#pragma unroll
    for (int c = 0; c < 16; c++) {
        const int col_local = 32 * t + 16 * ch + c;
        float v[8];
#pragma unroll
        for (int r = 0; r < 8; r++) v[r] = (c & 1) ? high(raw[r][c >> 1]) : low(raw[r][c >> 1]);
        if (FP8) {
            const int chunk = (warp * 2 + (rg >> 1)) ^ ((col_local >> 4) & 7);
            reinterpret_cast<uint2 *>(stage)[(col_local * 8 + chunk) * 2 + (rg & 1)] = make_uint2(cvt_rn_e4m3x4(v[3], v[2], v[1], v[0]), cvt_rn_e4m3x4(v[7], v[6], v[5], v[4]));
        } else {
            reinterpret_cast<uint32_t *>(stage)[col_local * 16 + (((warp ^ t) << 2) | rg)] = cvt_rn_e2m1x8(v);
        }
    }
    __syncthreads();
    constexpr int kChunks = FP8 ? 8 : 4;   // of 16 bytes a column
#pragma unroll
    for (int k = 0; k < kChunks; k++) {
        const int col_local = threadIdx.x / kChunks + 128 / kChunks * k, chunk = threadIdx.x % kChunks;
        const int64_t col = bx * 128 + col_local;
        if (col >= p.cols || by * 128 + (FP8 ? chunk >> 1 : chunk) * 32 >= p.rows) continue;
        const int at = chunk ^ (FP8 ? (col_local >> 4) & 7 : col_local >> 5);
        *reinterpret_cast<uint4 *>(p.q + col * p.ld_q + by * (16 * kChunks) + 16 * chunk) = reinterpret_cast<const uint4 *>(stage)[col_local * kChunks + at];
    }
    const int64_t col = bx * 128 + threadIdx.x;
    if (col < p.cols) {
        uint8_t *dst = p.scale + col * p.ld_s + by * 4;
        const uint32_t w = sc_stage[threadIdx.x];
#pragma unroll
        for (int b = 0; b < 4; b++)
            if (by * 128 + 32 * b < p.rows) dst[b] = (uint8_t)(w >> (8 * b));
    }
}

}  // namespace staged1d

// FP8: E4M3 payload (MXFP8), otherwise E2M1; transposed: the encoding of x^T.  Rounding to nearest.  The caller has checked its arguments.
template <bool FP8>
static fp4q_status launch_quantize1d_staged(Staged1dParams p, bool transposed, cudaStream_t stream)
{
    p.grid_x = ceil_div(p.cols, 128);
    const int64_t n_cta = p.grid_x * ceil_div(p.rows, 128);
    if (n_cta > 0x7FFFFFFF) return FP4Q_ERR_UNSUPPORTED;
    return launched(launch_dependent(transposed ? staged1d::quantize1d_t_staged_kernel<FP8> : staged1d::quantize1d_staged_kernel<FP8>,
                                     dim3((unsigned)n_cta), 128, stream, p));
}

}  // namespace fp4q
