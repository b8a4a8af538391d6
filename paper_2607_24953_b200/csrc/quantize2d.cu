// fp4q_quantize2d: 2D-block (32x32) FP4 quantization with dual-layout pack, sm_100a.
//
// One pass over HBM: 2 B/element read, 0.5 + 0.5 B/element written, 1 B per 1024 elements of scale.
// A CTA of 4 warps owns a 128x128 element block; a warp owns 32 rows x 128 columns (four 32x32
// blocks side by side); 8 lanes own one 32x32 block, each lane 8 rows x 16 consecutive columns
// (one 256-bit load per row, all eight issued before anything else).  While the loads are in flight
// the lane draws its Philox bytes (they do not depend on the data) and parks them in shared memory.
// The block maximum is reduced with warp shuffles over the 8 lanes, the E2M1 codes come from the
// hardware converts, the row-major payload goes straight to global memory (8 B per lane and row,
// 64 B contiguous per row and warp) and the transposed payload is built with an in-register 8x8
// nibble transpose, staged through 8 KB of shared memory and written as 64 B contiguous segments.
// CTAs whose tile lies fully inside a 32-byte aligned tensor run a check-free body, its ragged edges and tensors on 16-byte
// boundaries a general body with the same arithmetic; tensors whose rows start anywhere have a kernel that stages its
// tile (quantize2d_staged_kernel).
//
// Rounding: x 2^-e (exact in FP32) goes through the hardware converts cvt.rn.satfinite.e2m1x2.f32
// (nearest even) or cvt.rs.satfinite.e2m1x4.f32 (stochastic).  The stochastic convert adds 16 random bits
// below the kept mantissa bit and truncates; the elements that land in nibbles 0 and 2 take the upper 8
// of their 16 bits from rbits[23:16] and rbits[31:24] and the lower 8 from rbits[7:0] and rbits[15:8]
// (the other two inputs reuse the same bits in reversed order).  With the lower bytes zero and only
// those two inputs used, the instruction computes exactly "up iff floor(256 p) + r8 >= 256" for two
// elements at a time: the element's random byte is routed into place with one PRMT.  Blocks that
// contain non-finite values take a scalar path that rounds on the fp16 bit pattern of |x| 2^(-e-14)
// (magnitude code in bits 11..9, position between neighbours in bits 8..0).
#include <cuda_bf16.h>

#include "common.cuh"
#include "quant_device.cuh"
#include "staged_tile.cuh"

namespace fp4q {

struct Quant2dParams {
    const uint16_t *x;
    int64_t rows, cols, ld_x;
    uint8_t *q_rm;
    int64_t ld_rm;
    uint8_t *q_t;
    int64_t ld_t;
    uint8_t *scale;
    int64_t ld_s;
    int64_t grid_x;           // CTAs along the column direction
    uint32_t tensor_id;
    uint32_t flags;
    int x_vec_ok;             // 2: x 32-byte aligned, ld_x % 16 == 0 (256-bit loads); 1: 16-byte aligned, ld_x % 8 == 0
    int waits;                // the kernel waits for its predecessor before it reads (0: a later tensor of a multi-tensor call)
    int rng_aligned;          // nearest, or cols % 16 == 0 and index not transposed: one Philox block per 16-element segment
    PhiloxRoundKeys keys;
};

__device__ __noinline__ uint32_t philox_byte(const Quant2dParams &p, uint64_t idx)
{
    uint32_t o[4];
    const uint64_t blk = idx >> 4;
    philox4x32_10((uint32_t)blk, (uint32_t)(blk >> 32), p.tensor_id, 0u, p.keys, o);
    const uint32_t w = (idx >> 2) & 3;
    const uint32_t word = w == 0 ? o[0] : w == 1 ? o[1] : w == 2 ? o[2] : o[3];
    return (word >> (8 * (idx & 3))) & 0xFFu;
}

// In-register transpose of an 8x8 matrix of nibbles: a[r] holds row r (nibble c = column c);
// on return a[c] holds column c (nibble r = row r).
__device__ __forceinline__ void transpose8x8_nibbles(uint32_t a[8])
{
#pragma unroll
    for (int r = 0; r < 4; r++) {   // swap 4x4 quadrants (16-bit halves between rows r and r+4)
        const uint32_t lo = __byte_perm(a[r], a[r + 4], 0x5410), hi = __byte_perm(a[r], a[r + 4], 0x7632);
        a[r] = lo; a[r + 4] = hi;
    }
#pragma unroll
    for (int q = 0; q < 4; q++) {   // swap 2x2 blocks (bytes between rows r and r+2)
        const int r = (q & 1) + 4 * (q >> 1);
        const uint32_t lo = __byte_perm(a[r], a[r + 2], 0x6240), hi = __byte_perm(a[r], a[r + 2], 0x7351);
        a[r] = lo; a[r + 2] = hi;
    }
#pragma unroll
    for (int r = 0; r < 8; r += 2) {  // swap single nibbles between rows r and r+1
        const uint32_t lo = (a[r] & 0x0F0F0F0Fu) | ((a[r + 1] & 0x0F0F0F0Fu) << 4);
        const uint32_t hi = ((a[r] >> 4) & 0x0F0F0F0Fu) | (a[r + 1] & 0xF0F0F0F0u);
        a[r] = lo; a[r + 1] = hi;
    }
}

// FP32 sources (fp4q_quantize2d_multi_f32): a segment is rounded to BF16 as it arrives, to nearest even like a BF16 copy of the tensor,
// and everything after that is the same.
__device__ __forceinline__ uint32_t pack_bf16(uint32_t lo, uint32_t hi)
{
    const __nv_bfloat162 b = __floats2bfloat162_rn(__uint_as_float(lo), __uint_as_float(hi));
    return *reinterpret_cast<const uint32_t *>(&b);
}
__device__ __forceinline__ void load_segment_f32(const Quant2dParams &p, int64_t i, int64_t j0, uint32_t out[8])
{
    const float *src = reinterpret_cast<const float *>(p.x) + i * p.ld_x + j0;
    const bool row_ok = i < p.rows;
#pragma unroll
    for (int q = 0; q < 4; q++) {
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (row_ok && j0 + 4 * q + 4 <= p.cols) {
            v = load_global(reinterpret_cast<const uint4 *>(src) + q);
        } else if (row_ok) {
            uint32_t e[4];
#pragma unroll
            for (int k = 0; k < 4; k++) e[k] = j0 + 4 * q + k < p.cols ? __float_as_uint(load_global(src + 4 * q + k)) : 0u;
            v = make_uint4(e[0], e[1], e[2], e[3]);
        }
        out[2 * q] = pack_bf16(v.x, v.y);
        out[2 * q + 1] = pack_bf16(v.z, v.w);
    }
}

__device__ __forceinline__ void load_segment(const Quant2dParams &p, int64_t i, int64_t j0, uint32_t out[8])
{
    if (i >= p.rows || j0 >= p.cols) {
#pragma unroll
        for (int k = 0; k < 8; k++) out[k] = 0u;
        return;
    }
    const uint16_t *src = p.x + i * p.ld_x + j0;
    if (p.x_vec_ok == 2 && j0 + 16 <= p.cols) {
        asm volatile("ld.global.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=r"(out[0]), "=r"(out[1]), "=r"(out[2]), "=r"(out[3]), "=r"(out[4]), "=r"(out[5]), "=r"(out[6]),
                       "=r"(out[7])
                     : "l"(src));
    } else if (p.x_vec_ok && j0 + 16 <= p.cols) {
        const uint4 a = load_global(reinterpret_cast<const uint4 *>(src));
        const uint4 b = load_global(reinterpret_cast<const uint4 *>(src) + 1);
        out[0] = a.x; out[1] = a.y; out[2] = a.z; out[3] = a.w;
        out[4] = b.x; out[5] = b.y; out[6] = b.z; out[7] = b.w;
    } else {
#pragma unroll
        for (int k = 0; k < 8; k++) {
            const uint32_t lo = (j0 + 2 * k < p.cols) ? (uint32_t)load_global(src + 2 * k) : 0u;
            const uint32_t hi = (j0 + 2 * k + 1 < p.cols) ? (uint32_t)load_global(src + 2 * k + 1) : 0u;
            out[k] = lo | (hi << 16);
        }
    }
}

// ---- staged tiles: tensors whose rows start anywhere (odd pitch, unaligned base) or whose 16-element segments straddle
// Philox blocks (cols % 16 != 0).
//
// Per-element 16-bit loads cost 128 load instructions a lane, and one Philox call per element sixteen times the
// arithmetic.  Here a warp copies its 32 rows as aligned 16-byte pieces (17 cover 128 elements at any offset) into its own
// staging rows with cp.async and draws the nine Philox blocks that each row's 128 elements touch, once per warp, while they are on
// their way; each lane reads its segments back with three 128-bit shared loads a row and shifts them, and their random bytes, into
// place.  Bound by instructions (1537 and 2515 a warp with checks at every row, 714 and 1356 of the kernel for aligned rows) and by the
// phases of a CTA, which only other CTAs overlap.  So no row is checked by itself: segments are read as they are staged, what lies
// beyond the matrix is zeroed for all of a lane's rows at once where there is any, and only the stores ask.  us, nearest / stochastic, every row
// checked and now: 4099 x 2731 11.4 / 15.5 -> 9.7 / 13.5 (5.1 at the measured copy bandwidth), 16384 x 2731 33.2 / 45.2 -> 28.9 / 39.7, 9001 x 8191
// 50.7 / 70.0 -> 44.5 / 60.7, 300 x 777 5.5 / 6.9 -> 4.4 / 5.8, 7 x 7 4.4 / 5.9 -> 3.4 / 4.8.  (A body without checks for whole tiles beside the
// checked one gains as much on large matrices but loses 2-11 % on small ones and ones of many edge tiles, whose SMs run both.)

// The Philox blocks that the warp's 32 rows of 128 elements touch, nine per row: each lane draws the one in which its own segment
// of each of its eight rows starts (`own`, 128 apart) and the ninth of the row that has its number (`ninth`).  A segment's bytes
// run on into the block of its right neighbour, or into the ninth.  Loops that also stop at the last row cost whole tiles 1-2 %.
__device__ __forceinline__ void draw_row_blocks(const Quant2dParams &p, int64_t tile_row0, int64_t tile_col0, int rg, int seg, uint4 *own, uint4 *ninth, int lane)
{
    if (tile_row0 >= p.rows) return;
    uint64_t idx = (uint64_t)(tile_row0 + 8 * rg) * (uint64_t)p.cols + (uint64_t)tile_col0;
#pragma unroll 1
    for (int r = 0; r < 9; r++) {
        if (r == 8) idx = (uint64_t)(tile_row0 + lane) * (uint64_t)p.cols + (uint64_t)tile_col0;
        const uint64_t blk = (idx >> 4) + (r < 8 ? seg : 8);
        uint32_t R[4];
        philox4x32_10((uint32_t)blk, (uint32_t)(blk >> 32), p.tensor_id, 0u, p.keys, R);
        *(r < 8 ? own + 128 * r : ninth + 4 * (lane & 7) + (lane >> 3)) = make_uint4(R[0], R[1], R[2], R[3]);
        idx += (uint64_t)p.cols;
    }
}

// A segment's 16 random bytes; off: the row's offset into its first Philox block (0 .. 15).
__device__ __forceinline__ void read_staged_random(const uint4 &a, const uint4 &b, uint32_t off, uint32_t R[4])
{
    uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    const bool by2 = off & 8, by1 = off & 4;
#pragma unroll
    for (int k = 0; k < 6; k++) w[k] = by2 ? w[k + 2] : w[k];
#pragma unroll
    for (int k = 0; k < 5; k++) w[k] = by1 ? w[k + 1] : w[k];
#pragma unroll
    for (int k = 0; k < 4; k++) R[k] = __funnelshift_r(w[k], w[k + 1], 8 * (off & 3));
}

// The 16 random bytes of the row segment starting at element (i, j0), one Philox call per element: the slow
// generic path of the transposed index.
__device__ __forceinline__ void segment_random_bytes(const Quant2dParams &p, int64_t i, int64_t j0, uint32_t R[4])
{
#pragma unroll
    for (int w = 0; w < 4; w++) {
        uint32_t word = 0;
#pragma unroll 1
        for (int b = 0; b < 4; b++) {
            const int64_t j = j0 + 4 * w + b;
            if (j < p.cols) {
                const uint64_t idx = (p.flags & FP4Q_INDEX_TRANSPOSED)
                                         ? (uint64_t)j * (uint64_t)p.rows + (uint64_t)i
                                         : (uint64_t)i * (uint64_t)p.cols + (uint64_t)j;
                word |= philox_byte(p, idx) << (8 * b);
            }
        }
        R[w] = word;
    }
}

// FAST = the CTA's 128x128 tile lies fully inside the tensor, rows are 32-byte aligned (256-bit loads) and
// one Philox block covers each 16-element segment: no per-row bounds or path checks remain in the hot loop.
// BLK = block size: 32 (the method), or 16 / 64 for the block-size study.  A 16x16 block is two lanes (8 rows x 16
// columns each), a 64x64 block sixteen lanes in each of two neighbouring warps, which exchange their maxima through
// `xchg`.  With BLK = 64 the scale is still written once per 32x32 tile (four equal entries per block), so that the
// tensor feeds the GEMMs as it stands; with BLK = 16 the scale matrix has one entry per 16x16 block.
// STAGED = the tile goes through staging rows (above); the transposed payload's staging (qt_stage) then takes their place.
// EDGES = a tile of a tensor that is read directly and not made of whole 32-byte aligned tiles only: rows are not checked one by one
// here either.  us, nearest / stochastic, every row checked and now: 300 x 768 3.6 / 4.9 -> 2.8 / 3.7, 1000 x 2048 3.8 / 5.4 -> 3.05 / 4.0, 3000 x 3008
// 5.1 / 7.8 -> 4.7 / 6.6, 4099 x 2720 6.6 / 9.3 -> 6.0 / 8.5, on 16-byte boundaries 16384 x 4096 40.4 / 54.0 -> 35.6 / 47.6.  Tensors of whole tiles keep a
// kernel with the checked body beside them: the body for whole tiles rounds stochastically 3 % slower when compiled beside the other
// one, and 1 % alone (16384 x 11008 84.9, 87.9 and 86.4).
template <int MODE, bool FAST, int BLK, bool STAGED = false, int F32 = 0, bool EDGES = false>
__device__ __forceinline__ void quantize_tile(const Quant2dParams &p, uint4 *qt_stage, uint4 *rnd_stage, uint32_t *xchg, uint4 *staging = nullptr)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int t = lane >> 3;          // which of the warp's four 32x32 blocks
    const int rg = (lane >> 1) & 3;   // group of 8 rows inside the block
    const int ch = lane & 1;          // 16-column half of the block
    const int64_t bx = (int64_t)blockIdx.x % p.grid_x, by = (int64_t)blockIdx.x / p.grid_x;
    const int64_t tile_row0 = by * 128 + warp * 32, tile_col0 = bx * 128 + t * 32;
    const int64_t row0 = tile_row0 + rg * 8, col0 = tile_col0 + ch * 16;
    const bool tile_exists = FAST || (tile_row0 < p.rows && tile_col0 < p.cols);
    const int n_rows = FAST ? 8 : (int)max((int64_t)0, min((int64_t)8, p.rows - row0));   // of this lane's

    // Staged tensors of few rows: warps without rows (in a tensor of 32 rows three of a CTA's four) only meet the others; us, nearest /
    // stochastic, with everything done for them and now: 32 x 1000001 54.7 / 79.4 -> 42.5 / 56, 4 x 65537 6.6 / 8.6 -> 4.7 / 6.1; other sizes lose 1 %.
    // And of one or two rows the other six are not rounded: 1 x 5001 stochastic 4.95 -> 4.37.
    const bool idle = STAGED && tile_row0 >= p.rows, few = STAGED && p.rows <= 2;
    uint32_t raw[8][8];
    if (F32 && FAST) {
        const float *src = reinterpret_cast<const float *>(p.x) + row0 * p.ld_x + col0;
        uint32_t wide[8][16];
#pragma unroll
        for (int r = 0; r < 8; r++) {
            if (F32 == 2) {
#pragma unroll
                for (int h = 0; h < 2; h++)
                    asm volatile("ld.global.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                                 : "=r"(wide[r][8 * h]), "=r"(wide[r][8 * h + 1]), "=r"(wide[r][8 * h + 2]), "=r"(wide[r][8 * h + 3]),
                                   "=r"(wide[r][8 * h + 4]), "=r"(wide[r][8 * h + 5]), "=r"(wide[r][8 * h + 6]), "=r"(wide[r][8 * h + 7])
                                 : "l"(src + r * p.ld_x + 8 * h));
            } else {
#pragma unroll
                for (int h = 0; h < 4; h++)
                    asm volatile("ld.global.v4.b32 {%0,%1,%2,%3}, [%4];"
                                 : "=r"(wide[r][4 * h]), "=r"(wide[r][4 * h + 1]), "=r"(wide[r][4 * h + 2]), "=r"(wide[r][4 * h + 3])
                                 : "l"(src + r * p.ld_x + 4 * h));
            }
        }
#pragma unroll
        for (int r = 0; r < 8; r++)
#pragma unroll
            for (int k = 0; k < 8; k++) raw[r][k] = pack_bf16(wide[r][2 * k], wide[r][2 * k + 1]);
    } else if (F32) {
#pragma unroll
        for (int r = 0; r < 8; r++) load_segment_f32(p, row0 + r, col0, raw[r]);
    } else if (FAST) {
        const uint16_t *src = p.x + row0 * p.ld_x + col0;
#pragma unroll
        for (int r = 0; r < 8; r++)
            asm volatile("ld.global.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                         : "=r"(raw[r][0]), "=r"(raw[r][1]), "=r"(raw[r][2]), "=r"(raw[r][3]), "=r"(raw[r][4]),
                           "=r"(raw[r][5]), "=r"(raw[r][6]), "=r"(raw[r][7])
                         : "l"(src + r * p.ld_x));
    } else if (STAGED) {
        uint8_t *stage = reinterpret_cast<uint8_t *>(staging) + warp * kStageWarpBytes;
        stage_tile_rows(p, tile_row0, bx * 128, stage, lane);
        if (MODE == FP4Q_ROUND_STOCHASTIC)   // while the copies are on their way
            draw_row_blocks(p, tile_row0, bx * 128, rg, 2 * t + ch, rnd_stage + threadIdx.x, rnd_stage + 8 * 128 + 32 * warp, lane);
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();
        if (!idle) {
#pragma unroll
            for (int r = 0; r < 8; r++) read_staged_row_uncut(p, tile_row0, bx * 128, stage, lane, r, raw[r]);
        }
        cut_staged_rows(raw, n_rows, (int)max((int64_t)0, min((int64_t)16, p.cols - col0)));
    } else if (EDGES && p.x_vec_ok && col0 + 16 <= p.cols) {
        const uint16_t *src = p.x + row0 * p.ld_x + col0;
#pragma unroll
        for (int r = 0; r < 8; r++)
#pragma unroll
            for (int k = 0; k < 8; k++) raw[r][k] = 0u;
        if (p.x_vec_ok == 2) {
#pragma unroll
            for (int r = 0; r < 8; r++)
                if (r < n_rows)
                    asm volatile("ld.global.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                                 : "=r"(raw[r][0]), "=r"(raw[r][1]), "=r"(raw[r][2]), "=r"(raw[r][3]), "=r"(raw[r][4]),
                                   "=r"(raw[r][5]), "=r"(raw[r][6]), "=r"(raw[r][7])
                                 : "l"(src + r * p.ld_x));
        } else {
#pragma unroll
            for (int r = 0; r < 8; r++)
                if (r < n_rows) {
                    const uint4 a = load_global(reinterpret_cast<const uint4 *>(src + r * p.ld_x)), b = load_global(reinterpret_cast<const uint4 *>(src + r * p.ld_x) + 1);
                    raw[r][0] = a.x; raw[r][1] = a.y; raw[r][2] = a.z; raw[r][3] = a.w;
                    raw[r][4] = b.x; raw[r][5] = b.y; raw[r][6] = b.z; raw[r][7] = b.w;
                }
        }
    } else {
#pragma unroll
        for (int r = 0; r < 8; r++) load_segment(p, row0 + r, col0, raw[r]);
    }

    // The random bytes do not depend on the data: draw them while the loads are in flight and park them in
    // shared memory (each thread reads back only what it wrote), in a rolled loop that keeps the code small.
    if (MODE == FP4Q_ROUND_STOCHASTIC && !STAGED && (FAST || p.rng_aligned)) {
        uint64_t idx = (uint64_t)row0 * (uint64_t)p.cols + (uint64_t)col0;
#pragma unroll 2
        for (int r = 0; r < 8; r++) {
            uint32_t R[4];
            const uint64_t blk = idx >> 4;
            philox4x32_10((uint32_t)blk, (uint32_t)(blk >> 32), p.tensor_id, 0u, p.keys, R);
            rnd_stage[r * 128 + threadIdx.x] = make_uint4(R[0], R[1], R[2], R[3]);
            idx += (uint64_t)p.cols;
        }
    }

    // block maximum: packed BF16 |.| max with NaN propagation, so that any non-finite entry shows
    // up in the result and routes the block to the scalar path
    __nv_bfloat162 m2 = __float2bfloat162_rn(0.0f);
#pragma unroll
    for (int r = 0; r < 8; r++)
#pragma unroll
        for (int k = 0; k < 8; k++)
            m2 = __hmax2_nan(m2, __habs2(*reinterpret_cast<const __nv_bfloat162 *>(&raw[r][k])));
    constexpr int kShflLo = BLK == 16 ? 2 : 1, kShflHi = BLK == 16 ? 2 : BLK == 32 ? 4 : 8;   // lanes of one block
#pragma unroll
    for (int s = kShflLo; s <= kShflHi; s <<= 1) {
        uint32_t other = __shfl_xor_sync(0xFFFFFFFFu, *reinterpret_cast<uint32_t *>(&m2), s);
        m2 = __hmax2_nan(m2, *reinterpret_cast<__nv_bfloat162 *>(&other));
    }
    const __nv_bfloat16 m1 = __hmax_nan(m2.x, m2.y);
    uint32_t mbits = (uint32_t)(*reinterpret_cast<const uint16_t *>(&m1)) & 0x7FFFu;
    bool nonfinite64 = false;
    if (BLK == 64) {
        // the other 32 rows of the block belong to the neighbouring warp: both maxima (with NaN propagation, and over
        // finite entries only) cross through shared memory, unconditionally, so that every thread reaches the barrier
        uint32_t fm = 0;
#pragma unroll
        for (int r = 0; r < 8; r++)
#pragma unroll
            for (int k = 0; k < 8; k++) {
                const uint32_t lo = raw[r][k] & 0x7FFFu, hi = (raw[r][k] >> 16) & 0x7FFFu;
                if (lo < 0x7F80u && lo > fm) fm = lo;
                if (hi < 0x7F80u && hi > fm) fm = hi;
            }
#pragma unroll
        for (int s = 1; s <= 8; s <<= 1) {
            const uint32_t other = __shfl_xor_sync(0xFFFFFFFFu, fm, s);
            fm = other > fm ? other : fm;
        }
        if ((lane & 15) == 0) {
            xchg[(warp * 2 + (t >> 1)) * 2] = mbits;
            xchg[(warp * 2 + (t >> 1)) * 2 + 1] = fm;
        }
        __syncthreads();
        const uint32_t om = xchg[((warp ^ 1) * 2 + (t >> 1)) * 2], of = xchg[((warp ^ 1) * 2 + (t >> 1)) * 2 + 1];
        fm = of > fm ? of : fm;
        nonfinite64 = mbits >= 0x7F80u || om >= 0x7F80u;
        mbits = nonfinite64 ? fm : (om > mbits ? om : mbits);
    }

    const bool nonfinite = BLK == 64 ? nonfinite64 : mbits >= 0x7F80u;
    if (BLK != 64 && __any_sync(0xFFFFFFFFu, nonfinite)) {
        // maximum over the finite entries only
        uint32_t fm = 0;
#pragma unroll
        for (int r = 0; r < 8; r++)
#pragma unroll
            for (int k = 0; k < 8; k++) {
                const uint32_t lo = raw[r][k] & 0x7FFFu, hi = (raw[r][k] >> 16) & 0x7FFFu;
                if (lo < 0x7F80u && lo > fm) fm = lo;
                if (hi < 0x7F80u && hi > fm) fm = hi;
            }
#pragma unroll
        for (int s = kShflLo; s <= kShflHi; s <<= 1) {
            const uint32_t other = __shfl_xor_sync(0xFFFFFFFFu, fm, s);
            fm = other > fm ? other : fm;
        }
        if (nonfinite) mbits = fm;
    }

    const int code = scale_code_from_max(mbits);
    const float inv = inv_scale(code);
    if (BLK == 16) {
        if ((lane & 2) == 0 && row0 < p.rows && col0 < p.cols) p.scale[(row0 >> 4) * p.ld_s + (col0 >> 4)] = (uint8_t)code;
    } else if (tile_exists && (lane & 7) == 0) {
        p.scale[(tile_row0 >> 5) * p.ld_s + (tile_col0 >> 5)] = (uint8_t)code;
    }

    const uint4 *next_block = rnd_stage + (2 * t + ch < 7 ? threadIdx.x + (ch ? 7 : 1) : 8 * 128 + 32 * warp + rg);
    const int next_step = 2 * t + ch < 7 ? 128 : 4;
    const uint32_t off0 = (uint32_t)row0 * (uint32_t)p.cols;   // a tile starts on a multiple of 128
    auto staged_random = [&](int r, uint32_t R[4]) {
        read_staged_random(rnd_stage[r * 128 + threadIdx.x], next_block[r * next_step], (off0 + r * (uint32_t)p.cols) & 15u, R);
    };
    uint32_t W[8][2];
    uint8_t *dst_rm = p.q_rm + row0 * p.ld_rm + (col0 >> 1);
    if (idle) {   // nothing of it is written, transposed either
    } else if ((FAST || STAGED || EDGES) && !nonfinite) {
        // hot loop: no path selection, and no bounds checks but at the store
        const int n_store = tile_exists ? n_rows : 0;
#pragma unroll
        for (int r = 0; r < 8; r++) {
            if (STAGED && r == 2 && few) {
#pragma unroll
                for (int z = 2; z < 8; z++) W[z][0] = W[z][1] = 0u;
                break;
            }
            uint32_t R[4] = {0u, 0u, 0u, 0u};
            if (MODE == FP4Q_ROUND_STOCHASTIC) {
                if (STAGED) {
                    staged_random(r, R);
                } else {
                    const uint4 v = rnd_stage[r * 128 + threadIdx.x];
                    R[0] = v.x; R[1] = v.y; R[2] = v.z; R[3] = v.w;
                }
            }
            round_segment<MODE>(raw[r], inv, R, W[r]);
            if (FAST || r < n_store) *reinterpret_cast<uint2 *>(dst_rm + r * p.ld_rm) = make_uint2(W[r][0], W[r][1]);
        }
    } else {
#pragma unroll
        for (int r = 0; r < 8; r++) {
            const int64_t i = row0 + r;
            if (!tile_exists || i >= p.rows) {
                W[r][0] = W[r][1] = 0u;
                continue;
            }
            uint32_t R[4] = {0u, 0u, 0u, 0u};
            if (MODE == FP4Q_ROUND_STOCHASTIC) {
                if (STAGED) {
                    staged_random(r, R);
                } else if (FAST || EDGES || p.rng_aligned) {
                    const uint4 v = rnd_stage[r * 128 + threadIdx.x];
                    R[0] = v.x; R[1] = v.y; R[2] = v.z; R[3] = v.w;
                } else {
                    segment_random_bytes(p, i, col0, R);
                }
            }
            if (!nonfinite) {
                round_segment<MODE>(raw[r], inv, R, W[r]);
            } else {
                const uint2 w = round_segment_scalar<MODE>(make_uint4(raw[r][0], raw[r][1], raw[r][2], raw[r][3]),
                                                           make_uint4(raw[r][4], raw[r][5], raw[r][6], raw[r][7]),
                                                           make_uint4(R[0], R[1], R[2], R[3]), inv_scale_f16_aligned(code));
                W[r][0] = w.x;
                W[r][1] = w.y;
            }
            *reinterpret_cast<uint2 *>(dst_rm + r * p.ld_rm) = make_uint2(W[r][0], W[r][1]);
        }
    }

    if (p.q_t == nullptr) return;

    // transposed payload: per lane two 8x8 nibble blocks -> 16 words (one per column, 8 rows each)
    uint32_t *stage = reinterpret_cast<uint32_t *>(qt_stage);
    if (STAGED) __syncthreads();   // every warp has read its rows
    if (!idle)
#pragma unroll
    for (int g = 0; g < 2; g++) {
        uint32_t a[8];
#pragma unroll
        for (int r = 0; r < 8; r++) a[r] = W[r][g];
        transpose8x8_nibbles(a);
#pragma unroll
        for (int c = 0; c < 8; c++) {
            const int col_local = 32 * t + 16 * ch + 8 * g + c;
            // word index inside the 64-byte row: 4*(source warp) + rg, with the 16-byte chunk index
            // XORed by the column's block index so that a warp's stores spread over the banks
            stage[col_local * 16 + (((warp ^ t) << 2) | rg)] = a[c];
        }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const int row_local = (threadIdx.x >> 2) + 32 * k;   // transposed row = source column; its block index is k
        const int chunk = threadIdx.x & 3;                    // 32 source rows = one source warp
        const int64_t col = bx * 128 + row_local;
        if (FAST || (col < p.cols && by * 128 + chunk * 32 < p.rows)) {
            const uint4 v = qt_stage[row_local * 4 + (chunk ^ k)];
            *reinterpret_cast<uint4 *>(p.q_t + col * p.ld_t + by * 64 + chunk * 16) = v;
        }
    }
}

// EDGES: see quantize_tile; what comes here otherwise is made of whole tiles, has the transposed index or is a few rows.
template <int MODE, int BLK, bool EDGES, int CTAS = 4>   // CTAS: an SM
__global__ void __launch_bounds__(128, CTAS) quantize2d_kernel(const __grid_constant__ Quant2dParams p)
{
    __shared__ uint4 qt_stage[128 * 4];   // 128 transposed rows x 64 B (four 16-byte chunks, XOR-swizzled)
    __shared__ uint4 rnd_stage[MODE == FP4Q_ROUND_STOCHASTIC ? 8 * 128 : 1];   // per thread: 8 rows x 16 random bytes
    __shared__ uint32_t xchg[BLK == 64 ? 16 : 1];   // 64x64 blocks: maxima of the four warps' two half blocks
    if (p.waits) wait_for_predecessor();
    admit_successor();
    const int64_t bx = (int64_t)blockIdx.x % p.grid_x, by = (int64_t)blockIdx.x / p.grid_x;
    const bool full = p.x_vec_ok == 2 && p.rng_aligned && (by + 1) * 128 <= p.rows && (bx + 1) * 128 <= p.cols;
    if (full) quantize_tile<MODE, true, BLK>(p, qt_stage, rnd_stage, xchg);
    else quantize_tile<MODE, false, BLK, false, 0, EDGES>(p, qt_stage, rnd_stage, xchg);
    // The later tensors of a multi-tensor call do not read what the call's earlier ones wrote, so they did not wait; they
    // wait here, after their own stores, so that the grids still COMPLETE in launch order and whatever is enqueued after the
    // call sees every tensor of it.
    if (!p.waits) wait_for_predecessor();
}

// Every tile of a tensor whose rows start anywhere or whose segments straddle Philox blocks.  With the random blocks in memory of their
// own they are drawn while the rows are on their way; the transposed payload's staging takes the place of the rows, so that 53 KB
// and 128 registers allow four CTAs per SM, like the aligned kernel.  To nearest 36 KB and 96 registers allow five: us, four and five,
// 4099 x 2731 9.7 and 8.7, 16384 x 2731 29.0 and 28.2, 9001 x 8191 44.6 and 43.1, 32 x 1000001 42.2 and 37.8, 300 x 777 4.33 and 4.29 (six spill).
template <int MODE> constexpr int kStagedSmem = 4 * kStageWarpBytes + (MODE == FP4Q_ROUND_STOCHASTIC ? (8 * 128 + 4 * 32) * 16 : 0);
static_assert(4 * kStageWarpBytes >= 128 * 4 * 16, "the transposed payload's staging fits in the rows");
template <int MODE, int BLK = 32>
__global__ void __launch_bounds__(128, MODE == FP4Q_ROUND_NEAREST ? 5 : 4) quantize2d_staged_kernel(const __grid_constant__ Quant2dParams p)
{
    extern __shared__ uint4 dynamic_stage[];
    __shared__ uint32_t xchg[BLK == 64 ? 16 : 1];
    if (p.waits) wait_for_predecessor();
    admit_successor();
    quantize_tile<MODE, false, BLK, true>(p, dynamic_stage, dynamic_stage + 4 * kStageWarpBytes / 16, xchg, dynamic_stage);
    if (!p.waits) wait_for_predecessor();   // as in quantize2d_kernel
}

// FP32 source, rows on 16-byte boundaries: 5 bytes an element in one pass instead of 6 for a BF16 copy and 3 for its quantizer.  The
// loads of a lane's eight rows in flight take 128 registers beside everything else: three CTAs an SM instead of four.  The layer's
// pass, with a BF16 copy of its FP32 weight and without: 128 x 256 x 256 84.6 -> 77.8 us, 8192 x 2048 x 2048 97.2 -> 95.0.  Rows on 16 but
// not 32 bytes take 128-bit loads instead of 256-bit ones; through the body that checks every element they lost to the copy from
// some 10 million elements on.  us, 32 activation rows and the weight, copy / checked / now: 2048 x 2052 10.8 / 8.5 / 8.1,
// 4096 x 4100 31.9 / 29.8 / 20.3, 11008 x 4100 75.7 / 81.8 / 45.7.  The layer rounds its operands to nearest; stochastic rounding of rows
// that straddle Philox blocks (cols % 16 != 0) draws a block per element here, and the copy is the faster way: 4096 x 4100 158.8 / 37.4.
template <int MODE, int ROWS>   // ROWS: 2 = rows on 32 bytes, 1 = on 16
__global__ void __launch_bounds__(128, 3) quantize2d_f32_kernel(const __grid_constant__ Quant2dParams p)
{
    __shared__ uint4 qt_stage[128 * 4];
    __shared__ uint4 rnd_stage[MODE == FP4Q_ROUND_STOCHASTIC ? 8 * 128 : 1];
    if (p.waits) wait_for_predecessor();
    admit_successor();
    const int64_t bx = (int64_t)blockIdx.x % p.grid_x, by = (int64_t)blockIdx.x / p.grid_x;
    const bool full = p.rng_aligned && (by + 1) * 128 <= p.rows && (bx + 1) * 128 <= p.cols;
    if (full) quantize_tile<MODE, true, 32, false, ROWS>(p, qt_stage, rnd_stage, nullptr);
    else quantize_tile<MODE, false, 32, false, ROWS>(p, qt_stage, rnd_stage, nullptr);
    if (!p.waits) wait_for_predecessor();   // as in quantize2d_kernel
}

typedef void (*Quant2dKernel)(const Quant2dParams);

// Rows on vector boundaries and, with stochastic rounding, segments on Philox blocks are read directly: on 32-byte boundaries
// by the check-free body, on 16-byte ones by 128-bit loads, where these reach the rows' ends.  us, nearest / stochastic,
// direct and staged: 4096 x 4096 in a pitch of 4104 10.6 / 13.6 and 11.4 / 16.8, 2048 x 2048 in 2056 4.4 / 5.5 and 5.1 / 7.0, 16384 x 4096 35.6 / 47.6 and
// 39.0 / 54.5; with a last segment that is not full, which is read by elements: 4099 x 2728 nearest 11.9 and 8.7, 300 x 776 5.7 and
// 4.4, 16 x 10008 5.9 and 3.9, 1 x 10008 2.9 and 3.3.  Anything else is staged, except for the transposed index, whose random bytes run down
// the columns.
// A few rows in many tiles are read directly too, in the kernel whose body checks every row and rounds only those that exist; us, nearest /
// stochastic, all eight of a lane (or staged) and checked: 1 x 1000016 33.9 / 65.6 -> 28.0 / 52.8, 3 x 1000008 38.6 / 63.6 -> 31.2 / 63.6, 5 x 1000016
// 34.2 / 65.9 -> 32.8 / 62.5, 2 x 100016 5.6 / 9.1 -> 5.2 / 8.2, 1 x 10016 2.9 / 3.9 -> 2.8 / 3.6, but 7 x 1000016 34.4 / 66.1 and 35.9 / 67.5, 5 x 100016
// 5.65 / 9.1 and 6.0 / 9.7, 3 x 10016 2.9 / 3.8 and 3.0 / 4.0.
static Quant2dKernel quantize2d_kernel_for(const Quant2dParams &p, bool sr, int *smem)
{
    const int64_t n_cta = ceil_div(p.rows, 128) * ceil_div(p.cols, 128);
    const bool few = p.rows == 1 || (p.rows <= 5 && 300 * p.rows <= n_cta);
    const bool direct = p.x_vec_ok && p.rng_aligned && (p.x_vec_ok == 2 || p.cols % 16 == 0 || p.rows <= 2 || few);
    const bool transposed_index = sr && (p.flags & FP4Q_INDEX_TRANSPOSED), staged = !direct && !transposed_index;
    const bool edges = direct && !transposed_index && !few && (p.x_vec_ok != 2 || p.rows % 128 != 0 || p.cols % 128 != 0);
    const int which = (p.flags & FP4Q_BLOCK_16) ? 1 : (p.flags & FP4Q_BLOCK_64) ? 2 : 0;
    constexpr int N = FP4Q_ROUND_NEAREST, S = FP4Q_ROUND_STOCHASTIC;
    static const Quant2dKernel kernels[3][2][3] = {
        {{quantize2d_kernel<N, 32, false>, quantize2d_kernel<N, 16, false>, quantize2d_kernel<N, 64, false>},
         {quantize2d_kernel<S, 32, false>, quantize2d_kernel<S, 16, false>, quantize2d_kernel<S, 64, false>}},
        {{quantize2d_kernel<N, 32, true>, quantize2d_kernel<N, 16, true>, quantize2d_kernel<N, 64, true>},
         {quantize2d_kernel<S, 32, true>, quantize2d_kernel<S, 16, true>, quantize2d_kernel<S, 64, true>}},
        {{quantize2d_staged_kernel<N>, quantize2d_staged_kernel<N, 16>, quantize2d_staged_kernel<N, 64>},
         {quantize2d_staged_kernel<S>, quantize2d_staged_kernel<S, 16>, quantize2d_staged_kernel<S, 64>}}};
    // Nearest, where the grid is more than one or two rounds of four CTAs on 148 SMs: five.  us, four and five: edges 4099 x 2720 6.0 and 5.3, 4099 x 4096
    // 7.8 and 7.4, 16384 x 4096 in a pitch of 4104 35.6 and 34.6, but 3000 x 3008 (576 CTAs) 4.6 and 4.7, 300 x 768 2.8 and 2.9; whole tiles 8192 x 4096
    // 15.9 and 15.0, 4096 x 11008 24.2 and 23.0, 16384 x 4096 32.6 and 31.9, but 4096 x 4096 (1024), everything in L2, 6.9 and 7.2.  64 x 64 blocks, which only
    // the study of block sizes uses, have not been tried with five.
    static const Quant2dKernel five[2][2] = {{quantize2d_kernel<N, 32, false, 5>, quantize2d_kernel<N, 16, false, 5>},
                                             {quantize2d_kernel<N, 32, true, 5>, quantize2d_kernel<N, 16, true, 5>}};
    *smem = !staged ? 0 : sr ? kStagedSmem<FP4Q_ROUND_STOCHASTIC> : kStagedSmem<FP4Q_ROUND_NEAREST>;
    if (!staged && !sr && which < 2 && n_cta > (edges ? 592 : 1184)) return five[edges][which];
    return kernels[staged ? 2 : edges][sr][which];
}

static fp4q_status launch_quantizer(Quant2dKernel kernel, int64_t n_cta, int smem, cudaStream_t stream, const Quant2dParams &p, bool later)
{
    // More than 48 KB are asked for by each launch: an attribute of the kernel on the current device, whose setting costs 0.2 us.
    if (smem > 48 * 1024 && cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) return launched(cudaErrorUnknown);
    return launched(launch_dependent(kernel, dim3((unsigned)n_cta), 128, stream, p, later, smem));
}

}  // namespace fp4q

using namespace fp4q;

// Argument checks and kernel parameters of one tensor.  *n_cta = 0 for an empty tensor (nothing to launch).
static fp4q_status prepare_quantize2d(const void *x_bf16, int64_t rows, int64_t cols, int64_t ld_x, const fp4q_tensor *out,
                                      fp4q_round mode, uint64_t seed, uint32_t tensor_id, uint32_t flags, Quant2dParams &p,
                                      int64_t *n_cta)
{
    *n_cta = 0;
    if (rows < 0 || cols < 0) return FP4Q_ERR_SHAPE;
    if (mode != FP4Q_ROUND_NEAREST && mode != FP4Q_ROUND_STOCHASTIC) return FP4Q_ERR_UNSUPPORTED;
    if (flags & ~(FP4Q_INDEX_TRANSPOSED | FP4Q_BLOCK_16 | FP4Q_BLOCK_64)) return FP4Q_ERR_UNSUPPORTED;
    if ((flags & FP4Q_BLOCK_16) && (flags & FP4Q_BLOCK_64)) return FP4Q_ERR_UNSUPPORTED;
    const int sgran = (flags & FP4Q_BLOCK_16) ? 16 : 32;   // granularity of the scale matrix
    if (!out) return FP4Q_ERR_NULL;
    if (out->rows != rows || out->cols != cols) return FP4Q_ERR_SHAPE;
    if (rows == 0 || cols == 0) return FP4Q_OK;
    if (!x_bf16 || !out->q_rm || !out->scale) return FP4Q_ERR_NULL;
    if (ld_x < cols || out->ld_rm < round_up(cols, 32) / 2 || out->ld_s < ceil_div(cols, sgran)) return FP4Q_ERR_SHAPE;
    if (out->q_t && out->ld_t < round_up(rows, 32) / 2) return FP4Q_ERR_SHAPE;
    if (!aligned(x_bf16, 2) || !aligned(out->q_rm, 16) || out->ld_rm % 16 != 0) return FP4Q_ERR_ALIGN;
    if (out->q_t && (!aligned(out->q_t, 16) || out->ld_t % 16 != 0)) return FP4Q_ERR_ALIGN;

    p.x = static_cast<const uint16_t *>(x_bf16);
    p.rows = rows; p.cols = cols; p.ld_x = ld_x;
    p.q_rm = out->q_rm; p.ld_rm = out->ld_rm;
    p.q_t = out->q_t; p.ld_t = out->ld_t;
    p.scale = out->scale; p.ld_s = out->ld_s;
    p.grid_x = ceil_div(cols, 128);
    p.tensor_id = tensor_id;
    p.flags = flags;
    p.x_vec_ok = (aligned(x_bf16, 32) && ld_x % 16 == 0) ? 2 : (aligned(x_bf16, 16) && ld_x % 8 == 0) ? 1 : 0;
    p.rng_aligned = mode == FP4Q_ROUND_NEAREST || (cols % 16 == 0 && !(flags & FP4Q_INDEX_TRANSPOSED));
    philox_round_keys(seed, p.keys);
    *n_cta = p.grid_x * ceil_div(rows, 128);
    if (*n_cta > 0x7FFFFFFF) return FP4Q_ERR_UNSUPPORTED;
    return FP4Q_OK;
}

extern "C" fp4q_status fp4q_quantize2d(const void *x_bf16, int64_t rows, int64_t cols, int64_t ld_x,
                                       const fp4q_tensor *out, fp4q_round mode, uint64_t seed,
                                       uint32_t tensor_id, uint32_t flags, void *stream)
{
    Quant2dParams p;
    int64_t n_cta;
    if (fp4q_status st = prepare_quantize2d(x_bf16, rows, cols, ld_x, out, mode, seed, tensor_id, flags, p, &n_cta)) return st;
    if (n_cta == 0) return FP4Q_OK;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    p.waits = 1;
    int smem;
    const Quant2dKernel kernel = quantize2d_kernel_for(p, mode == FP4Q_ROUND_STOCHASTIC, &smem);
    return launch_quantizer(kernel, n_cta, smem, s, p, false);
}

static fp4q_status quantize2d_jobs(const fp4q_quantize_job *jobs, const uint8_t *is_f32, int32_t n_jobs, fp4q_round mode, uint64_t seed, void *stream)
{
    if (n_jobs < 0) return FP4Q_ERR_SHAPE;
    if (n_jobs > 0 && !jobs) return FP4Q_ERR_NULL;
    const bool sr = mode == FP4Q_ROUND_STOCHASTIC;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // First pass: every job is checked before the first launch, so that an argument error leaves the stream untouched.
    // Second pass: one launch of the one-tensor kernel per tensor; the tensors are independent, so a launch after the first does not
    // wait for the one before it and begins beside its last wave instead of after it (what two streams would give, in one stream).
    for (int pass = 0; pass < 2; pass++) {
        bool first = true;
        for (int32_t j = 0; j < n_jobs; j++) {
            const bool f32 = is_f32 && is_f32[j];
            if (jobs[j].flags & (FP4Q_BLOCK_16 | FP4Q_BLOCK_64)) return FP4Q_ERR_UNSUPPORTED;   // 32 x 32 blocks only
            Quant2dParams p;
            int64_t n_cta;
            if (fp4q_status st = prepare_quantize2d(jobs[j].x_bf16, jobs[j].rows, jobs[j].cols, jobs[j].ld_x, jobs[j].out, mode, seed,
                                                    jobs[j].tensor_id, jobs[j].flags, p, &n_cta))
                return st;
            if (n_cta == 0) continue;
            if (f32) {
                if (!aligned(jobs[j].x_bf16, 16) || jobs[j].ld_x % 4) return FP4Q_ERR_ALIGN;
                p.x_vec_ok = aligned(jobs[j].x_bf16, 32) && jobs[j].ld_x % 8 == 0 ? 2 : 1;
            }
            if (pass == 0) continue;
            p.waits = first;
            int smem = 0;
            static const Quant2dKernel f32_kernels[2][2] = {
                {quantize2d_f32_kernel<FP4Q_ROUND_NEAREST, 1>, quantize2d_f32_kernel<FP4Q_ROUND_NEAREST, 2>},
                {quantize2d_f32_kernel<FP4Q_ROUND_STOCHASTIC, 1>, quantize2d_f32_kernel<FP4Q_ROUND_STOCHASTIC, 2>}};
            const Quant2dKernel kernel = f32 ? f32_kernels[sr][p.x_vec_ok - 1] : quantize2d_kernel_for(p, sr, &smem);
            if (fp4q_status st = launch_quantizer(kernel, n_cta, smem, s, p, !first)) return st;
            first = false;
        }
    }
    return FP4Q_OK;
}

extern "C" fp4q_status fp4q_quantize2d_multi(const fp4q_quantize_job *jobs, int32_t n_jobs, fp4q_round mode, uint64_t seed,
                                             void *stream)
{
    return quantize2d_jobs(jobs, nullptr, n_jobs, mode, seed, stream);
}

extern "C" fp4q_status fp4q_quantize2d_multi_f32(const fp4q_quantize_job *jobs, const uint8_t *is_f32, int32_t n_jobs, fp4q_round mode,
                                                 uint64_t seed, void *stream)
{
    if (n_jobs > 0 && !is_f32) return FP4Q_ERR_NULL;
    return quantize2d_jobs(jobs, is_f32, n_jobs, mode, seed, stream);
}
