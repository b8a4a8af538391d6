// A warp's 32 rows x 128 columns of a BF16 matrix whose rows start anywhere, copied as aligned 16-byte pieces (17 cover 128 elements at any
// offset) into its own staging rows with cp.async and read back as the 16-element segments that a lane of the quantizers holds.
#pragma once

#include "common.cuh"

namespace fp4q {

constexpr int kStageRowBytes = 272;                        // 17 pieces
constexpr int kStageRows4 = 4 * kStageRowBytes + 32;       // the rows r, 8 + r, 16 + r, 24 + r, which one load instruction reads
constexpr int kStageWarpBytes = 8 * kStageRows4;

// Row r of row group rg.  The extra 32 bytes after the second of four rows make the offsets 0, 1, 4, 5 (in 16-byte units,
// modulo 8), so that the eight lanes of one shared-memory pass (four row groups x two column halves, 32 bytes apart)
// read eight different bank groups.
__device__ __forceinline__ int stage_row_offset(int r, int rg) { return r * kStageRows4 + rg * kStageRowBytes + (rg >> 1) * 32; }

static __device__ __noinline__ void stage_first_piece(uint32_t dst, uintptr_t g, uintptr_t lo, uintptr_t hi)
{
    uint32_t w[4];
#pragma unroll
    for (int k = 0; k < 8; k++) {
        const uintptr_t s = g + 2 * k;
        const uint32_t e = s >= lo && s < hi ? (uint32_t)load_global(reinterpret_cast<const uint16_t *>(s)) : 0u;
        w[k >> 1] = k & 1 ? w[k >> 1] | e << 16 : e;
    }
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]) : "memory");
}

// Starts the copies (the caller waits).  Tiles whose pieces all lie inside the tensor need no checks.
template <typename P>   // P: x, rows, cols, ld_x
__device__ __forceinline__ void stage_tile_rows(const P &p, int64_t tile_row0, int64_t tile_col0, uint8_t *stage, int lane)
{
    const uintptr_t lo = reinterpret_cast<uintptr_t>(p.x), hi = reinterpret_cast<uintptr_t>(p.x + (p.rows - 1) * p.ld_x + p.cols);
    const uintptr_t a0 = reinterpret_cast<uintptr_t>(p.x + tile_row0 * p.ld_x + tile_col0), pitch = 2 * (uintptr_t)p.ld_x;
    const uint32_t dst0 = (uint32_t)__cvta_generic_to_shared(stage) + 16 * (lane & 15);
    if (tile_row0 + 32 <= p.rows && tile_col0 + 128 <= p.cols && (a0 & ~(uintptr_t)15) >= lo && ((a0 + 31 * pitch) & ~(uintptr_t)15) + kStageRowBytes <= hi) {
        uintptr_t a = a0 + (lane >> 4) * pitch;
#pragma unroll
        for (int k = 0; k < 16; k++) {   // two rows of 16 pieces per step, the 17th pieces of all rows last
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                         ::"r"(dst0 + stage_row_offset((2 * k) & 7, k >> 2) + (lane >> 4) * kStageRows4), "l"((a & ~(uintptr_t)15) + 16 * (lane & 15)) : "memory");
            a += 2 * pitch;
        }
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                     ::"r"((uint32_t)__cvta_generic_to_shared(stage) + stage_row_offset(lane & 7, lane >> 3) + 256), "l"(((a0 + lane * pitch) & ~(uintptr_t)15) + 256)
                     : "memory");
        return;
    }
    // At the tensor's ends: pieces that hold nothing of a row are left out, one that reaches past the last element is copied as far as that,
    // one that starts before the first goes by loads.
    const uint32_t row_bytes = 2 * (uint32_t)(p.cols - tile_col0 < 128 ? p.cols - tile_col0 : 128);
    const int n_rows = (int)(p.rows - tile_row0 < 32 ? p.rows - tile_row0 : 32);
    if (n_rows <= 0) return;
    auto piece = [&](uintptr_t a, uint32_t c, uint32_t dst) {
        const uintptr_t g = (a & ~(uintptr_t)15) + c;
        if (c >= (uint32_t)(a & 15) + row_bytes) return;
        if (g >= lo) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(g), "r"((int)(hi - g < 16 ? hi - g : 16)) : "memory");
        else stage_first_piece(dst, g, lo, hi);
    };
    uintptr_t a = a0 + (lane >> 4) * pitch;
#pragma unroll 2
    for (int k = 0; k < 16; k++, a += 2 * pitch)
        if (2 * k + (lane >> 4) < n_rows) piece(a, 16 * (lane & 15), dst0 + stage_row_offset((2 * k) & 7, k >> 2) + (lane >> 4) * kStageRows4);
    if (lane < n_rows) piece(a0 + lane * pitch, 256, (uint32_t)__cvta_generic_to_shared(stage) + stage_row_offset(lane & 7, lane >> 3) + 256);
}

// One row's segment (16 elements) of the staged tile; off: the row's offset into its first piece, in bytes.
__device__ __forceinline__ void read_staged_segment(const uint8_t *src, uint32_t off, uint32_t out[8])
{
    uint32_t w[12];
#pragma unroll
    for (int q = 0; q < 3; q++) {
        const uint4 v = reinterpret_cast<const uint4 *>(src)[q];
        w[4 * q] = v.x; w[4 * q + 1] = v.y; w[4 * q + 2] = v.z; w[4 * q + 3] = v.w;
    }
    const bool by2 = off & 8, by1 = off & 4;
#pragma unroll
    for (int k = 0; k < 10; k++) w[k] = by2 ? w[k + 2] : w[k];
#pragma unroll
    for (int k = 0; k < 9; k++) w[k] = by1 ? w[k + 1] : w[k];
#pragma unroll
    for (int k = 0; k < 8; k++) out[k] = __funnelshift_r(w[k], w[k + 1], 8 * (off & 2));
}

// Segment r of lane's eight as it is staged, without a look at the matrix's ends: cut_staged_rows does that for all eight at once.
template <typename P>
__device__ __forceinline__ void read_staged_row_uncut(const P &p, int64_t tile_row0, int64_t tile_col0, const uint8_t *stage, int lane, int r, uint32_t out[8])
{
    const int seg = 2 * (lane >> 3) + (lane & 1), rg = (lane >> 1) & 3;
    const uint32_t a = (uint32_t)reinterpret_cast<uintptr_t>(p.x + tile_row0 * p.ld_x + tile_col0) + 16 * rg * (uint32_t)p.ld_x;
    read_staged_segment(stage + stage_row_offset(r, rg) + 32 * seg, (a + 2 * r * (uint32_t)p.ld_x) & 15, out);
}
// Zeros in place of what lies beyond the matrix; n_rows (0 .. 8), n_cols (0 .. 16): what there is of this lane's.
__device__ __forceinline__ void cut_staged_rows(uint32_t (&raw)[8][8], int n_rows, int n_cols)
{
    if (n_rows == 8 && n_cols == 16) return;
#pragma unroll
    for (int k = 0; k < 8; k++) {
        const uint32_t keep = 2 * k + 2 <= n_cols ? 0xFFFFFFFFu : 2 * k < n_cols ? 0xFFFFu : 0u;
#pragma unroll
        for (int r = 0; r < 8; r++) raw[r][k] = r < n_rows ? raw[r][k] & keep : 0u;
    }
}

// Segment r of lane's eight (rows rg * 8 + r, columns 32 t + 16 ch .. + 15; t = lane / 8, rg = lane / 2 % 4, ch = lane % 2) of the staged tile;
// what lies beyond the matrix reads as zero.
template <typename P>
__device__ __forceinline__ void read_staged_row(const P &p, int64_t tile_row0, int64_t tile_col0, const uint8_t *stage, int lane, int r, uint32_t out[8])
{
    const int seg = 2 * (lane >> 3) + (lane & 1), rg = (lane >> 1) & 3;
    const int64_t row = tile_row0 + 8 * rg + r, col0 = tile_col0 + 16 * seg;
    if (row < p.rows && col0 < p.cols) {
        const uint32_t off = (uint32_t)(reinterpret_cast<uintptr_t>(p.x + row * p.ld_x + tile_col0) & 15);
        read_staged_segment(stage + stage_row_offset(r, rg) + 32 * seg, off, out);
        if (col0 + 16 > p.cols) {   // what follows the row's last element belongs to the next row
            const int n = (int)(p.cols - col0);
#pragma unroll
            for (int k = 0; k < 8; k++) out[k] = 2 * k + 2 <= n ? out[k] : 2 * k < n ? out[k] & 0xFFFFu : 0u;
        }
    } else {
#pragma unroll
        for (int k = 0; k < 8; k++) out[k] = 0u;
    }
}

}  // namespace fp4q
