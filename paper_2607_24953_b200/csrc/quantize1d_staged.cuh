// 1D-block quantizers of matrices whose rows start anywhere, or that are not made of whole tiles (quantize1d_staged.cu).
#pragma once

#include "common.cuh"

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

// Which matrices come here, by their elements.  Rows that start anywhere, blocks along the rows: reading them element by element takes 2.2 us and
// 2 a million elements, staged tiles 5 and 0.45 (300 x 777 3.4 / 5.1, 1999 x 1003 6.2 / 5.4, 4099 x 5001 38.8 / 14.6).  The transpose of what is not made
// of whole tiles: rows on words have a kernel that is the better one for matrices that are over soon (2048 x 2752 5.7 / 7.6, 3000 x 3000
// 12.5 / 10.0); others 300 x 777 8.3 / 5.4, 1999 x 2731 11.3 / 8.3.
constexpr int64_t kStagedRowsFrom = 3 << 19, kStagedTransposeFrom = 6 << 20;

// fp8: E4M3 payload (MXFP8), otherwise E2M1; transposed: the encoding of x^T.  Rounding to nearest.  The caller has checked its arguments.
fp4q_status launch_quantize1d_staged(Staged1dParams p, bool fp8, bool transposed, cudaStream_t stream);

// UE8M0 code of MXFP8's truncation-free scale: the smallest e with 448 * 2^e >= M, from the BF16 magnitude bits of M.
__device__ __forceinline__ int e4m3_scale_code(uint32_t mbits)
{
    const int be = (int)(mbits >> 7), m7 = (int)(mbits & 0x7F);
    const int code = be == 0 ? 0 : be - 8 + (m7 > 0x60 ? 1 : 0);
    return code < 0 ? 0 : code;
}

}  // namespace fp4q
