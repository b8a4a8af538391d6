// Block-scaled tcgen05 GEMMs for sm_100a: C[M,N] = A[M,K] * B[N,K]^T with both operands
// contraction-contiguous ("K-major"), FP32 accumulation in tensor memory.
//
//   kind::mxf4      E2M1 payload, 2 codes per byte, one UE8M0 scale per 32x32 block of the source tensor
//                   (the 2D-block format): the hardware's per-row, per-32-element scale for row r and
//                   contraction block kb is scale[r/32][kb] or, for a transposed view, scale[kb][r/32].
//   kind::mxf8f6f4  E4M3 payload, one UE8M0 scale per row and 32 contraction elements (MXFP8).
//
// Persistent kernel, one CTA per SM, 12 warps.  Dense products of more than 128 rows, grouped weight gradients and grouped rows
// on 256-row boundaries, or on 128-row ones where that pays, run as clusters of two CTAs that share a 256x256 tile through cta_group::2 MMAs (each CTA holds 128
// rows of the accumulator, loads its own 128 A rows and half of the B rows); everything else uses one CTA per 128x256 tile.
//   warp 0      TMA producer: per stage the A tile (128 rows x 128 B) and the B tile (256 or 128 rows x 128 B),
//               128B swizzle
//   warp 1      MMA issuer: stays converged, one elected lane issues per stage 6 tcgen05.cp (scale images -> TMEM),
//               4 tcgen05.mma and the tcgen05.commit that frees the slot; in the second CTA of a pair it reports
//               that CTA's per-row scale images to the leader
//   warp 2      MXFP8 and long dense FP4 products on pairs: watcher, polls the slots' "full" barriers (several at a time), the scale images
//               and the accumulator's "empty" barrier and meets the MMA warp at a named barrier per stage (elsewhere the
//               MMA warp looks for itself); per-row FP4 kinds: second scale image builder
//   warp 3      scale image builder: per unit of 16 stages (4 or 2 with per-row images) loads the scale bytes and writes the
//               images tcgen05.cp reads in place (double-buffered); 2D-block scales as replicated 8-row images,
//               per-row scales as real 32-row images
//   warps 4-11  epilogue: tcgen05.ld of the 128x256 FP32 accumulator (each warp 32 lanes x 128 columns),
//               release of the accumulator as soon as it sits in registers, then convert and store (through staging
//               rows and TMA stores; one CTA with MXFP8: 256-bit stores)
// A ring of three or four (one CTA: 48 KB of operands per stage) or four or five (pair: 32 KB) shared-memory stages, by kind
// (Cfg), is guarded by mbarriers; the scale columns in TMEM form a ring of the same depth.  Every mbarrier wait is bounded: when a limit
// is hit the CTA records FP4Q_ERR_TIMEOUT in the workspace, releases the MMA warp from its named barriers, stops
// issuing work and leaves through the normal exit (TMEM is freed).
#include <atomic>
#include <cstdlib>
#include <cuda.h>
#include <cuda_bf16.h>

#include "common.cuh"
#include "quant_device.cuh"

namespace fp4q {

constexpr int BM = 128, BN = 256;            // per-CTA accumulator: 128 rows x 256 columns (a CTA pair covers 256 x 256)
constexpr int kMaxStages = 6;
constexpr int kAStageBytes = BM * 128;
constexpr int kMaxGroupsShared = 1023;       // grouped contraction: boundaries kept in shared memory up to this many groups
constexpr int kMaxGroupsSorted = 256;        // grouped contraction: up to this many groups may be taken longest first (launch_gemm_impl says when)
constexpr int kMaxGroupsPaired = 3071;       // paired rows: groups whose first tiles and numbers of pairs fit where the images will be
constexpr int kMaxRowTilesShared = 2048;     // grouped rows: group of each 128-row tile kept in shared memory up to this many tiles
constexpr int kSmemTail = 512;               // barriers, TMEM base, abort flag, scale scratch (one per loader warp)
// 2D-block scales: the scale images of a whole unit (up to 16 stages = 4096 contraction elements of one tile) are
// built once, ahead of time, and tcgen05.cp reads them in place.  Per 128-element chunk the compact form is one
// 16-byte row for A [row tile 0..3][block 0..3] and two for B (row tiles 0..3, 4..7); an image is such a row
// replicated over the 8 rows of one core matrix (128 B), which a descriptor with a zero stride between 8-row
// groups presents as the 32 identical rows tcgen05.cp.32x128b expects.  Per stage: 6 images = 768 B.
constexpr int kCacheChunks = 32;             // chunks per unit
constexpr int kUnitStagesMxf4 = kCacheChunks / 2;
// Per-row scales (MXFP8): a stage covers 4 contraction blocks; its three images (A rows, B rows 0..127, B rows
// 128..255) are real 32-row x 16-byte images (512 B each), row l holding rows l, l+32, l+64, l+96 of the operand.
// A unit is 4 stages (16 blocks, one 16-byte piece of every row's scales): half of the other kinds' 12 KB buffers, which
// pays for one more ring stage.
constexpr int kUnitStagesMxf8 = 4;
constexpr int kImageStageBytesMxf8 = 1536;
constexpr int kImageStageBytes = 768;        // A chunk 0, A chunk 1, B chunk 0 (rows 0..127, 128..255), B chunk 1 (same)
constexpr int kCompactBytes = kCacheChunks * 48;
// mxf4 with per-row scales: a stage has two chunks of four blocks.  The 1D-block operand has real images, A 2 x 512 B or B (256 rows)
// 4 x 512 B per stage, the 2D-block operand replicated ones like above, B 4 x 128 B or A 2 x 128 B.
constexpr int kUnitStagesMxf4R = 4;
constexpr int kImageStageBytesMxf4RA = 1024 + 512, kImageStageBytesMxf4RB = 256 + 2048;
// mxf4nvf4 with 16-element scale vectors (tensors quantized in 16 x 16 blocks): every MMA (64 contraction elements)
// has its own image per 128 operand rows - four scale bytes per row - so a stage holds A 4 x 512 B and B 8 x 512 B
constexpr int kUnitStagesMxf4B16 = 2;
constexpr int kImageStageBytesMxf4B16 = 6144;
// Epilogue staging of the pair kernel: each of the 8 epilogue warps owns 32 rows x 128 bytes, written from registers
// (128-byte swizzle: the 16-byte pieces of 8 rows fall into different banks) and drained by a TMA store, which keeps
// the output off the load/store unit that the MMA warp's instructions also pass through.
constexpr int kStagingWarpBytes = 32 * 128;

// CTAS = 1: one CTA per 128x256 tile, it loads all 256 B rows.  CTAS = 2: a cluster of two CTAs shares a 256x256
// tile through cta_group::2 MMAs; each CTA loads its own 128 A rows and half of the B rows, which halves the
// B-operand shared-memory and L2 traffic per CTA and leaves room for two more ring stages.
// KIND_MXF4: FP4 payloads, 2D-block scales on both operands (replicated scale images).  KIND_MXF8: E4M3 payloads,
// per-row scales.  KIND_MXF4RA, KIND_MXF4RB: FP4 payloads with per-row scale images for one operand - A or B quantized in 1D blocks (the
// paper's activation layout) - next to a 2D-block operand with replicated ones: in row-major order (B of the forward product) and
// seen transposed (A of the weight gradient).
// KIND_MXF4B16: FP4 payloads of tensors quantized in 16 x 16 blocks (block-size study): 16-element scale vectors
// (kind::mxf4nvf4, scale_vec::4X, UE8M0 scales), real images whose upper and lower 16 rows are equal.
enum { KIND_MXF4 = 0, KIND_MXF8 = 1, KIND_MXF4RA = 2, KIND_MXF4RB = 3, KIND_MXF4B16 = 4 };
__host__ __device__ constexpr bool kind_fp4(int kind) { return kind != KIND_MXF8; }

// Per-row scale images are rebuilt every 4 stages (2 with 16 x 16 blocks), and the global-memory latency of the bytes they are made of
// (about 3000 cycles under the operand traffic) exceeds the time such a unit runs.  The kernels for those kinds therefore fetch the
// bytes two units ahead with cp.async into raw buffers (no registers are held meanwhile); the pair kernel also keeps a third image
// buffer, because the way from "the MMAs have finished with a buffer" to "the leader may copy the next unit out of it" (commit to
// both CTAs, build, report to the leader) is longer than one unit as well.
template <int KIND, int CTAS>
struct Cfg {
    static constexpr bool kRowImages = KIND != KIND_MXF4;
    // Image builder warps: the per-row FP4 kinds, whose units are 4 or 2 stages, have two that take turns (one warp needs
    // 1500-2500 cycles for a unit, all of it latency); their MMA warp waits for itself and needs no watcher.
    static constexpr int kBuilders = kRowImages && KIND != KIND_MXF8 ? 2 : 1;
    static constexpr int kImageBufs = (CTAS == 2 && kRowImages) ? (KIND == KIND_MXF4B16 ? 4 : 3) : 2;
    static constexpr int kRawBufs = kRowImages ? (KIND == KIND_MXF4B16 ? 4 : 2) : 0;
    // The output leaves through staging rows and TMA stores wherever shared memory allows (everything but the
    // one-CTA kernel of MXFP8).  In the one-CTA kernel of the 2D kind - grouped products with short
    // contractions - plain stores of the 64 KB tile filled the SM's path to L2 and the TMA loads issued meanwhile
    // took 6500-8000 cycles instead of 3000; the staging costs that kernel its fourth ring stage.
    static constexpr bool kTmaStores = CTAS == 2 || KIND != KIND_MXF8;
    static constexpr int kStages = CTAS == 2 ? (KIND == KIND_MXF4RB || KIND == KIND_MXF4B16 ? 4 : 5) : (kTmaStores ? 3 : 4);
    static constexpr int kUnitStages = KIND == KIND_MXF4 ? kUnitStagesMxf4 : KIND == KIND_MXF8 ? kUnitStagesMxf8
                                       : KIND == KIND_MXF4B16 ? kUnitStagesMxf4B16 : kUnitStagesMxf4R;   // stages whose scale images are built together
    static constexpr int kImageStage = KIND == KIND_MXF4 ? kImageStageBytes : KIND == KIND_MXF8 ? kImageStageBytesMxf8 : KIND == KIND_MXF4B16 ? kImageStageBytesMxf4B16
                                       : KIND == KIND_MXF4RA ? kImageStageBytesMxf4RA : kImageStageBytesMxf4RB;
    static constexpr int kBufBytes = kUnitStages * kImageStage;   // an image buffer
    // A raw buffer: A's bytes, then B's, in entries of one row each, a word longer than the row's bytes of a unit (RowFetch); a 2D-block
    // operand's entries are its row tiles or, seen transposed, the unit's 32 blocks.
    static constexpr int kRawA = KIND == KIND_MXF8 ? 128 * 20 : KIND == KIND_MXF4RA ? 128 * 36 : KIND == KIND_MXF4RB ? 32 * 8 : 32 * 12;
    static constexpr int kRawB = KIND == KIND_MXF8 ? 256 * 20 : KIND == KIND_MXF4RA ? 8 * 36 + 32 : KIND == KIND_MXF4RB ? 256 * 36 : 32 * 20;
    static constexpr int kRawBytes = kRawA + kRawB;
    static constexpr int kSortedBytes = KIND == KIND_MXF4RA || KIND == KIND_MXF4RB ? 256 : KIND == KIND_MXF4B16 ? 768 : 0;   // a builder's 2D-block bytes as image rows
    static constexpr int kSmemCache = kRowImages ? kImageBufs * kBufBytes + kRawBufs * kRawBytes + kBuilders * kSortedBytes : kCompactBytes + kImageBufs * kBufBytes;
    static constexpr int kBRows = CTAS == 2 ? 128 : 256;
    static constexpr int kBStageBytes = kBRows * 128;
    static constexpr int kSmemOperands = kStages * (kAStageBytes + kBStageBytes);
    static constexpr int kSmemScales = (kSmemCache + 1023) / 1024 * 1024;
    static constexpr int kSmemStaging = kTmaStores ? 8 * kStagingWarpBytes : 0;
    static constexpr int kSmemGroups = (CTAS == 1 || KIND == KIND_MXF4) ? (kMaxGroupsShared + 1) * 4 + kMaxGroupsSorted * 2 : 0;   // grouped products: group tables
    static_assert(kSmemGroups == 0 || (kMaxGroupsShared + 1) * 4 >= kMaxRowTilesShared * 2, "group table");
    static constexpr int kSmemBytes = 1024 + kSmemOperands + kSmemScales + kSmemStaging + kSmemTail + kSmemGroups;
    static_assert(kSmemBytes <= 227 * 1024, "shared memory budget");
};
// Dense products and grouped rows: row tiles per rasterisation group.  With grouped rows a group's A rows and the weights of the
// few experts they belong to stay in L2 for the whole sweep over the columns (expert layer, 139520 rows, one group of all
// row tiles -> groups of 16: 768 x 2048 fwd/dgrad 142/207 -> 126/166 us, 2048 x 768 199/144 -> 158/128; 8 and 32 within 2 %).
constexpr int kRasterM = 16;
constexpr int kShortStages = 48;   // a short product: up to so many ring stages per CTA or pair (launch_gemm, launch_gemm_impl)
constexpr int kThreads = 384;
constexpr int kTmemCols = 512;
constexpr int kTmemSfBase = 256;
// scale columns per ring stage: SFA at +0 (+4 per chunk), SFB at +8 (+8 per chunk); with 16-element scale vectors
// SFA at +0 (+4 per MMA), SFB at +16 (+8 per MMA)
template <int KIND> struct SfCols { static constexpr int kStride = KIND == KIND_MXF4B16 ? 48 : 32; };
static_assert(kTmemSfBase + 5 * SfCols<KIND_MXF4>::kStride <= kTmemCols && kTmemSfBase + 4 * SfCols<KIND_MXF4B16>::kStride <= kTmemCols,
              "tensor memory budget: 256 accumulator columns + one scale slot per ring stage");
constexpr uint32_t kWaitLimit = 1u << 22;       // default number of polls after which a wait gives up (workspace word 2 overrides it)
// Longest suspension of one suspending poll: without it the limit is the system's, and a number of polls bounds nothing.  With
// 2^22 polls a wait gives up after about four seconds at the latest.
constexpr uint32_t kSuspendNs = 1000;
constexpr int kRelaxedNs = 64, kLazyNs = 256;   // back-off between polls of roles with slack
// Developer diagnostic (off by default): -DFP4Q_TRACE makes CTA 0 add up clock64() intervals of its roles in
// registers and leave them in the workspace's padding words (status[16 + 2*slot], 64-bit each).
#ifdef FP4Q_TRACE
#define TRACE_DECL(n) long long n = 0
#define TRACE_T0(t) long long t = clock64()
#define TRACE_ADD(acc, t) do { long long t_now = clock64(); acc += t_now - t; t = t_now; } while (0)
#define TRACE_OUT(p, slot, v) do { if (blockIdx.x == 0) reinterpret_cast<long long *>(p.status + 16)[slot] = (v); } while (0)
#ifdef FP4Q_TRACE_EVENTS
__device__ long long g_trace_events[2][8][512][2];   // [CTA 0/1][kind][stream index][clock64, globaltimer]
#define TRACE_EV(kind, idx) do { if (blockIdx.x < 2 && (idx) < 512) { long long gt; asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(gt)); \
    g_trace_events[blockIdx.x][kind][idx][0] = clock64(); g_trace_events[blockIdx.x][kind][idx][1] = gt; } } while (0)
extern "C" int fp4q_debug_events(void *host) { return (int)cudaMemcpyFromSymbol(host, g_trace_events, sizeof(g_trace_events)); }
#else
#define TRACE_EV(kind, idx)
#endif
#else
#define TRACE_EV(kind, idx)
#define TRACE_DECL(n)
#define TRACE_T0(t)
#define TRACE_ADD(acc, t)
#define TRACE_OUT(p, slot, v)
#endif
constexpr uint8_t kScalePad = 127;           // UE8M0 code of 1.0 for scale slots beyond the tensor (their payload is 0)

// MODE_PAIRED_ROWS: grouped rows on pairs where groups start on multiples of 128 rows: two row tiles of one group a pair, the last alone if
// the group has an odd number (the second CTA then loads nothing for A and stores nothing).
enum { MODE_DENSE = 0, MODE_GROUPED_ROWS = 1, MODE_GROUPED_K = 2, MODE_PAIRED_ROWS = 3 };

struct ScaleView {
    const uint8_t *ptr;
    int64_t stride_row;   // 2D blocks: bytes between consecutive row tiles (of 32 or 16 rows); per-row scales: between consecutive rows
    int64_t stride_kb;    // bytes between consecutive contraction blocks of 32
    int32_t n_row;        // 2D blocks: number of row tiles; per-row scales: number of rows
    int32_t n_kb;         // number of contraction blocks
    int32_t words;        // 2D blocks: ptr and the pitch are multiples of four bytes and offsets fit in 32 bits; set by the launch
};

// Division by a number that the launch knows, as a multiplication (Granlund and Montgomery, "Division by invariant integers using
// multiplication", 1994): with s = ceil(log2 d) and m = ceil(2^(31+s) / d), n / d = n m >> (31 + s) for every n < 2^31.
struct Divisor {
    uint32_t m, shift;
    __host__ __device__ __forceinline__ int32_t operator()(int32_t n) const { return (int32_t)((uint64_t)(uint32_t)n * m >> shift); }
};
static Divisor divisor(int32_t d)
{
    uint32_t s = 0;
    while (((int64_t)1 << s) < d) s++;
    return Divisor{(uint32_t)((((uint64_t)1 << (31 + s)) + (uint64_t)d - 1) / (uint64_t)d), 31 + s};
}

struct GemmParams {
    ScaleView sfa, sfb;
    void *C;
    int64_t ldc;
    int32_t M, N, K;                 // per-problem output rows, output columns, contraction length (elements)
    int32_t m_tiles, n_tiles, n_tile_total;   // m_tiles counts rows of 128 * ctas
    int32_t ctas;                    // CTAs per tile (1, or 2 for cta_group::2 pairs)
    int32_t raster_m;                // tile order: groups of raster_m row tiles, within a group row tile fastest
    Divisor by_problem, by_group, by_raster, by_tail;   // m_tiles * n_tiles; raster_m * n_tiles; raster_m; row tiles of the last group if it is smaller
    int32_t out_f32, accumulate;
    int32_t padded;                  // the output's rows may be filled up to 16 bytes
    int32_t tail_col;                // EPI_TAIL: first column of a row's last bytes, fewer than 16, which TMA stores do not write; INT32_MIN: none
    int32_t wide_stores;             // output base and row pitch are 32-byte aligned: 256-bit stores (whole sectors)
    int32_t mode, n_groups;
    int32_t rows_pair_aligned;       // grouped rows: every group starts on a multiple of 256 rows (caller's statement)
    const int64_t *row_offsets;
    int32_t b_rows_per_group;        // grouped rows: B row offset per group (forward)
    int32_t b_k_per_group;           // grouped rows: B contraction offset per group (dgrad)
    int32_t sort_groups;             // grouped contraction: take the groups longest first
    int32_t warps_meet;              // grouped contraction: epilogue warps start a tile together
    uint32_t *status;
    // quantizing epilogue (EPI_QUANT): the output leaves as a 2D-block FP4 tensor instead of BF16/FP32
    uint8_t *q_rm, *q_t, *q_scale;
    int64_t q_ld_rm, q_ld_t, q_ld_s;
    int32_t q_mode;                  // FP4Q_ROUND_NEAREST or FP4Q_ROUND_STOCHASTIC
    uint32_t q_tensor_id;
    PhiloxRoundKeys q_keys;
};

enum { EPI_STORE = 0, EPI_QUANT = 1, EPI_TAIL = 2 };   // TAIL: rows of the output end inside 16 bytes, which TMA stores would fill

struct Tile {
    int32_t a_row0, b_row0, b_load_row0, a_k0, b_k0, k_len, c_row0, c_col0, m_valid, n_valid;
};

// ---------------------------------------------------------------------------------------- PTX helpers

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.b32 %0, 1, 0, p;\n}"
                 : "=r"(ok) : "r"(bar), "r"(parity), "r"(kSuspendNs) : "memory");
    return ok != 0;
}

// Non-blocking probe of a barrier phase (the try_wait form may suspend the thread for a while).
__device__ __forceinline__ bool mbar_test_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.b32 %0, 1, 0, p;\n}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// One lane of a converged warp.
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile("{\n .reg .pred P;\n elect.sync _|P, 0xFFFFFFFF;\n selp.b32 %0, 1, 0, P;\n}" : "=r"(p));
    return p != 0;
}
// Named barrier on which the MMA warp and the warp that watches a ring slot for it meet (64 threads).  Both sides use the waiting
// form: with a non-waiting arrival a watcher that has given up, and only counts the remaining stages, could complete a barrier phase on
// its own and leave the MMA warp without a partner.  It says so with its arrival; returns whether the stage may be used.
__device__ __forceinline__ bool named_meet(uint32_t id, bool usable)
{
    uint32_t r;
    asm volatile("{\n .reg .pred p, q;\n setp.ne.u32 p, %2, 0;\n bar.red.and.pred q, %1, 64, p;\n selp.u32 %0, 1, 0, q;\n}" : "=r"(r) : "r"(id), "r"((uint32_t)usable) : "memory");
    return r != 0u;
}

// Bounded wait.  Returns false when the limit ran out (the timeout is then recorded) or when another
// role of this CTA has already given up, which it looks for after every suspension and after every 256th probe.  Every poll
// of an mbarrier is a shared-memory transaction that competes with the tensor core's operand reads and with the other
// roles' waits: a suspended thread makes one in kSuspendNs at most.
template <int BACKOFF_NS, bool PROBE = false>
__device__ __forceinline__ bool mbar_wait_impl(uint32_t bar, uint32_t parity, volatile uint32_t *abort_flag, uint32_t *status,
                                               uint64_t limit, uint32_t where)
{
    for (uint64_t it = 1; ; it++) {
        if (PROBE ? mbar_test_wait(bar, parity) : mbar_try_wait(bar, parity)) return true;
        if (BACKOFF_NS > 0) __nanosleep(BACKOFF_NS);
        if ((!PROBE || ((uint32_t)it & 255u) == 0u) && *abort_flag) return false;
        if (it >= limit) break;   // after the first poll: a wait that need not wait does not wait for the limit's load either
    }
    *abort_flag = 1u;
    if (atomicCAS(status, 0u, (uint32_t)FP4Q_ERR_TIMEOUT) == 0u) status[1] = where;
    return false;
}
__device__ __noinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile uint32_t *abort_flag, uint32_t *status, uint64_t limit,
                                       uint32_t where)
{
    return mbar_wait_impl<0>(bar, parity, abort_flag, status, limit, where);
}
// For the end of an aborted launch, when the abort flag is set already: 256 polls, a third of a millisecond at most.
__device__ __noinline__ void mbar_drain(uint32_t bar)
{
    for (int it = 0; it < 256 && !mbar_try_wait(bar, 0u); it++) __nanosleep(kLazyNs);
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int32_t x, int32_t y, uint32_t bar)
{
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar) : "memory");
}

// The same load issued by either CTA of a pair: the bytes are counted on the barrier at this address in the
// pair's leader CTA (cta_group::2 permits the barrier to live in the peer).
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap *map, int32_t x, int32_t y, uint32_t leader_bar)
{
    asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(leader_bar) : "memory");
}
// shared::cluster address of this CTA's shared-memory location `addr` as seen in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t cluster_addr(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// What such an arrival announces lies in this CTA's own shared memory or tensor memory and was made visible to the asynchronous proxy
// or fenced before; the other CTA only issues the instructions that read it here.  Release at the default scope, this CTA, orders the
// two, as an assumption about the hardware: that an SM has performed its own stores and the fence behind them before a later
// arrival of the same thread leaves it.  PTX's memory model does not promise it; there, only release and acquire that both
// reach the cluster order one CTA's writes before another's reads, and the waits on these barriers have the default scope too.
// Were it wrong, a pair's MMAs would read scale images of the second CTA that are not written yet, or overwrite an accumulator that is
// still being read: wrong results and no error.  Release at cluster scope for the images costs a product 0.45 to 0.6 us (forward
// 2048 x 2048 x 2048 9.9 -> 10.4, 8192 x 2048 x 2048 20.5 -> 21.0, 16384 x 4096 x 4096 94.5 -> 95.2; 16 x 16 blocks there 116.8 -> 121.5).
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_bar)
{
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}
__device__ __forceinline__ uint32_t cluster_ctarank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// The kernel's first barrier, which every warp passes at a place of its own: behind it the mbarriers of the CTA, or of both CTAs of
// a pair, exist.  In a pair warps arrive ahead of time (warp 4, which initializes them, after its fence.mbarrier_init), so that the
// way from one CTA to the other is under way while a role prepares what needs nobody else.  Only warp 1 arrives late: behind its
// allocation of tensor memory, with release, because the leader's scale copies and MMAs write the other CTA's tensor memory and
// nothing else puts them behind that CTA's allocation.  us, that arrival ahead of the allocation too and behind it: FP4 products level
// (2048 x 2048 x 2048 8.1 / 8.3 / 9.3 and 8.1 / 8.1 / 9.2), per-row kinds 1 to 1.5 % for small ones (16 x 16 blocks 8192 x 2048 x 2048 22.6 / 22.2 / 19.7 and
// 22.9 / 22.4 / 20.0, MXFP8 there 29.8 and 30.2).  In one CTA nobody waits for the builders, which come late and have a barrier of
// their own with warp 4.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
template <int CTAS, int BUILDERS, bool BUILDER = false>
__device__ __forceinline__ void start_sync()
{
    if (CTAS == 2) cluster_wait();
    else if (BUILDER) asm volatile("bar.sync 12, %0;" ::"n"(32 + 32 * BUILDERS) : "memory");
    else asm volatile("bar.sync 13, %0;" ::"n"(kThreads - 32 * BUILDERS) : "memory");
}

// TMA stores out of shared memory (bulk async-group completion).
__device__ __forceinline__ void tma_store_2d(const CUtensorMap *map, int32_t x, int32_t y, uint32_t src)
{
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];" ::"l"(map), "r"(x), "r"(y), "r"(src) : "memory");
}
__device__ __forceinline__ void tma_reduce_add_2d(const CUtensorMap *map, int32_t x, int32_t y, uint32_t src)
{
    asm volatile("cp.reduce.async.bulk.tensor.2d.global.shared::cta.add.tile.bulk_group [%0, {%1, %2}], [%3];" ::"l"(map), "r"(x), "r"(y), "r"(src) : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read_all() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }

__device__ __forceinline__ void tcgen05_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tcgen05_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }

template <int CTAS>
__device__ __forceinline__ void tcgen05_commit(uint32_t bar)
{
    if (CTAS == 1) {
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
    } else {   // arrives on the barrier at this offset in both CTAs of the pair
        asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                     ::"r"(bar), "h"((uint16_t)3) : "memory");
    }
}
template <int CTAS>
__device__ __forceinline__ void tcgen05_cp_32x128b_warpx4(uint32_t taddr, uint64_t sdesc)
{
    if (CTAS == 1) asm volatile("tcgen05.cp.cta_group::1.32x128b.warpx4 [%0], %1;" ::"r"(taddr), "l"(sdesc) : "memory");
    else asm volatile("tcgen05.cp.cta_group::2.32x128b.warpx4 [%0], %1;" ::"r"(taddr), "l"(sdesc) : "memory");
}

template <int KIND, int CTAS>
__device__ __forceinline__ void tcgen05_mma_block_scaled(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                                         uint32_t sfa_tmem, uint32_t sfb_tmem, uint32_t accumulate)
{
    if (KIND == KIND_MXF4B16 && CTAS == 2) {
        asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                     " tcgen05.mma.cta_group::2.kind::mxf4nvf4.block_scale.scale_vec::4X [%0], %1, %2, %3, [%5], [%6], p;\n}"
                     ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(sfa_tmem), "r"(sfb_tmem)
                     : "memory");
    } else if (KIND == KIND_MXF4B16) {
        asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                     " tcgen05.mma.cta_group::1.kind::mxf4nvf4.block_scale.scale_vec::4X [%0], %1, %2, %3, [%5], [%6], p;\n}"
                     ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(sfa_tmem), "r"(sfb_tmem)
                     : "memory");
    } else if (kind_fp4(KIND) && CTAS == 2) {
        asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                     " tcgen05.mma.cta_group::2.kind::mxf4.block_scale.scale_vec::2X [%0], %1, %2, %3, [%5], [%6], p;\n}"
                     ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(sfa_tmem), "r"(sfb_tmem)
                     : "memory");
    } else if (kind_fp4(KIND)) {
        asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                     " tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], %1, %2, %3, [%5], [%6], p;\n}"
                     ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(sfa_tmem), "r"(sfb_tmem)
                     : "memory");
    } else if (CTAS == 2) {
        asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                     " tcgen05.mma.cta_group::2.kind::mxf8f6f4.block_scale.scale_vec::1X [%0], %1, %2, %3, [%5], [%6], p;\n}"
                     ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(sfa_tmem), "r"(sfb_tmem)
                     : "memory");
    } else {
        asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                     " tcgen05.mma.cta_group::1.kind::mxf8f6f4.block_scale.scale_vec::1X [%0], %1, %2, %3, [%5], [%6], p;\n}"
                     ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(sfa_tmem), "r"(sfb_tmem)
                     : "memory");
    }
}

// Shared-memory matrix descriptor, K-major operand tile stored as rows of 128 B with the 128-byte swizzle
// (8-row groups 1024 B apart).
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t addr)
{
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | (1ull << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
// Descriptor of a replicated scale image: 8 rows of 16 B; the stride between 8-row groups is zero, so the 32 rows
// tcgen05.cp reads are four passes over the same 128 bytes.
__device__ __forceinline__ uint64_t smem_desc_scale_image_rep(uint32_t addr)
{
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | (1ull << 46);
}
// Descriptor of a scale image: 32 rows of 16 B, contiguous (no swizzle; 8-row groups 128 B apart).
__device__ __forceinline__ uint64_t smem_desc_scale_image(uint32_t addr)
{
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(128 >> 4) << 32) | (1ull << 46);
}

// Instruction descriptor of the block-scaled MMA: formats, K-major operands, N, UE8M0 scales, M, scale byte ids.
template <int KIND, int CTAS>
__device__ __forceinline__ uint32_t instr_desc(uint32_t a_sf_id, uint32_t b_sf_id)
{
    const uint32_t fmt = kind_fp4(KIND) ? 1u : 0u;   // mxf4: E2M1 = 1; mxf8f6f4: E4M3 = 0
    return (b_sf_id << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(BN >> 3) << 17) | (1u << 23) |
           ((uint32_t)((BM * CTAS) >> 4) << 24) | (a_sf_id << 29);
}

#define FP4Q_TMEM_LD_X32(taddr, v)                                                                              \
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "                                                      \
                 "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"                                      \
                 "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"                     \
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), \
                   "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]),      \
                   "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]),    \
                   "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]),    \
                   "=r"(v[29]), "=r"(v[30]), "=r"(v[31])                                                         \
                 : "r"(taddr))

// ---------------------------------------------------------------------------------------- tile decoding

// Grouped products need their group once per tile.  Searching the boundaries is a chain of dependent loads (seven
// for 128 groups), and in the TMA producer every load queues behind the copies it has just issued (about 500 cycles
// each): 4000 cycles per tile, more than a tile with a short contraction runs.  So the CTA fills a table in shared
// memory before its roles start (`goffs`, 4 KB, null when the problem is too large for it or the kernel's
// configuration has no room): with grouped rows the group of every 128-row tile as 16 bits (one load per tile),
// with a grouped contraction a 32-bit copy of the boundaries, with paired rows a word for every pair: its first row tile (16 bits),
// its group (15) and whether it has that tile only (1).

__device__ __forceinline__ int find_group(const int64_t *offs, const int32_t *goffs, int n_groups, int64_t row)
{
    int lo = 0, hi = n_groups;      // largest g with offs[g] <= row
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        const int64_t v = goffs ? (int64_t)goffs[mid] : load_global(offs + mid);
        if (v <= row) lo = mid; else hi = mid;
    }
    return lo;
}

// need: NEED_ALL; NEED_OUTPUT leaves out the B operand's position, with grouped rows the group lookup, which only the
// producer and the scale builder need; NEED_LENGTH, the contraction length alone, is for the MMA issuer and the watcher: a lookup in
// the MMA warp (shared-memory reads behind its pending MMAs) costs about 1900 cycles per tile.
// m_tiles: p.m_tiles but for paired rows, whose number only the boundaries tell.
enum { NEED_LENGTH = 0, NEED_OUTPUT = 1, NEED_ALL = 2 };
// One warp runs an instruction in about five cycles and every role decodes its tiles.  us, with integer divisions and with multiplications:
// 2048 x 2048 x 2048 10.4 / 10.6 / 11.9 -> 10.3 / 10.4 / 11.7, 16 groups of 9088 rows 768 x 1440 16.6 / 14.2 / 23.7 -> 16.0 / 13.4 / 22.9, quantized
// output 8192 x 5632 x 2048 61.4 -> 58.2.
// GROUPS: what a kernel is made for.  Dense products' tiles are decoded without the group branches, which cost the builders of the
// per-row kinds 3-8 % of a product (1D activations at 4096 x 4096 x 4096: 45.8 us without, 49.7 us with), one CTA's smallest ones 0.3 us
// (128 x 256 x 256 6.1 / 5.8) and quantized outputs 3-5 % (2048 x 2048 x 2048 12.4 / 11.7, 8192 x 5632 x 2048 56.6 / 55.2).
enum { GROUPS_NONE = 0, GROUPS_ANY = 1, GROUPS_PAIRED = 2, GROUPS_CUT = 3 };   // PAIRED: any, and paired rows; CUT: weight gradients of experts whose rows end within a box of 32
template <int GROUPS>
__device__ __forceinline__ void decode_tile(const GemmParams &p, int tile, int rank, Tile &t, int m_tiles, const int32_t *goffs, const uint16_t *gorder, int need = NEED_ALL)
{
    const int mode = GROUPS != GROUPS_NONE ? p.mode : MODE_DENSE;
    const int per_problem = m_tiles * p.n_tiles;
    const int nth = mode == MODE_GROUPED_K ? p.by_problem(tile) : 0, g = mode == MODE_GROUPED_K && gorder ? (int)gorder[nth] : nth;
    const int local = tile - nth * per_problem;
    // Tiles that run at the same time (consecutive indices) cover raster_m row tiles x a few column tiles, and
    // the sweep over column tiles finishes before the next group of row tiles starts: the group's A rows stay
    // in L2 for the whole sweep instead of the whole A operand being streamed once per wave.
    const int per_group = p.raster_m * p.n_tiles;
    const int grp_m = p.by_group(local), in_grp = local - grp_m * per_group;
    const int m0 = grp_m * p.raster_m, gsz = min(p.raster_m, m_tiles - m0);
    const int n_blk = gsz == p.raster_m ? p.by_raster(in_grp) : GROUPS == GROUPS_PAIRED && mode == MODE_PAIRED_ROWS ? in_grp / gsz : p.by_tail(in_grp), m_blk = m0 + (in_grp - n_blk * gsz);
    t.a_row0 = (m_blk * p.ctas + rank) * BM;
    t.b_row0 = n_blk * BN;
    t.b_load_row0 = t.b_row0 + (p.ctas == 2 ? rank * 128 : 0);
    t.a_k0 = t.b_k0 = 0;
    t.k_len = p.K;
    t.c_row0 = t.a_row0;
    t.c_col0 = t.b_row0;
    t.m_valid = min(BM, p.M - t.a_row0);
    t.n_valid = min(BN, p.N - t.b_row0);
    if (GROUPS == GROUPS_PAIRED && mode == MODE_PAIRED_ROWS) {
        if (need == NEED_LENGTH) return;
        const uint32_t e = (uint32_t)goffs[m_blk], alone = e >> 31;
        t.a_row0 = t.c_row0 = ((int)(e & 0xFFFFu) + (alone ? 0 : rank)) * BM;
        t.m_valid = alone && rank ? 0 : min(BM, p.M - t.a_row0);
        const int grp = (int)(e >> 16 & 0x7FFFu);
        t.b_row0 += grp * p.b_rows_per_group;
        t.b_load_row0 += grp * p.b_rows_per_group;
        t.b_k0 = grp * p.b_k_per_group;
    } else if (mode == MODE_GROUPED_ROWS) {
        if (need != NEED_ALL) return;
        const int grp = goffs ? (int)reinterpret_cast<const uint16_t *>(goffs)[t.a_row0 / BM]
                              : find_group(p.row_offsets, nullptr, p.n_groups, (int64_t)t.a_row0);
        t.b_row0 += grp * p.b_rows_per_group;
        t.b_load_row0 += grp * p.b_rows_per_group;
        t.b_k0 = grp * p.b_k_per_group;
    } else if (mode == MODE_GROUPED_K) {
        const int64_t k0 = goffs ? (int64_t)goffs[g] : load_global(p.row_offsets + g), k1 = goffs ? (int64_t)goffs[g + 1] : load_global(p.row_offsets + g + 1);
        t.a_k0 = t.b_k0 = (int32_t)k0;
        t.k_len = (int32_t)(k1 - k0);
        t.c_row0 = g * p.M + t.a_row0;
    }
}

// ---------------------------------------------------------------------------------------- scale images

// The stream of ring stages one CTA of a dense product works through: its tiles in order, each with its contraction stages.
struct StageIter {
    int tile, step, rank, it, n_it;
    Tile t;
    __device__ __forceinline__ void seek(const GemmParams &p, int stage_elems)
    {
        while (tile < p.n_tile_total) {
            decode_tile<GROUPS_NONE>(p, tile, rank, t, p.m_tiles, nullptr, nullptr, NEED_LENGTH);
            n_it = (t.k_len + stage_elems - 1) / stage_elems;
            if (n_it > 0) { it = 0; return; }
            tile += step;
        }
        n_it = 0;
    }
    __device__ __forceinline__ void init(const GemmParams &p, int first, int step_, int rank_, int stage_elems)
    {
        tile = first; step = step_; rank = rank_; it = 0;
        seek(p, stage_elems);
    }
    __device__ __forceinline__ bool valid(const GemmParams &p) const { return tile < p.n_tile_total; }
    __device__ __forceinline__ void next(const GemmParams &p, int stage_elems)
    {
        if (++it >= n_it) { tile += step; seek(p, stage_elems); }
    }
};

__device__ __forceinline__ void ldg_b32(const uint8_t *ptr, uint32_t &w)
{
    asm volatile("ld.global.b32 %0, [%1];" : "=r"(w) : "l"(ptr));
}

// Rows of a 4x4 byte matrix given by its columns: w[k] holds byte rt of column k in byte lane rt.
__device__ __forceinline__ uint4 transpose4x4_bytes(uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3)
{
    const uint32_t t0 = __byte_perm(w0, w1, 0x5140), t1 = __byte_perm(w2, w3, 0x5140);
    const uint32_t t2 = __byte_perm(w0, w1, 0x7362), t3 = __byte_perm(w2, w3, 0x7362);
    return make_uint4(__byte_perm(t0, t1, 0x5410), __byte_perm(t0, t1, 0x7632), __byte_perm(t2, t3, 0x5410),
                      __byte_perm(t2, t3, 0x7632));
}

// mxf4 / 2D blocks: a stage covers 8 contraction blocks (two chunks of 4).  For 128 operand rows and one chunk the
// scale image is 32 identical rows of 16 bytes [row tile 0..3][block 0..3]; A needs 2 such rows per stage (one per
// chunk), B (256 rows) 4.
//
// A unit has as many chunks as a warp has lanes: lane c loads the scale bytes of chunk c, four words for every four row tiles, and
// holds whole image rows.  All of a unit's loads are in flight together, and the next unit's while a unit is written.  A product's
// first MMA waits for its first unit, and a tile with a short contraction for its own: with the loads of A and B one after the
// other, then a pass through shared memory, then stores that met in the same banks, the first unit took 3300-6700 cycles from
// the first operand load on and every later one 4000-5000; now 1300-2800 and 1500.  One warp runs an instruction in about five
// cycles, so their number counts as well.
// w[i]: row-major scales: blocks kb..kb+3 of row tile rt0 + i; transposed view (stride_kb != 1): row tiles of group i / 4 of
// block kb + i % 4.
enum { SCALES_WHOLE = 0, SCALES_SHIFTED = 1, SCALES_GATHER = 2 };

// Where word i of lane's chunk starts, and how many bytes exist from there on.  Rows and blocks beyond the tensor take the place of
// ones that exist (their payload is zero, any finite scale will do).
__device__ __forceinline__ const uint8_t *chunk_word(const ScaleView &v, int rt0, int kb, int kb0, int i, int &n)
{
    if (v.stride_kb != 1) {
        const int rt = rt0 + (i & ~3) < v.n_row ? rt0 + (i & ~3) : rt0 < v.n_row ? rt0 : 0;   // 0: the second CTA of a pair, all of whose rows lie beyond
        n = v.n_row - rt;
        return v.ptr + min(kb + (i & 3), v.n_kb - 1) * v.stride_kb + rt;
    }
    if (kb >= v.n_kb) kb = kb0;
    n = v.n_kb - kb;
    return v.ptr + min(rt0 + i, v.n_row - 1) * v.stride_row + kb;
}
// An aligned word that reaches past an end of the scale matrix, which occupies the bytes lo .. hi - 1.
__device__ __noinline__ uint32_t load_end_word(const uint8_t *src, const uint8_t *lo, const uint8_t *hi)
{
    uint32_t w = 0;
#pragma unroll
    for (int e = 0; e < 4; e++)
        if (src + e >= lo && src + e < hi) w |= (uint32_t)load_global(src + e) << (8 * e);
    return w;
}
// Loads a unit's words of G groups of four row tiles: as they are, where all start on words and exist; otherwise, of a full unit, up
// to two aligned words each, which place_chunk_scales shifts into place when they are needed.  One lane a chunk, that is some
// four hundred instructions whatever the unit's length, so units that are not full are gathered by all lanes instead (12 words a
// chunk, 128 a round; SCALES_GATHER, nothing is loaded yet).  us, 161 x 2731, forward / input gradient, one lane a chunk and
// gathered: contraction of 1281 (a unit of 12 chunks) 11.7 / 11.2 and 9.4 / 9.5, of 2305 (20) 12.9 / 12.6 and 11.2 / 11.3, of 3585 (30)
// 14.7 / 14.4 and 13.7 / 13.8, of 4095 (32, full) 12.4 / 13.0 and 13.0 / 13.6.
template <int G>
__device__ __forceinline__ int fetch_chunk_scales(const ScaleView &v, int rt0, int kb0, int n_real, int n_chunks, uint32_t (&w)[4 * G], uint32_t (&next)[4 * G], int lane)
{
    const bool tr = v.stride_kb != 1;
    // The first unit's loads are on the way to a product's first MMA, in code that runs once, so they take few instructions: offsets of 32
    // bits and one branch for the view instead of a choice at each load.  A transposed view starts on a
    // tile's rows and a row-major view's blocks on a unit's, so both start on words where the matrix does.  us, with 64-bit offsets and
    // with these, forward / input gradient: 128 x 256 x 256 5.55 / 5.56 -> 5.44 / 5.40, 2048 x 2048 x 2048 8.13 / 8.33 -> 7.99 / 8.15, 16
    // groups of 9088 rows 768 x 1440 14.0 / 13.95 -> 13.9 / 13.4, 32 of 18560 768 x 1700 20.2 / 24.75 -> 20.2 / 23.6.
    if (v.words && rt0 + 4 * G <= v.n_row && kb0 + 4 * n_real <= v.n_kb) {
        if (lane < n_chunks) {   // a whole number of stages: the chunk that fills up the last one takes the first chunk's scales
            const uint32_t pitch = (uint32_t)(tr ? v.stride_kb : v.stride_row), kb = (uint32_t)(lane < n_real ? kb0 + 4 * lane : kb0);
            const uint8_t *src = v.ptr + (tr ? kb * pitch + rt0 : rt0 * pitch + kb);
            if (tr) {
#pragma unroll
                for (int i = 0; i < 4 * G; i++) ldg_b32(src + (uint32_t)((i & 3) * pitch + (i & ~3)), w[i]);
            } else {
#pragma unroll
                for (int i = 0; i < 4 * G; i++) ldg_b32(src + (uint32_t)(i * pitch), w[i]);
            }
        }
        return SCALES_WHOLE;
    }
    const int64_t pitch = tr ? v.stride_kb : v.stride_row;
    if (n_chunks < kCacheChunks) return SCALES_GATHER;
    const uint8_t *end = v.ptr + (tr ? (v.n_kb - 1) * pitch + v.n_row : (v.n_row - 1) * pitch + v.n_kb);
    if (lane < n_chunks) {
#pragma unroll
        for (int i = 0; i < 4 * G; i++) {
            int n;
            const uint8_t *a = chunk_word(v, rt0, kb0 + 4 * lane, kb0, i, n);
            const int mis = (int)(reinterpret_cast<uintptr_t>(a) & 3);
            a -= mis;
            next[i] = 0u;
            if (a >= v.ptr && a + 4 <= end) ldg_b32(a, w[i]);
            else w[i] = load_end_word(a, v.ptr, end);
            if (mis + n > 4 && mis != 0) {
                if (a + 8 <= end) ldg_b32(a + 4, next[i]);
                else next[i] = load_end_word(a + 4, v.ptr, end);
            }
        }
    }
    return SCALES_SHIFTED;
}
template <int G>
__device__ __forceinline__ void place_chunk_scales(const ScaleView &v, int rt0, int kb0, uint32_t (&w)[4 * G], const uint32_t (&next)[4 * G], int lane)
{
#pragma unroll
    for (int i = 0; i < 4 * G; i++) {
        int n;
        const uint8_t *a = chunk_word(v, rt0, kb0 + 4 * lane, kb0, i, n);
        const uint32_t keep = n < 4 ? (1u << (8 * n)) - 1u : 0xFFFFFFFFu;
        w[i] = (__funnelshift_r(w[i], next[i], 8 * (uint32_t)(reinterpret_cast<uintptr_t>(a) & 3)) & keep) | (kScalePad * 0x01010101u & ~keep);
    }
}
// The 16-byte image row [row tile][block] of a group's four words.
__device__ __forceinline__ uint4 chunk_image_row(const ScaleView &v, const uint32_t *w)
{
    return v.stride_kb != 1 ? transpose4x4_bytes(w[0], w[1], w[2], w[3]) : make_uint4(w[0], w[1], w[2], w[3]);
}

// Units at the ends of a scale matrix, or of scales that start on any byte, but for full ones.  The words of the operands that need it,
// item q a (chunk, row tile) of A's four row tiles or, after them, of B's eight, spread over the lanes and gathered in shared
// memory as rows of 16 bytes.  Slots beyond the tensor hold the pad byte.
template <bool GROUPED>
__device__ __forceinline__ void gather_scale_rows(const GemmParams &p, const Tile &t, int k0, bool need_a, bool need_b, int n_chunks, uint32_t *dst, int lane)
{
    const int n_a = need_a ? 4 * n_chunks : 0, n = n_a + (need_b ? 8 * n_chunks : 0);
    for (int base = 0; base < n; base += 32 * 4) {
        uint32_t b[4][4];
#pragma unroll
        for (int j = 0; j < 4; j++) {   // loads of four items in flight before anything is used
            // One item a lane is all of a short unit, and grouped products of one stage a tile pay for every instruction: 8704 x 256 x 2080 in
            // 8 groups, input gradient 16.5 -> 15.4 us.  (Dense ones, 0.3 % slower with it, do without.)
            if (GROUPED && j == 1 && base + 32 >= n) break;
            const int q = base + 32 * j + lane;
            const bool is_a = q < n_a;
            const int i = is_a ? q : q - n_a, chunk = is_a ? i >> 2 : i >> 3, rt = is_a ? i & 3 : i & 7;
            const ScaleView &v = is_a ? p.sfa : p.sfb;
            const int row = ((is_a ? t.a_row0 : t.b_row0) >> 5) + rt, kb = (((is_a ? t.a_k0 : t.b_k0) + k0) >> 5) + 4 * chunk;
            const uint8_t *src = v.ptr + (int64_t)row * v.stride_row + (int64_t)kb * v.stride_kb;
            const int n_bytes = q < n && row < v.n_row ? v.n_kb - kb : 0;
#pragma unroll
            for (int k = 0; k < 4; k++) {
                b[j][k] = kScalePad;
                asm volatile("{\n .reg .pred p;\n setp.gt.s32 p, %2, %3;\n @p ld.global.u8 %0, [%1];\n}" : "+r"(b[j][k]) : "l"(src), "r"(n_bytes), "r"(k));
                src += v.stride_kb;
            }
        }
#pragma unroll
        for (int j = 0; j < 4; j++) {
            if (GROUPED && j == 1 && base + 32 >= n) break;
            const int q = base + 32 * j + lane;
            if (q < n) dst[q < n_a ? q : 4 * kCacheChunks + q - n_a] = b[j][0] | b[j][1] << 8 | b[j][2] << 16 | b[j][3] << 24;
        }
    }
    __syncwarp();
}

// ---------------------------------------------------------------------------------------- epilogue store

// The transposed payload of blocks jp and jp + 1 of a warp's four (32 x 32 codes each), out of the row-major codes in its staging rows (32 rows of
// 64 bytes in the 64-byte swizzle): a lane transposes the 8 x 8 codes of eight rows and one word, in registers, and writes eight columns'
// words to their rows of 16 bytes behind them.  The order of a lane's rows and columns differs from its neighbours' by what the byte permutations
// select, so that two lanes meet in a bank instead of four (loads) or eight (stores).  An exchange through 16 shuffles a block took three times the
// instructions; us, nearest / stochastic: 2048 x 2048 x 2048 11.8 / 12.8 -> 11.5 / 12.6, 8192 x 2048 x 2048 24.9 / 29.5 -> 23.9 / 28.2, 8192 x 5632 x 2048
// 54.1 / 65.8 -> 51.3 / 61.9, 16384 x 4096 x 4096, where the rounding is hidden, 104.4 / 115.0 -> 103.4 / 115.8.
__device__ __forceinline__ void transpose_staged_codes(uint32_t stg, int jp, int lane)
{
    const uint32_t b = (uint32_t)lane >> 4, g = ((uint32_t)lane >> 2) & 3u, m = (uint32_t)lane & 3u;   // block, rows 8 g .., columns 8 m ..
    const uint32_t src = stg + 512 * g + 128 * g + 16 * ((jp + b) ^ g) + 4 * m;
    uint32_t a[8];   // a[i] is row 8 g + (i ^ 2 g); row r has its 16-byte pieces XORed by r / 2 % 4
#pragma unroll
    for (int i = 0; i < 8; i++) asm volatile("ld.shared.b32 %0, [%1];" : "=r"(a[i]) : "r"(src ^ (uint32_t)(64 * i + 16 * (i >> 1))) : "memory");
    // Which columns come out first (m), and which of two rows comes first in a word (g).
    const uint32_t first4 = g & 2 ? 0x1054u : 0x5410u, second4 = first4 ^ 0x2222u, lo4 = m & 2 ? second4 : first4, hi4 = lo4 ^ 0x2222u;
    const uint32_t first2 = g & 1 ? 0x2604u : 0x6240u, second2 = first2 ^ 0x1111u, lo2 = m & 1 ? second2 : first2, hi2 = lo2 ^ 0x1111u;
#pragma unroll
    for (int r = 0; r < 4; r++) {   // 16-bit halves between rows r and r + 4
        const uint32_t lo = __byte_perm(a[r], a[r + 4], lo4), hi = __byte_perm(a[r], a[r + 4], hi4);
        a[r] = lo; a[r + 4] = hi;
    }
#pragma unroll
    for (int q = 0; q < 4; q++) {   // bytes between rows r and r + 2
        const int r = (q & 1) + 4 * (q >> 1);
        const uint32_t lo = __byte_perm(a[r], a[r + 2], lo2), hi = __byte_perm(a[r], a[r + 2], hi2);
        a[r] = lo; a[r + 2] = hi;
    }
#pragma unroll
    for (int r = 0; r < 8; r += 2) {   // nibbles between rows r and r + 1
        const uint32_t lo = (a[r] & 0x0F0F0F0Fu) | ((a[r + 1] & 0x0F0F0F0Fu) << 4), hi = ((a[r] >> 4) & 0x0F0F0F0Fu) | (a[r + 1] & 0xF0F0F0F0u);
        a[r] = lo; a[r + 1] = hi;
    }
    const uint32_t dst = stg + 2048 + 512 * (jp + b) + 128 * m + 4 * g + 32 * m;   // a[k] is column 8 m + (k ^ 2 m)
#pragma unroll
    for (int k = 0; k < 8; k++) asm volatile("st.shared.b32 [%0], %1;" ::"r"(dst ^ (uint32_t)(k << 4)), "r"(a[k]) : "memory");
}

// One round of the epilogue: 32 words per lane (this lane's row, 128 bytes) into the warp's swizzled staging rows, then one
// TMA store (kind 0: BF16 bytes, 1: FP32 bytes, 2: FP32 add-reduction) of the 32 x 128 B box; fresh: staging rows that no store reads.
// TAIL: a box of nothing but a row's last elements (store_row_tail) is not stored.
// CUT: n_rows of the box may be fewer than 32, with other rows of the output behind them (a grouped weight gradient is a stack of
// matrices of any number of rows).  Such a box leaves by the lanes' own stores, in kernels that nothing else runs: compiled into those
// of all grouped products they took 0.7 % on average, input gradients of ragged widths 1-3 %.  (So did a map with the group
// as its outermost dimension, which clips the box: input gradients 38.0 -> 39.8, 24.6 -> 25.5 us.)
template <bool CUT, bool TAIL>
__device__ __forceinline__ void stage_and_store(const GemmParams &p, const CUtensorMap *map, const uint32_t *w, uint32_t stg_row, uint32_t swz,
                                                uint32_t stg, int col, int32_t y, int kind, int lane, bool fresh, int n_rows)
{
    if (!fresh) {
        if (lane == 0) bulk_wait_read_all();   // the previous round's store has read the staging rows
        __syncwarp();
    }
#pragma unroll
    for (int c = 0; c < 8; c++)
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(stg_row + ((c ^ swz) << 4)), "r"(w[4 * c]), "r"(w[4 * c + 1]),
                     "r"(w[4 * c + 2]), "r"(w[4 * c + 3]) : "memory");
    if (CUT && n_rows < 32) {
        __syncwarp();
        const int c = col + (kind == 0 ? 2 : 1) * lane, n = p.N - c;   // this lane's word of a row, and what there is of its columns
#pragma unroll 1
        for (int r = 0; r < n_rows; r++) {
            uint32_t x;
            asm volatile("ld.shared.b32 %0, [%1];" : "=r"(x) : "r"(stg + r * 128 + ((((uint32_t)lane >> 2) ^ (r & 7)) << 4) + 4 * (lane & 3)) : "memory");
            const int64_t at = ((int64_t)y + r) * p.ldc + c;
            if (kind == 0) {
                if (n > 0) static_cast<uint16_t *>(p.C)[at] = (uint16_t)x;
                if (n > 1) static_cast<uint16_t *>(p.C)[at + 1] = (uint16_t)(x >> 16);
            } else if (n > 0) {
                float *dst = static_cast<float *>(p.C) + at;
                if (kind == 2) atomicAdd(dst, __uint_as_float(x));
                else *dst = __uint_as_float(x);
            }
        }
        __syncwarp();
        return;
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic-proxy writes -> TMA store
    __syncwarp();
    if (lane == 0 && !(TAIL && col == p.tail_col)) {
        if (kind == 2) tma_reduce_add_2d(map, col, y, stg);                 // x in FP32 elements
        else tma_store_2d(map, col * (kind == 1 ? 4 : 2), y, stg);          // x in bytes
        bulk_commit();
    }
}

// A row's last elements, n (1 .. 7) from column p.tail_col on, out of the 16 bytes of staging that hold them.  A TMA store writes whole pieces of 16 bytes,
// whatever the map's element type: with a map that ends inside one, it writes zeros over what follows the row's last column.  Kernels of
// their own (EPI_TAIL), since the few instructions behind a tile cost others up to 3 %, and only for outputs whose padding is not theirs to
// fill; us, with those zeros and without: 1999 x 1003 x 2731 forward 10.5 / 10.8, 16384 x 1003 x 2721 24.6 / 25.2, 9001 x 4095 x 2049 43.8 / 44.7, 849 x 67 x 169
// 5.7 / 6.0; where the output is not in L2, sectors that are written in part cost more (7296 x 490 x 1664 8.4 / 9.6).
__device__ __forceinline__ void store_row_tail(const GemmParams &p, int64_t row, uint32_t src)
{
    uint32_t x[4];
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3]) : "r"(src) : "memory");
    const int n = p.N - p.tail_col;
    const int64_t at = row * p.ldc + p.tail_col;   // on 16 bytes
    if (p.out_f32) {
        float *dst = static_cast<float *>(p.C) + at;
        if (p.accumulate) {
#pragma unroll
            for (int i = 0; i < 3; i++)
                if (i < n) atomicAdd(dst + i, __uint_as_float(x[i]));
        } else {
            if (n & 2) *reinterpret_cast<uint2 *>(dst) = make_uint2(x[0], x[1]);
            if (n & 1) dst[n - 1] = __uint_as_float(n & 2 ? x[2] : x[0]);
        }
    } else {
        uint16_t *dst = static_cast<uint16_t *>(p.C) + at;
        if (n & 4) *reinterpret_cast<uint2 *>(dst) = make_uint2(x[0], x[1]);
        if (n & 2) *reinterpret_cast<uint32_t *>(dst + (n & 4)) = n & 4 ? x[2] : x[0];
        if (n & 1) dst[n - 1] = (uint16_t)(n & 4 ? (n & 2 ? x[3] : x[2]) : (n & 2 ? x[1] : x[0]));
    }
}

// One whole 32-byte sector per lane (a 16-byte store leaves half a sector to a second transaction).
__device__ __forceinline__ void st_global_v8(void *dst, const uint32_t *w)
{
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "r"(w[0]), "r"(w[1]), "r"(w[2]),
                 "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]) : "memory");
}

__device__ __forceinline__ void store_row_chunk(const GemmParams &p, int64_t row, int col0, int n_cols_valid,
                                                const uint32_t v[32])
{
    // 32 consecutive accumulator columns of one output row, starting at column col0
    if (n_cols_valid <= 0) return;
    if (p.out_f32) {
        float *dst = static_cast<float *>(p.C) + row * p.ldc + col0;
        if (n_cols_valid >= 32 && p.wide_stores && !p.accumulate) {
#pragma unroll
            for (int q = 0; q < 4; q++) st_global_v8(dst + 8 * q, v + 8 * q);
        } else if (n_cols_valid >= 32) {
#pragma unroll
            for (int q = 0; q < 8; q++) {
                float4 o = make_float4(__uint_as_float(v[4 * q]), __uint_as_float(v[4 * q + 1]),
                                       __uint_as_float(v[4 * q + 2]), __uint_as_float(v[4 * q + 3]));
                if (p.accumulate) {
                    const float4 old = *reinterpret_cast<const float4 *>(dst + 4 * q);
                    o.x += old.x; o.y += old.y; o.z += old.z; o.w += old.w;
                }
                *reinterpret_cast<float4 *>(dst + 4 * q) = o;
            }
        } else {
#pragma unroll
            for (int q = 0; q < 32; q++)
                if (q < n_cols_valid) dst[q] = __uint_as_float(v[q]) + (p.accumulate ? dst[q] : 0.0f);
        }
    } else {
        __nv_bfloat16 *dst = static_cast<__nv_bfloat16 *>(p.C) + row * p.ldc + col0;
        if (n_cols_valid >= 32 && p.wide_stores) {
            uint32_t w[16];
#pragma unroll
            for (int e = 0; e < 16; e++) {
                const __nv_bfloat162 b = __floats2bfloat162_rn(__uint_as_float(v[2 * e]), __uint_as_float(v[2 * e + 1]));
                w[e] = *reinterpret_cast<const uint32_t *>(&b);
            }
            st_global_v8(dst, w);
            st_global_v8(dst + 16, w + 8);
        } else if (n_cols_valid >= 32) {
#pragma unroll
            for (int q = 0; q < 4; q++) {
                uint32_t w[4];
#pragma unroll
                for (int e = 0; e < 4; e++) {
                    const __nv_bfloat162 b = __floats2bfloat162_rn(__uint_as_float(v[8 * q + 2 * e]),
                                                                   __uint_as_float(v[8 * q + 2 * e + 1]));
                    w[e] = *reinterpret_cast<const uint32_t *>(&b);
                }
                *reinterpret_cast<uint4 *>(dst + 8 * q) = make_uint4(w[0], w[1], w[2], w[3]);
            }
        } else {
#pragma unroll
            for (int q = 0; q < 32; q++)
                if (q < n_cols_valid) dst[q] = __float2bfloat16_rn(__uint_as_float(v[q]));
        }
    }
}

// Position in a ring of image buffers: buffer index and the parity of the barrier phase that goes with it.
struct BufRing {
    uint32_t buf = 0, phase = 0;
    __device__ __forceinline__ void next(uint32_t n) { if (++buf == n) { buf = 0; phase ^= 1u; } }
};

// The stream of scale units (kUnitStages stages of one tile) a CTA works through.
template <int GROUPS>
struct UnitIter {
    int tile, step, rank, k0, m_tiles, n_total;
    Tile t;
    const int32_t *goffs = nullptr;
    const uint16_t *gorder = nullptr;
    __device__ __forceinline__ void seek(const GemmParams &p)
    {
        while (tile < n_total) {
            decode_tile<GROUPS>(p, tile, rank, t, m_tiles, goffs, gorder);
            if (k0 < t.k_len) return;
            tile += step;
            k0 = 0;
        }
    }
    __device__ __forceinline__ void init(const GemmParams &p, int first, int step_, int rank_, int m_tiles_, int n_total_)
    {
        m_tiles = m_tiles_; n_total = n_total_;
        tile = first; step = step_; rank = rank_; k0 = 0;
        seek(p);
    }
    __device__ __forceinline__ bool valid(const GemmParams &p) const { return tile < n_total; }
    __device__ __forceinline__ void next(const GemmParams &p, int unit_elems)
    {
        k0 += unit_elems;
        if (k0 >= t.k_len) { tile += step; k0 = 0; seek(p); }   // a tile is decoded once: its three divisions took longer than a unit's images
    }
};

// ---- scale images of the per-row kinds

__device__ __forceinline__ void cp_async16(uint32_t dst, const uint8_t *src, int src_bytes)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const uint8_t *src, int src_bytes)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const uint8_t *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ uint32_t lds32(const uint8_t *p) { return *reinterpret_cast<const uint32_t *>(p); }

// A row's bytes from src on, which may lie on any byte, as WORDS aligned words from the one that holds the first.  The matrix
// occupies the bytes lo .. hi - 1 and src is one of them; INSIDE: so are all bytes of the words.
template <int WORDS, bool INSIDE>
__device__ __forceinline__ void fetch_row(uint32_t dst, const uint8_t *src, const uint8_t *lo, const uint8_t *hi)
{
    const uint8_t *a = src - (reinterpret_cast<uintptr_t>(src) & 3);
    if (INSIDE) {
#pragma unroll
        for (int k = 0; k < WORDS; k++) cp_async4(dst + 4 * k, a + 4 * k);
        return;
    }
    const int n = (int)min((int64_t)(4 * WORDS), (int64_t)(hi - a));   // bytes before the matrix's end
    if (a < lo) asm volatile("st.shared.b32 [%0], %1;" ::"r"(dst), "r"(load_end_word(a, lo, hi)) : "memory");
    else cp_async4(dst, a, min(n, 4));
#pragma unroll
    for (int k = 1; k < WORDS; k++) cp_async4(dst + 4 * k, 4 * k < n ? a + 4 * k : a, max(0, min(n - 4 * k, 4)));
}
// Word k of such a row, whose first byte is byte `mis` of the first word; bytes from n_valid on are not the row's.
__device__ __forceinline__ uint32_t row_word(uint32_t lo, uint32_t hi, uint32_t mis, int k, int n_valid)
{
    const int n = n_valid - 4 * k;
    const uint32_t w = __funnelshift_r(lo, hi, 8 * mis);
    return n >= 4 ? w : n <= 0 ? 0u : w & ((1u << (8 * n)) - 1u);
}

// Per-row scales: BYTES scale bytes of each of the NQ x 32 rows from row0 on, row row0 + lane + 32 q one of lane's.  Rows on 16-byte
// boundaries are copied as they are, others word by word in entries of one word more and shifted when they are read.  (Loads
// by each piece, with a wait for it, were ten times the code and did not run ahead: MXFP8 forward 1999 x 1003 x 2731, 86 blocks a row, 68.4 ->
// 18.2 us, 300 x 777 x 1234 35.3 -> 12.7, 1D activations there 21.5 / 22.9 -> 11.4 / 12.5 and 12.0 / 20.1 -> 8.3 / 10.4.)  Rows beyond the tensor take
// the place of the last (their payload is zero, any finite scale will do), bytes beyond a row's last become zero.
template <int NQ, int BYTES>
struct RowFetch {
    const uint8_t *src[NQ];
    __device__ __forceinline__ static bool wide(const ScaleView &v) { return ((reinterpret_cast<uintptr_t>(v.ptr) | (uintptr_t)v.stride_row) & 15) == 0; }
    __device__ __forceinline__ void set(const ScaleView &v, int row0, int lane)
    {
#pragma unroll
        for (int q = 0; q < NQ; q++) src[q] = v.ptr + (int64_t)min(row0 + lane + 32 * q, v.n_row - 1) * v.stride_row;
    }
    __device__ __forceinline__ void fetch(const ScaleView &v, int kb0, uint32_t raw, int lane) const
    {
        if (wide(v)) {
#pragma unroll
            for (int q = 0; q < NQ; q++)
#pragma unroll
                for (int h = 0; h < BYTES / 16; h++) {
                    const int n = max(0, min(16, v.n_kb - kb0 - 16 * h));
                    cp_async16(raw + (32 * q + lane) * BYTES + 16 * h, src[q] + kb0 + (n > 0 ? 16 * h : 0), n);
                }
            return;
        }
        constexpr int kWords = BYTES / 4 + 1;
        const uint8_t *hi = v.ptr + (int64_t)(v.n_row - 1) * v.stride_row + v.n_kb;
        raw += 4 * kWords * lane;
        if (__all_sync(0xFFFFFFFFu, src[0] + kb0 >= v.ptr + 3 && src[NQ - 1] + kb0 + 4 * kWords <= hi)) {
#pragma unroll
            for (int q = 0; q < NQ; q++) fetch_row<kWords, true>(raw + 128 * kWords * q, src[q] + kb0, v.ptr, hi);
        } else {
#pragma unroll
            for (int q = 0; q < NQ; q++) fetch_row<kWords, false>(raw + 128 * kWords * q, src[q] + kb0, v.ptr, hi);
        }
    }
    // w[q]: the words of row row0 + lane + 32 q, of any tile whose bytes have landed
    __device__ __forceinline__ static void read(const ScaleView &v, int row0, int kb0, const uint8_t *raw, int lane, uint32_t (*w)[BYTES / 4])
    {
        if (wide(v)) {
#pragma unroll
            for (int q = 0; q < NQ; q++)
#pragma unroll
                for (int h = 0; h < BYTES / 16; h++) {
                    const uint4 x = reinterpret_cast<const uint4 *>(raw + (32 * q + lane) * BYTES)[h];
                    w[q][4 * h] = x.x; w[q][4 * h + 1] = x.y; w[q][4 * h + 2] = x.z; w[q][4 * h + 3] = x.w;
                }
            return;
        }
        constexpr int kWords = BYTES / 4 + 1;
#pragma unroll
        for (int q = 0; q < NQ; q++) {
            const uint32_t mis = ((uint32_t)reinterpret_cast<uintptr_t>(v.ptr) + (uint32_t)min(row0 + lane + 32 * q, v.n_row - 1) * (uint32_t)v.stride_row + (uint32_t)kb0) & 3;
            const uint8_t *e = raw + 4 * kWords * (32 * q + lane);
            uint32_t x[kWords];
#pragma unroll
            for (int k = 0; k < kWords; k++) x[k] = lds32(e + 4 * k);
#pragma unroll
            for (int k = 0; k < BYTES / 4; k++) w[q][k] = row_word(x[k], x[k + 1], mis, k, v.n_kb - kb0);
        }
    }
};

// 2D-block scales in a per-row kind: TILES row tiles by 32 blocks, an entry a row tile or, seen transposed, a block.  Like a per-row
// operand's rows they are copied as they are where their entries start on 16 (transposed: TILES) bytes, otherwise word by word in entries of
// one word more.
template <int TILES, bool TR>
__device__ __forceinline__ bool wide_blocks(const ScaleView &v)
{
    return ((reinterpret_cast<uintptr_t>(v.ptr) | (uintptr_t)(TR ? v.stride_kb : v.stride_row)) & (TR ? TILES - 1 : 15)) == 0;
}
template <int TILES, bool TR>
__device__ __forceinline__ void fetch_blocks(const ScaleView &v, int rt0, int kb0, uint32_t raw, int lane)
{
    if (TR) {
        const int n = max(0, min(TILES, v.n_row - rt0));
        const uint8_t *src = v.ptr + (int64_t)min(kb0 + lane, v.n_kb - 1) * v.stride_kb + (n > 0 ? rt0 : 0);
        if (wide_blocks<TILES, TR>(v)) asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(raw + lane * TILES), "l"(src), "n"(TILES), "r"(n) : "memory");
        else fetch_row<TILES / 4 + 1, false>(raw + lane * (TILES + 4), src, v.ptr, v.ptr + (int64_t)(v.n_kb - 1) * v.stride_kb + v.n_row);
    } else if (wide_blocks<TILES, TR>(v)) {
        if (lane < 2 * TILES) {
            const int h = 16 * (lane & 1), n = max(0, min(16, v.n_kb - kb0 - h));
            cp_async16(raw + lane * 16, v.ptr + (int64_t)min(rt0 + (lane >> 1), v.n_row - 1) * v.stride_row + kb0 + (n > 0 ? h : 0), n);
        }
    } else if (lane < TILES) {
        const uint8_t *src = v.ptr + (int64_t)min(rt0 + lane, v.n_row - 1) * v.stride_row + kb0;
        fetch_row<9, false>(raw + lane * 36, src, v.ptr, v.ptr + (int64_t)(v.n_row - 1) * v.stride_row + v.n_kb);
    }
}
// The same, landed, as words of four blocks: store(row tile, chunk of four blocks, word).
template <int TILES, bool TR, typename F>
__device__ __forceinline__ void sort_blocks(const ScaleView &v, int rt0, int kb0, const uint8_t *raw, int lane, F store)
{
    const uint32_t p0 = (uint32_t)reinterpret_cast<uintptr_t>(v.ptr);
    const bool wide = wide_blocks<TILES, TR>(v);
    if (TR) {   // a lane transposes four blocks' bytes of four row tiles
        if (lane < 2 * TILES) {
            const int h = lane % (TILES / 4), c = lane / (TILES / 4);
            uint32_t m[4];
            if (wide) {
#pragma unroll
                for (int i = 0; i < 4; i++) m[i] = lds32(raw + (4 * c + i) * TILES + 4 * h);
            } else {
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    const uint8_t *e = raw + (4 * c + i) * (TILES + 4) + 4 * h;
                    const uint32_t mis = (p0 + (uint32_t)min(kb0 + 4 * c + i, v.n_kb - 1) * (uint32_t)v.stride_kb + (uint32_t)(rt0 < v.n_row ? rt0 : 0)) & 3;
                    m[i] = row_word(lds32(e), lds32(e + 4), mis, h, v.n_row - rt0);
                }
            }
            const uint4 t = transpose4x4_bytes(m[0], m[1], m[2], m[3]);
            store(4 * h, c, t.x); store(4 * h + 1, c, t.y); store(4 * h + 2, c, t.z); store(4 * h + 3, c, t.w);
        }
    } else if (wide) {
        if (lane < 2 * TILES) {
            const int rt = lane >> 1, c = 4 * (lane & 1);
            const uint4 x = *reinterpret_cast<const uint4 *>(raw + lane * 16);
            store(rt, c, x.x); store(rt, c + 1, x.y); store(rt, c + 2, x.z); store(rt, c + 3, x.w);
        }
    } else {
#pragma unroll
        for (int i = 0; i < TILES / 4; i++) {
            const int rt = (lane + 32 * i) % TILES, c = (lane + 32 * i) / TILES;
            const uint32_t mis = (p0 + (uint32_t)min(rt0 + rt, v.n_row - 1) * (uint32_t)v.stride_row + (uint32_t)kb0) & 3;
            const uint8_t *e = raw + rt * 36 + 4 * c;
            store(rt, c, row_word(lds32(e), lds32(e + 4), mis, c, v.n_kb - kb0));
        }
    }
}

// What bounds these kinds is how fast a warp, whose work is all latency, turns a unit's bytes into images.  A 2D-block operand's are
// therefore transposed by one lane each (not all by every lane), and in KIND_MXF4RA / RB it has replicated images, whose 16-byte rows
// are a quarter of the real images' bytes; that also pays for the fifth ring stage of RA.  us, 8192 x 5632 x 2048: 1D activations
// forward / weight gradient 51.0 / 52.3 -> 47.7 / 48.4 (16384 x 4096 x 4096 121 / 130 -> 109 / 123), 16 x 16 blocks 53.5 / 47.6 / 55.1 -> 53.0 / 45.1 /
// 50.8.  With the image rows read back from shared memory only when their buffer was free, 16 x 16 forward 2048 x 2048 x 2048 took 10.7 instead
// of 10.0.
// A builder's unit of a per-row kind, in three steps: fetch() starts the copies of a unit's bytes, read() takes them out of the raw
// buffer into registers, write() makes the images, of which nothing but stores is left when their buffer falls free.  `sorted` is the
// builder's own: 2D-block bytes as 16-byte image rows.
template <int KIND, int CTAS>
struct RowBuilder {
    static constexpr int kRawA = Cfg<KIND, CTAS>::kRawA;
    static constexpr bool kRowsA = KIND == KIND_MXF8 || KIND == KIND_MXF4RA, kRowsB = KIND == KIND_MXF8 || KIND == KIND_MXF4RB;
    static constexpr int kBytes = KIND == KIND_MXF8 ? 16 : 32, kShift = KIND == KIND_MXF4B16 ? 4 : 5;   // a unit's blocks; log2 of a block's length
    RowFetch<kRowsA ? 4 : 1, kBytes> a;
    RowFetch<kRowsB ? 8 : 1, kBytes> b;
    uint32_t w[KIND == KIND_MXF4B16 ? 1 : (kRowsA ? 4 : 0) + (kRowsB ? 8 : 0)][kBytes / 4];   // per-row operands, A's rows first
    uint4 block_rows[KIND == KIND_MXF4B16 ? 24 : KIND == KIND_MXF4RA ? 4 : KIND == KIND_MXF4RB ? 2 : 1];   // 2D-block operands' image rows

    __device__ __forceinline__ void set(const GemmParams &p, const Tile &t, int lane)
    {
        if (kRowsA) a.set(p.sfa, t.a_row0, lane);
        if (kRowsB) b.set(p.sfb, t.b_row0, lane);
    }
    __device__ __forceinline__ void fetch(const GemmParams &p, const Tile &t, int k0, uint8_t *raw, int lane) const
    {
        const int kb0 = k0 >> kShift;
        const uint32_t ra = smem_u32(raw), rb = ra + kRawA;
        if (kRowsA) a.fetch(p.sfa, kb0, ra, lane);
        if (kRowsB) b.fetch(p.sfb, kb0, rb, lane);
        if (KIND == KIND_MXF4RA) fetch_blocks<8, false>(p.sfb, t.b_row0 >> 5, kb0, rb, lane);
        if (KIND == KIND_MXF4RB) fetch_blocks<4, true>(p.sfa, t.a_row0 >> 5, kb0, ra, lane);
        if (KIND == KIND_MXF4B16) {
            if (p.sfa.stride_kb != 1) fetch_blocks<8, true>(p.sfa, t.a_row0 >> 4, kb0, ra, lane);
            else fetch_blocks<8, false>(p.sfa, t.a_row0 >> 4, kb0, ra, lane);
            if (p.sfb.stride_kb != 1) fetch_blocks<16, true>(p.sfb, t.b_row0 >> 4, kb0, rb, lane);
            else fetch_blocks<16, false>(p.sfb, t.b_row0 >> 4, kb0, rb, lane);
        }
    }
    __device__ __forceinline__ void read(const GemmParams &p, const Tile &t, int k0, const uint8_t *raw, uint8_t *sorted, int lane)
    {
        const int kb0 = k0 >> kShift;
        uint32_t *s = reinterpret_cast<uint32_t *>(sorted);
        if (kRowsA) a.read(p.sfa, t.a_row0, kb0, raw, lane, w);
        if (kRowsB) b.read(p.sfb, t.b_row0, kb0, raw + kRawA, lane, w + (kRowsA ? 4 : 0));
        // [chunk][row tile], that is a chunk's one or two image rows
        if (KIND == KIND_MXF4RA) sort_blocks<8, false>(p.sfb, t.b_row0 >> 5, kb0, raw + kRawA, lane, [&](int rt, int c, uint32_t x) { s[8 * c + rt] = x; });
        if (KIND == KIND_MXF4RB) sort_blocks<4, true>(p.sfa, t.a_row0 >> 5, kb0, raw, lane, [&](int rt, int c, uint32_t x) { s[4 * c + rt] = x; });
        if (KIND == KIND_MXF4B16) {
            // operand rows l + 32 q of image row l lie in row tile 2 q + l / 16: [MMA][half of the lanes][q]
            auto sa = [&](int rt, int c, uint32_t x) { s[8 * c + 4 * (rt & 1) + (rt >> 1)] = x; };
            auto sb = [&](int rt, int c, uint32_t x) { s[64 + 16 * c + 8 * (rt & 1) + (rt >> 1)] = x; };
            if (p.sfa.stride_kb != 1) sort_blocks<8, true>(p.sfa, t.a_row0 >> 4, kb0, raw, lane, sa);
            else sort_blocks<8, false>(p.sfa, t.a_row0 >> 4, kb0, raw, lane, sa);
            if (p.sfb.stride_kb != 1) sort_blocks<16, true>(p.sfb, t.b_row0 >> 4, kb0, raw + kRawA, lane, sb);
            else sort_blocks<16, false>(p.sfb, t.b_row0 >> 4, kb0, raw + kRawA, lane, sb);
        }
        if (KIND == KIND_MXF8) return;
        __syncwarp();
        const uint4 *rows = reinterpret_cast<const uint4 *>(sorted);
        if (KIND == KIND_MXF4B16) {
            const int hi = lane >> 4;
#pragma unroll
            for (int j = 0; j < 8; j++) {   // MMA j % 4 of stage j / 4
                block_rows[3 * j] = rows[2 * j + hi];                       // A
                block_rows[3 * j + 1] = rows[16 + 4 * j + 2 * hi];          // B rows 0..127
                block_rows[3 * j + 2] = rows[16 + 4 * j + 2 * hi + 1];      // B rows 128..255
            }
        } else {
#pragma unroll
            for (int i = 0; i < (KIND == KIND_MXF4RA ? 4 : 2); i++) block_rows[i] = rows[4 * i + (lane >> 3)];
        }
    }
    __device__ __forceinline__ void write(int n_stages, uint8_t *images, int lane) const
    {
        constexpr int kStage = Cfg<KIND, CTAS>::kImageStage;
        if (KIND == KIND_MXF4B16) {
#pragma unroll
            for (int j = 0; j < 8; j++) {
                if (j >= 4 * n_stages) break;
                uint4 *img = reinterpret_cast<uint4 *>(images + (j >> 2) * kStage) + lane;
                img[32 * (j & 3)] = block_rows[3 * j];
                img[128 + 64 * (j & 3)] = block_rows[3 * j + 1];
                img[160 + 64 * (j & 3)] = block_rows[3 * j + 2];
            }
            return;
        }
        if (KIND == KIND_MXF4RA || KIND == KIND_MXF4RB) {   // replicated images: lane writes one of the eight copies of every fourth row
            constexpr int kRows = KIND == KIND_MXF4RA ? 2 : 1, kFirst = KIND == KIND_MXF4RA ? 1024 : 0;   // image rows per chunk
#pragma unroll
            for (int i = 0; i < 2 * kRows; i++) {
                const int k = 4 * i + (lane >> 3), c = k / kRows;
                *reinterpret_cast<uint4 *>(images + (c >> 1) * kStage + kFirst + (c & 1) * 128 * kRows + (k % kRows) * 128 + (lane & 7) * 16) = block_rows[i];
            }
        }
#pragma unroll
        for (int st = 0; st < 4; st++) {   // real images
            if (st >= n_stages) break;
            uint4 *img = reinterpret_cast<uint4 *>(images + st * kStage + (KIND == KIND_MXF4RB ? 256 : 0)) + lane;
            if (KIND == KIND_MXF8) {
                img[0] = make_uint4(w[0][st], w[1][st], w[2][st], w[3][st]);            // A
                img[32] = make_uint4(w[4][st], w[5][st], w[6][st], w[7][st]);           // B rows 0..127
                img[64] = make_uint4(w[8][st], w[9][st], w[10][st], w[11][st]);         // B rows 128..255
            } else {
#pragma unroll
                for (int c = 0; c < 2; c++)
#pragma unroll
                    for (int r = 0; r < (KIND == KIND_MXF4RB ? 2 : 1); r++) {
                        const int j = 2 * st + c, q = 4 * r;
                        img[(KIND == KIND_MXF4RB ? 64 : 32) * c + 32 * r] = make_uint4(w[q][j], w[q + 1][j], w[q + 2][j], w[q + 3][j]);
                    }
            }
        }
    }
};

// ---------------------------------------------------------------------------------------- kernel

// WATCH: warp 2 looks at the ring's barriers for the MMA warp and the two meet at a named barrier per stage; otherwise the
// MMA warp looks for itself, at the next stage's before it issues a stage.  launch_gemm() says which is used where.
// GROUPS: see decode_tile; grouped products exist for 2D-block scales only, and their kernels have no watcher.
template <int KIND, int CTAS, int EPI, bool WATCH, int GROUPS>
__global__ void __launch_bounds__(kThreads, 1)
gemm_block_scaled_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                         const __grid_constant__ CUtensorMap tmC, const __grid_constant__ CUtensorMap tmD,
                         const __grid_constant__ GemmParams p)
{
    constexpr int kStageElems = kind_fp4(KIND) ? 256 : 128;   // contraction elements per stage (128 B per row)
    constexpr int kMmaK = kind_fp4(KIND) ? 64 : 32;           // contraction elements per MMA (32 B per row)
    constexpr int kElemsPerByte = kind_fp4(KIND) ? 2 : 1;
    constexpr int kStages = Cfg<KIND, CTAS>::kStages;
    constexpr int kBStageBytes = Cfg<KIND, CTAS>::kBStageBytes;
    constexpr int kUnitStages = Cfg<KIND, CTAS>::kUnitStages, kImageStage = Cfg<KIND, CTAS>::kImageStage;
    constexpr int kBufBytes = Cfg<KIND, CTAS>::kBufBytes;
    constexpr bool kGrouped = GROUPS != GROUPS_NONE;
    static_assert(!kGrouped || (KIND == KIND_MXF4 && !WATCH), "grouped products");

    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t *smem_a = smem;
    uint8_t *smem_b = smem + kStages * kAStageBytes;
    uint8_t *smem_compact = smem + Cfg<KIND, CTAS>::kSmemOperands;   // 2D blocks: gathered scale rows of the unit being built ...
    uint8_t *smem_images = smem_compact + (Cfg<KIND, CTAS>::kRowImages ? 0 : kCompactBytes);   // ... and the buffers of ready scale images (any kind)
    uint8_t *smem_raw_scales = smem_images + Cfg<KIND, CTAS>::kImageBufs * kBufBytes;   // per-row scales: bytes in flight
    uint8_t *smem_staging = smem_compact + Cfg<KIND, CTAS>::kSmemScales;   // 1024-byte aligned (pair kernel only)
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem_staging + Cfg<KIND, CTAS>::kSmemStaging);
    // bars[0..5] full, bars[6..11] empty, bars[12] accumulator full, bars[13] accumulator empty,
    // bars[18] tensor pipe drained (abort path), bars[24..27] scale images full, bars[28..31] scale images empty,
    // bars[32..35] (leader of a pair) the second CTA's scale images full - one of each per image buffer
    uint32_t *tmem_base_slot = reinterpret_cast<uint32_t *>(bars + 21);
    volatile uint32_t *abort_flag = reinterpret_cast<volatile uint32_t *>(bars + 21) + 1;
    volatile uint32_t *acc_seen = reinterpret_cast<volatile uint32_t *>(bars + 22);   // the epilogue's verdict on its wait for the accumulator
    int32_t *goffs_smem = reinterpret_cast<int32_t *>(reinterpret_cast<uint8_t *>(bars) + kSmemTail);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t bar_full = smem_u32(bars), bar_empty = smem_u32(bars + kMaxStages);
    const uint32_t bar_acc_full = smem_u32(bars + 12), bar_acc_empty = smem_u32(bars + 13);
    const uint32_t bar_cache_full = smem_u32(bars + 24), bar_cache_empty = smem_u32(bars + 28);
    const uint32_t bar_drain = smem_u32(bars + 18), bar_peer_cache_full = smem_u32(bars + 32);
    constexpr int kImageBufs = Cfg<KIND, CTAS>::kImageBufs;

    // In a pair, rank 0 leads: it owns the "full" and "accumulator empty" barriers and issues every tcgen05.mma.
    const int rank = CTAS == 2 ? (int)cluster_ctarank() : 0;
    const bool leader = rank == 0;
    const int first_tile = blockIdx.x / CTAS, tile_step = gridDim.x / CTAS;

    // Roles start as soon as each can.  With initialization, tensor memory, a barrier and only then decoding and loads one after the
    // other, the first operand load left 2900 cycles after a pair's first instruction and the first MMA 6100; now 1500 and 5300.  us:
    // 2048 x 2048 x 2048 9.6 / 9.9 / 11.2 -> 9.5 / 9.6 / 10.9, quantized output 12.6 -> 12.3, 1D activations 11.0 -> 10.4, 300 x 777 x 1234 9.1 / 8.9 /
    // 9.8 -> 8.8 / 8.7 / 9.4.
    constexpr int kBuilders = Cfg<KIND, CTAS>::kBuilders;
    if (warp == 4) {   // an epilogue warp has time
        // One barrier a lane.  A stage's "full" barrier takes the producer's expect_tx arrival (in a pair the leader's, which announces
        // both CTAs' bytes: the second CTA's loads complete on the leader's barrier), the accumulator's "empty" barrier one
        // arrival per epilogue warp (of both CTAs of a pair), every other one commit or one builder.
        if (lane < 21 || lane >= 24) mbar_init(smem_u32(bars + lane), lane == 13 ? 8 * CTAS : 1);
        if (lane < 4) mbar_init(smem_u32(bars + 32 + lane), 1);
        if (lane == 0) *abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        __threadfence_block();   // the flag, ahead of the relaxed arrival
        __syncwarp();
        if (CTAS == 2) cluster_arrive_relaxed();
        else asm volatile("bar.arrive 12, %0;" ::"n"(32 + 32 * kBuilders) : "memory");   // for the builders
        if (lane == 0) {
            if (Cfg<KIND, CTAS>::kTmaStores) asm volatile("prefetch.tensormap [%0];" ::"l"(&tmC) : "memory");
            if (EPI == EPI_QUANT) asm volatile("prefetch.tensormap [%0];" ::"l"(&tmD) : "memory");
        }
        __syncwarp();
    } else if (CTAS == 2 && warp != 1) {
        cluster_arrive_relaxed();
    }
    if (warp == 0) {
        if (lane == 0) {
            asm volatile("prefetch.tensormap [%0];" ::"l"(&tmA) : "memory");
            asm volatile("prefetch.tensormap [%0];" ::"l"(&tmB) : "memory");
        }
        __syncwarp();
    }
    if (warp == 1) {
        if (CTAS == 1) {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_base_slot)),
                         "r"(kTmemCols) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        } else {
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_base_slot)),
                         "r"(kTmemCols) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
            tcgen05_fence_before();
            cluster_arrive();
        }
    }
    // Everything above touches this CTA only; from here on the kernel reads what its predecessor in the stream wrote.  Its own
    // successor is let in by its end (launch_dependent says why).
    wait_for_predecessor();
    // Poll limit of every bounded wait (workspace word 2; 0 = the default) and the development hook of word 3 (n > 0:
    // the producer of CTA 0 leaves out its n-th stage load, so that a test can watch a wait run out and the kernel
    // leave through its timeout path without anything faulting or spinning for long).
    const uint32_t wait_limit_word = load_global(p.status + 2), withhold_load = blockIdx.x == 0 ? load_global(p.status + 3) : 0u;
    const uint64_t wait_limit = wait_limit_word != 0u ? wait_limit_word : kWaitLimit;
    // grouped products: a 32-bit copy of the group boundaries for the per-tile lookups of every role
    const int n_row_tiles = (p.M + BM - 1) / BM;
    const bool goffs_ok = kGrouped && Cfg<KIND, CTAS>::kSmemGroups > 0 &&
                          ((GROUPS == GROUPS_PAIRED && p.mode == MODE_PAIRED_ROWS) || (p.mode == MODE_GROUPED_K && p.n_groups <= kMaxGroupsShared) ||
                           (p.mode == MODE_GROUPED_ROWS && n_row_tiles <= kMaxRowTilesShared && p.n_groups <= 65535));
    if (goffs_ok && p.mode == MODE_GROUPED_K)
        for (int g = threadIdx.x; g <= p.n_groups; g += kThreads) goffs_smem[g] = (int32_t)load_global(p.row_offsets + g);
    if (goffs_ok && p.mode == MODE_GROUPED_ROWS) {
        // A search in global memory is up to four misses one after the other: boundaries of more than one 128-byte line are copied
        // first, to where the images will be.  us, forward / input gradient: 64 groups of 20608 rows 768 x 2048 30.4 / 36.0 -> 30.0 / 35.3,
        // 128 of 41856 50.4 / 64.2 -> 49.8 / 63.3; within a line 8 of 2560 512 x 256 7.1 / 7.3 -> 7.2 / 7.4.
        int32_t *bounds = reinterpret_cast<int32_t *>(smem_images);
        const bool copy = p.n_groups > 16 && (p.n_groups + 1) * (int)sizeof(int32_t) <= Cfg<KIND, CTAS>::kImageBufs * kBufBytes;
        if (copy) {
            for (int g = threadIdx.x; g <= p.n_groups; g += kThreads) bounds[g] = (int32_t)load_global(p.row_offsets + g);
            __syncthreads();
        }
        for (int i = threadIdx.x; i < n_row_tiles; i += kThreads)
            reinterpret_cast<uint16_t *>(goffs_smem)[i] = (uint16_t)find_group(p.row_offsets, copy ? bounds : nullptr, p.n_groups, (int64_t)i * BM);
    }
    int m_tiles = p.m_tiles, n_tile_total = p.n_tile_total;
    if (GROUPS == GROUPS_PAIRED && p.mode == MODE_PAIRED_ROWS) {
        // Groups' first row tiles, their numbers of pairs added up, then every pair looks its group up.  Offsets that are not as the caller
        // states go to some tile or other, but to no other memory.
        int32_t *start = reinterpret_cast<int32_t *>(smem_images), *first = start + p.n_groups + 1;
        for (int g = threadIdx.x; g <= p.n_groups; g += kThreads)
            start[g] = g == 0 ? 0 : g == p.n_groups ? n_row_tiles : (int32_t)max((int64_t)0, min((int64_t)n_row_tiles, (load_global(p.row_offsets + g) + BM - 1) / BM));
        __syncthreads();
        if (warp == 4) {
            const int per_lane = (p.n_groups + 31) / 32, g0 = min(lane * per_lane, p.n_groups), g1 = min(g0 + per_lane, p.n_groups);
            int sum = 0;
            for (int g = g0; g < g1; g++) sum += (max(0, start[g + 1] - start[g]) + 1) >> 1;
            int before = sum;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int other = __shfl_up_sync(0xFFFFFFFFu, before, d);
                if (lane >= d) before += other;
            }
            before -= sum;
            for (int g = g0; g < g1; g++) {
                first[g] = before;
                before += (max(0, start[g + 1] - start[g]) + 1) >> 1;
            }
            if (lane == 31) first[p.n_groups] = min(before, kMaxGroupsShared + 1);
        }
        __syncthreads();
        m_tiles = first[p.n_groups];
        n_tile_total = m_tiles * p.n_tiles;
        for (int i = threadIdx.x; i < m_tiles; i += kThreads) {
            const int g = find_group(nullptr, first, p.n_groups, i), rt = start[g] + 2 * (i - first[g]);
            goffs_smem[i] = (int32_t)((uint32_t)rt | (uint32_t)g << 16 | (rt + 1 >= start[g + 1] ? 0x80000000u : 0u));
        }
    }
    const int32_t *goffs = goffs_ok ? goffs_smem : nullptr;
    // Grouped contraction: the groups longest first.  Their tiles go round the CTAs in turn, so that in any other order a CTA
    // that meets several of the long ones finishes last.
    uint16_t *gorder = nullptr;
    if (goffs_ok && p.sort_groups) {
        gorder = reinterpret_cast<uint16_t *>(goffs_smem + kMaxGroupsShared + 1);
        __syncthreads();
        for (int g = threadIdx.x; g < p.n_groups; g += kThreads) {
            const int len = goffs_smem[g + 1] - goffs_smem[g];
            int before = 0;
#pragma unroll 4
            for (int h = 0; h < p.n_groups; h++) {
                const int other = goffs_smem[h + 1] - goffs_smem[h];
                before += other > len || (other == len && h < g);
            }
            gorder[before] = (uint16_t)g;
        }
    }
    if (goffs_ok) __syncthreads();

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        // One stage at a time: wait for its slot (the suspending form, by the whole warp: a wait in a lane-0 branch cost
        // 2-4 % of a dense product, probing three slots per round as much again), then issue its loads.
        const uint32_t lbar0 = CTAS == 1 ? bar_full : cluster_addr(bar_full, 0), a0 = smem_u32(smem_a), b0 = smem_u32(smem_b);
        uint32_t stage = 0, phase = 0;
        bool ok = true;
        const bool issuer = elect_one();
        TRACE_DECL(c_empty); TRACE_DECL(c_issue);
        TRACE_T0(tt);
        int ev_j = 0;
        bool started = false;
        for (int tile = first_tile; ok && tile < n_tile_total; tile += tile_step) {
            Tile t;
            decode_tile<GROUPS>(p, tile, rank, t, m_tiles, goffs, gorder);
            const int32_t ya = kGrouped && t.m_valid <= 0 ? p.M : t.a_row0;   // a CTA without rows: zeros from beyond the tensor
            const int n_it = (t.k_len + kStageElems - 1) / kStageElems;
            int xa = t.a_k0 / kElemsPerByte, xb = t.b_k0 / kElemsPerByte;
            if (!started) start_sync<CTAS, kBuilders>();
            started = true;
#pragma unroll 1
            for (int it = 0; it < n_it; it++, xa += 128, xb += 128) {
                ok = mbar_wait_impl<0>(bar_empty + 8 * stage, phase ^ 1u, abort_flag, p.status, wait_limit, 0x100u + stage);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                TRACE_ADD(c_empty, tt);
                if (lane == 0) TRACE_EV(0, ev_j);
                if (issuer && !(withhold_load != 0u && (uint32_t)ev_j + 1u == withhold_load)) {
                    const uint32_t lbar = lbar0 + 8 * stage;
                    if (CTAS == 1) {
                        mbar_arrive_expect_tx(lbar, kAStageBytes + kBStageBytes);
                        tma_load_2d(a0 + stage * kAStageBytes, &tmA, xa, ya, lbar);
                        tma_load_2d(b0 + stage * kBStageBytes, &tmB, xb, t.b_load_row0, lbar);
                    } else {
                        // Both CTAs' bytes are counted on the leader's barrier, which the leader arms for all of them.
                        // (A remote mbarrier.arrive per stage by a thread of the second CTA costs ~1200 cycles each
                        // and cannot be pipelined; letting the TMA unit signal the remote barrier costs nothing.)
                        if (leader) mbar_arrive_expect_tx(bar_full + 8 * stage, 2 * (kAStageBytes + kBStageBytes));
                        tma_load_2d_pair(a0 + stage * kAStageBytes, &tmA, xa, ya, lbar);
                        tma_load_2d_pair(b0 + stage * kBStageBytes, &tmB, xb, t.b_load_row0, lbar);
                    }
                }
                if (lane == 0) TRACE_EV(1, ev_j);
                ev_j++;
                if (++stage == kStages) { stage = 0; phase ^= 1u; }
                TRACE_ADD(c_issue, tt);
            }
        }
        if (!started) start_sync<CTAS, kBuilders>();
        if (!ok) {   // give copies already in flight time to land before the CTA's shared memory is released
            for (int i = 0; i < 200; i++) __nanosleep(1000);
        }
        if (lane == 0) { TRACE_OUT(p, 0, c_empty); TRACE_OUT(p, 1, c_issue); }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer (the leader CTA of a pair)
        // The warp stays converged and one elected lane issues the tcgen05 instructions: their descriptors then live
        // in uniform registers, and a scale copy costs about ten cycles of the issuing thread instead of fifty.
        // A shared-memory access of this warp queues behind its own pending MMAs: a wait for the next stage right after a
        // stage was issued stalls the tensor pipe for 200-300 cycles even when the stage is there.  So either a watcher warp
        // looks at the barriers and hands over through a named barrier (WATCH), or this warp probes the next stage's
        // barriers BEFORE it issues a stage and waits afterwards only if they were not complete.  All lanes wait: a
        // lane-0 branch around the wait costs as much as the wait.
        uint32_t stage = 0, full_phase = 0, acc_empty_phase = 0;
        tcgen05_fence_before();
        __syncwarp();
        if (CTAS == 2) asm volatile("bar.arrive 14, 288;" ::: "memory");   // tensor memory is there: for the epilogue warps
        start_sync<CTAS, kBuilders>();
        tcgen05_fence_after();
        const uint32_t tmem_base = *tmem_base_slot;
        // mma_ok: no wait for a stage has run out.  Afterwards the remaining stages are issued unseen, but their slots are not given back: the
        // producers would announce a slot's next bytes on a barrier that still waits for the last ones, which is undefined.  (One
        // predicate on that commit and the watcher's word with its arrival: within 0.3 % of a product; nothing issued at all, 0.5 to 1 %.)
        bool mma_ok = true;
        bool ready = false;   // !WATCH: the next stage has been seen complete
        BufRing ring;   // image buffer of the current unit
        const bool issuer = elect_one();
        int ev_j = 0;
        TRACE_DECL(c_acc); TRACE_DECL(c_sync); TRACE_DECL(c_issue);
        TRACE_T0(tt);
        for (int tile = first_tile; leader && tile < n_tile_total; tile += tile_step) {
            Tile t;
            decode_tile<GROUPS>(p, tile, rank, t, m_tiles, goffs, gorder, NEED_LENGTH);
            const int n_it = (t.k_len + kStageElems - 1) / kStageElems;
            if (n_it == 0) continue;
            TRACE_ADD(c_acc, tt);
            for (int it = 0; it < n_it; it++) {
                if (WATCH) {
                    mma_ok = named_meet(1 + stage, true);   // the watcher has seen the operands and both scale images of this stage
                } else {
                    if (it == 0) {
                        if (mma_ok) mma_ok = mbar_wait_impl<0>(bar_acc_empty, acc_empty_phase ^ 1u, abort_flag, p.status, wait_limit, 0x200u);
                        acc_empty_phase ^= 1u;
                    }
                    if (!ready) {
                        if ((it & (kUnitStages - 1)) == 0) {
                            if (mma_ok) mma_ok = mbar_wait_impl<0>(bar_cache_full + 8 * ring.buf, ring.phase, abort_flag, p.status, wait_limit, 0x510u + ring.buf);
                            if (CTAS == 2 && mma_ok)
                                mma_ok = mbar_wait_impl<0>(bar_peer_cache_full + 8 * ring.buf, ring.phase, abort_flag, p.status, wait_limit, 0x520u + ring.buf);
                        }
                        if (mma_ok) mma_ok = mbar_wait_impl<0>(bar_full + 8 * stage, full_phase, abort_flag, p.status, wait_limit, 0x300u + stage);
                    }
                    const uint32_t ns = stage + 1 == kStages ? 0u : stage + 1;
                    ready = mbar_test_wait(bar_full + 8 * ns, ns == 0 ? full_phase ^ 1u : full_phase);
                    if (it == n_it - 1 || ((it + 1) & (kUnitStages - 1)) == 0) {   // the next stage starts a unit
                        BufRing nu = ring;
                        nu.next(kImageBufs);
                        ready = ready && mbar_test_wait(bar_cache_full + 8 * nu.buf, nu.phase);
                        if (CTAS == 2) ready = ready && mbar_test_wait(bar_peer_cache_full + 8 * nu.buf, nu.phase);
                    }
                    __syncwarp();
                }
                tcgen05_fence_after();
                TRACE_ADD(c_sync, tt);
                if (lane == 0) TRACE_EV(2, ev_j);
                if (issuer) {
                    const uint32_t sf_tmem = tmem_base + kTmemSfBase + stage * SfCols<KIND>::kStride;
                    const uint32_t img = smem_u32(smem_images + ring.buf * kBufBytes + (it & (kUnitStages - 1)) * kImageStage);
                    if (KIND == KIND_MXF4B16) {
#pragma unroll
                        for (int i = 0; i < 4; i++) {
                            tcgen05_cp_32x128b_warpx4<CTAS>(sf_tmem + 4 * i, smem_desc_scale_image(img + 512 * i));
                            tcgen05_cp_32x128b_warpx4<CTAS>(sf_tmem + 16 + 8 * i, smem_desc_scale_image(img + 2048 + 1024 * i));
                            tcgen05_cp_32x128b_warpx4<CTAS>(sf_tmem + 20 + 8 * i, smem_desc_scale_image(img + 2560 + 1024 * i));
                        }
                    } else if (KIND == KIND_MXF8) {
                        tcgen05_cp_32x128b_warpx4<CTAS>(sf_tmem, smem_desc_scale_image(img));
                        tcgen05_cp_32x128b_warpx4<CTAS>(sf_tmem + 8, smem_desc_scale_image(img + 512));
                        tcgen05_cp_32x128b_warpx4<CTAS>(sf_tmem + 12, smem_desc_scale_image(img + 1024));
                    } else {
                        constexpr bool kRealA = KIND == KIND_MXF4RA, kRealB = KIND == KIND_MXF4RB;   // the other images are replicated
                        constexpr uint32_t kA = kRealA ? 512 : 128, kB = kRealB ? 512 : 128;
#pragma unroll
                        for (int c = 0; c < 2; c++) {
                            tcgen05_cp_32x128b_warpx4<CTAS>(sf_tmem + 4 * c, kRealA ? smem_desc_scale_image(img + kA * c) : smem_desc_scale_image_rep(img + kA * c));
                            const uint32_t b = img + 2 * kA + 2 * kB * c;
                            tcgen05_cp_32x128b_warpx4<CTAS>(sf_tmem + 8 + 8 * c, kRealB ? smem_desc_scale_image(b) : smem_desc_scale_image_rep(b));
                            tcgen05_cp_32x128b_warpx4<CTAS>(sf_tmem + 12 + 8 * c, kRealB ? smem_desc_scale_image(b + kB) : smem_desc_scale_image_rep(b + kB));
                        }
                    }
                    const uint64_t adesc = smem_desc_sw128(smem_u32(smem_a + stage * kAStageBytes));
                    const uint64_t bdesc = smem_desc_sw128(smem_u32(smem_b + stage * kBStageBytes));
                    const int k_left = t.k_len - it * kStageElems;
                    const int n_mma = min(4, (k_left + kMmaK - 1) / kMmaK);
#pragma unroll
                    for (int i = 0; i < 4; i++) {
                        if (i < n_mma) {
                            if (KIND == KIND_MXF4B16) {   // one 32-bit scale column entry per row and MMA: all four bytes are used
                                tcgen05_mma_block_scaled<KIND, CTAS>(tmem_base, adesc + 2 * i, bdesc + 2 * i, instr_desc<KIND, CTAS>(0u, 0u),
                                                                     sf_tmem + 4 * i, sf_tmem + 16 + 8 * i, (it > 0 || i > 0) ? 1u : 0u);
                                continue;
                            }
                            const int chunk = kind_fp4(KIND) ? (i >> 1) : 0;
                            const uint32_t sf_id = kind_fp4(KIND) ? 2u * (i & 1) : (uint32_t)i;
                            tcgen05_mma_block_scaled<KIND, CTAS>(tmem_base, adesc + 2 * i, bdesc + 2 * i,
                                                                 instr_desc<KIND, CTAS>(sf_id, sf_id), sf_tmem + 4 * chunk,
                                                                 sf_tmem + 8 + 8 * chunk, (it > 0 || i > 0) ? 1u : 0u);
                        }
                    }
                    if (mma_ok) tcgen05_commit<CTAS>(bar_empty + 8 * stage);
                    if (it == n_it - 1) tcgen05_commit<CTAS>(bar_acc_full);
                    if ((it & (kUnitStages - 1)) == kUnitStages - 1 || it == n_it - 1)
                        tcgen05_commit<CTAS>(bar_cache_empty + 8 * ring.buf);   // the unit's images have been copied
                }
                if ((it & (kUnitStages - 1)) == kUnitStages - 1 || it == n_it - 1) ring.next(kImageBufs);
                TRACE_ADD(c_issue, tt);
                if (lane == 0) TRACE_EV(3, ev_j);
                ev_j++;
                if (++stage == kStages) { stage = 0; full_phase ^= 1u; }
            }
        }
        if (KIND != KIND_MXF4 && CTAS == 2 && !leader) {
            // Per-row scales, second CTA of a pair, whose MMA warp has nothing else to do: report each unit of scale images the
            // builders have finished to the leader, which issues the scale copies of both CTAs.
            bool fwd_ok = true;
            BufRing fr;
            UnitIter<GROUPS_NONE> un;
            for (un.init(p, first_tile, tile_step, rank, m_tiles, n_tile_total); fwd_ok && un.valid(p); un.next(p, kUnitStages * kStageElems), fr.next(kImageBufs)) {
                fwd_ok = __all_sync(0xFFFFFFFFu, mbar_wait_impl<0>(bar_cache_full + 8 * fr.buf, fr.phase, abort_flag, p.status, wait_limit, 0x530u + fr.buf));
                if (fwd_ok && issuer) mbar_arrive_cluster(cluster_addr(bar_peer_cache_full + 8 * fr.buf, 0));
            }
            __syncwarp();
        }
        if (leader && *abort_flag) {
            // Some role gave up, and this warp has run through the remaining stages.  The second CTA, whose producer waits for slots that
            // are not given back, is told; and before tensor memory is freed the tensor pipe is idle (a bounded wait).
            if (CTAS == 2 && lane == 0)
                asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cluster_addr(smem_u32(const_cast<const uint32_t *>(abort_flag)), 1)), "r"(1u) : "memory");
            if (issuer) tcgen05_commit<CTAS>(bar_drain);
            __syncwarp();
            if (lane == 0) mbar_drain(bar_drain);
            __syncwarp();
            // Loads of either CTA may still be on their way: hold the pair (the other roles wait at the final barrier) until they
            // have landed.
            for (int i = 0; i < 200; i++) __nanosleep(1000);
        }
        if (lane == 0) { TRACE_OUT(p, 2, c_acc); TRACE_OUT(p, 3, c_sync); TRACE_OUT(p, 4, c_issue); }
    } else if (warp == 3 || (warp == 2 && Cfg<KIND, CTAS>::kBuilders == 2)) {
        // ------------------------------------------------------------------ scale image builder
        // 2D-block scales: per unit (up to 16 stages of one tile) loads the scale bytes as 16-byte rows, one lane a chunk, and
        // replicates each row into its image; per-row scales: loads the unit's scale words and
        // writes the 32-row images directly.  Two image buffers alternate, so the next unit is built while
        // the current one runs: all global-memory latency of the scale path is paid here, off the per-stage
        // critical path, and nothing has to be written per stage.  A buffer is free again once the MMA warp's
        // commit reports that the last scale copy out of it has completed.  In a pair each CTA builds the images
        // of its own 128 A rows and of all 256 B rows.
        // At its end a builder waits until its last buffer is free: the MMA warp's commits, which arrive at both CTAs of a pair, come in
        // order and that one is the last.
        BufRing ring;
        bool ok = true;
        if (KIND != KIND_MXF4) {
            // per-row scales: the raw bytes of the next kOwnRaw units are in flight (cp.async) while a unit is turned into
            // images.  Two builders take every other unit and have raw buffers of their own.
            constexpr int kRawBytes = Cfg<KIND, CTAS>::kRawBytes, kSorted = Cfg<KIND, CTAS>::kSortedBytes;
            constexpr int kOwnRaw = Cfg<KIND, CTAS>::kRawBufs > 0 ? Cfg<KIND, CTAS>::kRawBufs / kBuilders : 1;
            uint8_t *raw = smem_raw_scales + (3 - warp) * (kOwnRaw * kRawBytes + kSorted);
            UnitIter<GROUPS_NONE> ahead, cur;
            ahead.init(p, first_tile, tile_step, rank, m_tiles, n_tile_total);
            if (warp == 2) {   // the second builder starts with the second unit
                if (ahead.valid(p)) ahead.next(p, kUnitStages * kStageElems);
                ring.next(kImageBufs);
            }
            cur = ahead;
            RowBuilder<KIND, CTAS> rb;
            int rows_tile = -1;
            uint32_t raw_buf = 0;
            BufRing used;
            bool any = false;
#pragma unroll 1
            for (int i = -kOwnRaw;; i++) {   // unit i of this builder is made, unit i + kOwnRaw is fetched
                uint8_t *own = raw + raw_buf * kRawBytes;
                if (++raw_buf == kOwnRaw) raw_buf = 0;
                if (i >= 0) {
                    if (!cur.valid(p)) break;
                    asm volatile("cp.async.wait_group %0;" ::"n"(kOwnRaw - 1) : "memory");   // this unit's bytes have landed
                    __syncwarp();
                    rb.read(p, cur.t, cur.k0, own, raw + kOwnRaw * kRawBytes, lane);
                    __syncwarp();   // the raw buffer and the sorted rows are free
                }
                if (ahead.valid(p)) {
                    if (ahead.tile != rows_tile) {
                        rb.set(p, ahead.t, lane);
                        rows_tile = ahead.tile;
                    }
                    rb.fetch(p, ahead.t, ahead.k0, own, lane);
                    for (int n = 0; n < kBuilders; n++)
                        if (ahead.valid(p)) ahead.next(p, kUnitStages * kStageElems);
                }
                asm volatile("cp.async.commit_group;" ::: "memory");   // one group in any case
                if (i < 0) {
                    if (i == -1) start_sync<CTAS, kBuilders, true>();
                    continue;
                }
                ok = mbar_wait_impl<0>(bar_cache_empty + 8 * ring.buf, ring.phase ^ 1u, abort_flag, p.status, wait_limit, 0x500u + ring.buf);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                rb.write(min(kUnitStages, (cur.t.k_len - cur.k0 + kStageElems - 1) / kStageElems), smem_images + ring.buf * kBufBytes, lane);
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic-proxy writes -> tcgen05.cp
                __syncwarp();
                // In the second CTA of a pair the arrival is forwarded to the leader by warp 1: the remote arrival
                // stalls its issuing thread for about a thousand cycles, which this warp spends on the next unit.
                if (lane == 0) mbar_arrive(bar_cache_full + 8 * ring.buf);
                used = ring;
                any = true;
                for (int n = 0; n < kBuilders; n++) {
                    ring.next(kImageBufs);
                    if (cur.valid(p)) cur.next(p, kUnitStages * kStageElems);
                }
            }
            asm volatile("cp.async.wait_all;" ::: "memory");
            if (ok && any) mbar_wait_impl<0>(bar_cache_empty + 8 * used.buf, used.phase, abort_flag, p.status, wait_limit, 0x540u);
        }
        if (KIND == KIND_MXF4) {
            UnitIter<GROUPS> un;   // the unit whose scale bytes are being loaded
            un.goffs = goffs;
            un.gorder = gorder;
            un.init(p, first_tile, tile_step, rank, m_tiles, n_tile_total);
            uint32_t wa[4] = {}, wb[8] = {};
            uint32_t next_a[4] = {}, next_b[8] = {};
            int how_a = SCALES_WHOLE, how_b = SCALES_WHOLE;
            int n_chunks = 0;                // of the unit that is loaded; 0: none
            // A unit is written while the next one's loads are in flight; the first is written before anything else is looked at.
            // In a pair the leader's multicast commits release the buffers.  Whether a remote arrival wakes a suspended thread is not
            // specified: this wait probes (where the other roles suspend on such barriers, they look again after kSuspendNs at the latest).
            bool started = false;
            BufRing used;
            for (int unit = 0, fetched = 0;;) {
                const int n = n_chunks;
                uint4 row_a, row_b0, row_b1;
                if (n > 0) {
                    const int kb_a = (un.t.a_k0 + un.k0) >> 5, kb_b = (un.t.b_k0 + un.k0) >> 5;
                    if (how_a == SCALES_SHIFTED) place_chunk_scales<1>(p.sfa, un.t.a_row0 >> 5, kb_a, wa, next_a, lane);
                    if (how_b == SCALES_SHIFTED) place_chunk_scales<2>(p.sfb, un.t.b_row0 >> 5, kb_b, wb, next_b, lane);
                    row_a = chunk_image_row(p.sfa, wa);
                    row_b0 = chunk_image_row(p.sfb, wb);
                    row_b1 = chunk_image_row(p.sfb, wb + 4);
                    if (how_a == SCALES_GATHER || how_b == SCALES_GATHER) {
                        gather_scale_rows<kGrouped>(p, un.t, un.k0, how_a == SCALES_GATHER, how_b == SCALES_GATHER, n, reinterpret_cast<uint32_t *>(smem_compact), lane);
                        const uint4 *gathered = reinterpret_cast<const uint4 *>(smem_compact);
                        if (how_a == SCALES_GATHER) row_a = gathered[lane];
                        if (how_b == SCALES_GATHER) { row_b0 = gathered[kCacheChunks + 2 * lane]; row_b1 = gathered[kCacheChunks + 2 * lane + 1]; }
                        __syncwarp();
                    }
                }
                n_chunks = 0;
                if (n == 0 || unit > 0) {
                    if (fetched++) un.next(p, kUnitStages * kStageElems);
                    if (un.valid(p)) {
                        const int n_real = min(kCacheChunks, (un.t.k_len - un.k0 + 127) >> 7);
                        n_chunks = (n_real + 1) & ~1;   // whole stages
                        how_a = fetch_chunk_scales<1>(p.sfa, un.t.a_row0 >> 5, (un.t.a_k0 + un.k0) >> 5, n_real, n_chunks, wa, next_a, lane);
                        how_b = fetch_chunk_scales<2>(p.sfb, un.t.b_row0 >> 5, (un.t.b_k0 + un.k0) >> 5, n_real, n_chunks, wb, next_b, lane);
                    } else if (n == 0) {
                        break;
                    }
                }
                if (!started) start_sync<CTAS, kBuilders, true>();   // the first unit's loads are on their way
                started = true;
                if (n == 0) continue;
                const int buf = ring.buf;
                if (unit >= kImageBufs) {   // the first units' buffers have never been used
                    ok = mbar_wait_impl<kRelaxedNs, CTAS == 2>(bar_cache_empty + 8 * buf, ring.phase ^ 1u, abort_flag, p.status, wait_limit, 0x500u + buf);
                    ok = __all_sync(0xFFFFFFFFu, ok);
                    if (!ok) break;
                }
                if (lane < n) {
                    uint8_t *images = smem_images + buf * kBufBytes + (lane >> 1) * kImageStageBytes + (lane & 1) * 128;
                    uint4 *img_a = reinterpret_cast<uint4 *>(images), *img_b = reinterpret_cast<uint4 *>(images + 256 + (lane & 1) * 128);
                    // the lanes' images lie 128 bytes apart: each starts with another of the eight rows, so that eight lanes cover all banks
#pragma unroll
                    for (int i = 0; i < 8; i++) {
                        const int r = (i + lane) & 7;
                        img_a[r] = row_a;
                        img_b[r] = row_b0;
                        img_b[8 + r] = row_b1;
                    }
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic-proxy writes -> tcgen05.cp
                __syncwarp();
                if (lane == 0) {   // 16-stage units leave time for the second CTA's own (slow) remote arrival
                    TRACE_EV(5, unit);
                    if (CTAS == 1 || leader) mbar_arrive(bar_cache_full + 8 * buf);
                    else mbar_arrive_cluster(cluster_addr(bar_peer_cache_full + 8 * buf, 0));
                }
                used = ring;
                ring.next(kImageBufs);
                unit++;
            }
            if (!started) start_sync<CTAS, kBuilders, true>();
            else if (ok) mbar_wait_impl<kRelaxedNs, CTAS == 2>(bar_cache_empty + 8 * used.buf, used.phase, abort_flag, p.status, wait_limit, 0x540u);
        }
    } else if (warp == 2) {
        // ------------------------------------------------------------------ watcher
        // Follows the stream of stages (one CTA, or the leader of a pair; the second CTA's warp idles).  For each
        // it waits for the ring slot's "full" barrier (the operand bytes of both CTAs), at the first stage of a
        // unit for the unit's scale images (of both CTAs), and at the first stage of a tile for the accumulator
        // to be drained; then it meets the MMA warp at the slot's named barrier.  After a timeout they meet at every remaining
        // stage all the same, so that the MMA warp, which cannot time out on a named barrier, always runs to its end.
        StageIter sg;
        sg.init(p, first_tile, tile_step, rank, kStageElems);
        start_sync<CTAS, kBuilders>();
        uint32_t stage = 0, phase = 0, acc_phase = 0;
        BufRing ring;   // image buffer of the current unit
        bool ok = true;
        TRACE_DECL(c_meet); TRACE_DECL(c_poll);
        TRACE_T0(tt);
        int ev_j = 0;
        bool unit_seen = false;   // the next unit's scale images have been seen complete
        uint32_t ahead = 0;   // stages after the current one whose "full" barrier is already known to be complete
        while (WATCH && leader && sg.valid(p)) {
            if (lane == 0) TRACE_EV(4, ev_j);
            if (ahead > 0) {
                ahead--;
            } else {
                if (ok) {   // all lanes probe (a lane-0 branch and the broadcast of its result slowed the hand-over by 2-4 %)
                    if ((sg.it & (kUnitStages - 1)) == 0 && !unit_seen) {
                        // both CTAs' images of this unit: the two barriers probed together (the latencies overlap)
                        const uint32_t b0 = bar_cache_full + 8 * ring.buf, b1 = (CTAS == 2 ? bar_peer_cache_full : bar_cache_full) + 8 * ring.buf;
                        for (uint32_t spin = 0; ; spin++) {
                            uint32_t q0, q1;
                            asm volatile("{\n .reg .pred p0, p1;\n"
                                         " mbarrier.test_wait.parity.shared::cta.b64 p0, [%2], %4;\n"
                                         " mbarrier.test_wait.parity.shared::cta.b64 p1, [%3], %4;\n"
                                         " selp.b32 %0, 1, 0, p0;\n selp.b32 %1, 1, 0, p1;\n}"
                                         : "=r"(q0), "=r"(q1) : "r"(b0), "r"(b1), "r"(ring.phase) : "memory");
                            if (q0 && q1) break;
                            if (spin >= wait_limit) {
                                ok = false;
                                *abort_flag = 1u;
                                if (atomicCAS(p.status, 0u, (uint32_t)FP4Q_ERR_TIMEOUT) == 0u) p.status[1] = (q0 ? 0x520u : 0x510u) + ring.buf;
                                break;
                            }
                            if ((spin & 255u) == 255u && *abort_flag) { ok = false; break; }
                        }
                    }
                    if ((sg.it & (kUnitStages - 1)) == 0) unit_seen = false;
                    // Whether the next unit's images are in place is looked up ahead of time, so that a unit boundary
                    // costs no extra probe on the critical path: with short units (per-row scales) the two barriers
                    // ride along with every probe of the ring slots below; with 16-stage units one look in the second
                    // half of the unit is enough, and the slot probes stay as light as they can be.
                    BufRing nu = ring;
                    nu.next(kImageBufs);
                    const uint32_t nb0 = bar_cache_full + 8 * nu.buf, nb1 = (CTAS == 2 ? bar_peer_cache_full : bar_cache_full) + 8 * nu.buf;
                    if (KIND == KIND_MXF4 && ok && (sg.it & (kUnitStages - 1)) >= kUnitStages / 2 && !unit_seen)
                        unit_seen = mbar_test_wait(nb0, nu.phase) && (CTAS == 1 || mbar_test_wait(nb1, nu.phase));
                    if (ok && sg.it == 0) ok = mbar_wait_impl<0, true>(bar_acc_empty, acc_phase ^ 1u, abort_flag, p.status, wait_limit, 0x200u);
                    if (ok) {
                        // A probe of an mbarrier takes this warp a few hundred cycles even when the phase is long
                        // complete, more than the MMA warp needs per stage.  So the slot's "full" barrier and those of
                        // the next three slots are probed in one go (the latencies overlap); slots found complete are
                        // handed over later without another look.  Only stages of the same unit qualify: they need
                        // nothing but their "full" barrier.
                        const int left = min(kUnitStages - 1 - (sg.it & (kUnitStages - 1)), sg.n_it - 1 - sg.it);
                        uint32_t sl[4], ph[4];
                        sl[0] = stage; ph[0] = phase;
#pragma unroll
                        for (int q = 1; q < 4; q++) {
                            sl[q] = sl[q - 1] + 1 == kStages ? 0u : sl[q - 1] + 1;
                            ph[q] = sl[q] == 0 ? ph[q - 1] ^ 1u : ph[q - 1];
                        }
                        uint32_t r0 = 0, r1 = 0, r2 = 0, r3 = 0, r4 = 0, r5 = 0;
                        for (uint32_t spin = 0; ; spin++) {
                            if (KIND == KIND_MXF4)
                                asm volatile("{\n .reg .pred p0, p1, p2, p3;\n"
                                             " mbarrier.test_wait.parity.shared::cta.b64 p0, [%4], %5;\n"
                                             " mbarrier.test_wait.parity.shared::cta.b64 p1, [%6], %7;\n"
                                             " mbarrier.test_wait.parity.shared::cta.b64 p2, [%8], %9;\n"
                                             " mbarrier.test_wait.parity.shared::cta.b64 p3, [%10], %11;\n"
                                             " selp.b32 %0, 1, 0, p0;\n selp.b32 %1, 1, 0, p1;\n selp.b32 %2, 1, 0, p2;\n selp.b32 %3, 1, 0, p3;\n}"
                                             : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                                             : "r"(bar_full + 8 * sl[0]), "r"(ph[0]), "r"(bar_full + 8 * sl[1]), "r"(ph[1]),
                                               "r"(bar_full + 8 * sl[2]), "r"(ph[2]), "r"(bar_full + 8 * sl[3]), "r"(ph[3]) : "memory");
                            else
                            asm volatile("{\n .reg .pred p0, p1, p2, p3, p4, p5;\n"
                                         " mbarrier.test_wait.parity.shared::cta.b64 p0, [%6], %7;\n"
                                         " mbarrier.test_wait.parity.shared::cta.b64 p1, [%8], %9;\n"
                                         " mbarrier.test_wait.parity.shared::cta.b64 p2, [%10], %11;\n"
                                         " mbarrier.test_wait.parity.shared::cta.b64 p3, [%12], %13;\n"
                                         " mbarrier.test_wait.parity.shared::cta.b64 p4, [%14], %16;\n"
                                         " mbarrier.test_wait.parity.shared::cta.b64 p5, [%15], %16;\n"
                                         " selp.b32 %0, 1, 0, p0;\n selp.b32 %1, 1, 0, p1;\n selp.b32 %2, 1, 0, p2;\n selp.b32 %3, 1, 0, p3;\n"
                                         " selp.b32 %4, 1, 0, p4;\n selp.b32 %5, 1, 0, p5;\n}"
                                         : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3), "=r"(r4), "=r"(r5)
                                         : "r"(bar_full + 8 * sl[0]), "r"(ph[0]), "r"(bar_full + 8 * sl[1]), "r"(ph[1]),
                                           "r"(bar_full + 8 * sl[2]), "r"(ph[2]), "r"(bar_full + 8 * sl[3]), "r"(ph[3]),
                                           "r"(nb0), "r"(nb1), "r"(nu.phase) : "memory");
                            if (r0) break;
                            if (spin >= wait_limit) {
                                ok = false;
                                *abort_flag = 1u;
                                if (atomicCAS(p.status, 0u, (uint32_t)FP4Q_ERR_TIMEOUT) == 0u) p.status[1] = 0x300u + stage;
                                break;
                            }
                            if ((spin & 255u) == 255u && *abort_flag) { ok = false; break; }
                        }
                        ahead = !ok ? 0u : (left >= 1 && r1) ? ((left >= 2 && r2) ? ((left >= 3 && r3) ? 3u : 2u) : 1u) : 0u;
                        if (r4 && r5) unit_seen = true;
                    }
                }
                ahead = __reduce_min_sync(0xFFFFFFFFu, ahead);   // what every lane has seen
            }
            ok = __all_sync(0xFFFFFFFFu, ok);
            TRACE_ADD(c_poll, tt);
            if (lane == 0) TRACE_EV(6, ev_j);
            ev_j++;
            named_meet(1 + stage, ok);   // rendezvous: the MMA warp is at most one stage behind
            TRACE_ADD(c_meet, tt);
            if (sg.it == 0) acc_phase ^= 1u;
            if ((sg.it & (kUnitStages - 1)) == kUnitStages - 1 || sg.it == sg.n_it - 1) ring.next(kImageBufs);
            if (++stage == kStages) { stage = 0; phase ^= 1u; }
            sg.next(p, kStageElems);
        }
        __syncwarp();
        if (lane == 0) { TRACE_OUT(p, 6, c_meet); TRACE_OUT(p, 7, c_poll); }
    } else if (warp >= 4) {
        // ------------------------------------------------------------------ epilogue
        const int quarter = warp & 3;            // TMEM lanes 32*quarter .. +31 (hardware: warp id mod 4)
        const int half = (warp - 4) >> 2;        // accumulator columns 128*half .. +127
        start_sync<CTAS, kBuilders>();
        if (CTAS == 2) asm volatile("bar.sync 14, 288;" ::: "memory");
        tcgen05_fence_after();
        const uint32_t tmem_base = *tmem_base_slot;
        uint32_t acc_phase = 0;
        bool ok = true, arrived = false;
        int ev_t = 0;
        TRACE_DECL(c_wait); TRACE_DECL(c_ld); TRACE_DECL(c_store);
        TRACE_T0(tt);
        for (int tile = first_tile; ok && tile < n_tile_total; tile += tile_step) {
            Tile t;
            decode_tile<GROUPS>(p, tile, rank, t, m_tiles, goffs, gorder, NEED_OUTPUT);
            const bool last = tile + tile_step >= n_tile_total;   // of this CTA
            const int row_in_tile = 32 * quarter + lane;
            const int64_t row = (int64_t)t.c_row0 + row_in_tile;
            const bool row_ok = row_in_tile < t.m_valid;
            uint32_t v[4][32];
            if (t.k_len > 0) {
                // this wait spans a whole tile (every other one spans a few stages at most): its limit grows with the
                // tile's contraction length, so that a very long contraction cannot run into it on a healthy run
                const uint64_t tile_limit = wait_limit * (uint64_t)(1 + (t.k_len >> 12));
                // Every warp waits for itself (the suspending form: polling warps keep the shared-memory unit busy enough to slow every other
                // role's waits).  With one thread waiting and the warps meeting at a named barrier behind it, us: 2048 x 4096 x 4096 quantized
                // 20.5 / 19.7, 8192 x 2048 x 2048 19.3 / 19.4 / 16.8 -> 18.3 / 18.4 / 16.7, 1D activations there 20.2 / 19.5 -> 19.5 / 19.4, 16 x 16 blocks 23.2 / 23.1 /
                // 20.0 -> 22.3 / 22.0 / 19.8, 16384 x 4096 x 4096 98.3 / 98.4 / 104.6 -> 94.7 / 94.7 / 103.8.  Weight gradients of short groups, bound by
                // their writes, lose when warps drift apart (36352 rows in 128 groups, 1408 x 2048, 271 -> 316; 16640 in 128, 512 x 2048 99 ->
                // 113), so there they still meet.
                if (kGrouped && p.warps_meet) {
                    if (warp == 4 && lane == 0) {
                        ok = mbar_wait(bar_acc_full, acc_phase, abort_flag, p.status, tile_limit, 0x404u);
                        acc_seen[acc_phase] = ok ? 1u : 0u;   // one word per phase: a warp is at most one tile behind
                    }
                    __syncwarp();
                    asm volatile("bar.sync 15, 256;" ::: "memory");
                    ok = acc_seen[acc_phase] != 0u;
                } else {
                    ok = mbar_wait(bar_acc_full, acc_phase, abort_flag, p.status, tile_limit, 0x404u);
                    ok = __all_sync(0xFFFFFFFFu, ok);
                }
                TRACE_ADD(c_wait, tt);
                if (lane == 0) TRACE_EV(7, 16 * ev_t + 2 * (warp - 4));
                if (!ok) break;
                acc_phase ^= 1u;
                tcgen05_fence_after();
                const uint32_t taddr = tmem_base + ((uint32_t)(32 * quarter) << 16) + 128u * half;
                FP4Q_TMEM_LD_X32(taddr, v[0]);
                FP4Q_TMEM_LD_X32(taddr + 32, v[1]);
                FP4Q_TMEM_LD_X32(taddr + 64, v[2]);
                FP4Q_TMEM_LD_X32(taddr + 96, v[3]);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                tcgen05_fence_before();
                __syncwarp();
                // The accumulator now lives in registers.  Behind the last one nobody waits for the accumulator, and this warp has nothing
                // to do with the other CTA any more: it lets the pair go while its output leaves.  The arrival is relaxed: all that has to be
                // over before tensor memory is freed is this warp's reads of it, which wait::ld has completed and which the tcgen05
                // fences before the arrival and before the deallocation order (PTX's own examples pair these fences with relaxed
                // arrivals).  Release costs products of 8 us 2 % (2048 x 2048 x 2048 8.1 / 8.1 / 9.15 -> 8.3 / 8.3 / 9.4).
                if (last) {
                    if (CTAS == 2) cluster_arrive_relaxed();
                    else asm volatile("bar.arrive 14, 288;" ::: "memory");
                    arrived = true;
                } else if (lane == 0) {   // the leader's MMA thread waits for both CTAs
                    if (CTAS == 1 || leader) mbar_arrive(bar_acc_empty);
                    else mbar_arrive_cluster(cluster_addr(bar_acc_empty, 0));
                }
                TRACE_ADD(c_ld, tt);
                if (lane == 0) TRACE_EV(7, 16 * ev_t + 2 * (warp - 4) + 1);
                ev_t++;
            } else {
#pragma unroll
                for (int j = 0; j < 4; j++)
#pragma unroll
                    for (int q = 0; q < 32; q++) v[j][q] = 0u;
            }
            if (EPI == EPI_QUANT) {
                // The output tile leaves as 2D-block FP4: each warp owns four 32x32 blocks (its 32 rows x 32 columns
                // per chunk).  The accumulator is rounded to BF16 first, so the result equals fp4q_quantize2d applied
                // to the BF16 output of the plain product: block maximum over the warp, truncation-free scale, E2M1
                // codes by the same converts, row-major payload from the lane's own row, transposed payload from the staged
                // row-major codes; both leave through the staging rows and TMA stores.
                const int64_t row_g = (int64_t)t.c_row0 + row_in_tile;
                const int row0_blk = t.c_row0 + 32 * quarter;
                // staging: 32 rows x 64 B of row-major payload (64-byte swizzle) and 128 rows x 16 B of transposed payload
                uint8_t *stg = smem_staging + (warp - 4) * kStagingWarpBytes;
                const uint32_t stg_rm = smem_u32(stg) + lane * 64, swz = (uint32_t)((lane >> 1) & 3);
                const bool any = row0_blk < p.M && t.c_col0 + 128 * half < p.N;   // warp-uniform: something to write
                if (any) {
                    if (lane == 0) bulk_wait_read_all();   // the previous tile's stores have read the staging rows
                    __syncwarp();
                }
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const int col0 = t.c_col0 + 128 * half + 32 * j;
                    if (col0 >= p.N || row0_blk >= p.M) continue;   // warp-uniform
                    // The maximum as in the quantizer: packed |.| with NaN propagation (a fifth of the instructions of a comparison per
                    // element), so that a non-finite entry shows in the result and sends the block through the careful pass.  us, the two
                    // builds replayed in turn, forward nearest / stochastic: 300 x 768 x 1232 12.8 / 14.2 -> 12.1 / 13.4, 8192 x 2048 x 2048 31.5 /
                    // 36.4 -> 28.5 / 33.2, 8192 x 5632 x 2048 70.2 / 80.6 -> 62.5 / 73.1.  From 16 stages a tile on the epilogue is hidden and the
                    // gain with it: 16384 x 4096 x 4096 117.4 / 119.6 -> 117.8 / 119.4, and 16384 x 11008 x 4096 loses with stochastic rounding,
                    // 280.8 / 320.3 -> 278.9 / 325.0, for a reason that is not known.
                    uint32_t raw[16];
                    __nv_bfloat162 m2 = __float2bfloat162_rn(0.0f);
#pragma unroll
                    for (int e = 0; e < 16; e++) {
                        const __nv_bfloat162 b = __floats2bfloat162_rn(__uint_as_float(v[j][2 * e]), __uint_as_float(v[j][2 * e + 1]));
                        raw[e] = *reinterpret_cast<const uint32_t *>(&b);
                        m2 = __hmax2_nan(m2, __habs2(b));
                    }
                    const __nv_bfloat16 m1 = __hmax_nan(m2.x, m2.y);
                    uint32_t mx = __reduce_max_sync(0xFFFFFFFFu, (uint32_t)(*reinterpret_cast<const uint16_t *>(&m1)) & 0x7FFFu);
                    const bool nonfinite = mx >= 0x7F80u;
                    if (nonfinite) {
                        mx = 0;
#pragma unroll
                        for (int e = 0; e < 16; e++) {
                            const uint32_t m0 = raw[e] & 0x7FFFu, m1b = (raw[e] >> 16) & 0x7FFFu;
                            mx = max(mx, max(m0 >= 0x7F80u ? 0u : m0, m1b >= 0x7F80u ? 0u : m1b));
                        }
                        mx = __reduce_max_sync(0xFFFFFFFFu, mx);
                    }
                    const int code = scale_code_from_max(mx);
                    uint32_t W[4];
#pragma unroll
                    for (int sg = 0; sg < 2; sg++) {
                        uint32_t R[4] = {0u, 0u, 0u, 0u};
                        if (p.q_mode == FP4Q_ROUND_STOCHASTIC) {
                            const uint64_t blk = (uint64_t)(row_g * p.N + col0 + 16 * sg) >> 4;   // N % 16 == 0
                            philox4x32_10((uint32_t)blk, (uint32_t)(blk >> 32), p.q_tensor_id, 0u, p.q_keys, R);
                        }
                        if (nonfinite) {
                            const uint4 lo = make_uint4(raw[8 * sg], raw[8 * sg + 1], raw[8 * sg + 2], raw[8 * sg + 3]);
                            const uint4 hi = make_uint4(raw[8 * sg + 4], raw[8 * sg + 5], raw[8 * sg + 6], raw[8 * sg + 7]);
                            const uint4 rn = make_uint4(R[0], R[1], R[2], R[3]);
                            const uint2 w = p.q_mode == FP4Q_ROUND_STOCHASTIC
                                                ? round_segment_scalar<FP4Q_ROUND_STOCHASTIC>(lo, hi, rn, inv_scale_f16_aligned(code))
                                                : round_segment_scalar<FP4Q_ROUND_NEAREST>(lo, hi, rn, inv_scale_f16_aligned(code));
                            W[2 * sg] = w.x;
                            W[2 * sg + 1] = w.y;
                        } else if (p.q_mode == FP4Q_ROUND_STOCHASTIC) {
                            round_segment<FP4Q_ROUND_STOCHASTIC>(raw + 8 * sg, inv_scale(code), R, W + 2 * sg);
                        } else {
                            round_segment<FP4Q_ROUND_NEAREST>(raw + 8 * sg, inv_scale(code), R, W + 2 * sg);
                        }
                    }
                    if (lane == 0) p.q_scale[(int64_t)(row0_blk >> 5) * p.q_ld_s + (col0 >> 5)] = (uint8_t)code;
                    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(stg_rm + (((uint32_t)j ^ swz) << 4)), "r"(W[0]), "r"(W[1]),
                                 "r"(W[2]), "r"(W[3]) : "memory");
                }
                if (any && p.q_t != nullptr) {
                    __syncwarp();
                    transpose_staged_codes(smem_u32(stg), 0, lane);
                    if (t.c_col0 + 128 * half + 64 < p.N) transpose_staged_codes(smem_u32(stg), 2, lane);
                }
                if (any) {
                    // both payloads leave by TMA stores, which clip at the tensors' edges (rows past T, columns past N)
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) {
                        tma_store_2d(&tmC, (t.c_col0 + 128 * half) >> 1, row0_blk, smem_u32(stg));
                        if (p.q_t != nullptr) tma_store_2d(&tmD, row0_blk >> 1, t.c_col0 + 128 * half, smem_u32(stg) + 2048);
                        bulk_commit();
                    }
                }
            } else if (Cfg<KIND, CTAS>::kTmaStores) {
                // 128 bytes per row and round - 64 BF16 or 32 FP32 columns - go
                // through this warp's staging rows and leave by a TMA store, which clips rows and columns past the
                // output's edge.  With accumulation the store is the TMA's FP32 add-reduction.
                if (t.m_valid > 32 * quarter) {
                    // A round waits for the one before it to have left the staging rows, about 1000 cycles.  The CTA's last tile, whose output
                    // nothing runs beside, takes the ring's stages instead, a place for every round: no load or MMA will use them again.
                    // With this, pairs whose CTAs part after the last accumulator is read, and stores that are only waited for until
                    // they have read shared memory, us: 2048 x 2048 x 2048 9.3 / 9.4 / 10.9 -> 8.3 / 8.5 / 9.7, weight gradients of 128 x 256 x 256 8.2 -> 6.9,
                    // 8192 x 2048 x 2048 18.3 -> 17.0.  (One fence and one thread's four stores behind the last round: 8.4 -> 9.0.)
                    static_assert(Cfg<KIND, CTAS>::kSmemOperands >= 8 * 4 * kStagingWarpBytes, "the last tile's rounds fit in the ring");
                    const uint32_t stg0 = last ? smem_u32(smem) + (warp - 4) * 4 * kStagingWarpBytes : smem_u32(smem_staging) + (warp - 4) * kStagingWarpBytes;
                    const uint32_t swz = (uint32_t)(lane & 7);
                    const int32_t y = t.c_row0 + 32 * quarter;
                    const int n_rows = t.m_valid - 32 * quarter;
                    if (p.out_f32) {
#pragma unroll
                        for (int h = 0; h < 4; h++) {
                            const int col_in_tile = 128 * half + 32 * h;
                            const uint32_t stg = last ? stg0 + h * kStagingWarpBytes : stg0;
                            if (col_in_tile < t.n_valid)
                                stage_and_store<GROUPS == GROUPS_CUT, EPI == EPI_TAIL>(p, &tmC, v[h], stg + lane * 128, swz, stg, t.c_col0 + col_in_tile, y, p.accumulate ? 2 : 1, lane, last, n_rows);
                        }
                    } else {
#pragma unroll
                        for (int h = 0; h < 2; h++) {
                            const int col_in_tile = 128 * half + 64 * h;
                            if (col_in_tile >= t.n_valid) continue;
                            uint32_t w[32];
#pragma unroll
                            for (int e = 0; e < 32; e++) {
                                const __nv_bfloat162 b = __floats2bfloat162_rn(__uint_as_float(v[2 * h + (e >> 4)][(2 * e) & 31]),
                                                                               __uint_as_float(v[2 * h + (e >> 4)][(2 * e + 1) & 31]));
                                w[e] = *reinterpret_cast<const uint32_t *>(&b);
                            }
                            const uint32_t stg = last ? stg0 + h * kStagingWarpBytes : stg0;
                            stage_and_store<GROUPS == GROUPS_CUT, EPI == EPI_TAIL>(p, &tmC, w, stg + lane * 128, swz, stg, t.c_col0 + col_in_tile, y, 0, lane, last, n_rows);
                        }
                    }
                    // The last box of a row is the one that lies in the staging rows now (or in its own place of the ring).
                    const uint32_t tail = (uint32_t)p.tail_col - (uint32_t)(t.c_col0 + 128 * half);
                    if (EPI == EPI_TAIL && tail < 128u && row_ok && !(GROUPS == GROUPS_CUT && n_rows < 32)) {
                        const uint32_t byte = tail << (p.out_f32 ? 2 : 1);
                        store_row_tail(p, row, stg0 + (last ? byte >> 7 : 0u) * kStagingWarpBytes + lane * 128 + (((byte >> 4 & 7u) ^ swz) << 4));
                    }
                }
            } else if (row_ok) {
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const int col_in_tile = 128 * half + 32 * j;
                    store_row_chunk(p, row, t.c_col0 + col_in_tile, t.n_valid - col_in_tile, v[j]);
                }
            }
            TRACE_ADD(c_store, tt);
        }
        if (!arrived) {   // the last tile was not computed, or has no contraction
            tcgen05_fence_before();
            __syncwarp();
            if (CTAS == 2) cluster_arrive();
            else asm volatile("bar.arrive 14, 288;" ::: "memory");
        }
        // The stores have read their staging rows; what they write is there when the grid has completed.
        if ((Cfg<KIND, CTAS>::kTmaStores || EPI == EPI_QUANT) && lane == 0) bulk_wait_read_all();
        if (warp == 4 && lane == 0) { TRACE_OUT(p, 10, c_wait); TRACE_OUT(p, 11, c_ld); TRACE_OUT(p, 12, c_store); }
        __syncwarp();
    }

    // Shared memory and tensor memory of a pair stay until both CTAs have done with them.  Epilogue warps have arrived already.
    if (CTAS == 2) {
        if (warp < 4) {
            __syncwarp();
            cluster_arrive();
        }
        cluster_wait();
    } else if (warp == 1) {
        asm volatile("bar.sync 14, 288;" ::: "memory");
    }
    if (warp == 1) {
        tcgen05_fence_after();
        const uint32_t tmem_base = *tmem_base_slot;
        if (CTAS == 1)
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
        else
            asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
    }
}

// ---------------------------------------------------------------------------------------- host side

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_tiled_fn()
{
    static const EncodeTiledFn fn = [] {   // several threads may make their first product at the same time: all but one wait
        void *ptr = nullptr;
        cudaDriverEntryPointQueryResult qres;
        const bool found = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess && qres == cudaDriverEntryPointSuccess;
        return found ? reinterpret_cast<EncodeTiledFn>(ptr) : nullptr;
    }();
    return fn;
}
// The encoder wants a context on the calling thread, which the runtime binds with the thread's first call that needs one; a thread whose first
// call is a product has made none.
static bool encode_tiled(CUtensorMap *map, CUtensorMapDataType type, int rank, void *base, const cuuint64_t *dims, const cuuint64_t *strides,
                         const cuuint32_t *box, CUtensorMapSwizzle swizzle, CUtensorMapL2promotion promotion)
{
    const EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    const cuuint32_t estr[5] = {1u, 1u, 1u, 1u, 1u};
    auto encode = [&] {
        return fn(map, type, (cuuint32_t)rank, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle, promotion, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    };
    CUresult r = encode();
    int dev;
    if (r == CUDA_ERROR_INVALID_CONTEXT && cudaGetDevice(&dev) == cudaSuccess && cudaSetDevice(dev) == cudaSuccess) r = encode();
    return r == CUDA_SUCCESS;
}

// Operand tile map: a [rows, row_bytes] byte matrix with pitch ld_bytes, box = 128 B x box_rows, 128B swizzle.
static bool make_operand_map(CUtensorMap *map, const void *base, int64_t rows, int64_t row_bytes, int64_t ld_bytes,
                             int box_rows)
{
    const cuuint64_t dims[2] = {(cuuint64_t)row_bytes, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)ld_bytes};
    const cuuint32_t box[2] = {128u, (cuuint32_t)box_rows};
    return encode_tiled(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void *>(base), dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B);
}

// Output map for the TMA stores: box = 128 bytes x 32 rows, 128-byte swizzle.  Plain stores address the
// output as bytes; accumulation uses the TMA add-reduction, which needs the element type (FP32, 32 per box row).  cols: where
// rows must not be filled up to 16 bytes, whole pieces of these (store_row_tail has the rest), or none, and then no store uses the map.
static bool make_output_map(CUtensorMap *map, void *base, int64_t rows, int64_t cols, int64_t ld, bool f32, bool reduce)
{
    const int64_t esize = f32 ? 4 : 2;
    const cuuint64_t row_bytes = (cuuint64_t)(cols > 0 ? cols * esize : 16);
    const cuuint64_t dims[2] = {reduce ? row_bytes / 4 : row_bytes, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)(ld * esize)};
    const cuuint32_t box[2] = {reduce ? 32u : 128u, 32u};
    return encode_tiled(map, reduce ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, base, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B,
                        CU_TENSOR_MAP_L2_PROMOTION_NONE);
}

// Plain byte matrix [rows, row_bytes] with pitch ld_bytes as a store target.
static bool make_byte_map(CUtensorMap *map, void *base, int64_t rows, int64_t row_bytes, int64_t ld_bytes, int box_bytes,
                          int box_rows, CUtensorMapSwizzle swizzle)
{
    const cuuint64_t dims[2] = {(cuuint64_t)row_bytes, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)ld_bytes};
    const cuuint32_t box[2] = {(cuuint32_t)box_bytes, (cuuint32_t)box_rows};
    return encode_tiled(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, base, dims, strides, box, swizzle, CU_TENSOR_MAP_L2_PROMOTION_NONE);
}

struct Operand {
    const uint8_t *payload;
    int64_t rows, row_bytes, ld_bytes;
    ScaleView sf;
};

constexpr int kMaxDevices = 64;   // per-device host state (attributes set, SM counts, static workspace address); threads that find it unset all set the same

static int current_device()
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return -1;
    return dev;
}

static int sm_count(int dev)
{
    static std::atomic<int> known[kMaxDevices];
    int n = known[dev].load(std::memory_order_relaxed);
    if (n == 0) {
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 148;
        known[dev].store(n, std::memory_order_relaxed);
    }
    return n;
}

// Most row tiles that pairs can have with grouped rows on multiples of 128: a group with an odd number has one alone.
static int64_t paired_tiles(const GemmParams &p)
{
    const int64_t rows = ceil_div(p.M, BM);
    return (rows + (p.n_groups < rows ? p.n_groups : rows)) / 2;
}

template <int KIND, int CTAS, int EPI, bool WATCH, int GROUPS = GROUPS_NONE>
static fp4q_status launch_gemm_impl(const Operand &A, const Operand &B, GemmParams &p, void *stream)
{
    CUtensorMap tmA, tmB, tmC;
    if (GROUPS == GROUPS_NONE && p.mode != MODE_DENSE) return FP4Q_ERR_UNSUPPORTED;
    const int64_t out_rows = p.mode == MODE_GROUPED_K ? (int64_t)p.n_groups * p.M : p.M;
    if (!make_operand_map(&tmA, A.payload, A.rows, A.row_bytes, A.ld_bytes, BM)) return FP4Q_ERR_CUDA;
    CUtensorMap tmD = tmA;   // second output map: only the quantizing epilogue has one
    if (EPI == EPI_QUANT) {
        // row-major payload [T, ceil32(N)/2] bytes, box 64 B x 32 rows (64-byte swizzle); transposed payload
        // [N, ceil32(T)/2] bytes, box 16 B x 128 rows
        if (!make_byte_map(&tmC, p.q_rm, p.M, round_up(p.N, 32) / 2, p.q_ld_rm, 64, 32, CU_TENSOR_MAP_SWIZZLE_64B)) return FP4Q_ERR_CUDA;
        if (p.q_t && !make_byte_map(&tmD, p.q_t, p.N, round_up(p.M, 32) / 2, p.q_ld_t, 16, 128, CU_TENSOR_MAP_SWIZZLE_NONE)) return FP4Q_ERR_CUDA;
    } else {
        const int32_t whole = EPI == EPI_TAIL ? p.N / (p.out_f32 ? 4 : 8) * (p.out_f32 ? 4 : 8) : p.N;   // columns in whole pieces of 16 bytes
        p.tail_col = whole < p.N ? whole : INT32_MIN;
        if (!make_output_map(&tmC, p.C, out_rows, whole, p.ldc, p.out_f32 != 0, p.accumulate != 0)) return FP4Q_ERR_CUDA;
    }
    if (!make_operand_map(&tmB, B.payload, B.rows, B.row_bytes, B.ld_bytes, Cfg<KIND, CTAS>::kBRows)) return FP4Q_ERR_CUDA;
    p.ctas = CTAS;
    p.m_tiles = (int32_t)ceil_div(p.M, BM * CTAS);
    p.n_tile_total = p.m_tiles * p.n_tiles * (p.mode == MODE_GROUPED_K ? p.n_groups : 1);
    p.raster_m = p.mode != MODE_GROUPED_K ? (p.m_tiles < kRasterM ? p.m_tiles : kRasterM) : p.m_tiles;
    if (p.mode == MODE_PAIRED_ROWS) {   // as many as there can be
        p.m_tiles = (int32_t)paired_tiles(p);
        p.n_tile_total = p.m_tiles * p.n_tiles;
        p.raster_m = kRasterM;
    }
#ifdef FP4Q_TRACE
    if (const char *g = getenv("FP4Q_DEBUG_RASTER")) { p.raster_m = atoi(g); if (p.raster_m > p.m_tiles) p.raster_m = p.m_tiles; }
#endif

    const int32_t tail = p.m_tiles % p.raster_m;
    p.by_problem = divisor(p.m_tiles * p.n_tiles);
    p.by_group = divisor(p.raster_m * p.n_tiles);
    p.by_raster = divisor(p.raster_m);
    p.by_tail = divisor(tail != 0 ? tail : 1);
    const int dev = current_device();
    if (dev < 0) return FP4Q_ERR_CUDA;
    static std::atomic<bool> attr_set[kMaxDevices];   // the attribute is a property of (kernel, device): one flag per device and instantiation
    if (!attr_set[dev].load(std::memory_order_relaxed)) {
        if (cudaFuncSetAttribute(gemm_block_scaled_kernel<KIND, CTAS, EPI, WATCH, GROUPS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 Cfg<KIND, CTAS>::kSmemBytes) != cudaSuccess)
            return FP4Q_ERR_CUDA;
        attr_set[dev].store(true, std::memory_order_relaxed);
    }
    int slots = sm_count(dev) / CTAS;   // CTAs or pairs that run at a time
#ifdef FP4Q_TRACE
    if (const char *g = getenv("FP4Q_DEBUG_SLOTS")) slots = atoi(g);   // development only: use fewer SMs
#endif
    const int grid = CTAS * (p.n_tile_total < slots ? p.n_tile_total : slots);
    constexpr int kElems = kind_fp4(KIND) ? 256 : 128;
    const int64_t tile_stages = ceil_div(p.K, kElems);   // a grouped contraction: of one output tile over all groups
    const int64_t n_stages = p.mode == MODE_GROUPED_K ? (int64_t)p.m_tiles * p.n_tiles * (tile_stages + p.n_groups) : p.n_tile_total * tile_stages;
    // Longest first costs every CTA a sort before its first load, quadratic in the groups (1.8 us at 128, 4.4 us at 256), and runs
    // the groups that are bound by MMAs apart from those that are bound by output.  It pays for groups of two stages and more
    // on average in products that last: at least half a stage a slot for every group.  us, as they come and longest first,
    // Zipf lengths: 139520 rows x 768 x 2048 in 128 groups 244-248 / 239, 32768 in 64 103 / 98, 16384 in 32 55-57 / 53;
    // below the line 65536 x 256 x 512 in 128 38 / 41, 131072 x 256 x 512 in 256 65-69 / 76, 4096 x 128 x 256 in 256 12 / 16.
    p.sort_groups = p.mode == MODE_GROUPED_K && p.n_groups <= kMaxGroupsSorted && p.K >= 512 * (int64_t)p.n_groups &&
                    2 * n_stages >= (int64_t)p.n_groups * slots;
    p.warps_meet = p.mode == MODE_GROUPED_K && p.K < 512 * (int64_t)p.n_groups;   // two stages a group on average
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = Cfg<KIND, CTAS>::kSmemBytes;
    cfg.stream = static_cast<cudaStream_t>(stream);
    // Short products start beside the end of a quantizer before them: up to 48 stages, about 25 us, per CTA or pair.  Passes of
    // quantizers and products, without and with, us: 2048 x 4096 x 4096 (28 stages) 102.8 / 97.6, 1D activations 2048 x 4096 x 4096
    // 32.5 / 29.3; nothing changes from 4096 x 4096 x 4096 (55 stages) on, except that CTAs of long products are placed as SMs
    // fall free instead of in order, and tiles that share operands end up far apart (all three products of 16384 x 11008 x 4096
    // with their quantizers 1039 / 1084).  In a captured graph the one-CTA products of the smallest layers lose (4 experts of 512
    // tokens in all 31.7 / 33.4, 128 x 256 x 256 31.0 / 31.9), so only those on pairs take part there.
    cudaLaunchAttribute attr[2];
    cfg.attrs = attr;
    if (CTAS == 2) {
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = CTAS;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.numAttrs = 1;
    }
    if (n_stages <= kShortStages * (int64_t)slots && !(CTAS == 1 && capturing(cfg.stream))) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
    }
    return launched(cudaLaunchKernelEx(&cfg, gemm_block_scaled_kernel<KIND, CTAS, EPI, WATCH, GROUPS>, tmA, tmB, tmC, tmD, p));
}

// Whether a view's words can be loaded with offsets of 32 bits: a unit reads less than 16 pitches past the last row's start.
static ScaleView scale_view(ScaleView v)
{
    const bool tr = v.stride_kb != 1;
    const int64_t pitch = tr ? v.stride_kb : v.stride_row, n = tr ? v.n_kb : v.n_row;
    v.words = aligned(v.ptr, 4) && pitch % 4 == 0 && pitch >= 0 && pitch <= 0xFFFFFFFFll / (n + 16);
    return v;
}

// Argument checks common to every product: everything that can be refused is refused here, before any work is enqueued.
static fp4q_status check_gemm_args(const Operand &A, const Operand &B, const GemmParams &p, const void *ws, size_t ws_bytes)
{
    if (!ws || ws_bytes < sizeof(Workspace)) return FP4Q_ERR_WORKSPACE;
    if (!aligned(ws, 256)) return FP4Q_ERR_ALIGN;
    if (!aligned(A.payload, 16) || !aligned(B.payload, 16) || A.ld_bytes % 16 || B.ld_bytes % 16) return FP4Q_ERR_ALIGN;
    const size_t esize = p.out_f32 ? 4 : 2;
    if (!aligned(p.C, 16) || (p.ldc * esize) % 16) return FP4Q_ERR_ALIGN;
    return FP4Q_OK;
}

// Whether grouped rows on multiples of 128 run on pairs.  A tile of a pair takes 0.83-0.9 of the time of one CTA's that does half as much (three
// stages 2.5 / 3.0 us, eight 4.75 / 5.4; nothing is gained with one or two), the table of pairs 0.7 us, and a group with an odd number of
// row tiles, every other one on average, a tile for half the work.  So the rounds of tiles are compared, 9 to 10.  us, one CTA and pairs,
// forward / input gradient: 272 row tiles in 32 groups, 768 x 2048 39.0 / 46.2 -> 34.5 / 44.7, 263 in 16 37.5 / 43.7 -> 32.5 / 41.2, 260 in 8, 1408 x 1024
// 38.4 / 36.9 -> 33.5 / 32.1, 36 in 8, 1408 x 1440 16.1 / 14.1 -> 13.9 / 13.1; left on one CTA: 327 in 128, 768 x 2048 50.0 / 62.8 and 49.9 / 64.4, 145 in 32,
// 768 x 1700 21.3 / 24.6 and 22.0 / 26.8, 257 in 4, 512 x 512 13.3 / 13.2 and 14.3 / 14.2.
static bool pairs_pay(const GemmParams &p)
{
    const int64_t rows = ceil_div(p.M, BM), groups = p.n_groups < rows ? p.n_groups : rows;
    if (p.K <= 512 || p.n_groups > kMaxGroupsPaired || paired_tiles(p) > kMaxGroupsShared + 1) return false;
    const int dev = current_device();
    const int64_t sms = dev < 0 ? 148 : sm_count(dev), pairs = (2 * rows + groups + 3) / 4;
    return 9 * ceil_div(pairs * p.n_tiles, sms / 2) + 2 <= 10 * ceil_div(rows * p.n_tiles, sms);
}

// With the epilogue that the output's rows ask for.
template <int KIND, int CTAS, bool WATCH, int GROUPS = GROUPS_NONE>
static fp4q_status launch_store(const Operand &A, const Operand &B, GemmParams &p, void *stream)
{
    if constexpr (Cfg<KIND, CTAS>::kTmaStores)
        if (GROUPS == GROUPS_CUT || (!p.padded && p.N % (p.out_f32 ? 4 : 8) != 0)) return launch_gemm_impl<KIND, CTAS, EPI_TAIL, WATCH, GROUPS>(A, B, p, stream);
    if constexpr (GROUPS == GROUPS_CUT) return FP4Q_ERR_UNSUPPORTED;
    else return launch_gemm_impl<KIND, CTAS, EPI_STORE, WATCH, GROUPS>(A, B, p, stream);
}

template <int KIND>
static fp4q_status launch_gemm(const Operand &A, const Operand &B, GemmParams &p, void *ws, size_t ws_bytes, void *stream)
{
    if (fp4q_status s = check_gemm_args(A, B, p, ws, ws_bytes)) return s;
    const size_t esize = p.out_f32 ? 4 : 2;
    if (p.n_tile_total <= 0) return FP4Q_OK;
    p.wide_stores = aligned(p.C, 32) && (p.ldc * esize) % 32 == 0;
    p.sfa = scale_view(A.sf);
    p.sfb = scale_view(B.sf);
    p.status = reinterpret_cast<uint32_t *>(ws);
    // Dense products (FP4 and MXFP8) with more than one row tile run as cta_group::2 pairs: 256x256 tiles, each CTA
    // loads half of the B rows; so does the grouped weight gradient, whose groups cut the contraction axis, not the
    // output rows of a tile, and grouped rows where every group starts on a multiple of 256 or where paired rows pay.
    // FP4Q_CTA_PAIRS=0 in the environment (read once, before the first GEMM call) selects the one-CTA kernel instead.
    static const bool use_pairs = [] { const char *e = getenv("FP4Q_CTA_PAIRS"); return !(e && e[0] == '0'); }();
    // The watcher pays in dense FP4 and MXFP8 products on pairs that last: with and without, 16384 x 4096 x 4096 FP4 102.6 / 103.5 / 98.0 and
    // 103.9 / 104.5 / 101.3 us, MXFP8 199.7 and 207.0.  FP4 products of up to 48 stages a pair are faster without it (2048 x 2048 x 2048 8.5 / 8.6 / 9.6
    // and 8.1 / 8.3 / 9.3, 512 x 1024 x 1024 6.8 / 6.6 / 7.2 and 6.5 / 6.3 / 7.0, 3000 x 3000 x 3000 16.8 / 16.9 / 18.5 and 16.5 / 16.7 / 18.2; from 55 stages on
    // between -1.5 and +1.4 %, from 80 on slower), MXFP8 ones are level.  Everything else has none: the short contractions of grouped
    // products (expert weight gradients 222 and 225 us without, 228 and 230 us with), the quantizing epilogue, whose warps it competes
    // with (113 and 116 us), and the per-row FP4 kinds, where its warp builds scale images instead.
    if constexpr (KIND == KIND_MXF4) {
        if (p.mode != MODE_DENSE) {
            if (use_pairs && p.M > BM && p.mode == MODE_GROUPED_ROWS && !p.rows_pair_aligned && pairs_pay(p)) p.mode = MODE_PAIRED_ROWS;
            if (p.mode == MODE_GROUPED_K && p.M % 32 != 0) {
                if (use_pairs && p.M > BM) return launch_store<KIND, 2, false, GROUPS_CUT>(A, B, p, stream);
                return launch_store<KIND, 1, false, GROUPS_CUT>(A, B, p, stream);
            }
            const bool pairs = p.mode == MODE_GROUPED_K || p.mode == MODE_PAIRED_ROWS || p.rows_pair_aligned;
            if (use_pairs && pairs && p.M > BM) return launch_store<KIND, 2, false, GROUPS_PAIRED>(A, B, p, stream);
            return launch_store<KIND, 1, false, GROUPS_ANY>(A, B, p, stream);
        }
    }
    if (use_pairs && p.M > BM) {
        if constexpr (KIND == KIND_MXF4) {
            const int dev = current_device();
            const int64_t pairs = dev < 0 ? 74 : sm_count(dev) / 2;
            if (ceil_div(p.M, 2 * BM) * p.n_tiles * ceil_div(p.K, 256) <= kShortStages * pairs) return launch_store<KIND, 2, false>(A, B, p, stream);
        }
        return launch_store<KIND, 2, KIND == KIND_MXF4 || KIND == KIND_MXF8>(A, B, p, stream);
    }
    return launch_store<KIND, 1, false>(A, B, p, stream);
}

static bool tensor_ok(const fp4q_tensor *t) { return t && t->rows >= 0 && t->cols >= 0; }

static fp4q_status check_groups(const fp4q_groups *g)
{
    if (!g) return FP4Q_OK;
    if (g->n_groups <= 0) return FP4Q_ERR_SHAPE;
    if (g->row_alignment != 0 && g->row_alignment != 128 && g->row_alignment != 256) return FP4Q_ERR_UNSUPPORTED;
    if (!g->row_offsets) return FP4Q_ERR_NULL;
    return FP4Q_OK;
}

// Row-major payload of a tensor [rows, cols] as an operand whose rows are the tensor's rows.
static Operand operand_rm(const fp4q_tensor *t)
{
    Operand o;
    o.payload = t->q_rm;
    o.rows = t->rows;
    o.row_bytes = round_up(t->cols, 32) / 2;
    o.ld_bytes = t->ld_rm;
    o.sf = ScaleView{t->scale, t->ld_s, 1, (int32_t)ceil_div(t->rows, 32), (int32_t)ceil_div(t->cols, 32)};
    return o;
}
// Transposed payload: operand rows are the tensor's columns, contraction runs over the tensor's rows.
static Operand operand_t(const fp4q_tensor *t)
{
    Operand o;
    o.payload = t->q_t;
    o.rows = t->cols;
    o.row_bytes = round_up(t->rows, 32) / 2;
    o.ld_bytes = t->ld_t;
    o.sf = ScaleView{t->scale, 1, t->ld_s, (int32_t)ceil_div(t->cols, 32), (int32_t)ceil_div(t->rows, 32)};
    return o;
}

static bool out_type_ok(fp4q_out dt)
{
    const int type = (int)dt & ~(int)FP4Q_OUT_PADDED;
    return type == FP4Q_OUT_BF16 || type == FP4Q_OUT_F32;
}
static bool out_type_f32(fp4q_out dt) { return ((int)dt & ~(int)FP4Q_OUT_PADDED) == FP4Q_OUT_F32; }
static void set_out_type(GemmParams &p, fp4q_out dt)
{
    p.out_f32 = out_type_f32(dt);
    p.padded = ((int)dt & (int)FP4Q_OUT_PADDED) != 0;
}

static void dense_tiles(GemmParams &p)
{
    p.m_tiles = (int32_t)ceil_div(p.M, BM);
    p.n_tiles = (int32_t)ceil_div(p.N, BN);
    p.n_tile_total = p.m_tiles * p.n_tiles;
}

}  // namespace fp4q

using namespace fp4q;

static const int64_t kMaxDim = 0x7FFFFFFF - 4096;

// The forward product's arguments turned into kernel parameters.  *noop is set when there is nothing to compute.
static fp4q_status prepare_fwd(const fp4q_tensor *X, const fp4q_tensor *W, void *Y, int64_t ldy, fp4q_out dt, const fp4q_groups *g,
                               GemmParams &p, bool *noop)
{
    *noop = false;
    if (!tensor_ok(X) || !tensor_ok(W)) return X && W ? FP4Q_ERR_SHAPE : FP4Q_ERR_NULL;
    if (fp4q_status s = check_groups(g)) return s;
    if (!out_type_ok(dt)) return FP4Q_ERR_UNSUPPORTED;
    if (X->cols != W->cols) return FP4Q_ERR_SHAPE;
    const int64_t T = X->rows, K = X->cols;
    const int64_t N = g ? W->rows / g->n_groups : W->rows;
    if (g && (W->rows % g->n_groups || N % 32)) return FP4Q_ERR_SHAPE;   // expert blocks must start on a 32-row tile
    if (T > kMaxDim || N > kMaxDim || K > kMaxDim || W->rows > kMaxDim) return FP4Q_ERR_UNSUPPORTED;
    if (T == 0 || N == 0) { *noop = true; return FP4Q_OK; }
    if (!Y || !X->q_rm || !W->q_rm || !X->scale || !W->scale) return FP4Q_ERR_NULL;
    if (ldy < N) return FP4Q_ERR_SHAPE;
    p = GemmParams{};
    p.C = Y; p.ldc = ldy; p.M = (int32_t)T; p.N = (int32_t)N; p.K = (int32_t)K;
    set_out_type(p, dt); p.accumulate = 0;
    dense_tiles(p);
    if (g) {
        p.mode = MODE_GROUPED_ROWS; p.n_groups = g->n_groups; p.row_offsets = g->row_offsets;
        p.rows_pair_aligned = g->row_alignment == 256;
        p.b_rows_per_group = (int32_t)N; p.b_k_per_group = 0;
    }
    return FP4Q_OK;
}

extern "C" fp4q_status fp4q_gemm_fwd(const fp4q_tensor *X, const fp4q_tensor *W, void *Y, int64_t ldy, fp4q_out dt,
                                     const fp4q_groups *g, void *ws, size_t ws_bytes, void *stream)
{
    GemmParams p;
    bool noop;
    if (fp4q_status s = prepare_fwd(X, W, Y, ldy, dt, g, p, &noop)) return s;
    if (noop) return FP4Q_OK;
    return launch_gemm<KIND_MXF4>(operand_rm(X), operand_rm(W), p, ws, ws_bytes, stream);
}

// C[M, N] = A B^T with the output leaving as the 2D-block FP4 tensor Cq (dense, pair kernel).
// Grouped form (g != NULL): b_rows_per_group / b_k_per_group as in the plain grouped products; the pair tiles need
// every group to start on a multiple of 256 rows.
static fp4q_status launch_gemm_quantized(const Operand &A, const Operand &B, int64_t M, int64_t N, int64_t K, const fp4q_tensor *Cq,
                                         fp4q_round mode, uint64_t seed, uint32_t tensor_id, const fp4q_groups *g,
                                         int32_t b_rows_per_group, int32_t b_k_per_group, void *ws, size_t ws_bytes, void *stream)
{
    if (mode != FP4Q_ROUND_NEAREST && mode != FP4Q_ROUND_STOCHASTIC) return FP4Q_ERR_UNSUPPORTED;
    if (fp4q_status s = check_groups(g)) return s;
    if (g && g->row_alignment != 256) return FP4Q_ERR_UNSUPPORTED;
    if (Cq->rows != M || Cq->cols != N) return FP4Q_ERR_SHAPE;
    if (M > kMaxDim || N > kMaxDim || K > kMaxDim) return FP4Q_ERR_UNSUPPORTED;
    if (N % 16 != 0) return FP4Q_ERR_UNSUPPORTED;   // one Philox block per 16-element row segment of the output
    if (M == 0 || N == 0) return FP4Q_OK;
    if (!A.payload || !B.payload || !A.sf.ptr || !B.sf.ptr || !Cq->q_rm || !Cq->scale) return FP4Q_ERR_NULL;
    if (Cq->ld_rm < round_up(N, 32) / 2 || Cq->ld_s < ceil_div(N, 32)) return FP4Q_ERR_SHAPE;
    if (Cq->q_t && Cq->ld_t < round_up(M, 32) / 2) return FP4Q_ERR_SHAPE;
    if (!aligned(Cq->q_rm, 16) || Cq->ld_rm % 16 != 0) return FP4Q_ERR_ALIGN;
    if (Cq->q_t && (!aligned(Cq->q_t, 16) || Cq->ld_t % 16 != 0)) return FP4Q_ERR_ALIGN;
    if (!ws || ws_bytes < sizeof(Workspace)) return FP4Q_ERR_WORKSPACE;
    if (!aligned(ws, 256)) return FP4Q_ERR_ALIGN;
    if (!aligned(A.payload, 16) || !aligned(B.payload, 16) || A.ld_bytes % 16 || B.ld_bytes % 16) return FP4Q_ERR_ALIGN;
    GemmParams p = {};
    p.M = (int32_t)M; p.N = (int32_t)N; p.K = (int32_t)K;
    dense_tiles(p);
    p.sfa = scale_view(A.sf); p.sfb = scale_view(B.sf);
    p.status = reinterpret_cast<uint32_t *>(ws);
    p.q_rm = Cq->q_rm; p.q_ld_rm = Cq->ld_rm;
    p.q_t = Cq->q_t; p.q_ld_t = Cq->ld_t;
    p.q_scale = Cq->scale; p.q_ld_s = Cq->ld_s;
    p.q_mode = (int32_t)mode; p.q_tensor_id = tensor_id;
    philox_round_keys(seed, p.q_keys);
    if (g) {
        p.mode = MODE_GROUPED_ROWS; p.n_groups = g->n_groups; p.row_offsets = g->row_offsets;
        p.rows_pair_aligned = 1;
        p.b_rows_per_group = b_rows_per_group; p.b_k_per_group = b_k_per_group;
    }
    if (g) return launch_gemm_impl<KIND_MXF4, 2, EPI_QUANT, false, GROUPS_ANY>(A, B, p, stream);
    return launch_gemm_impl<KIND_MXF4, 2, EPI_QUANT, false>(A, B, p, stream);
}

extern "C" fp4q_status fp4q_gemm_fwd_quantized(const fp4q_tensor *X, const fp4q_tensor *W, const fp4q_tensor *Yq, fp4q_round mode,
                                               uint64_t seed, uint32_t tensor_id, const fp4q_groups *g, void *ws, size_t ws_bytes,
                                               void *stream)
{
    if (!tensor_ok(X) || !tensor_ok(W) || !tensor_ok(Yq)) return X && W && Yq ? FP4Q_ERR_SHAPE : FP4Q_ERR_NULL;
    if (X->cols != W->cols) return FP4Q_ERR_SHAPE;
    if (g && g->n_groups > 0 && (W->rows % g->n_groups || (W->rows / g->n_groups) % 32)) return FP4Q_ERR_SHAPE;
    const int64_t N = g && g->n_groups > 0 ? W->rows / g->n_groups : W->rows;
    return launch_gemm_quantized(operand_rm(X), operand_rm(W), X->rows, N, X->cols, Yq, mode, seed, tensor_id, g, (int32_t)N, 0, ws,
                                 ws_bytes, stream);
}

extern "C" fp4q_status fp4q_gemm_dgrad_quantized(const fp4q_tensor *dY, const fp4q_tensor *W, const fp4q_tensor *dXq, fp4q_round mode,
                                                 uint64_t seed, uint32_t tensor_id, const fp4q_groups *g, void *ws, size_t ws_bytes,
                                                 void *stream)
{
    if (!tensor_ok(dY) || !tensor_ok(W) || !tensor_ok(dXq)) return dY && W && dXq ? FP4Q_ERR_SHAPE : FP4Q_ERR_NULL;
    const int64_t N = dY->cols;
    if (g && g->n_groups > 0 ? (W->rows != N * g->n_groups || N % 64) : (W->rows != N)) return FP4Q_ERR_SHAPE;
    return launch_gemm_quantized(operand_rm(dY), operand_t(W), dY->rows, W->cols, N, dXq, mode, seed, tensor_id, g, 0, (int32_t)N, ws,
                                 ws_bytes, stream);
}

extern "C" fp4q_status fp4q_gemm_dgrad(const fp4q_tensor *dY, const fp4q_tensor *W, void *dX, int64_t ldx, fp4q_out dt,
                                       const fp4q_groups *g, void *ws, size_t ws_bytes, void *stream)
{
    if (!tensor_ok(dY) || !tensor_ok(W)) return dY && W ? FP4Q_ERR_SHAPE : FP4Q_ERR_NULL;
    if (fp4q_status s = check_groups(g)) return s;
    if (!out_type_ok(dt)) return FP4Q_ERR_UNSUPPORTED;
    const int64_t T = dY->rows, N = dY->cols, K = W->cols;
    if (g ? (W->rows != N * g->n_groups) : (W->rows != N)) return FP4Q_ERR_SHAPE;
    if (g && N % 64) return FP4Q_ERR_UNSUPPORTED;   // a group's contraction range must end on an MMA boundary
    if (T > kMaxDim || N > kMaxDim || K > kMaxDim || W->rows > kMaxDim) return FP4Q_ERR_UNSUPPORTED;
    if (T == 0 || K == 0) return FP4Q_OK;
    if (!dX || !dY->q_rm || !W->q_t || !dY->scale || !W->scale) return FP4Q_ERR_NULL;
    if (ldx < K) return FP4Q_ERR_SHAPE;
    GemmParams p = {};
    p.C = dX; p.ldc = ldx; p.M = (int32_t)T; p.N = (int32_t)K; p.K = (int32_t)N;
    set_out_type(p, dt); p.accumulate = 0;
    dense_tiles(p);
    if (g) {
        p.mode = MODE_GROUPED_ROWS; p.n_groups = g->n_groups; p.row_offsets = g->row_offsets;
        p.rows_pair_aligned = g->row_alignment == 256;
        p.b_rows_per_group = 0; p.b_k_per_group = (int32_t)N;
    }
    return launch_gemm<KIND_MXF4>(operand_rm(dY), operand_t(W), p, ws, ws_bytes, stream);
}

extern "C" fp4q_status fp4q_gemm_wgrad(const fp4q_tensor *dY, const fp4q_tensor *X, void *dW, int64_t ldw, fp4q_out dt,
                                       int accumulate, const fp4q_groups *g, void *ws, size_t ws_bytes, void *stream)
{
    if (!tensor_ok(dY) || !tensor_ok(X)) return dY && X ? FP4Q_ERR_SHAPE : FP4Q_ERR_NULL;
    if (fp4q_status s = check_groups(g)) return s;
    if (!out_type_ok(dt)) return FP4Q_ERR_UNSUPPORTED;
    if (accumulate && !out_type_f32(dt)) return FP4Q_ERR_UNSUPPORTED;
    if (dY->rows != X->rows) return FP4Q_ERR_SHAPE;
    const int64_t T = dY->rows, N = dY->cols, K = X->cols;
    if (T > kMaxDim || N > kMaxDim || K > kMaxDim) return FP4Q_ERR_UNSUPPORTED;
    if (g && N * g->n_groups > kMaxDim) return FP4Q_ERR_UNSUPPORTED;
    if (N == 0 || K == 0) return FP4Q_OK;
    if (!dW || !dY->q_t || !X->q_t || !dY->scale || !X->scale) return FP4Q_ERR_NULL;
    if (ldw < K) return FP4Q_ERR_SHAPE;
    GemmParams p = {};
    p.C = dW; p.ldc = ldw; p.M = (int32_t)N; p.N = (int32_t)K; p.K = (int32_t)T;
    set_out_type(p, dt); p.accumulate = accumulate ? 1 : 0;
    dense_tiles(p);
    if (g) {
        p.mode = MODE_GROUPED_K; p.n_groups = g->n_groups; p.row_offsets = g->row_offsets;
        p.n_tile_total *= g->n_groups;
    }
    return launch_gemm<KIND_MXF4>(operand_t(dY), operand_t(X), p, ws, ws_bytes, stream);
}

extern "C" fp4q_status fp4q_mxfp8_qk(const uint8_t *xq, int64_t ld_xq, const uint8_t *xs, int64_t ld_xs, int64_t T,
                                     int64_t Kdim, const uint8_t *wq_q, const uint8_t *wq_s, const uint8_t *wk_q,
                                     const uint8_t *wk_s, int64_t ld_wq, int64_t ld_ws, int64_t N, void *Q_out,
                                     void *K_out, int64_t ldo, fp4q_out dt, void *ws, size_t ws_bytes, void *stream)
{
    if (T < 0 || N < 0 || Kdim < 0) return FP4Q_ERR_SHAPE;
    if (!out_type_ok(dt)) return FP4Q_ERR_UNSUPPORTED;
    if (T > kMaxDim || N > kMaxDim || Kdim > kMaxDim) return FP4Q_ERR_UNSUPPORTED;
    if (T == 0 || N == 0) return FP4Q_OK;
    if (!xq || !xs) return FP4Q_ERR_NULL;
    if ((wq_q && (!wq_s || !Q_out)) || (wk_q && (!wk_s || !K_out))) return FP4Q_ERR_NULL;
    const int64_t kpad = round_up(Kdim, 32), nkb = ceil_div(Kdim, 32);
    if (ld_xq < kpad || ld_wq < kpad || ld_xs < nkb || ld_ws < nkb || ldo < N) return FP4Q_ERR_SHAPE;
    Operand A;
    A.payload = xq; A.rows = T; A.row_bytes = kpad; A.ld_bytes = ld_xq;
    A.sf = ScaleView{xs, ld_xs, 1, (int32_t)T, (int32_t)nkb};
    const uint8_t *wq[2] = {wq_q, wk_q};
    const uint8_t *wsf[2] = {wq_s, wk_s};
    void *out[2] = {Q_out, K_out};
    for (int i = 0; i < 2; i++) {
        if (!wq[i]) continue;
        Operand B;
        B.payload = wq[i]; B.rows = N; B.row_bytes = kpad; B.ld_bytes = ld_wq;
        B.sf = ScaleView{wsf[i], ld_ws, 1, (int32_t)N, (int32_t)nkb};
        GemmParams p = {};
        p.C = out[i]; p.ldc = ldo; p.M = (int32_t)T; p.N = (int32_t)N; p.K = (int32_t)Kdim;
        set_out_type(p, dt);
        dense_tiles(p);
        if (fp4q_status s = launch_gemm<KIND_MXF8>(A, B, p, ws, ws_bytes, stream)) return s;
    }
    return FP4Q_OK;
}

extern "C" fp4q_status fp4q_mxfp8_gemm(const uint8_t *aq, int64_t ld_aq, const uint8_t *as, int64_t ld_as, int64_t M,
                                       const uint8_t *bq, int64_t ld_bq, const uint8_t *bs, int64_t ld_bs, int64_t N,
                                       int64_t Kdim, void *C, int64_t ldc, fp4q_out dt, void *ws, size_t ws_bytes,
                                       void *stream)
{
    if (M < 0 || N < 0 || Kdim < 0) return FP4Q_ERR_SHAPE;
    if (!out_type_ok(dt)) return FP4Q_ERR_UNSUPPORTED;
    if (M > kMaxDim || N > kMaxDim || Kdim > kMaxDim) return FP4Q_ERR_UNSUPPORTED;
    if (M == 0 || N == 0) return FP4Q_OK;
    if (!aq || !as || !bq || !bs || !C) return FP4Q_ERR_NULL;
    const int64_t kpad = round_up(Kdim, 32), nkb = ceil_div(Kdim, 32);
    if (ld_aq < kpad || ld_bq < kpad || ld_as < nkb || ld_bs < nkb || ldc < N) return FP4Q_ERR_SHAPE;
    Operand A, B;
    A.payload = aq; A.rows = M; A.row_bytes = kpad; A.ld_bytes = ld_aq;
    A.sf = ScaleView{as, ld_as, 1, (int32_t)M, (int32_t)nkb};
    B.payload = bq; B.rows = N; B.row_bytes = kpad; B.ld_bytes = ld_bq;
    B.sf = ScaleView{bs, ld_bs, 1, (int32_t)N, (int32_t)nkb};
    GemmParams p = {};
    p.C = C; p.ldc = ldc; p.M = (int32_t)M; p.N = (int32_t)N; p.K = (int32_t)Kdim;
    set_out_type(p, dt);
    dense_tiles(p);
    return launch_gemm<KIND_MXF8>(A, B, p, ws, ws_bytes, stream);
}

extern "C" fp4q_status fp4q_gemm_fwd_act1d(const uint8_t *xq, int64_t ld_xq, const uint8_t *xs, int64_t ld_xs, int64_t T,
                                           const fp4q_tensor *W, void *Y, int64_t ldy, fp4q_out dt, void *ws, size_t ws_bytes,
                                           void *stream)
{
    if (!tensor_ok(W)) return W ? FP4Q_ERR_SHAPE : FP4Q_ERR_NULL;
    if (T < 0) return FP4Q_ERR_SHAPE;
    if (!out_type_ok(dt)) return FP4Q_ERR_UNSUPPORTED;
    const int64_t N = W->rows, K = W->cols;
    if (T > kMaxDim || N > kMaxDim || K > kMaxDim) return FP4Q_ERR_UNSUPPORTED;
    if (T == 0 || N == 0) return FP4Q_OK;
    if (!Y || !xq || !xs || !W->q_rm || !W->scale) return FP4Q_ERR_NULL;
    if (ldy < N || ld_xq < round_up(K, 32) / 2 || ld_xs < ceil_div(K, 32)) return FP4Q_ERR_SHAPE;
    Operand A, B = operand_rm(W);
    A.payload = xq; A.rows = T; A.row_bytes = round_up(K, 32) / 2; A.ld_bytes = ld_xq;
    A.sf = ScaleView{xs, ld_xs, 1, (int32_t)T, (int32_t)ceil_div(K, 32)};
    GemmParams p = {};
    p.C = Y; p.ldc = ldy; p.M = (int32_t)T; p.N = (int32_t)N; p.K = (int32_t)K;
    set_out_type(p, dt);
    dense_tiles(p);
    return launch_gemm<KIND_MXF4RA>(A, B, p, ws, ws_bytes, stream);
}

extern "C" fp4q_status fp4q_gemm_wgrad_act1d(const fp4q_tensor *dY, const uint8_t *xtq, int64_t ld_xtq, const uint8_t *xts,
                                             int64_t ld_xts, int64_t K, void *dW, int64_t ldw, fp4q_out dt, int accumulate,
                                             void *ws, size_t ws_bytes, void *stream)
{
    if (!tensor_ok(dY)) return dY ? FP4Q_ERR_SHAPE : FP4Q_ERR_NULL;
    if (K < 0) return FP4Q_ERR_SHAPE;
    if (!out_type_ok(dt)) return FP4Q_ERR_UNSUPPORTED;
    if (accumulate && !out_type_f32(dt)) return FP4Q_ERR_UNSUPPORTED;
    const int64_t T = dY->rows, N = dY->cols;
    if (T > kMaxDim || N > kMaxDim || K > kMaxDim) return FP4Q_ERR_UNSUPPORTED;
    if (N == 0 || K == 0) return FP4Q_OK;
    if (!dW || !dY->q_t || !dY->scale || !xtq || !xts) return FP4Q_ERR_NULL;
    if (ldw < K || ld_xtq < round_up(T, 32) / 2 || ld_xts < ceil_div(T, 32)) return FP4Q_ERR_SHAPE;
    Operand A = operand_t(dY), B;
    B.payload = xtq; B.rows = K; B.row_bytes = round_up(T, 32) / 2; B.ld_bytes = ld_xtq;
    B.sf = ScaleView{xts, ld_xts, 1, (int32_t)K, (int32_t)ceil_div(T, 32)};
    GemmParams p = {};
    p.C = dW; p.ldc = ldw; p.M = (int32_t)N; p.N = (int32_t)K; p.K = (int32_t)T;
    set_out_type(p, dt); p.accumulate = accumulate ? 1 : 0;
    dense_tiles(p);
    return launch_gemm<KIND_MXF4RB>(A, B, p, ws, ws_bytes, stream);
}

// ------------------------------------------------------------------------------------------------------
// Products on tensors quantized in 16 x 16 blocks (block-size study): same payloads, scale matrix
// [ceil(rows/16), ceil(cols/16)], 16-element scale vectors in the MMA.  Dense only.
namespace fp4q {

static Operand operand_rm16(const fp4q_tensor *t)
{
    Operand o = operand_rm(t);
    o.sf = ScaleView{t->scale, t->ld_s, 1, (int32_t)ceil_div(t->rows, 16), (int32_t)ceil_div(t->cols, 16)};
    return o;
}
static Operand operand_t16(const fp4q_tensor *t)
{
    Operand o = operand_t(t);
    o.sf = ScaleView{t->scale, 1, t->ld_s, (int32_t)ceil_div(t->cols, 16), (int32_t)ceil_div(t->rows, 16)};
    return o;
}

// which: 0 forward (A = a.q_rm [M,K], B = b.q_rm [N,K]), 1 input gradient (A = a.q_rm [M,K'], B = b.q_t), 2 weight
// gradient (A = a.q_t, B = b.q_t)
static fp4q_status gemm_b16(int which, const fp4q_tensor *a, const fp4q_tensor *b, void *C, int64_t ldc, fp4q_out dt, int accumulate,
                            void *ws, size_t ws_bytes, void *stream)
{
    if (!tensor_ok(a) || !tensor_ok(b)) return a && b ? FP4Q_ERR_SHAPE : FP4Q_ERR_NULL;
    if (!out_type_ok(dt)) return FP4Q_ERR_UNSUPPORTED;
    if (accumulate && !out_type_f32(dt)) return FP4Q_ERR_UNSUPPORTED;
    int64_t M, N, K;
    if (which == 0) { if (a->cols != b->cols) return FP4Q_ERR_SHAPE; M = a->rows; N = b->rows; K = a->cols; }
    else if (which == 1) { if (a->cols != b->rows) return FP4Q_ERR_SHAPE; M = a->rows; N = b->cols; K = a->cols; }
    else { if (a->rows != b->rows) return FP4Q_ERR_SHAPE; M = a->cols; N = b->cols; K = a->rows; }
    if (M > kMaxDim || N > kMaxDim || K > kMaxDim) return FP4Q_ERR_UNSUPPORTED;
    if (M == 0 || N == 0) return FP4Q_OK;
    const uint8_t *pa = which == 2 ? a->q_t : a->q_rm, *pb = which == 0 ? b->q_rm : b->q_t;
    if (!C || !pa || !pb || !a->scale || !b->scale) return FP4Q_ERR_NULL;
    if (ldc < N) return FP4Q_ERR_SHAPE;
    GemmParams p = {};
    p.C = C; p.ldc = ldc; p.M = (int32_t)M; p.N = (int32_t)N; p.K = (int32_t)K;
    set_out_type(p, dt); p.accumulate = accumulate ? 1 : 0;
    dense_tiles(p);
    return launch_gemm<KIND_MXF4B16>(which == 2 ? operand_t16(a) : operand_rm16(a), which == 0 ? operand_rm16(b) : operand_t16(b), p, ws,
                                     ws_bytes, stream);
}

}  // namespace fp4q

extern "C" fp4q_status fp4q_gemm_fwd_b16(const fp4q_tensor *X, const fp4q_tensor *W, void *Y, int64_t ldy, fp4q_out dt, void *ws,
                                         size_t ws_bytes, void *stream)
{
    return gemm_b16(0, X, W, Y, ldy, dt, 0, ws, ws_bytes, stream);
}

extern "C" fp4q_status fp4q_gemm_dgrad_b16(const fp4q_tensor *dY, const fp4q_tensor *W, void *dX, int64_t ldx, fp4q_out dt, void *ws,
                                           size_t ws_bytes, void *stream)
{
    return gemm_b16(1, dY, W, dX, ldx, dt, 0, ws, ws_bytes, stream);
}

extern "C" fp4q_status fp4q_gemm_wgrad_b16(const fp4q_tensor *dY, const fp4q_tensor *X, void *dW, int64_t ldw, fp4q_out dt,
                                           int accumulate, void *ws, size_t ws_bytes, void *stream)
{
    return gemm_b16(2, dY, X, dW, ldw, dt, accumulate, ws, ws_bytes, stream);
}

// ------------------------------------------------------------------------------------------------------
// Forward product for callers that cannot allocate device memory.
//
// The GEMM kernel records device-side anomalies in a small workspace that the regular entry points take
// from the caller.  Code that runs where cudaMalloc is off limits -- a plug-in inside a host application
// that owns the device heap, a real-time loop that must not enter the allocator, a sandbox that only hands
// out pre-registered buffers -- has no way to supply one.  For those callers the workspace lives in the
// fixed array below, which every GPU that loads this library holds until the process exits.
namespace fp4q {

constexpr size_t kStaticWorkspaceBytes = 1024;   // stated maximum; the kernel's workspace must fit in it
static __device__ __align__(256) unsigned char g_static_workspace[kStaticWorkspaceBytes];

static std::atomic<void *> g_static_workspace_addr[kMaxDevices];   // device address of the array, per device

// In host code the array's name is only a handle: the device address has to be asked for, once per device,
// with that device current.
static fp4q_status static_workspace_address(void **out)
{
    const int dev = current_device();
    if (dev < 0) return FP4Q_ERR_CUDA;
    if (g_static_workspace_addr[dev] == nullptr) {
        void *ptr = nullptr;
        if (cudaGetSymbolAddress(&ptr, g_static_workspace) != cudaSuccess || ptr == nullptr) return FP4Q_ERR_CUDA;
        g_static_workspace_addr[dev] = ptr;
    }
    *out = g_static_workspace_addr[dev];
    return FP4Q_OK;
}

}  // namespace fp4q

extern "C" fp4q_status fp4q_gemm_fwd_static_workspace(const fp4q_tensor *X, const fp4q_tensor *W, void *Y, int64_t ldy,
                                                      fp4q_out dt, uint32_t *status_out, void *stream)
{
    if (fp4q_workspace_bytes() > kStaticWorkspaceBytes) return FP4Q_ERR_WORKSPACE;   // layout outgrew the array
    // every argument error is reported before anything is put on the stream
    GemmParams p;
    bool noop;
    if (fp4q_status s = prepare_fwd(X, W, Y, ldy, dt, nullptr, p, &noop)) return s;
    void *ws = nullptr;
    if (fp4q_status s = static_workspace_address(&ws)) return s;
    if (!noop)
        if (fp4q_status s = check_gemm_args(operand_rm(X), operand_rm(W), p, ws, kStaticWorkspaceBytes)) return s;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // the array keeps whatever the previous call left: the status words must start at zero
    if (cudaMemsetAsync(ws, 0, sizeof(Workspace), st) != cudaSuccess) return FP4Q_ERR_CUDA;
    if (!noop)
        if (fp4q_status s = launch_gemm<KIND_MXF4>(operand_rm(X), operand_rm(W), p, ws, kStaticWorkspaceBytes, stream)) return s;
    if (status_out &&
        cudaMemcpyAsync(status_out, ws, sizeof(uint32_t), cudaMemcpyDeviceToDevice, st) != cudaSuccess)
        return FP4Q_ERR_CUDA;
    return FP4Q_OK;
}
