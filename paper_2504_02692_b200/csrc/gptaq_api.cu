// C ABI of the GPTAQ layer solve: handle, argument checks, launch sequences.
// Every arithmetic step runs in the kernels of this library; the host code
// below only validates, carves the caller's workspace and enqueues launches.
#include "../../include/gptaq.h"

#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <utility>
#include <vector>

#include "kernels.cuh"
#include "simt_gemm.cuh"
#include "umma_gemm.cuh"
#include "tc_gemm.cuh"
#include "factor.cuh"
#include "narrow.cuh"
#include "quantize_block.cuh"

using namespace gptaq;

namespace {

constexpr size_t ALIGN = 256;
inline size_t round_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

enum Stage { STAGE_ACCUM = 0, STAGE_FACTORED = 1, STAGE_P = 2 };
constexpr int64_t ACT_ORDER_MAX_N = 57344;     // a weight row (float32) has to fit the shared memory of one CTA
constexpr int64_t P_ROWWISE_MAX_N = 16384;     // two rows (float32) in the shared memory of one CTA

}  // namespace

struct gptaq_ctx {
    int64_t n;
    int device;
    int num_sms;
    char *state;
    size_t state_bytes;
    char *ws;
    size_t ws_bytes;
    StateHeader *hd;
    float *H, *D;
    uint8_t *dead;         // dead-input flags in working (possibly sorted) column order
    uint8_t *dead_raw;     // ... in the caller's column order
    int *perm;             // act_order: working column c is the caller's column perm[c]
    bool act_order;
    int stage;
    int64_t tokens;
    int64_t launches;
    int stats_precision;   // GPTAQ_STATS_*
    bool tensor;           // float32-grade tensor-core GEMMs (fp16-split operands) for factor / P / trailing update
    bool split;            // ... for P / trailing update of the current factor (set by gptaq_factor)
    int terms;             // GPTAQ_TERM_* switches of gptaq_quantize
    bool static_groups;    // group grids from the original weights, per group of the caller's columns
    int clip_steps; float clip_min;   // clipping-range search of the grids
    // Statistics pipeline: the conversion of a token batch runs on the caller's stream, the
    // tensor-core product on `gemm_stream`, so that the (memory-bound) conversion of the next
    // batch overlaps the (tensor-bound) product of this one.  Two operand buffers alternate.
    cudaStream_t gemm_stream;
    cudaStream_t inv_stream;      // gptaq_factor: the rows of the inverse, beside the factorisation
    cudaEvent_t inv_ready, inv_done;
    cudaEvent_t conv_done[2], gemm_done[2];
    bool gemm_pending[2];
    bool relayout;         // the operand buffers change size: wait for the products in flight first
    int next_buf;
    // tensor maps of a buffer's operands (they lie in the workspace: only the padded token count and the layout matter)
    struct StatsMaps { CUtensorMap x, d, xlo, dlo, h, dxx, slots; int64_t kp, chunk; int narr; bool c_tma; } stats_maps[2];
    // partial sums of the cut tiles of the statistics products wait in the workspace (fix_args.scratch) until
    // the sums are needed or the cut changes; fix_pending: they have not been added to H / dXX^T yet
    bool fix_pending;
    StatsGemmArgs fix_args;
    bool d_upper_only;     // a token batch went in without the tiles of dXX^T below the diagonal
    // optional timing of the statistics kernel alone: one event pair per launch, on the stream it runs on
    bool kernel_timing;
    std::vector<std::pair<cudaEvent_t, cudaEvent_t>> timing_events;   // pool; the first timing_used are recorded
    size_t timing_used;
    std::string cuda_error;
};

namespace {

struct Layout {
    size_t h_off, d_off, dead_off, dead_raw_off, perm_off, total;
};

Layout state_layout(int64_t n) {
    Layout l;
    size_t mat = round_up((size_t)n * (size_t)n * sizeof(float), ALIGN);
    l.h_off = ALIGN;
    l.d_off = l.h_off + mat;
    l.dead_off = l.d_off + mat;
    l.dead_raw_off = l.dead_off + round_up((size_t)n, ALIGN);
    l.perm_off = l.dead_raw_off + round_up((size_t)n, ALIGN);
    l.total = l.perm_off + round_up((size_t)n * sizeof(int), ALIGN);
    return l;
}

// float32-grade tensor-core path (tc_gemm.cuh): widths whose float32 rows are 16-byte multiples (the epilogue's tensor
// map) and that are large enough for 128 x 256 tiles to pay.  The fp16 copies of n x n operands have a row pitch of their
// own, the next multiple of 8 (a TMA stride rule).
constexpr int64_t TC_MIN_N = 512;
inline bool tc_shape_ok(int64_t n) { return n >= TC_MIN_N && (n % 4) == 0; }
inline int64_t split_pitch(int64_t n) { return (n + 7) / 8 * 8; }

struct WsLayout {
    size_t t_off, rinv_off;
    size_t diag_off;        // copy of the next diagonal block
    size_t s_off[3];        // split operand matrices, fp16 hi then lo (n x split_pitch(n) each)
    size_t pan_off[2];      // split copy of factor panels, hi / lo: n x SUPER_NB fp16
    // [-Err | Wpre] of a launch: float32, its fp16 hi / lo parts (tensor cores), row scales
    size_t ew_off, ew_lo_off, rs_off, total;
    bool tensor;
};

// FP16-split factorisation: panels are grouped in super-panels of SUPER_NB columns; inside a super-panel
// the rank-128 update only touches the super-panel's remaining columns, the rest of the matrix receives
// one rank-SUPER_NB update per super-panel (8x less read-modify-write traffic, longer contractions)
constexpr int SUPER_NB = 8 * NB;
// The lazy-batch update of gptaq_quantize likewise: a launch of quant_block_kernel takes QB_SUPER columns (QB_W without the
// tensor cores), everything beyond them receives their errors at once.  The result does not depend on where the launches
// end, so the caller's block size does not set their width (128 x 128 with blocks of 32: 3 launches for 9, 67 -> 28 us).

WsLayout ws_layout(int64_t n, int64_t m_max) {
    WsLayout w;
    size_t nb = (size_t)((n + NB - 1) / NB);
    const size_t mat = round_up((size_t)n * (size_t)n * sizeof(float), ALIGN);
    w.tensor = tc_shape_ok(n);
    w.t_off = 0;
    w.rinv_off = w.t_off + mat;
    w.diag_off = w.rinv_off + round_up(nb * NB * NB * sizeof(float), ALIGN);
    size_t off = w.diag_off + round_up(NB * NB * sizeof(float), ALIGN);
    // S0 = U^T, S1 = U then P^T, S2 = dXX^T then O
    const size_t smat = round_up(2 * (size_t)n * (size_t)split_pitch(n) * sizeof(__half), ALIGN);
    for (int i = 0; i < 3; ++i) { w.s_off[i] = off; if (w.tensor) off += smat; }
    const size_t pan = (size_t)n * SUPER_NB * sizeof(__half);
    for (int i = 0; i < 2; ++i) { w.pan_off[i] = off; if (w.tensor) off += round_up(pan, ALIGN); }
    const size_t ew = round_up((size_t)m_max * 2 * (w.tensor ? QB_SUPER : QB_W) * sizeof(float), ALIGN);
    w.ew_off = off;
    w.ew_lo_off = off + ew;
    w.rs_off = off + (w.tensor ? 2 * ew : ew);
    w.total = w.rs_off + (w.tensor ? round_up((size_t)m_max * sizeof(float), ALIGN) : 0);
    return w;
}

gptaq_status_t cuda_fail(gptaq_ctx *h, cudaError_t e) {
    if (h) h->cuda_error = cudaGetErrorString(e);
    return GPTAQ_ERR_CUDA;
}

#define CU(call)                                             \
    do {                                                     \
        cudaError_t e__ = (call);                            \
        if (e__ != cudaSuccess) return cuda_fail(h, e__);    \
    } while (0)

#define LAUNCHED()                                           \
    do {                                                     \
        cudaError_t e__ = cudaGetLastError();                \
        if (e__ != cudaSuccess) return cuda_fail(h, e__);    \
        h->launches++;                                       \
    } while (0)

gptaq_status_t gemm(gptaq_ctx *h, const GemmProblem &p, bool a_rc, bool b_rc, cudaStream_t s, int early_ctas = 0) {
    if (p.M <= 0 || p.N <= 0 || p.nbatch <= 0) return GPTAQ_OK;
    cudaError_t e = launch_simt_gemm(p, a_rc, b_rc, s, early_ctas);
    if (e != cudaSuccess) return cuda_fail(h, e);
    h->launches++;
    return GPTAQ_OK;
}

#define OK(call)                                  \
    do {                                          \
        gptaq_status_t s__ = (call);              \
        if (s__ != GPTAQ_OK) return s__;          \
    } while (0)

// cuTensorMapEncodeTiled through the runtime's driver entry point (no link-time libcuda).
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

// fp16 matrix [rows][kp] (K contiguous), box = 64 x box_rows, 128-byte swizzle.
bool make_kmajor_map(CUtensorMap *map, const void *ptr, int64_t rows, int64_t kp, int box_rows) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {(cuuint64_t)kp, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)kp * 2};
    cuuint32_t box[2] = {(cuuint32_t)UBK, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void *>(ptr), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// A split operand (hi / lo arrays of the same shape) as seen by the tensor-core GEMM.
struct SplitOperand {
    const __half *hi, *lo;
    int64_t rows, cols, ld;
};

// __half matrix [rows][ld] with `cols` valid K-contiguous elements per row; box = 64 x box_rows.
bool make_f16_map(CUtensorMap *map, const void *ptr, int64_t rows, int64_t cols, int64_t ld, int box_rows) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    cuuint32_t box[2] = {(cuuint32_t)TBK, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void *>(ptr), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool make_operand_map(CUtensorMap *map, const __half *ptr, const SplitOperand &o, int box_rows) {
    return make_f16_map(map, ptr, o.rows, o.cols, o.ld, box_rows);
}

struct TcMaps {
    CUtensorMap a_hi, a_lo, b_hi, b_lo, b2_hi, b2_lo;
};

bool make_tc_maps(TcMaps *m, const SplitOperand &A, const SplitOperand &B, const SplitOperand *B2) {
    const SplitOperand &b2 = B2 ? *B2 : B;
    return make_operand_map(&m->a_hi, A.hi, A, TBM) && make_operand_map(&m->a_lo, A.lo, A, TBM) &&
           make_operand_map(&m->b_hi, B.hi, B, TBOX) && make_operand_map(&m->b_lo, B.lo, B, TBOX) &&
           make_operand_map(&m->b2_hi, b2.hi, b2, TBOX) && make_operand_map(&m->b2_lo, b2.lo, b2, TBOX);
}

// Launch with programmatic stream serialization where `pdl` is set: the kernel may be scheduled while its predecessor
// drains; it calls pdl_wait() before it touches anything the predecessor wrote.
// So start: the factorisation's chain (4 % of it at n = 4096; the damping up to 3 us up to n = 2052), the tensor-core products of
// gptaq_factor and gptaq_build_P and the correction matrix of narrow layers; the second pass of the statistics'
// conversion (2 to 4 us a call; back to back 4 calls of 4112 tokens at n = 1024 141 -> 135, of 2777 at n = 2052 392 -> 396);
// split copies and small float32 products of few CTAs (launch_split16, launch_simt_gemm); the column loop without tensor cores
// from its second launch on (launch_quant_block).  All else is launched plainly: the column loop on the tensor cores and its
// products (4 % slower so), column_loop_kernel, the statistics products, what a call begins with (copies, permutations, grids,
// maxima).
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(bool pdl, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
    cfg.attrs = attr; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

TcGemmArgs tc_args(float *C, int64_t ldc, int M, int N, int K, float alpha, float beta, int mode, int mask,
                   StateHeader *hd) {
    TcGemmArgs a;
    std::memset(&a, 0, sizeof(a));
    a.C = C; a.ldc = ldc; a.M = M; a.N = N; a.K = K; a.nbatch = 1;
    a.alpha = alpha; a.beta = beta; a.mode = mode; a.mask = mask; a.hd = hd;
    return a;
}

// float32 matrix C [M][ldc] with N valid columns as the target of bulk reductions: box = 32 x 128,
// 128-byte swizzle (the layout the epilogue writes its staging boxes in).
bool make_c_map(CUtensorMap *map, float *C, int64_t M, int64_t N, int64_t ldc) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {(cuuint64_t)N, (cuuint64_t)M};
    cuuint64_t strides[1] = {(cuuint64_t)ldc * 4};
    cuuint32_t box[2] = {32, (cuuint32_t)TBM};
    cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, C, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

cudaError_t launch_tc_gemm(const TcMaps &m, const TcGemmArgs &a_in, int num_sms, cudaStream_t s, bool pdl = true, bool beside = false) {
    if (a_in.M <= 0 || a_in.N <= 0 || a_in.nbatch <= 0) return cudaSuccess;
    TcGemmArgs a = a_in;
    const int bn = tc_tile_width(a, num_sms);
    const int64_t tiles = (int64_t)a.nbatch * ((a.M + TBM - 1) / TBM) * ((a.N + bn - 1) / bn);
    const int grid = (int)std::min<int64_t>(tiles, num_sms);
    a.sched = beside ? &a.hd->sched_counter2 : &a.hd->sched_counter;     // (two launches at the same time: one counter each)
    // "C += ...": bulk tensor reductions where the target qualifies for a tensor map (16-byte aligned base
    // and row pitch); scattered per-thread reductions otherwise
    CUtensorMap mapC = m.a_hi;       // placeholder, not dereferenced unless c_tma is set
    a.c_tma = 0;
    if (a.beta == 1.f && a.nbatch == 1 && !a.amax_out && (a.mask == TC_MASK_NONE || a.mask == TC_MASK_UPPER_KEEP) &&
        (reinterpret_cast<uintptr_t>(a.C) & 15) == 0 && (a.ldc & 3) == 0 && make_c_map(&mapC, a.C, a.M, a.N, a.ldc))
        a.c_tma = 1;
    return launch_pdl(pdl, bn == 256 ? tc_gemm_kernel<256> : bn == 128 ? tc_gemm_kernel<128> : tc_gemm_kernel<64>, dim3(grid),
                      dim3(TC_THREADS), tc_smem(bn), s, m.a_hi, m.a_lo, m.b_hi, m.b_lo, m.b2_hi, m.b2_lo, mapC, a);
}

// Slots of StateHeader::tc_amax (largest magnitudes of FP16-split operands).

cudaError_t launch_absmax(const AbsmaxArgs &a, const AbsmaxArgs &b, int num_sms, cudaStream_t s) {
    absmax_kernel<<<dim3(std::max(1, std::min(a.rows, 4 * num_sms)), 2), 256, 0, s>>>(a, b);
    return cudaGetLastError();
}

struct SplitBatch {
    int nbatch = 1;
    int64_t src_bstride = 0, dst_bstride = 0;
    int rows_last = 0, cols_last = 0;
};

// hi_t / lo_t non-null: the transposed form goes there in the same pass (transpose is then ignored)
Split16Args split16_args(const float *src, int64_t lds, __half *hi, __half *lo, int64_t ldd, int rows, int cols,
                         bool transpose, int mask, float scale, const unsigned *amax, const SplitBatch &b = SplitBatch(),
                         __half *hi_t = nullptr, __half *lo_t = nullptr, float *row_inv = nullptr) {
    Split16Args a;
    a.src = src; a.lds = lds; a.src_bstride = b.src_bstride; a.hi = hi; a.lo = lo; a.ldd = ldd;
    a.dst_bstride = b.dst_bstride;
    a.rows = rows; a.cols = cols; a.rows_last = b.rows_last; a.cols_last = b.cols_last; a.nbatch = b.nbatch;
    a.transpose = hi_t ? 2 : (transpose ? 1 : 0); a.mask = mask; a.scale = scale; a.amax = amax;
    a.hi_t = hi_t; a.lo_t = lo_t; a.row_inv = row_inv;
    return a;
}
// Starts early where that takes no more than a CTA per SM: those that are there before their turn hold the SMs that the product in
// front leaves free, several to an SM, and work there.  us plain / always early / by this rule: gptaq_build_P at n = 640
// 50 / 49 / 46, 768 54 / 64 / 52, 1024 64 / 72 / 64, 4096 356 / 362 / 356; gptaq_factor at n = 1536 417 / 424 / 418.
cudaError_t launch_split16(const Split16Args &a, int num_sms, cudaStream_t s, const Split16Args *second = nullptr) {
    if (a.rows <= 0 || a.cols <= 0 || a.nbatch <= 0) return cudaSuccess;
    dim3 grid((a.cols + 63) / 64, (a.rows + 63) / 64, a.nbatch + (second ? 1 : 0));
    const bool early = (int64_t)grid.x * grid.y * grid.z <= num_sms;
    return launch_pdl(early, split16_kernel, grid, dim3(256), 0, s, a, second ? *second : a);
}

// Scratch of the statistics kernel's K-split tail: at most one 128 x 256 partial tile per SM.
size_t stats_scratch_bytes(int num_sms) { return round_up((size_t)num_sms * UBM * UBN * sizeof(float), ALIGN); }
constexpr int MAX_SMS_FOR_SIZING = 256;

// fp16 operand arrays per converted batch: X^T, (X~ - X)^T, the low part of X^T, the low part of (X~ - X)^T
int stats_operand_arrays(int precision) {
    return precision == GPTAQ_STATS_FP16_SPLIT_FULL_TENSOR ? 4 : (precision == GPTAQ_STATS_FP16_SPLIT_TENSOR ? 3 : 2);
}

// Largest token chunk (multiple of 64) whose fp16 operand copies fit the workspace next to that scratch.
int64_t tc_chunk_tokens(const gptaq_ctx *h) {
    const int nbuf = stats_operand_arrays(h->stats_precision);
    int64_t per_token = 2 * nbuf * h->n * 2;   // two buffers of X^T, dX^T (and their low parts), fp16
    const size_t reserve = stats_scratch_bytes(h->num_sms);
    if (h->ws_bytes <= reserve + 2 * ALIGN) return 0;
    int64_t cap = (int64_t)((h->ws_bytes - reserve - 2 * ALIGN) / (size_t)per_token);
    cap = cap / UBK * UBK;
    return std::min<int64_t>(cap, 1 << 20);
}

bool tc_eligible(const gptaq_ctx *h) {
    // from 256 input channels on, and for exactly 128 (one half-empty pair tile per sum; the TMA boxes of 128
    // channels then cover the operand exactly)
    return h->stats_precision != GPTAQ_STATS_FP32 && (h->n >= UBN || h->n == UBM) && tc_chunk_tokens(h) >= UBK &&
           encode_tiled_fn() != nullptr;
}

// A small batch of a narrow layer takes the float32 products whatever the precision asked for: no conversions, one launch
// instead of three.  us a batch, float32 / tensor cores: n = 128 512 tokens 16 / 35, 2048 23 / 37, 4096 37 / 37; n = 256 512
// tokens 19 / 36, 1024 29 / 37, 2048 43 / 39; n = 384 512 tokens 31 / 35.  Batches after one another overlap on the tensor
// path (20 to 25 us each), so the line lies at half of where a single one would draw it.
constexpr int64_t STATS_FP32_WORK = (int64_t)1 << 25;          // tokens n^2

// Adds the waiting partial sums of the cut tiles to H / dXX^T, on the internal stream behind the products.
gptaq_status_t flush_partials(gptaq_ctx *h) {
    if (!h->fix_pending) return GPTAQ_OK;
    const StatsGemmArgs &ga = h->fix_args;
    stats_fixup_kernel<<<dim3((unsigned)(ga.ntiles - ga.full_tiles), FIXUP_SLABS), 256, 0, h->gemm_stream>>>(ga);
    LAUNCHED();
    h->fix_pending = false;
    CU(cudaEventRecord(h->gemm_done[0], h->gemm_stream));
    h->gemm_pending[0] = true;
    return GPTAQ_OK;
}

// Orders `s` after every statistics product still running on the internal stream.
gptaq_status_t join_statistics(gptaq_ctx *h, cudaStream_t s) {
    OK(flush_partials(h));
    for (int i = 0; i < 2; ++i)
        if (h->gemm_pending[i]) {
            CU(cudaStreamWaitEvent(s, h->gemm_done[i], 0));
            h->gemm_pending[i] = false;
        }
    return GPTAQ_OK;
}

// For a step that ends early because a CUDA call failed: `s` is ordered after all that the internal streams were given so
// far, so that whatever the caller does next (gptaq_reset, other use of its buffers) does not meet it.
gptaq_status_t join_after_error(gptaq_ctx *h, cudaStream_t s, gptaq_status_t st) {
    if (st != GPTAQ_OK) {
        if (cudaEventRecord(h->gemm_done[0], h->gemm_stream) == cudaSuccess) cudaStreamWaitEvent(s, h->gemm_done[0], 0);
        if (cudaEventRecord(h->inv_done, h->inv_stream) == cudaSuccess) cudaStreamWaitEvent(s, h->inv_done, 0);
    }
    return st;
}

gptaq_status_t accumulate_tc(gptaq_ctx *h, const float *X, const float *Xfp, int64_t tokens, int64_t ld,
                             cudaStream_t s) {
    const int n = (int)h->n;
    if (h->relayout) {
        OK(join_statistics(h, s));
        h->relayout = false;
    }
    const int64_t chunk = tc_chunk_tokens(h);
    // 256 x 256 tiles of H (upper) and of dXX^T (upper too, unless act_order will permute it)
    const int d_full = h->act_order ? 1 : 0;
    const int64_t ntiles = TileIter::total(n, d_full);
    if (!d_full) h->d_upper_only = true;
    const int npairs = std::max(1, h->num_sms / 2);         // CTA pairs (clusters of two)
    for (int64_t t0 = 0; t0 < tokens; t0 += chunk) {
        const int tk = (int)std::min<int64_t>(chunk, tokens - t0);
        const int kp = (tk + UBK - 1) / UBK * UBK;
        const int narr = stats_operand_arrays(h->stats_precision);
        const bool split = narr >= 3, splitd = narr == 4;
        const int buf = h->next_buf;
        h->next_buf ^= 1;
        const size_t buf_bytes = round_up((size_t)narr * n * (size_t)(chunk) * 2, ALIGN);
        __half *Xt = reinterpret_cast<__half *>(h->ws + (size_t)buf * buf_bytes);
        __half *dXt = Xt + (size_t)n * kp;
        __half *Xlo = split ? dXt + (size_t)n * kp : nullptr;
        __half *dXlo = splitd ? Xlo + (size_t)n * kp : nullptr;
        unsigned *amax = h->hd->amax[buf];
        cudaStream_t gs = h->gemm_stream;
        // this buffer was last read by the product issued two chunks ago
        if (h->gemm_pending[buf]) {
            CU(cudaStreamWaitEvent(s, h->gemm_done[buf], 0));
            h->gemm_pending[buf] = false;
        }
        ConvertArgs ca;
        ca.X = X + t0 * ld; ca.Xfp = Xfp + t0 * ld; ca.ld = ld; ca.tokens = tk; ca.n = n; ca.kp = kp;
        ca.Xt = Xt; ca.dXt = dXt; ca.Xlo = Xlo; ca.dXlo = dXlo; ca.amax = amax;
        dim3 cgrid(kp / 64, (n + 63) / 64);
        convert_transpose_kernel<0><<<cgrid, 256, 0, s>>>(ca);
        LAUNCHED();
        CU(launch_pdl(true, convert_transpose_kernel<1>, dim3(std::min<unsigned>(cgrid.x * cgrid.y, 4u * (unsigned)h->num_sms)), dim3(256),
                      0, s, ca));
        h->launches++;
        CU(cudaEventRecord(h->conv_done[buf], s));
        CU(cudaStreamWaitEvent(gs, h->conv_done[buf], 0));
        gptaq_ctx::StatsMaps &mp = h->stats_maps[buf];
        if (mp.kp != kp || mp.chunk != chunk || mp.narr != narr) {
            const __half *lo = split ? Xlo : Xt;    // unused maps still have to be valid
            const __half *dlo = splitd ? dXlo : dXt;
            mp.kp = 0;
            if (!make_kmajor_map(&mp.x, Xt, n, kp, UBM) || !make_kmajor_map(&mp.d, dXt, n, kp, UBM) ||
                !make_kmajor_map(&mp.xlo, lo, n, kp, UBM) || !make_kmajor_map(&mp.dlo, dlo, n, kp, UBM)) {
                h->cuda_error = "cuTensorMapEncodeTiled failed";
                return GPTAQ_ERR_CUDA;
            }
            // the targets of the sums: bulk reductions where the rows are 16-byte multiples (scattered reductions otherwise)
            float *scratch = reinterpret_cast<float *>(h->ws + 2 * buf_bytes);
            mp.c_tma = n % 4 == 0 && make_c_map(&mp.h, h->H, n, n, n) && make_c_map(&mp.dxx, h->D, n, n, n) &&
                       make_c_map(&mp.slots, scratch, (int64_t)h->num_sms * UBM, UBN, UBN);
            if (!mp.c_tma) mp.h = mp.dxx = mp.slots = mp.x;         // (placeholders, not dereferenced)
            mp.kp = kp; mp.chunk = chunk; mp.narr = narr;
        }
        StatsGemmArgs ga;
        ga.H = h->H; ga.D = h->D; ga.n = n; ga.kblocks = kp / UBK; ga.nseg_h = split ? 3 : 1; ga.nseg_d = splitd ? 3 : 1; ga.amax = amax; ga.hd = h->hd;
        // the last, partial wave of tiles is cut along K so that every pair has work
        ga.d_full = d_full;
        ga.ntiles = (int)ntiles;
        ga.full_tiles = (int)(ntiles / npairs) * npairs;
        ga.ksplit = 1;
        const int cut = (int)ntiles - ga.full_tiles;
        if (cut > 0) {
            const int by_pairs = npairs / cut, by_k = ga.kblocks / (2 * UCHUNK);
            ga.ksplit = std::max(1, std::min(std::min(by_pairs, by_k), 8));
        }
        ga.ksplit_d = 0;
        int cut_items = cut * ga.ksplit, cut_slots = cut * (ga.ksplit - 1);
        if (ga.full_tiles == 0 && ga.nseg_h != ga.nseg_d) {
            // fewer tiles than pairs, those of H several times as long as those of dXX^T (low parts of X): cut so that the
            // longest item is as short as it gets.  3001 tokens at n = 1416, 21 tiles of 141 and 21 of 47 K-blocks: a batch
            // 87 us as they are (none could be cut in the same number of items), 67 with two items and one.
            const int T = (n + UPM - 1) / UPM, nh = T * (T + 1) / 2, nd = (int)ntiles - nh;
            const int lh = ga.kblocks * ga.nseg_h, ld = ga.kblocks * ga.nseg_d;
            int best = INT32_MAX;
            for (int kd = 1; kd <= 8 && nh + nd * kd <= npairs; ++kd) {
                const int kh = std::min(8, (npairs - nd * kd) / nh);
                // (pieces of one accumulation chain at least)
                const int ph = std::max(1, std::min(kh, lh / UCHUNK)), pd = std::max(1, std::min(kd, ld / UCHUNK));
                const int longest = std::max((lh + ph - 1) / ph, (ld + pd - 1) / pd);
                if (longest < best) { best = longest; ga.ksplit = ph; ga.ksplit_d = pd; }
            }
            cut_items = nh * ga.ksplit + nd * ga.ksplit_d;
            cut_slots = cut_items - cut;
        }
        if (cut_slots == 0) { ga.full_tiles = (int)ntiles; ga.ksplit = 1; ga.ksplit_d = 0; cut_items = 0; }
        // scratch behind the two operand buffers (one partial 128 x 256 tile per CTA at most; the products
        // run one after the other on the internal stream, so one scratch serves both buffers)
        ga.scratch = reinterpret_cast<float *>(h->ws + 2 * buf_bytes);
        ga.c_tma = mp.c_tma ? 1 : 0;
        const int nitems = ga.full_tiles + cut_items;
        const int sgrid = 2 * std::min(nitems, npairs);
        std::pair<cudaEvent_t, cudaEvent_t> *tev = nullptr;
        if (h->kernel_timing) {
            if (h->timing_used == h->timing_events.size()) {
                std::pair<cudaEvent_t, cudaEvent_t> ev{nullptr, nullptr};
                CU(cudaEventCreate(&ev.first));
                CU(cudaEventCreate(&ev.second));
                h->timing_events.push_back(ev);
            }
            tev = &h->timing_events[h->timing_used++];
            CU(cudaEventRecord(tev->first, gs));
        }
        if (h->fix_pending && (h->fix_args.ksplit != ga.ksplit || h->fix_args.ksplit_d != ga.ksplit_d || h->fix_args.full_tiles != ga.full_tiles ||
                               h->fix_args.ntiles != ga.ntiles || h->fix_args.d_full != ga.d_full ||
                               h->fix_args.scratch != ga.scratch))
            OK(flush_partials(h));              // another cut: the slots change meaning
        if (cut_slots > 0 && !h->fix_pending) {
            CU(cudaMemsetAsync(ga.scratch, 0, (size_t)cut_slots * 2 * UBM * UBN * sizeof(float), gs));
            h->fix_args = ga;
            h->fix_pending = true;
        }
        stats_umma_kernel<<<sgrid, UMMA_THREADS, UMMA_SMEM, gs>>>(mp.x, mp.d, mp.xlo, mp.dlo, mp.h, mp.dxx, mp.slots, ga);
        LAUNCHED();
        if (tev) CU(cudaEventRecord(tev->second, gs));
        CU(cudaEventRecord(h->gemm_done[buf], gs));
        h->gemm_pending[buf] = true;
    }
    h->tokens += tokens;
    return GPTAQ_OK;
}

bool valid_block(int b) { return b == 32 || b == 64 || b == 128; }

// float32 matrix [n][n] in boxes of 32 x 32, as they lie.
bool make_box_map(CUtensorMap *map, const float *ptr, int64_t n) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {(cuuint64_t)n, (cuuint64_t)n};
    cuuint64_t strides[1] = {(cuuint64_t)n * 4};
    cuuint32_t box[2] = {32, 32};
    cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float *>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// What the column loop and the trailing update work on: the factor U, the matrix P, the
// dead-input flags, the device status header and the m x 2B scratch for [-Err | Wpre].
struct QuantizeTarget {
    int n;
    const float *U, *P;
    const uint8_t *dead;
    StateHeader *hd;
    float *EW;
    int64_t ew_floats;         // its size
    int num_sms;
    // tensor-core trailing update (null: plain float32 products): U^T and P^T as fp16 hi / lo (row pitch ldt,
    // lo = hi + n * ldt), each with the scale of its recorded maximum; EW is then m x 2 * SW wide (SW columns per
    // launch), EW16 holds its fp16 hi / lo parts (lo = hi + m * 2 * SW) with one scale per row
    const __half *UT16 = nullptr, *PT16 = nullptr;
    int64_t ldt = 0;
    __half *EW16 = nullptr;
    float *row_inv = nullptr;
    const unsigned *amax_u = nullptr, *amax_p = nullptr;
    // a second stream for one half of many rows (null: none), and two events
    cudaStream_t side = nullptr;
    cudaEvent_t fork = nullptr, join = nullptr;
    int terms = GPTAQ_TERM_ERR | GPTAQ_TERM_ASYM;   // which terms of the weight update are applied
    const int *perm = nullptr;                      // act_order: working column c is the caller's column perm[c]
    int clip_steps = 0; float clip_min = 1.f;       // clipping-range search of the grids (0 steps: min/max)
    const uint8_t *dead_orig = nullptr;             // static groups: dead-input flags in the caller's column order
    bool static_groups = false;
};

// One launch of quant_block_kernel: columns [i0, i1) of the loop for rows [r0, r1) of m, SW columns per launch at most.
// src: the caller's weights, read instead of W by a launch that takes all columns (or nullptr).
cudaError_t launch_quant_block(const QuantizeTarget &t, float *W, int64_t ldw, const void *src, int64_t lds, int w_dtype, int64_t r0, int64_t r1, int64_t m, int i0, int i1, int SW,
                               int bits, int group, int sym, uint8_t *codes, float *scales, float *zeros, int G,
                               bool static_groups, cudaStream_t s) {
    const bool far_form = t.UT16 != nullptr;
    const size_t nn = (size_t)t.n * t.ldt;
    QuantBlockArgs a;
    std::memset(&a, 0, sizeof(a));
    a.W = W; a.ldw = ldw; a.src = src; a.lds = lds; a.src_bf16 = src && w_dtype == GPTAQ_W_BF16; a.row_first = (int)r0; a.m = (int)r1; a.n = t.n; a.U = t.U; a.P = t.P; a.dead = t.dead;
    a.i0 = i0; a.i1 = i1; a.bw = far_form ? QB_W : SW;
    a.bits = bits; a.group = group; a.sym = sym;
    a.codes = codes; a.scales = scales; a.zeros = zeros; a.G = G;
    a.ew_ld = 2 * SW; a.ew_pre = SW;
    if (i1 < t.n) {
        a.EW = t.EW;
        if (far_form) { a.EWS_hi = t.EW16; a.EWS_lo = t.EW16 + (size_t)m * 2 * SW; a.row_inv = t.row_inv; }
    }
    a.amax_u = t.amax_u; a.amax_p = t.amax_p; a.hd = t.hd;
    a.err_scale = (t.terms & GPTAQ_TERM_ERR) ? 1.f : 0.f; a.asym_scale = (t.terms & GPTAQ_TERM_ASYM) ? 1.f : 0.f;
    a.perm = t.perm; a.clip_steps = t.clip_steps; a.clip_min = t.clip_min;
    CUtensorMap uh, ul, ph, pl, u32, p32;
    std::memset(&uh, 0, sizeof(uh)); ul = ph = pl = u32 = p32 = uh;
    // (rows of U and P by the TMA unit where they are 16-byte multiples)
    a.up_tma = t.n % 4 == 0 && ((reinterpret_cast<uintptr_t>(t.U) | reinterpret_cast<uintptr_t>(t.P)) & 15) == 0 &&
               make_box_map(&u32, t.U, t.n) && make_box_map(&p32, t.P, t.n);
    if (far_form && (!make_f16_map(&uh, t.UT16, t.n, t.n, t.ldt, 128) || !make_f16_map(&ul, t.UT16 + nn, t.n, t.n, t.ldt, 128) ||
                     !make_f16_map(&ph, t.PT16, t.n, t.n, t.ldt, 128) || !make_f16_map(&pl, t.PT16 + nn, t.n, t.n, t.ldt, 128)))
        return cudaErrorUnknown;
    // Few rows: CTAs of 16 while one round of them takes all rows (m, not this launch's share of it: two halves beside one another
    // are more than a round).  us a call with 32 and with 16: 64 x 1024 146 and 131, 512 x 1024 with groups 152 and 134, 1003 x 1416
    // 228 and 206, 2368 x 1416 249 and 232.  Without tensor cores a launch is a quarter as long and the products between two launches,
    // which start early, meet twice as many CTAs: 512 x 400 85 and 81, 777 x 400 88 and 85, 1003 x 400 91 and 95, hence a third of
    // the SMs.
    const bool few = m <= (int64_t)QB_ROWS_FEW * (far_form ? t.num_sms : t.num_sms / 3);
    const int rows = few ? QB_ROWS_FEW : QB_ROWS;
    const dim3 grid((unsigned)((r1 - r0 + rows - 1) / rows));
    const size_t smem = quant_block_smem_bytes(far_form, static_groups, rows);
    // Near form, more CTAs than SMs: two to an SM, one works while the other waits for its own chain, although each has 80
    // registers then and spills some (16384 rows of 400 columns 375 us, with one 390; 8192 of 1023 899, 907; static groups 416, 435
    // and 939, 972; with a grid every 32 columns 4768 rows of 500 columns 204, 213, 16384 of 1023 1740, 1770); below that
    // one, which has the registers of both (1023 columns: 2048 rows 355, two 408; 4736 rows 535, 584).
    const bool two = grid.x > (unsigned)t.num_sms;
    // Near form, from the second launch of a call on: it starts while the product before it drains, and reads U and P meanwhile
    // (1000 rows of 1024 columns 256 -> 242 us a call).  That takes two things: the first launch of a call is a plain one, so that
    // all that made U and P is done before the call's first kernel begins, in a captured graph too; and nothing in a call writes U or P.
    const bool pdl = !far_form && i0 > 0;
    auto launch = [&](auto kernel, int threads) { return launch_pdl(pdl, kernel, grid, dim3(threads), smem, s, uh, ul, ph, pl, u32, p32, a); };
    if (few) {
        if (far_form) return static_groups ? launch(quant_block_kernel<true, true, 1, QB_ROWS_FEW>, QB_THREADS_FAR) : launch(quant_block_kernel<true, false, 1, QB_ROWS_FEW>, QB_THREADS_FAR);
        return static_groups ? launch(quant_block_kernel<false, true, 1, QB_ROWS_FEW>, QB_THREADS_NEAR) : launch(quant_block_kernel<false, false, 1, QB_ROWS_FEW>, QB_THREADS_NEAR);
    }
    if (far_form) return static_groups ? launch(quant_block_kernel<true, true, 1>, QB_THREADS_FAR) : launch(quant_block_kernel<true, false, 1>, QB_THREADS_FAR);
    if (static_groups) return two ? launch(quant_block_kernel<false, true, 2>, QB_THREADS_NEAR) : launch(quant_block_kernel<false, true, 1>, QB_THREADS_NEAR);
    return two ? launch(quant_block_kernel<false, false, 2>, QB_THREADS_NEAR) : launch(quant_block_kernel<false, false, 1>, QB_THREADS_NEAR);
}

// Raises the shared-memory limits of the kernels of the column loop.
cudaError_t configure_quantize_kernels() {
    const cudaFuncAttribute attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e = cudaFuncSetAttribute(column_loop_kernel<4>, attr, 2 * 128 * 128 * (int)sizeof(float));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(column_loop_kernel<2>, attr, 2 * 64 * 64 * (int)sizeof(float));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(quant_block_kernel<true, true, 1>, attr, (int)quant_block_smem_bytes(true, true, QB_ROWS));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(quant_block_kernel<true, false, 1>, attr, (int)quant_block_smem_bytes(true, false, QB_ROWS));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(quant_block_kernel<false, true, 1>, attr, (int)quant_block_smem_bytes(false, true, QB_ROWS));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(quant_block_kernel<false, true, 2>, attr, (int)quant_block_smem_bytes(false, true, QB_ROWS));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(quant_block_kernel<false, false, 1>, attr, (int)quant_block_smem_bytes(false, false, QB_ROWS));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(quant_block_kernel<false, false, 2>, attr, (int)quant_block_smem_bytes(false, false, QB_ROWS));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(quant_block_kernel<true, true, 1, QB_ROWS_FEW>, attr, (int)quant_block_smem_bytes(true, true, QB_ROWS_FEW));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(quant_block_kernel<true, false, 1, QB_ROWS_FEW>, attr, (int)quant_block_smem_bytes(true, false, QB_ROWS_FEW));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(quant_block_kernel<false, true, 1, QB_ROWS_FEW>, attr, (int)quant_block_smem_bytes(false, true, QB_ROWS_FEW));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(quant_block_kernel<false, false, 1, QB_ROWS_FEW>, attr, (int)quant_block_smem_bytes(false, false, QB_ROWS_FEW));
    return e;
}

gptaq_status_t check_quantize_args(int64_t n, const void *d_W, int w_dtype, int64_t m, int64_t ldw, int bits,
                                   int group, int blocksize, const uint8_t *d_codes, const float *d_scales,
                                   const float *d_zeros, const float *d_Wq) {
    if (bits < 2 || bits > 8 || !valid_block(blocksize) || group < 0 ||
        (w_dtype != GPTAQ_W_FP32 && w_dtype != GPTAQ_W_BF16))
        return GPTAQ_ERR_UNSUPPORTED;
    if (group > 0 && (blocksize % group) != 0) return GPTAQ_ERR_UNSUPPORTED;
    if (m == 0) return GPTAQ_OK;
    if (!d_W || !d_codes || !d_scales || !d_zeros || ldw < n) return GPTAQ_ERR_INVALID_ARG;
    if (w_dtype == GPTAQ_W_BF16 && !d_Wq) return GPTAQ_ERR_INVALID_ARG;
    return GPTAQ_OK;
}

#define QLAUNCHED()                                          \
    do {                                                     \
        cudaError_t e__ = cudaGetLastError();                \
        if (e__ != cudaSuccess) { *err = e__; return GPTAQ_ERR_CUDA; } \
        ++*launches;                                         \
    } while (0)

// Rows per CTA of the column permutations: PERM_ROWS while two CTAs fit an SM, then fewer.
int perm_rows(int n, size_t element) { return std::max(1, std::min(PERM_ROWS, (int)(100 * 1024 / (n * element)))); }

// Algorithm 1, the blocked loop: launch sequence shared by the entry points that quantize.
gptaq_status_t quantize_core(const QuantizeTarget &t, void *d_W, int w_dtype, int64_t m, int64_t ldw,
                             int bits, int group, int sym, int blocksize, uint8_t *d_codes, float *d_scales,
                             float *d_zeros, float *d_Wq, cudaStream_t s, int64_t *launches, cudaError_t *err) {
    const int n = t.n;
    float *EW = t.EW;
    float *Wk = static_cast<float *>(d_W);
    int64_t ldk = ldw;
    // grids per output channel, per group of whole 32-column steps, or per column (static groups): quant_block_kernel.
    // Smaller groups take column_loop_kernel (one warp per row, any group).
    const bool static_groups = t.static_groups && group > 0;
    const bool steps = group <= 0 || (group % 32) == 0 || static_groups;
    const bool tensor = t.UT16 != nullptr;
    // columns per launch: as many as the slab holds (and the scratch has room for the errors of), else the caller's block
    const int SW = !steps ? blocksize : tensor ? QB_SUPER : (n <= QB_W || t.ew_floats >= m * 2 * QB_W) ? QB_W : blocksize;
    // A single launch for all columns reads the caller's weights itself, and makes the grids per channel of a single block (whose
    // columns are then a group like another): the copy or the grids' launch is 3 to 30 us a call (1003 x 128 with groups 21.3 -> 17.2,
    // 333 x 128 from bfloat16 19.5 -> 14.3, 512 x 512 with groups 60 -> 55, 8192 x 128 29.5 -> 24.6).
    const bool direct = steps && !t.perm && n <= SW;
    const bool grid_inside = direct && group <= 0 && n <= QB_W && t.clip_steps == 0;
    const int kernel_group = grid_inside ? QB_W : group;
    const void *src = nullptr;
    if (t.perm) {
        // working copy in sorted column order (the caller's d_Wq; checked to be a second buffer)
        const size_t esz = w_dtype == GPTAQ_W_BF16 ? sizeof(__nv_bfloat16) : sizeof(float);
        const int rows = perm_rows(n, esz);
        const unsigned grid = (unsigned)std::min<int64_t>((m + rows - 1) / rows, t.num_sms * 8);
        if (w_dtype == GPTAQ_W_BF16)
            gather_cols_kernel<__nv_bfloat16><<<grid, 256, rows * n * esz, s>>>(static_cast<const __nv_bfloat16 *>(d_W), ldw, d_Wq, n,
                                                                              (int)m, n, t.perm, nullptr, rows);
        else
            gather_cols_kernel<float><<<grid, 256, rows * n * esz, s>>>(static_cast<const float *>(d_W), ldw, d_Wq, n, (int)m, n,
                                                                      t.perm, nullptr, rows);
        QLAUNCHED();
        Wk = d_Wq; ldk = n;
    } else if (w_dtype == GPTAQ_W_BF16 || (d_Wq && d_Wq != d_W)) {
        Wk = d_Wq; ldk = n;
        if (direct) src = d_W;
        else if (group > 0) {
            const dim3 grid((unsigned)((n + 1023) / 1024), (unsigned)std::min<int64_t>((m + WIDEN_ROWS - 1) / WIDEN_ROWS, 65535));
            if (w_dtype == GPTAQ_W_BF16)
                widen_kernel<__nv_bfloat16><<<grid, 256, 0, s>>>(static_cast<const __nv_bfloat16 *>(d_W), ldw, d_Wq, n, (int)m, n);
            else widen_kernel<float><<<grid, 256, 0, s>>>(static_cast<const float *>(d_W), ldw, d_Wq, n, (int)m, n);
            QLAUNCHED();
        }
    }

    const int G = group > 0 ? (n + group - 1) / group : 1;
    if (static_groups) {
        // grids of the original weights (the caller's d_W in its own column order is still untouched)
        const unsigned sg_grid = (unsigned)(((int64_t)m * G + 7) / 8);
        if (w_dtype == GPTAQ_W_BF16)
            static_group_grid_kernel<__nv_bfloat16><<<sg_grid, 256, 0, s>>>(static_cast<const __nv_bfloat16 *>(d_W), ldw, (int)m, n,
                                                                           group, G, t.dead_orig, bits, sym, d_scales, d_zeros,
                                                                           t.clip_steps, t.clip_min);
        else
            static_group_grid_kernel<float><<<sg_grid, 256, 0, s>>>(static_cast<const float *>(d_W), ldw, (int)m, n, group, G,
                                                                   t.dead_orig, bits, sym, d_scales, d_zeros, t.clip_steps,
                                                                   t.clip_min);
        QLAUNCHED();
    }
    if (group <= 0 && !grid_inside) {
        // (from the caller's rows, with the working copy made on the way; in sorted order that exists already)
        const unsigned rg = (unsigned)((m + 7) / 8);
        const bool own = t.perm || Wk == d_W;
        float *copy = own || direct ? nullptr : Wk;
        if (w_dtype == GPTAQ_W_BF16 && !own)
            row_grid_kernel<__nv_bfloat16><<<rg, 256, 0, s>>>(static_cast<const __nv_bfloat16 *>(d_W), ldw, copy, ldk, (int)m, n, t.dead, bits,
                                                              sym, d_scales, d_zeros, t.clip_steps, t.clip_min);
        else
            row_grid_kernel<float><<<rg, 256, 0, s>>>(own ? Wk : static_cast<const float *>(d_W), own ? ldk : ldw, copy, ldk, (int)m, n, t.dead,
                                                      bits, sym, d_scales, d_zeros, t.clip_steps, t.clip_min);
        QLAUNCHED();
    }

    TcMaps maps;
    if (tensor) {
        const size_t nn = (size_t)n * t.ldt, me = (size_t)m * 2 * SW;
        const SplitOperand A{t.EW16, t.EW16 + me, m, 2 * SW, 2 * SW};
        const SplitOperand B{t.UT16, t.UT16 + nn, n, n, t.ldt}, B2{t.PT16, t.PT16 + nn, n, n, t.ldt};
        if (!make_tc_maps(&maps, A, B, &B2)) { *err = cudaErrorUnknown; return GPTAQ_ERR_CUDA; }
    }
    if (steps && tensor) {
        // More rows than one round of CTAs: two halves of the rows on two streams, so that one half's launches fill the SMs
        // that the last round of the other's leaves idle (16384 x 4096, four rounds for 3.5: 3455 us, in one piece
        // 3696; 5000 x 4096, two for 1.06: 1256, 1713).  Rows that one round takes gain nothing (4096 x 4096 1045, 1030).
        struct Part { int64_t r0, r1; cudaStream_t s; } parts[2] = {{0, m, s}, {m, m, t.side}};
        if (t.side && m > (int64_t)QB_ROWS * t.num_sms) {
            parts[0].r1 = parts[1].r0 = (m / 2 + TBM - 1) / TBM * TBM;
            *err = cudaEventRecord(t.fork, s);
            if (*err == cudaSuccess) *err = cudaStreamWaitEvent(t.side, t.fork, 0);
            if (*err != cudaSuccess) return GPTAQ_ERR_CUDA;
        }
        for (int i0 = 0; i0 < n; i0 += SW) {
            const int i1 = std::min(i0 + SW, n);
            for (const Part &p : parts) {
                if (p.r0 == p.r1) continue;
                *err = launch_quant_block(t, Wk, ldk, src, ldw, w_dtype, p.r0, p.r1, m, i0, i1, SW, bits, kernel_group, sym, d_codes, d_scales, d_zeros, G,
                                          static_groups, p.s);
                if (*err != cudaSuccess) return GPTAQ_ERR_CUDA;
                ++*launches;
                if (i1 >= n) continue;
                // W[:, i1:] += [-Err | Wpre] * [U[blk, i1:] ; P[blk, i1:]] on the tensor cores: B operand rows
                // are rows i1.. of U^T (first SW contraction steps) and of P^T (the next SW)
                TcGemmArgs g = tc_args(Wk + p.r0 * ldk + i1, ldk, (int)(p.r1 - p.r0), n - i1, 2 * SW, 1.f, 1.f, TC_FULL, TC_MASK_NONE, t.hd);
                g.a_row0 = (int)p.r0;
                g.b_row0 = i1; g.b_k0 = i0; g.k_split = SW; g.b2_k0 = i0;
                g.row_inv = t.row_inv + p.r0; g.amax_b = t.amax_u;
                *err = launch_tc_gemm(maps, g, t.num_sms, p.s, false, p.s == t.side);
                if (*err != cudaSuccess) return GPTAQ_ERR_CUDA;
                ++*launches;
            }
        }
        if (parts[1].r0 < parts[1].r1) {
            *err = cudaEventRecord(t.join, t.side);
            if (*err == cudaSuccess) *err = cudaStreamWaitEvent(s, t.join, 0);
            if (*err != cudaSuccess) return GPTAQ_ERR_CUDA;
        }
    } else for (int i0 = 0; i0 < n; i0 += SW) {
        const int i1 = std::min(i0 + SW, n);
        if (steps) {
            *err = launch_quant_block(t, Wk, ldk, src, ldw, w_dtype, 0, m, m, i0, i1, SW, bits, kernel_group, sym, d_codes, d_scales, d_zeros, G,
                                      static_groups, s);
            if (*err != cudaSuccess) return GPTAQ_ERR_CUDA;
            ++*launches;
        } else {
            ColumnLoopArgs a;
            a.W = Wk; a.ldw = ldk; a.m = (int)m; a.n = n; a.U = t.U; a.P = t.P; a.dead = t.dead;
            a.i0 = i0; a.bw = i1 - i0;
            a.bits = bits; a.group = group; a.sym = sym;
            a.codes = d_codes; a.scales = d_scales; a.zeros = d_zeros; a.G = G; a.EW = EW; a.hd = t.hd;
            a.amax_u = t.amax_u; a.amax_p = t.amax_p;
            a.perm = t.perm; a.clip_steps = t.clip_steps; a.clip_min = t.clip_min;
            a.err_scale = (t.terms & GPTAQ_TERM_ERR) ? 1.f : 0.f; a.asym_scale = (t.terms & GPTAQ_TERM_ASYM) ? 1.f : 0.f;
            const int nw = std::max(1, std::min(32, (int)((m + t.num_sms - 1) / t.num_sms)));
            const unsigned cl_grid = (unsigned)((m + nw - 1) / nw);
            const size_t cl_smem = 2 * (size_t)blocksize * blocksize * sizeof(float);
            const int T = blocksize / 32;
            if (T == 4) column_loop_kernel<4><<<cl_grid, nw * 32, cl_smem, s>>>(a);
            else if (T == 2) column_loop_kernel<2><<<cl_grid, nw * 32, cl_smem, s>>>(a);
            else column_loop_kernel<1><<<cl_grid, nw * 32, cl_smem, s>>>(a);
            QLAUNCHED();
            if (tensor && i1 < n) {
                // [-Err | rho Wpre] scaled row by row and split here (quant_block_kernel does so itself)
                rowscale_split16_kernel<<<(unsigned)((m + 7) / 8), 256, 0, s>>>(EW, 2 * SW, (int)m, 2 * SW, t.EW16,
                                                                              t.EW16 + (size_t)m * 2 * SW, t.row_inv);
                QLAUNCHED();
            }
        }
        if (i1 >= n) break;
        if (tensor) {
            // the same update behind column_loop_kernel
            TcGemmArgs g = tc_args(Wk + i1, ldk, (int)m, n - i1, 2 * SW, 1.f, 1.f, TC_FULL, TC_MASK_NONE, t.hd);
            g.b_row0 = i1; g.b_k0 = i0; g.k_split = SW; g.b2_k0 = i0;
            g.row_inv = t.row_inv; g.amax_b = t.amax_u;
            *err = launch_tc_gemm(maps, g, t.num_sms, s, false);
            if (*err != cudaSuccess) return GPTAQ_ERR_CUDA;
            ++*launches;
        } else {
            // W[:, i1:] += [-Err | Wpre] * [U[blk, i1:] ; P[blk, i1:]]   (lazy-batch update)
            Operand bop = make_operand(t.U + (int64_t)i0 * n + i1, 1, n);
            bop.p2 = t.P + (int64_t)i0 * n + i1;
            bop.k_split = SW;
            // (early up to four CTAs per SM, the column loop leaves most of the SMs free: 128 x 1024 194 us plain, 182 early; 256 x 1024,
            // 448 CTAs at first, 198 and 192; 512 x 1024, 896 CTAs, 213 and 224; 1000 x 1024 242 and 250)
            GemmProblem pt = make_problem(make_operand(EW, 2 * SW, 1), bop, Wk + i1, ldk, (int)m, n - i1, 2 * SW, 1.f, 1.f, GEMM_FULL);
            *err = launch_simt_gemm(pt, false, true, s, steps ? 4 * t.num_sms : 0);
            if (*err != cudaSuccess) return GPTAQ_ERR_CUDA;
            ++*launches;
        }
    }
    if (t.perm) {
        // dequantized weights back to the caller's column order
        const int rows = perm_rows(n, sizeof(float));
        const unsigned grid = (unsigned)std::min<int64_t>((m + rows - 1) / rows, t.num_sms * 8);
        unpermute_rows_kernel<<<grid, 256, rows * n * sizeof(float), s>>>(Wk, ldk, (int)m, n, t.perm, rows);
        QLAUNCHED();
    }
    return GPTAQ_OK;
}


// ---------------------------------------------------------------------------
// Built-in scratch of gptaq_quantize_static: one array per GPU that loads the library, held
// until the process exits.  Layout: status header | dead-input flags (all zero) | [-Err | Wpre].
// In host code the array's name is only a stand-in for the symbol, not a device address; the
// address that kernels may use is looked up once per device with cudaGetSymbolAddress.
// ---------------------------------------------------------------------------
constexpr size_t STATIC_FLAGS_OFFSET = 256;
constexpr size_t STATIC_EW_OFFSET = STATIC_FLAGS_OFFSET + GPTAQ_STATIC_MAX_N;
constexpr size_t STATIC_SCRATCH_BYTES = STATIC_EW_OFFSET + (size_t)GPTAQ_STATIC_SCRATCH_FLOATS * sizeof(float);
static_assert(STATIC_EW_OFFSET % 256 == 0, "scratch alignment");
static_assert(sizeof(StateHeader) <= STATIC_FLAGS_OFFSET, "header fits");

static __device__ __align__(256) unsigned char g_static_scratch[STATIC_SCRATCH_BYTES];

struct StaticScratch {
    bool ready;
    uint8_t *base;
    int num_sms;
};
constexpr int MAX_DEVICES = 64;
StaticScratch g_static_table[MAX_DEVICES];
std::mutex g_static_mutex;

__global__ void export_status_kernel(const StateHeader *hd, int64_t *out) {
    out[0] = hd->status;
    out[1] = hd->info;
}

// Set-up on first use, once per device, with that device current: resolves the device address
// of the scratch array and raises the shared-memory limit of the column-loop kernels.
cudaError_t static_scratch_for_current_device(StaticScratch **out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= MAX_DEVICES) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_static_mutex);
    StaticScratch &sc = g_static_table[dev];
    if (!sc.ready) {
        void *ptr = nullptr;
        e = cudaGetSymbolAddress(&ptr, g_static_scratch);
        if (e != cudaSuccess) return e;
        e = cudaDeviceGetAttribute(&sc.num_sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        e = configure_quantize_kernels();
        if (e != cudaSuccess) return e;
        sc.base = static_cast<uint8_t *>(ptr);
        sc.ready = true;
    }
    *out = &sc;
    return cudaSuccess;
}

}  // namespace

extern "C" {

size_t gptaq_state_bytes(int64_t n) {
    if (n <= 0) return 0;
    return state_layout(n).total;
}

size_t gptaq_workspace_bytes(int64_t n, int64_t m_max, int64_t max_batch_tokens, int blocksize) {
    if (n <= 0 || m_max < 0 || max_batch_tokens < 0 || !valid_block(blocksize)) return 0;
    // the fp16 operand copies of one token batch share the space of the later steps' scratch
    size_t kp = round_up((size_t)max_batch_tokens, (size_t)UBK);
    size_t xt = 2 * round_up(3 * (size_t)n * kp * 2, ALIGN) + stats_scratch_bytes(MAX_SMS_FOR_SIZING);
    return std::max(ws_layout(n, m_max).total, xt);
}

gptaq_status_t gptaq_create(gptaq_handle_t *out, int64_t n, void *d_state, size_t state_bytes,
                            void *d_workspace, size_t workspace_bytes, gptaq_stream_t stream) {
    if (!out) return GPTAQ_ERR_INVALID_ARG;
    *out = nullptr;
    if (n <= 0 || n > (int64_t)1 << 20 || !d_state || !d_workspace) return GPTAQ_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(d_state) % ALIGN) || (reinterpret_cast<uintptr_t>(d_workspace) % ALIGN))
        return GPTAQ_ERR_INVALID_ARG;
    Layout l = state_layout(n);
    if (state_bytes < l.total) return GPTAQ_ERR_WORKSPACE;
    if (workspace_bytes < ws_layout(n, 0).total) return GPTAQ_ERR_WORKSPACE;
    gptaq_ctx *h = new (std::nothrow) gptaq_ctx();
    if (!h) return GPTAQ_ERR_INVALID_ARG;
    h->n = n;
    h->state = static_cast<char *>(d_state);
    h->state_bytes = state_bytes;
    h->ws = static_cast<char *>(d_workspace);
    h->ws_bytes = workspace_bytes;
    h->hd = reinterpret_cast<StateHeader *>(h->state);
    h->H = reinterpret_cast<float *>(h->state + l.h_off);
    h->D = reinterpret_cast<float *>(h->state + l.d_off);
    h->dead = reinterpret_cast<uint8_t *>(h->state + l.dead_off);
    h->dead_raw = reinterpret_cast<uint8_t *>(h->state + l.dead_raw_off);
    h->perm = reinterpret_cast<int *>(h->state + l.perm_off);
    h->act_order = false;
    h->launches = 0;
    h->stats_precision = GPTAQ_STATS_FP16_SPLIT_TENSOR;
    h->tensor = tc_shape_ok(n) && encode_tiled_fn() != nullptr;
    h->terms = GPTAQ_TERM_ERR | GPTAQ_TERM_ASYM;
    h->clip_steps = 0; h->clip_min = 1.f;
    h->static_groups = false;
    h->kernel_timing = false;
    h->timing_used = 0;
    cudaError_t e = cudaGetDevice(&h->device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, h->device);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(invert_diag_block_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ID_SMEM);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(diag_factor_kernel<DF_LAST>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DF_SMEM_LAST);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(diag_factor_kernel<DF_BLOCK>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DF_SMEM);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(diag_factor_kernel<DF_WHOLE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DF_SMEM_WHOLE);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(panel_solve_kernel<2, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PS_SMEM);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(panel_solve_kernel<4, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PS_SMEM);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(panel_solve_kernel<4, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PS_SMEM);
    if (e == cudaSuccess) e = configure_quantize_kernels();
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(p_narrow_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)np_smem(NP_MAX_N));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(stats_umma_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)UMMA_SMEM);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(tc_gemm_kernel<256>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tc_smem(256));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(tc_gemm_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tc_smem(128));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(tc_gemm_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tc_smem(64));
    // the conversion of the next batch shares the SMs with the running product: both kernels ask for
    // the largest shared-memory carve-out, so that a conversion CTA fits beside a product CTA
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(stats_umma_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(convert_transpose_kernel<0>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(convert_transpose_kernel<1>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(unpermute_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ACT_ORDER_MAX_N * 4);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(gather_cols_kernel<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ACT_ORDER_MAX_N * 4);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(gather_cols_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ACT_ORDER_MAX_N * 4);
    if (e != cudaSuccess) {
        delete h;
        return GPTAQ_ERR_CUDA;
    }
    h->gemm_stream = h->inv_stream = nullptr;
    h->inv_ready = h->inv_done = nullptr;
    h->relayout = false;
    h->next_buf = 0;
    h->stats_maps[0].kp = h->stats_maps[1].kp = 0;
    h->fix_pending = false;
    h->d_upper_only = false;
    for (int i = 0; i < 2; ++i) { h->conv_done[i] = h->gemm_done[i] = nullptr; h->gemm_pending[i] = false; }
    {
        // highest priority: when a product and the conversion of the next batch become ready together, the
        // product's CTAs (one per SM, nearly all of its shared memory) are placed first and the conversion
        // fills the SMs that the product's last round of tiles leaves idle
        int prio_lo = 0, prio_hi = 0;
        e = cudaDeviceGetStreamPriorityRange(&prio_lo, &prio_hi);
        if (e == cudaSuccess) e = cudaStreamCreateWithPriority(&h->gemm_stream, cudaStreamNonBlocking, prio_hi);
    }
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&h->inv_stream, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&h->inv_ready, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&h->inv_done, cudaEventDisableTiming);
    for (int i = 0; i < 2 && e == cudaSuccess; ++i) {
        e = cudaEventCreateWithFlags(&h->conv_done[i], cudaEventDisableTiming);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&h->gemm_done[i], cudaEventDisableTiming);
    }
    if (e != cudaSuccess) {
        gptaq_destroy(h);
        return GPTAQ_ERR_CUDA;
    }
    gptaq_status_t st = gptaq_reset(h, stream);
    if (st != GPTAQ_OK) {
        gptaq_destroy(h);
        return st;
    }
    *out = h;
    return GPTAQ_OK;
}

gptaq_status_t gptaq_reset(gptaq_handle_t h, gptaq_stream_t stream) {
    if (!h) return GPTAQ_ERR_INVALID_ARG;
    Layout l = state_layout(h->n);
    OK(join_statistics(h, static_cast<cudaStream_t>(stream)));
    CU(cudaMemsetAsync(h->state, 0, l.total, static_cast<cudaStream_t>(stream)));
    h->stage = STAGE_ACCUM;
    h->tokens = 0;
    h->d_upper_only = false;
    return GPTAQ_OK;
}

gptaq_status_t gptaq_destroy(gptaq_handle_t h) {
    if (!h) return GPTAQ_ERR_INVALID_ARG;
    if (h->gemm_stream) {
        cudaStreamSynchronize(h->gemm_stream);
        cudaStreamDestroy(h->gemm_stream);
    }
    if (h->inv_stream) {
        cudaStreamSynchronize(h->inv_stream);
        cudaStreamDestroy(h->inv_stream);
    }
    if (h->inv_ready) cudaEventDestroy(h->inv_ready);
    if (h->inv_done) cudaEventDestroy(h->inv_done);
    for (int i = 0; i < 2; ++i) {
        if (h->conv_done[i]) cudaEventDestroy(h->conv_done[i]);
        if (h->gemm_done[i]) cudaEventDestroy(h->gemm_done[i]);
    }
    for (auto &ev : h->timing_events) { cudaEventDestroy(ev.first); cudaEventDestroy(ev.second); }
    delete h;
    return GPTAQ_OK;
}

gptaq_status_t gptaq_accumulate(gptaq_handle_t h, const float *d_X, const float *d_Xfp,
                                int64_t tokens, int64_t ld, gptaq_stream_t stream) {
    if (!h || tokens < 0 || tokens > INT32_MAX) return GPTAQ_ERR_INVALID_ARG;
    if (h->stage != STAGE_ACCUM) return GPTAQ_ERR_BAD_STATE;
    if (tokens == 0) return GPTAQ_OK;
    if (!d_X || !d_Xfp || ld < h->n) return GPTAQ_ERR_INVALID_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int n = (int)h->n;
    if (tc_eligible(h) && tokens > STATS_FP32_WORK / (h->n * h->n))
        return join_after_error(h, s, accumulate_tc(h, d_X, d_Xfp, tokens, ld, s));
    OK(join_statistics(h, s));
    // H (upper tiles) += X X^T
    Operand xa = make_operand(d_X, 1, ld);
    GemmProblem ph = make_problem(xa, xa, h->H, n, n, n, (int)tokens, 1.f, 1.f, GEMM_UPPER_TILES);
    // (narrow layers: with the second sum in one launch)
    GemmProblem both = ph;
    both.nbatch = 2; both.paired = 1; both.pair_mode = GEMM_FULL; both.pair_sub = d_Xfp; both.pair_C = h->D;
    if (simt_tiles(both) <= SIMT_SMALL_TILES) {
        OK(gemm(h, both, true, true, s));
        h->tokens += tokens;
        return GPTAQ_OK;
    }
    OK(gemm(h, ph, true, true, s));
    // dXX^T += (X~ - X) X^T, the difference taken in float32 at load time
    Operand da = xa;
    da.sub = d_Xfp;
    GemmProblem pd = make_problem(da, xa, h->D, n, n, n, (int)tokens, 1.f, 1.f, GEMM_FULL);
    OK(gemm(h, pd, true, true, s));
    h->tokens += tokens;
    return GPTAQ_OK;
}

gptaq_status_t gptaq_flush(gptaq_handle_t h, gptaq_stream_t stream) {
    if (!h) return GPTAQ_ERR_INVALID_ARG;
    return join_statistics(h, static_cast<cudaStream_t>(stream));
}

gptaq_status_t gptaq_accumulate_host(gptaq_handle_t h, const float *h_X, const float *h_Xfp,
                                     int64_t tokens, int64_t ld, void *d_stage, size_t stage_bytes,
                                     gptaq_stream_t stream) {
    if (!h || tokens < 0) return GPTAQ_ERR_INVALID_ARG;
    if (h->stage != STAGE_ACCUM) return GPTAQ_ERR_BAD_STATE;
    if (tokens == 0) return GPTAQ_OK;
    if (!h_X || !h_Xfp || !d_stage || ld < h->n) return GPTAQ_ERR_INVALID_ARG;
    size_t one = (size_t)tokens * (size_t)h->n * sizeof(float);
    if (stage_bytes < 2 * one) return GPTAQ_ERR_WORKSPACE;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    float *dx = static_cast<float *>(d_stage);
    float *dxfp = dx + (size_t)tokens * (size_t)h->n;
    size_t rowb = (size_t)h->n * sizeof(float);
    CU(cudaMemcpy2DAsync(dx, rowb, h_X, (size_t)ld * sizeof(float), rowb, (size_t)tokens,
                         cudaMemcpyHostToDevice, s));
    CU(cudaMemcpy2DAsync(dxfp, rowb, h_Xfp, (size_t)ld * sizeof(float), rowb, (size_t)tokens,
                         cudaMemcpyHostToDevice, s));
    return gptaq_accumulate(h, dx, dxfp, tokens, h->n, stream);
}

// gptaq_factor behind its argument checks.
static gptaq_status_t factor_core(gptaq_ctx *h, float damp, cudaStream_t s) {
    OK(join_statistics(h, s));
    const int n = (int)h->n;
    const int nb = (n + NB - 1) / NB;
    WsLayout wl = ws_layout(h->n, 0);
    float *T = reinterpret_cast<float *>(h->ws + wl.t_off);
    float *Rinv = reinterpret_cast<float *>(h->ws + wl.rinv_off);
    float *H = h->H;

    const float inv_tokens = (float)(1.0 / (double)h->tokens);
    if (nb == 1 && !h->act_order) {
        DiagFactorArgs da = {};
        da.src = H; da.lds = n; da.n = n; da.H = H; da.hd = h->hd;
        da.inv_tokens = inv_tokens; da.damp = damp; da.dead = h->dead_raw; da.dead_working = h->dead;
        CUtensorMap none;
        std::memset(&none, 0, sizeof(none));
        CU(launch_pdl(false, diag_factor_kernel<DF_WHOLE>, dim3(1), dim3(DF_THREADS), DF_SMEM_WHOLE, s, none, none, da));
        h->launches++;
        h->split = false;
        h->stage = STAGE_FACTORED;
        return GPTAQ_OK;
    }
    diag_stats_kernel<<<1, 1024, 0, s>>>(H, n, inv_tokens, damp, h->hd, h->dead_raw, h->act_order ? nullptr : h->dead);
    LAUNCHED();
    if (h->act_order) {
        // columns in order of decreasing diag(H): dXX^T and H are permuted on both sides, through T (H stays there until it
        // is scaled)
        rank_desc_kernel<<<(n + RANK_COLS - 1) / RANK_COLS, 256, 0, s>>>(H, n, inv_tokens, h->dead_raw, h->perm, h->dead);
        LAUNCHED();
        const int rows = perm_rows(n, sizeof(float));
        gather_cols_kernel<float><<<std::min((n + rows - 1) / rows, h->num_sms * 8), 256, rows * n * sizeof(float), s>>>(h->D, n, T, n, n, n, h->perm, h->perm, rows);
        LAUNCHED();
        CU(cudaMemcpyAsync(h->D, T, (size_t)n * n * sizeof(float), cudaMemcpyDeviceToDevice, s));
        permute_symmetric_kernel<<<dim3((n + 255) / 256, n), 256, 0, s>>>(H, T, n, h->perm);
        LAUNCHED();
    }
    CU(launch_pdl(true, scale_damp_kernel, dim3((n + 63) / 64, (n + 15) / 16), dim3(256), 0, s, static_cast<const float *>(h->act_order ? T : H),
                  H, n, static_cast<const StateHeader *>(h->hd), static_cast<const uint8_t *>(h->dead)));
    h->launches++;

    // Rank updates and the inverse on split operands, with damping: the rows of R lie between sqrt(lambda) and
    // sqrt(max diag H_d), those of its inverse between 1 / sqrt of these, and as lambda = damp * mean(diag) the two are at most
    // sqrt(n / damp) apart (453 at n = 2052, damp = 0.01), while the parts keep their 22 bits down to 2^-17 of the largest entry.
    // Without damping nothing bounds them: plain float32 (units of the inputs that span 1e4, relative error of U at n = 2052
    // 1.9e-6 with split rank updates, 2.2e-7 without; n = 1024 / 2052 / 4096 / 8192 split 0.29, 1.26, 2.37,
    // 8.5 ms when that was last built, plain now 0.29, 0.95, 2.81, 14.1).
    const bool split = h->tensor && damp > 0.f;
    // reverse Cholesky H_d = R R^T, R upper, from the last block column upwards
    __half *pan_hi = split ? reinterpret_cast<__half *>(h->ws + wl.pan_off[0]) : nullptr;
    __half *pan_lo = split ? reinterpret_cast<__half *>(h->ws + wl.pan_off[1]) : nullptr;
    TcMaps pan_maps;
    std::memset(static_cast<void *>(&pan_maps), 0, sizeof(pan_maps));
    if (split) {
        const SplitOperand pan{pan_hi, pan_lo, n, SUPER_NB, SUPER_NB};
        if (!make_tc_maps(&pan_maps, pan, pan, nullptr)) { h->cuda_error = "cuTensorMapEncodeTiled failed"; return GPTAQ_ERR_CUDA; }
    }
    float *next_diag = reinterpret_cast<float *>(h->ws + wl.diag_off);
    // rank-NB (or super-panel) update of the columns to the left of panel p, on stream `us` with at most `sms` CTAs
    auto update = [&](int p, cudaStream_t us, int sms) -> gptaq_status_t {
        const int b0 = p * NB;
        const int s0 = b0 / SUPER_NB * SUPER_NB;
        if (split && b0 >= TC_MIN_N) {
            const unsigned *am = h->hd->tc_amax + AMAX_PAN;
            if (b0 > s0) {
                // inside the super-panel: A[0:b0, s0:b0] -= R[0:b0, blk] R[s0:b0, blk]^T  (upper part)
                TcGemmArgs g = tc_args(H + s0, n, b0, b0 - s0, NB, -1.f, 1.f, TC_UPPER_TILES, TC_MASK_UPPER_KEEP, h->hd);
                g.diag_off = s0; g.a_k0 = g.b_k0 = b0 - s0; g.b_row0 = s0;
                g.amax_a = g.amax_b = am;
                CU(launch_tc_gemm(pan_maps, g, sms, us));
            } else {
                // super-panel [s0, s1) done: A[0:s0, 0:s0] -= R[0:s0, s0:s1] R[0:s0, s0:s1]^T  (upper part)
                const int s1 = std::min(s0 + SUPER_NB, nb * NB);
                TcGemmArgs g = tc_args(H, n, s0, s0, s1 - s0, -1.f, 1.f, TC_UPPER_TILES, TC_MASK_UPPER_KEEP, h->hd);
                g.amax_a = g.amax_b = am;
                CU(launch_tc_gemm(pan_maps, g, sms, us));
            }
            h->launches++;
            return GPTAQ_OK;
        }
        // A[0:b0, 0:b0] -= R[0:b0, blk] R[0:b0, blk]^T  (upper part)
        Operand rp = make_operand(H + b0, n, 1);
        GemmProblem ps = make_problem(rp, rp, H, n, b0, b0, std::min(NB, n - b0), -1.f, 1.f, GEMM_UPPER_TILES);
        // (early where it has a CTA per SM at most: gptaq_factor 384 120 -> 116, 777 293 -> 286, 1027 434 -> 428 us)
        return gemm(h, ps, false, false, us, h->num_sms);
    };
    auto factor_diag = [&](int p, const float *src, int64_t lds, int syrk, int pan_col0) -> gptaq_status_t {
        DiagFactorArgs da = {};
        da.src = src; da.lds = lds; da.n = n; da.b0 = p * NB; da.Rdiag = Rinv + (size_t)p * NB * NB;
        da.syrk = syrk; da.pan_col0 = pan_col0; da.hd = h->hd;
        // (a second CTA inverts the block before; block 0 has its own inverse to make, block 1 is inverted beside it)
        da.H = H; da.inv_b0 = (p + 1) * NB; da.inv_Rdiag = da.Rdiag + NB * NB;
        CU(launch_pdl(true, p ? diag_factor_kernel<DF_BLOCK> : diag_factor_kernel<DF_LAST>, dim3(p > 0 && p + 1 < nb ? 2 : 1), dim3(DF_THREADS),
                      p ? DF_SMEM : DF_SMEM_LAST, s, pan_maps.a_hi, pan_maps.a_lo, da));
        h->launches++;
        return GPTAQ_OK;
    };
    // U = R^-1 of each diagonal block of SUPER_NB columns, a row of NB x NB blocks at a time and beside the factorisation:
    //   U[p, p] = R_pp^-1 (beside the next diagonal block),   U[p, > p] = -U[p, p] T[p, > p],   T[i, > i] = R[i, > i] U[> i, > i]
    // T gathers the products of a row of U as soon as that row is there (rows i < p of the super-panel at once, 128 contraction
    // steps each), so that little is left when the last block is factored.  Plain float32 products.
    // R is overwritten: row p comes after panel p is solved, hence after the update that reads it.  Nothing of this is put on
    // the chain's own stream, where every event costs 4 us.
    // These products start early where they have at most a CTA per SM: more of them sit on SMs that the chain's kernels beside
    // them want whole (gptaq_factor, us plain / always early / so: n = 512 136 / 134 / 134, 1024 249 / 252 / 247,
    // 2048 561 / 578 / 559, 4096 1268 / 1313 / 1266).
    cudaStream_t is = nb > 1 ? h->inv_stream : s;
    auto inverse_row = [&](int p) -> gptaq_status_t {
        const int b0 = p * NB, b1 = b0 + NB, e1 = std::min(b0 / SUPER_NB * SUPER_NB + SUPER_NB, n);
        if (b1 >= e1) return GPTAQ_OK;
        GemmProblem pu = make_problem(make_operand(H + (int64_t)b0 * n + b0, n, 1), make_operand(T + (int64_t)b0 * n + b1, 1, n),
                                      H + (int64_t)b0 * n + b1, n, NB, e1 - b1, NB, -1.f, 0.f, GEMM_TRI_LEFT);
        return gemm(h, pu, false, true, is, h->num_sms);
    };
    // T[i, p ..] += R[i, p] U[p, p ..] for the rows i < p of the super-panel (the columns of block p receive their first term)
    auto inverse_gather = [&](int p) -> gptaq_status_t {
        const int b0 = p * NB, q0 = b0 / SUPER_NB * SUPER_NB, e1 = std::min(q0 + SUPER_NB, n);
        if (b0 == q0) return GPTAQ_OK;
        GemmProblem pt = make_problem(make_operand(H + (int64_t)q0 * n + b0, n, 1), make_operand(H + (int64_t)b0 * n + b0, 1, n),
                                      T + (int64_t)q0 * n + b0, n, b0 - q0, e1 - b0, std::min(NB, n - b0), 1.f, 1.f, GEMM_FULL);
        pt.fresh = NB;
        return gemm(h, pt, false, true, is, h->num_sms);
    };
    // Rows of a panel may be read before the diagonal kernel in front of it has finished, because the update that made them is
    // waited for by an event.  In a captured graph that event becomes an edge of the same programmatic kind as the one from
    // the diagonal kernel, and the rows would be read before the update has written them.
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    const bool plain_stream = cudaStreamIsCapturing(s, &capture) == cudaSuccess && capture == cudaStreamCaptureStatusNone;
    bool diag_done = false;                     // the diagonal block of this panel was factored beside the last update
    for (int p = nb - 1; p >= 0; --p) {
        const int b0 = p * NB;
        const int s0 = split ? b0 / SUPER_NB * SUPER_NB : b0;      // first column of this panel's super-panel
        if (!diag_done) OK(factor_diag(p, H + (int64_t)b0 * n + b0, n, 0, 0));
        const bool early = diag_done && plain_stream;        // (diag_done: the update of this panel's columns was waited for)
        diag_done = false;
        if (p == 0) break;
        const bool ahead = split && b0 > s0;   // the next panel is in the same super-panel: its block needs this panel only
        PanelSolveArgs pa;
        pa.H = H; pa.n = n; pa.b0 = b0; pa.Rdiag = Rinv + (size_t)p * NB * NB;
        pa.pan_hi = pan_hi; pa.pan_lo = pan_lo;
        pa.pan_ld = SUPER_NB; pa.pan_col0 = b0 - s0; pa.hd = h->hd;
        pa.next_diag = ahead ? next_diag : nullptr;
        pa.early = early ? 1 : 0;
        // a warp per 2 (4) rows while that fills no SM beyond PS_WORKERS warps, per 8 rows beyond; as few warps per CTA as give
        // every SM at most one CTA
        const int most = PS_WORKERS * h->num_sms, rows = b0 / 2 <= most ? 2 : b0 / 4 <= most ? 4 : 8;
        const int groups = b0 / rows;
        pa.workers = std::max(1, std::min(PS_WORKERS, (groups + h->num_sms - 1) / h->num_sms));
        const int slabs = std::min((groups + pa.workers - 1) / pa.workers, h->num_sms);
        const dim3 pg(slabs + (ahead ? 1 : 0));
        CU(launch_pdl(true, rows == 2 ? panel_solve_kernel<2, 1> : rows == 4 ? panel_solve_kernel<4, 1> : panel_solve_kernel<4, 2>, pg,
                      dim3(PS_THREADS), PS_SMEM, s, pa));
        h->launches++;
        CU(cudaEventRecord(h->inv_ready, s));
        CU(cudaStreamWaitEvent(is, h->inv_ready, 0));
        if (ahead) {
            // the update on the internal stream, the next diagonal block (and this one's inverse) beside it on two SMs left free
            // (p = 1: block 0 is all that the update would reach)
            if (p > 1) {
                CU(cudaStreamWaitEvent(h->gemm_stream, h->inv_ready, 0));
                OK(update(p, h->gemm_stream, h->num_sms - 2));
                CU(cudaEventRecord(h->gemm_done[0], h->gemm_stream));
            }
            OK(factor_diag(p - 1, next_diag, NB, 1, b0 - s0));
            if (p > 1) CU(cudaStreamWaitEvent(s, h->gemm_done[0], 0));
            diag_done = true;
        } else OK(update(p, s, h->num_sms));
        // (block p + 1 was inverted beside block p)
        if (p + 1 < nb) {
            OK(inverse_row(p + 1));
            OK(inverse_gather(p + 1));
        }
        if (p == 1) {
            // Row 1 of the inverse need not wait for block 0: block 1 is inverted beside it by a kernel of its own, and block 0 by its own
            // diagonal kernel (gptaq_factor, us: both behind block 0 n = 384 114, 500 154, 640 162, 777 284, 2048 549; so 108, 147, 156,
            // 277, 545).
            // (on the rows' own stream where no row is under way there, one event less)
            cudaStream_t bs = nb > 2 ? h->gemm_stream : is;
            if (bs != is) CU(cudaStreamWaitEvent(bs, h->inv_ready, 0));
            invert_diag_block_kernel<<<1, ID_THREADS, ID_SMEM, bs>>>(H, n, NB, Rinv + NB * NB);
            LAUNCHED();
            if (bs != is) {
                CU(cudaEventRecord(h->conv_done[0], bs));
                CU(cudaStreamWaitEvent(is, h->conv_done[0], 0));
            }
            OK(inverse_row(1));
            OK(inverse_gather(1));
        }
    }
    if (nb > 1) {
        CU(cudaEventRecord(h->inv_done, is));
        CU(cudaStreamWaitEvent(s, h->inv_done, 0));
    }
    is = s;
    OK(inverse_row(0));

    // U beyond the diagonal blocks of SUPER_NB columns, by doubling:
    // inv([[A, B], [0, C]]) = [[A^-1, -A^-1 B C^-1], [0, C^-1]]
    for (int64_t sz = SUPER_NB; sz < n; sz *= 2) {
        const int np = (int)((n - sz + 2 * sz - 1) / (2 * sz));
        const int tail = (int)(n - (2 * sz * (np - 1) + sz));
        const int64_t bstride = 2 * sz * ((int64_t)n + 1);
        if (split) {
            // The two products on the tensor cores with FP16-split operands.  Ranges: B holds entries of R
            // (bounded like the panels), the inverted blocks are bounded by 1 / sqrt(lambda), the
            // intermediate T records its own maximum in the first product's epilogue.
            const int64_t ldt = split_pitch(n);
            const size_t nn = (size_t)n * ldt;
            __half *A1 = reinterpret_cast<__half *>(h->ws + wl.s_off[0]);     // left operands, K-major at their own coordinates
            __half *B2 = reinterpret_cast<__half *>(h->ws + wl.s_off[1]);     // transposed right operands
            unsigned *am = h->hd->tc_amax;
            const SplitOperand Aop{A1, A1 + nn, n, n, ldt}, Bop{B2, B2 + nn, n, n, ldt};
            TcMaps m16;
            if (!make_tc_maps(&m16, Aop, Bop, nullptr)) { h->cuda_error = "cuTensorMapEncodeTiled failed"; return GPTAQ_ERR_CUDA; }
            SplitBatch sb; sb.nbatch = np; sb.src_bstride = bstride; sb.dst_bstride = 2 * sz * (ldt + 1);
            SplitBatch sbt = sb; sbt.cols_last = tail;
            SplitBatch sbc = sb; sbc.rows_last = tail; sbc.cols_last = tail;
            CU(cudaMemsetAsync(am + AMAX_T, 0, sizeof(unsigned), s));
            CU(launch_split16(split16_args(H + sz, n, A1 + sz, A1 + nn + sz, ldt, (int)sz, (int)sz, false, SPLIT_ALL, 1.f, am + AMAX_PAN, sbt), h->num_sms, s));
            CU(launch_split16(split16_args(H + sz * n + sz, n, B2 + sz * ldt + sz, B2 + nn + sz * ldt + sz, ldt, (int)sz, (int)sz, true,
                                           SPLIT_UPPER, 1.f, am + AMAX_INV, sbc), h->num_sms, s));
            TcGemmArgs g1 = tc_args(T + sz, n, (int)sz, (int)sz, (int)sz, 1.f, 0.f, TC_TRI_RIGHT, TC_MASK_NONE, h->hd);
            g1.nbatch = np; g1.c_bstride = bstride; g1.N_last = tail; g1.K_last = tail;
            g1.a_row0 = 0; g1.a_row_bs = (int)(2 * sz); g1.a_k0 = (int)sz; g1.a_k_bs = (int)(2 * sz);
            g1.b_row0 = (int)sz; g1.b_row_bs = (int)(2 * sz); g1.b_k0 = (int)sz; g1.b_k_bs = (int)(2 * sz);
            g1.amax_a = am + AMAX_PAN; g1.amax_b = am + AMAX_INV; g1.amax_out = am + AMAX_T;
            CU(launch_tc_gemm(m16, g1, h->num_sms, s));
            CU(launch_split16(split16_args(H, n, A1, A1 + nn, ldt, (int)sz, (int)sz, false, SPLIT_UPPER, 1.f, am + AMAX_INV, sb), h->num_sms, s));
            CU(launch_split16(split16_args(T + sz, n, B2 + sz * ldt, B2 + nn + sz * ldt, ldt, (int)sz, (int)sz, true, SPLIT_ALL, 1.f, am + AMAX_T, sbt), h->num_sms, s));
            TcGemmArgs g2 = tc_args(H + sz, n, (int)sz, (int)sz, (int)sz, -1.f, 0.f, TC_TRI_LEFT, TC_MASK_NONE, h->hd);
            g2.nbatch = np; g2.c_bstride = bstride; g2.N_last = tail;
            g2.a_row0 = 0; g2.a_row_bs = (int)(2 * sz); g2.a_k0 = 0; g2.a_k_bs = (int)(2 * sz);
            g2.b_row0 = (int)sz; g2.b_row_bs = (int)(2 * sz); g2.b_k0 = 0; g2.b_k_bs = (int)(2 * sz);
            g2.amax_a = am + AMAX_INV; g2.amax_b = am + AMAX_T;
            CU(launch_tc_gemm(m16, g2, h->num_sms, s));
            h->launches += 6;
            continue;
        }
        // plain float32 products
        // T = B * C^-1
        GemmProblem p1 = make_problem(make_operand(H + sz, n, 1),
                                      make_operand(H + sz * n + sz, 1, n), T + sz, n,
                                      (int)sz, (int)sz, (int)sz, 1.f, 0.f, GEMM_TRI_RIGHT);
        p1.nbatch = np; p1.batchA = p1.batchB = p1.batchC = bstride;
        p1.batchN_last = tail; p1.batchK_last = tail;
        OK(gemm(h, p1, false, true, s));
        // B <- -A^-1 * T
        GemmProblem p2 = make_problem(make_operand(H, n, 1), make_operand(T + sz, 1, n), H + sz, n,
                                      (int)sz, (int)sz, (int)sz, -1.f, 0.f, GEMM_TRI_LEFT);
        p2.nbatch = np; p2.batchA = p2.batchB = p2.batchC = bstride;
        p2.batchN_last = tail;
        OK(gemm(h, p2, false, true, s));
    }
    // Without damping the columns of U go with the reciprocal units of the inputs, and in the contractions of P and of the
    // lazy-batch update the parts' range (2^-39 of the largest entry) is off by the ratio of the units.  Widths that are
    // 4 mod 8 take plain float32 then; the others keep the split operands at any damping.
    h->split = h->tensor && (damp > 0.f || n % 8 == 0);
    h->stage = STAGE_FACTORED;
    return GPTAQ_OK;
}

gptaq_status_t gptaq_factor(gptaq_handle_t h, float damp, gptaq_stream_t stream) {
    if (!h || !(damp >= 0.f) || !std::isfinite(damp)) return GPTAQ_ERR_INVALID_ARG;
    if (h->stage != STAGE_ACCUM || h->tokens <= 0) return GPTAQ_ERR_BAD_STATE;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    return join_after_error(h, s, factor_core(h, damp, s));
}

gptaq_status_t gptaq_build_P(gptaq_handle_t h, float alpha, gptaq_stream_t stream) {
    if (!h || !std::isfinite(alpha)) return GPTAQ_ERR_INVALID_ARG;
    if (h->stage != STAGE_FACTORED) return GPTAQ_ERR_BAD_STATE;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int n = (int)h->n;
    WsLayout wl = ws_layout(h->n, 0);
    float *O = reinterpret_cast<float *>(h->ws + wl.t_off);
    if (h->split) {
        // Every operand is scaled by a power of two into the fp16 range, so its largest magnitude is recorded first (by a
        // reduction kernel for U and dXX^T, by the producing GEMM's epilogue for O and P).  dXX^T and O have a scale per
        // row: a row goes with the unit of the input that it belongs to, and with one scale for the whole matrix the rows of
        // inputs 1e4 below the largest kept 13 of their 22 bits.
        // Workspace: S[0] = U^T (kept for gptaq_quantize), S[1] = U, then P^T (kept), S[2] = dXX^T, then O; the row scales lie
        // where gptaq_factor had the diagonal blocks of R.
        const int64_t ldt = split_pitch(n);
        const size_t nn = (size_t)n * ldt;
        __half *UT16 = reinterpret_cast<__half *>(h->ws + wl.s_off[0]);
        __half *U16 = reinterpret_cast<__half *>(h->ws + wl.s_off[1]);
        __half *A16 = reinterpret_cast<__half *>(h->ws + wl.s_off[2]);
        unsigned *am = h->hd->tc_amax;
        const float inv_tokens = (float)(1.0 / (double)h->tokens);
        unsigned *amax_d = reinterpret_cast<unsigned *>(h->ws + wl.rinv_off), *amax_o = amax_d + n;
        float *inv_d = reinterpret_cast<float *>(amax_o + n), *inv_o = inv_d + n;
        CU(cudaMemsetAsync(am + AMAX_U, 0, 2 * sizeof(unsigned), s));      // slots U, P
        // (of dXX^T only the entries above the diagonal reach O: row j of U starts at column j and M_U keeps j > i)
        CU(launch_absmax({h->H, n, n, n, SPLIT_UPPER, 1.f, am + AMAX_U, nullptr, nullptr},
                         {h->D, n, n, n, SPLIT_STRICT_UPPER, inv_tokens, nullptr, amax_d, amax_o}, h->num_sms, s));
        // U and U^T in one pass, dXX^T in the same launch
        const Split16Args split_d = split16_args(h->D, n, A16, A16 + nn, ldt, n, n, false, SPLIT_STRICT_UPPER, inv_tokens, amax_d, SplitBatch(),
                                                 nullptr, nullptr, inv_d);
        CU(launch_split16(split16_args(h->H, n, U16, U16 + nn, ldt, n, n, false, SPLIT_UPPER, 1.f, am + AMAX_U, SplitBatch(), UT16, UT16 + nn), h->num_sms, s, &split_d));
        h->launches += 2;
        const SplitOperand Uop{U16, U16 + nn, n, n, ldt}, UTop{UT16, UT16 + nn, n, n, ldt};
        const SplitOperand Aop{A16, A16 + nn, n, n, ldt};
        TcMaps maps;
        // O = ((dXX^T / tokens) U^T) .* M_U  (contraction over k >= column, U[a][k] = 0 below)
        if (!make_tc_maps(&maps, Aop, Uop, nullptr)) { h->cuda_error = "cuTensorMapEncodeTiled failed"; return GPTAQ_ERR_CUDA; }
        TcGemmArgs go = tc_args(O, n, n, n, n, 1.f, 0.f, TC_O, TC_MASK_STRICT_ZERO, h->hd);
        go.row_inv = inv_d; go.amax_b = am + AMAX_U; go.row_amax_out = amax_o;
        CU(launch_tc_gemm(maps, go, h->num_sms, s));
        CU(launch_split16(split16_args(O, n, A16, A16 + nn, ldt, n, n, false, SPLIT_STRICT_UPPER, 1.f, amax_o, SplitBatch(), nullptr,
                                       nullptr, inv_o), h->num_sms, s));
        // P = alpha * O U  (B operand rows are rows of U^T)
        if (!make_tc_maps(&maps, Aop, UTop, nullptr)) { h->cuda_error = "cuTensorMapEncodeTiled failed"; return GPTAQ_ERR_CUDA; }
        TcGemmArgs gp = tc_args(h->D, n, n, n, n, alpha, 0.f, TC_P, TC_MASK_STRICT_ZERO, h->hd);
        gp.row_inv = inv_o; gp.amax_b = am + AMAX_U; gp.amax_out = am + AMAX_P;
        CU(launch_tc_gemm(maps, gp, h->num_sms, s));
        // P^T for the lazy-batch updates of gptaq_quantize, over the copy of U that is no longer needed
        CU(launch_split16(split16_args(h->D, n, U16, U16 + nn, ldt, n, n, true, SPLIT_STRICT_UPPER, 1.f, am + AMAX_P), h->num_sms, s));
        h->launches += 4;
        h->stage = STAGE_P;
        return GPTAQ_OK;
    }
    const float scale = (float)((double)alpha / (double)h->tokens);
    if (n <= NP_MAX_N) {
        CU(launch_pdl(true, p_narrow_kernel, dim3((n + NP_ROWS - 1) / NP_ROWS), dim3(NP_THREADS), np_smem(n), s, h->D,
                      static_cast<const float *>(h->H), n, scale));
        h->launches++;
        h->stage = STAGE_P;
        return GPTAQ_OK;
    }
    // O = (dXX^T U^T) .* M_U
    GemmProblem po = make_problem(make_operand(h->D, n, 1), make_operand(h->H, n, 1), O, n, n, n, n,
                                  1.f, 0.f, GEMM_O);
    OK(gemm(h, po, false, false, s));
    // P = (alpha / tokens) * O U
    GemmProblem pp = make_problem(make_operand(O, n, 1), make_operand(h->H, 1, n), h->D, n, n, n, n,
                                  scale, 0.f, GEMM_P);
    OK(gemm(h, pp, false, true, s));
    h->stage = STAGE_P;
    return GPTAQ_OK;
}

gptaq_status_t gptaq_build_P_rowwise(gptaq_handle_t h, float alpha, gptaq_stream_t stream) {
    if (!h || !std::isfinite(alpha)) return GPTAQ_ERR_INVALID_ARG;
    if (h->stage != STAGE_FACTORED) return GPTAQ_ERR_BAD_STATE;
    if (h->n > P_ROWWISE_MAX_N) return GPTAQ_ERR_UNSUPPORTED;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int n = (int)h->n;
    CU(cudaFuncSetAttribute(p_rowwise_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(2 * P_ROWWISE_MAX_N * sizeof(float))));
    p_rowwise_kernel<<<n, PR_THREADS, 2 * (size_t)n * sizeof(float), s>>>(h->D, h->H, n, (float)((double)alpha / (double)h->tokens));
    LAUNCHED();
    // the operand copies that gptaq_quantize reads, as gptaq_build_P leaves them
    WsLayout wl = ws_layout(h->n, 0);
    if (h->split) {
        const int64_t ldt = split_pitch(n);
        const size_t nn = (size_t)n * ldt;
        __half *UT16 = reinterpret_cast<__half *>(h->ws + wl.s_off[0]);
        __half *PT16 = reinterpret_cast<__half *>(h->ws + wl.s_off[1]);
        unsigned *am = h->hd->tc_amax;
        CU(cudaMemsetAsync(am + AMAX_U, 0, 2 * sizeof(unsigned), s));
        CU(launch_absmax({h->H, n, n, n, SPLIT_UPPER, 1.f, am + AMAX_U, nullptr, nullptr},
                         {h->D, n, n, n, SPLIT_STRICT_UPPER, 1.f, am + AMAX_P, nullptr, nullptr}, h->num_sms, s));
        const Split16Args split_p = split16_args(h->D, n, PT16, PT16 + nn, ldt, n, n, true, SPLIT_STRICT_UPPER, 1.f, am + AMAX_P);
        CU(launch_split16(split16_args(h->H, n, UT16, UT16 + nn, ldt, n, n, true, SPLIT_UPPER, 1.f, am + AMAX_U), h->num_sms, s, &split_p));
        h->launches += 2;
    }
    h->stage = STAGE_P;
    return GPTAQ_OK;
}

gptaq_status_t gptaq_quantize(gptaq_handle_t h, void *d_W, int w_dtype, int64_t m, int64_t ldw,
                              int bits, int group, int sym, int blocksize,
                              uint8_t *d_codes, float *d_scales, float *d_zeros, float *d_Wq,
                              gptaq_stream_t stream) {
    if (!h || m < 0 || m > INT32_MAX) return GPTAQ_ERR_INVALID_ARG;
    if (h->stage != STAGE_P) return GPTAQ_ERR_BAD_STATE;
    gptaq_status_t st = check_quantize_args(h->n, d_W, w_dtype, m, ldw, bits, group, blocksize, d_codes,
                                            d_scales, d_zeros, d_Wq);
    if (st != GPTAQ_OK || m == 0) return st;
    if (h->act_order && (!d_Wq || d_Wq == d_W)) return GPTAQ_ERR_INVALID_ARG;
    WsLayout wl = ws_layout(h->n, m);
    if (h->ws_bytes < wl.total) return GPTAQ_ERR_WORKSPACE;
    QuantizeTarget t;
    t.n = (int)h->n; t.U = h->H; t.P = h->D; t.dead = h->dead; t.hd = h->hd;
    t.EW = reinterpret_cast<float *>(h->ws + wl.ew_off);
    t.ew_floats = (int64_t)((wl.ew_lo_off - wl.ew_off) / sizeof(float));
    t.num_sms = h->num_sms;
    t.terms = h->terms;
    t.perm = h->act_order ? h->perm : nullptr;
    t.clip_steps = h->clip_steps; t.clip_min = h->clip_min;
    t.static_groups = h->static_groups; t.dead_orig = h->dead_raw;
    t.side = h->gemm_stream; t.fork = h->conv_done[0]; t.join = h->gemm_done[0];
    // fp16-split updates, plain float32 products otherwise
    // (groups of fewer than 32 columns update block by block, and blocks of 32 columns are no whole K-block of 64)
    const bool f16 = h->split && ((blocksize % 64) == 0 || group <= 0 || (group % 32) == 0 || h->static_groups);
    if (f16) {
        t.ldt = split_pitch(h->n);
        t.UT16 = reinterpret_cast<const __half *>(h->ws + wl.s_off[0]);
        t.PT16 = reinterpret_cast<const __half *>(h->ws + wl.s_off[1]);
        t.EW16 = reinterpret_cast<__half *>(h->ws + wl.ew_lo_off);
        t.row_inv = reinterpret_cast<float *>(h->ws + wl.rs_off);
        t.amax_u = h->hd->tc_amax + AMAX_U; t.amax_p = h->hd->tc_amax + AMAX_P;
    }
    cudaError_t e = cudaSuccess;
    st = quantize_core(t, d_W, w_dtype, m, ldw, bits, group, sym, blocksize, d_codes, d_scales, d_zeros, d_Wq,
                       static_cast<cudaStream_t>(stream), &h->launches, &e);
    if (st == GPTAQ_ERR_CUDA) h->cuda_error = cudaGetErrorString(e);
    return join_after_error(h, static_cast<cudaStream_t>(stream), st);
}

size_t gptaq_quantize_stage_bytes(int64_t m, int64_t n, int group) {
    if (m < 0 || n <= 0 || group < 0) return 0;
    size_t G = group > 0 ? (size_t)((n + group - 1) / group) : 1;
    return round_up((size_t)m * n * sizeof(float), ALIGN) + round_up((size_t)m * n, ALIGN) +
           2 * round_up((size_t)m * G * sizeof(float), ALIGN);
}

gptaq_status_t gptaq_quantize_host(gptaq_handle_t h, const float *h_W, int64_t m, int64_t ldw,
                                   int bits, int group, int sym, int blocksize,
                                   uint8_t *h_codes, float *h_scales, float *h_zeros, float *h_Wq,
                                   void *d_stage, size_t stage_bytes, gptaq_stream_t stream) {
    if (!h || m < 0) return GPTAQ_ERR_INVALID_ARG;
    if (h->stage != STAGE_P) return GPTAQ_ERR_BAD_STATE;
    if (m == 0) return GPTAQ_OK;
    if (!h_W || !h_codes || !h_scales || !h_zeros || !d_stage || ldw < h->n || group < 0)
        return GPTAQ_ERR_INVALID_ARG;
    if (stage_bytes < gptaq_quantize_stage_bytes(m, h->n, group)) return GPTAQ_ERR_WORKSPACE;
    const size_t n = (size_t)h->n;
    const size_t G = group > 0 ? (n + group - 1) / group : 1;
    char *base = static_cast<char *>(d_stage);
    float *dW = reinterpret_cast<float *>(base);
    uint8_t *dC = reinterpret_cast<uint8_t *>(base + round_up((size_t)m * n * sizeof(float), ALIGN));
    float *dS = reinterpret_cast<float *>(reinterpret_cast<char *>(dC) + round_up((size_t)m * n, ALIGN));
    float *dZ = reinterpret_cast<float *>(reinterpret_cast<char *>(dS) + round_up((size_t)m * G * sizeof(float), ALIGN));
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    CU(cudaMemcpy2DAsync(dW, n * sizeof(float), h_W, (size_t)ldw * sizeof(float), n * sizeof(float),
                         (size_t)m, cudaMemcpyHostToDevice, s));
    OK(gptaq_quantize(h, dW, GPTAQ_W_FP32, m, (int64_t)n, bits, group, sym, blocksize, dC, dS, dZ, nullptr,
                      stream));
    CU(cudaMemcpyAsync(h_codes, dC, (size_t)m * n, cudaMemcpyDeviceToHost, s));
    CU(cudaMemcpyAsync(h_scales, dS, (size_t)m * G * sizeof(float), cudaMemcpyDeviceToHost, s));
    CU(cudaMemcpyAsync(h_zeros, dZ, (size_t)m * G * sizeof(float), cudaMemcpyDeviceToHost, s));
    if (h_Wq) CU(cudaMemcpyAsync(h_Wq, dW, (size_t)m * n * sizeof(float), cudaMemcpyDeviceToHost, s));
    return GPTAQ_OK;
}

gptaq_status_t gptaq_quantize_static(const float *d_U, const float *d_P, int64_t n, void *d_W, int w_dtype,
                                     int64_t m, int64_t ldw, int bits, int group, int sym, int blocksize,
                                     uint8_t *d_codes, float *d_scales, float *d_zeros, float *d_Wq,
                                     int64_t *d_status, gptaq_stream_t stream) {
    if (!d_U || !d_P || n <= 0 || m < 0 || m > INT32_MAX) return GPTAQ_ERR_INVALID_ARG;
    gptaq_status_t st = check_quantize_args(n, d_W, w_dtype, m, ldw, bits, group, blocksize, d_codes, d_scales,
                                            d_zeros, d_Wq);
    if (st != GPTAQ_OK) return st;
    // the limits of the built-in scratch come before anything touches the device
    if (n > GPTAQ_STATIC_MAX_N || (int64_t)m * 2 * blocksize > GPTAQ_STATIC_SCRATCH_FLOATS)
        return GPTAQ_ERR_WORKSPACE;
    if (m == 0) return GPTAQ_OK;
    StaticScratch *sc = nullptr;
    cudaError_t e = static_scratch_for_current_device(&sc);
    if (e != cudaSuccess) return GPTAQ_ERR_CUDA;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // every call shares the array and finds the last call's contents: the status header and
    // the all-zero dead-input flags have to start from zero
    e = cudaMemsetAsync(sc->base, 0, STATIC_EW_OFFSET, s);
    if (e != cudaSuccess) return GPTAQ_ERR_CUDA;
    QuantizeTarget t;
    t.n = (int)n; t.U = d_U; t.P = d_P;
    t.hd = reinterpret_cast<StateHeader *>(sc->base);
    t.dead = sc->base + STATIC_FLAGS_OFFSET;
    t.EW = reinterpret_cast<float *>(sc->base + STATIC_EW_OFFSET);
    t.ew_floats = GPTAQ_STATIC_SCRATCH_FLOATS;
    t.num_sms = sc->num_sms;
    int64_t launches = 0;
    st = quantize_core(t, d_W, w_dtype, m, ldw, bits, group, sym, blocksize, d_codes, d_scales, d_zeros, d_Wq, s,
                       &launches, &e);
    if (st != GPTAQ_OK) return st;
    if (d_status) {
        export_status_kernel<<<1, 1, 0, s>>>(t.hd, d_status);
        if (cudaGetLastError() != cudaSuccess) return GPTAQ_ERR_CUDA;
    }
    return GPTAQ_OK;
}

gptaq_status_t gptaq_sync_status(gptaq_handle_t h, int64_t *info, gptaq_stream_t stream) {
    if (!h) return GPTAQ_ERR_INVALID_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    OK(join_statistics(h, s));
    StateHeader hd;
    CU(cudaMemcpyAsync(&hd, h->hd, sizeof(hd), cudaMemcpyDeviceToHost, s));
    CU(cudaStreamSynchronize(s));
    if (info) *info = hd.info;
    return static_cast<gptaq_status_t>(hd.status);
}

float *gptaq_H(gptaq_handle_t h) { return h ? h->H : nullptr; }
float *gptaq_D(gptaq_handle_t h) { return h ? h->D : nullptr; }
const float *gptaq_U(gptaq_handle_t h) { return (h && h->stage != STAGE_ACCUM) ? h->H : nullptr; }
const float *gptaq_P(gptaq_handle_t h) { return (h && h->stage == STAGE_P) ? h->D : nullptr; }

gptaq_status_t gptaq_selftest_bounded_wait(gptaq_handle_t h, double seconds, gptaq_stream_t stream) {
    if (!h || !(seconds > 0.0) || seconds > 2.0) return GPTAQ_ERR_INVALID_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int khz = 0;
    CU(cudaDeviceGetAttribute(&khz, cudaDevAttrClockRate, h->device));
    bounded_wait_selftest_kernel<<<1, 32, 0, s>>>(h->hd, (long long)(seconds * 1e3 * (double)khz));
    LAUNCHED();
    return GPTAQ_OK;
}
int64_t gptaq_tokens(gptaq_handle_t h) { return h ? h->tokens : -1; }

gptaq_status_t gptaq_set_tokens(gptaq_handle_t h, int64_t tokens) {
    if (!h || tokens < 0) return GPTAQ_ERR_INVALID_ARG;
    if (h->stage != STAGE_ACCUM) return GPTAQ_ERR_BAD_STATE;
    h->tokens = tokens;
    return GPTAQ_OK;
}

gptaq_status_t gptaq_set_stats_precision(gptaq_handle_t h, int precision) {
    if (!h) return GPTAQ_ERR_INVALID_ARG;
    if (precision != GPTAQ_STATS_FP16_TENSOR && precision != GPTAQ_STATS_FP32 &&
        precision != GPTAQ_STATS_FP16_SPLIT_TENSOR && precision != GPTAQ_STATS_FP16_SPLIT_FULL_TENSOR)
        return GPTAQ_ERR_UNSUPPORTED;
    if (h->stage != STAGE_ACCUM) return GPTAQ_ERR_BAD_STATE;
    if (precision != h->stats_precision) h->relayout = true;
    h->stats_precision = precision;
    return GPTAQ_OK;
}

gptaq_status_t gptaq_set_act_order(gptaq_handle_t h, int enable) {
    if (!h) return GPTAQ_ERR_INVALID_ARG;
    if (h->stage != STAGE_ACCUM) return GPTAQ_ERR_BAD_STATE;
    if (enable && h->n > ACT_ORDER_MAX_N) return GPTAQ_ERR_UNSUPPORTED;
    // the permutation needs the part of dXX^T below the diagonal, which earlier batches did not accumulate
    if (enable && !h->act_order && h->d_upper_only) return GPTAQ_ERR_BAD_STATE;
    h->act_order = enable != 0;
    return GPTAQ_OK;
}

gptaq_status_t gptaq_set_static_groups(gptaq_handle_t h, int enable) {
    if (!h) return GPTAQ_ERR_INVALID_ARG;
    h->static_groups = enable != 0;
    return GPTAQ_OK;
}

const int32_t *gptaq_perm(gptaq_handle_t h) { return (h && h->act_order && h->stage != STAGE_ACCUM) ? h->perm : nullptr; }

gptaq_status_t gptaq_set_clip_search(gptaq_handle_t h, int steps, float min_ratio) {
    if (!h) return GPTAQ_ERR_INVALID_ARG;
    if (steps < 0 || steps > 1024) return GPTAQ_ERR_UNSUPPORTED;
    if (steps > 0 && !(min_ratio > 0.f && min_ratio < 1.f)) return GPTAQ_ERR_INVALID_ARG;
    h->clip_steps = steps;
    h->clip_min = steps > 0 ? min_ratio : 1.f;
    return GPTAQ_OK;
}

gptaq_status_t gptaq_set_update_terms(gptaq_handle_t h, int terms) {
    if (!h) return GPTAQ_ERR_INVALID_ARG;
    if (terms & ~(GPTAQ_TERM_ERR | GPTAQ_TERM_ASYM)) return GPTAQ_ERR_UNSUPPORTED;
    h->terms = terms;
    return GPTAQ_OK;
}

int gptaq_recommended_stats_precision(int64_t n, int64_t total_tokens) {
    // fp16 rounding of X perturbs U by about 5e-5 * sqrt(n/k) / ((1 - sqrt(n/k))^2 + damp):
    // below 1e-4 with margin once there are 16 tokens per input channel.
    return (n > 0 && total_tokens >= 16 * n) ? GPTAQ_STATS_FP16_TENSOR : GPTAQ_STATS_FP16_SPLIT_TENSOR;
}

int64_t gptaq_launch_count(gptaq_handle_t h) { return h ? h->launches : -1; }

gptaq_status_t gptaq_set_kernel_timing(gptaq_handle_t h, int enable) {
    if (!h) return GPTAQ_ERR_INVALID_ARG;
    h->kernel_timing = enable != 0;
    return GPTAQ_OK;
}

gptaq_status_t gptaq_stats_kernel_time(gptaq_handle_t h, double *ms_total, int64_t *launches) {
    if (!h || !ms_total || !launches) return GPTAQ_ERR_INVALID_ARG;
    double total = 0.0;
    for (size_t i = 0; i < h->timing_used; ++i) {
        CU(cudaEventSynchronize(h->timing_events[i].second));
        float ms = 0.f;
        CU(cudaEventElapsedTime(&ms, h->timing_events[i].first, h->timing_events[i].second));
        total += ms;
    }
    *ms_total = total;
    *launches = (int64_t)h->timing_used;
    h->timing_used = 0;
    return GPTAQ_OK;
}

const char *gptaq_status_string(gptaq_status_t s) {
    switch (s) {
        case GPTAQ_OK: return "ok";
        case GPTAQ_ERR_INVALID_ARG: return "invalid argument";
        case GPTAQ_ERR_BAD_STATE: return "call out of order";
        case GPTAQ_ERR_WORKSPACE: return "buffer too small";
        case GPTAQ_ERR_NOT_SPD: return "damped H is not positive definite";
        case GPTAQ_ERR_NONFINITE: return "non-finite value";
        case GPTAQ_ERR_TIMEOUT: return "bounded device wait ran out";
        case GPTAQ_ERR_UNSUPPORTED: return "unsupported argument combination";
        case GPTAQ_ERR_CUDA: return "CUDA runtime error";
    }
    return "unknown status";
}

const char *gptaq_last_cuda_error(gptaq_handle_t h) { return h ? h->cuda_error.c_str() : ""; }

}  // extern "C"
