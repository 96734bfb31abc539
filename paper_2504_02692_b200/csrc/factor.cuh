// The reverse Cholesky factorisation H_d = R R^T (R upper), panel by panel of NB columns from the right:
//
//   diag_factor_kernel   one CTA: the NB x NB diagonal block (and the inverses of its 32 x 32 diagonal sub-blocks);
//   panel_solve_kernel   the rows above: R[0:b0, blk] = A[0:b0, blk] R_pp^-T, in place and as split parts;
//   the rank-NB update of the columns to the left (tc_gemm_kernel, simt kernels).
//
// The chain diagonal -> solve -> update -> next diagonal bounds narrow and ordinary layers, and of it the diagonal block
// (128 dependent pivots).  Where the next block belongs to the same super-panel its diagonal kernel does not wait for the
// update: it takes a copy of the block from before the update and subtracts this panel's contribution itself (one
// 128 x 128 x 128 product on the tensor cores), so that the update runs beside it on another stream.
// A panel of a 1024-wide layer is 28 us of the chain, from one diagonal kernel's start to the next one's: the diagonal block 19 (14.5
// of them the factorisation, 3 until the block is loaded and updated), the rows above it 7, the launches between.  Its inverse is made
// beside the next block and the rows of U are gathered as they come, block 1's beside block 0, which inverts itself: behind the last
// block only row 0 of U is left (n = 384 114 -> 108 us, 777 284 -> 277).  A layer of one block is a single launch (n = 128 36 -> 31).
// The inverse as a kernel of its own behind the update (11 us on one SM) and one pivot at a time made a panel 33 us, every CTA of one
// kernel factoring the diagonal block first and the update on the chain 45.  gptaq_factor, us, in that last form: n = 1024 404,
// 2052 1118, 4096 2036; in the one between 292, 731, 1396; now 246, 653, 1255 to 1275.
#pragma once
#include "tc_gemm.cuh"

namespace gptaq {

constexpr int NB = 128;
constexpr int FP_LD = NB + 4;
constexpr int FP_YLD = 36;

// The 32-step recurrences below run in four rounds of 8 unrolled steps over register arrays that move up by 8 after a
// round: unrolled over all 32 steps the code of this file's roles exceeds the instruction cache (about 30 KB; beyond it a
// warp executes one instruction in three cycles), which cost more than the dependent chains themselves.
template <typename T>
__device__ __forceinline__ void move_up8(T (&d)[32]) {
#pragma unroll
    for (int j = 31; j >= 8; --j) d[j] = d[j - 8];
#pragma unroll
    for (int j = 0; j < 8; ++j) d[j] = 0.f;
}

// x R^T = a for one row (a: 32 entries) against an upper triangular 32 x 32 block R given by its transpose (Rt[k][i] =
// R[i][k], pitch FP_LD) and its reciprocal diagonal; emit(k, x_k) receives the results from k = 31 down.
// The same recurrence with a = unit vector e_l gives column l of R^-1.  ready(k) is called before columns k .. k - 7 are
// read (k = 31, 23, ..).
template <typename Ready, typename Emit>
__device__ __forceinline__ void solve32(float (&a)[32], const float *Rt, const float *dinv, Ready ready, Emit emit) {
#pragma unroll 1
    for (int k0 = 24; k0 >= 0; k0 -= 8) {
        // a[24 + e] is entry k0 + e
#pragma unroll
        for (int e = 7; e >= 0; --e) {
            const int k = k0 + e;
            if (e == 7) ready(k);
            const float x = a[24 + e] * dinv[k];
            emit(k, x);
            // entries below k: 24 + e - 1 .. 24 - k0; the rest (below entry 0) reads up to 24 words ahead of the row in shared
            // memory and is never used
            const float *col = Rt + k * FP_LD + k0 - 24;
#pragma unroll
            for (int j4 = 5 + (e + 3) / 4; j4 >= 0; --j4) {
                const float4 r = *reinterpret_cast<const float4 *>(col + 4 * j4);
                a[4 * j4 + 0] = fmaf(-x, r.x, a[4 * j4 + 0]);
                a[4 * j4 + 1] = fmaf(-x, r.y, a[4 * j4 + 1]);
                a[4 * j4 + 2] = fmaf(-x, r.z, a[4 * j4 + 2]);
                a[4 * j4 + 3] = fmaf(-x, r.w, a[4 * j4 + 3]);
            }
        }
        move_up8(a);
    }
}

// Eight columns of the block factorisation, for the rows that a warp holds one per lane (d[24 + e]: entry of the row in column
// e of the eight).  Leader: the eight rows of the columns' own diagonal block are among them (lanes l0 .. l0 + 7); every lane
// reads that 8 x 8 block (through `gs`, 64 words) and factors it by itself, so that the chain from pivot to pivot is a
// reciprocal root (hardware estimate and one Newton step, to about one ulp), a scaling and one FMA, in registers.
// col[k * FP_LD + i] receives R[i][k] for the lanes up to the diagonal, dinv[k] the reciprocal roots.  x: the row's results.
// A pivot that is not a positive normal number counts as 1; returns the first such column (-1: none).
__device__ __forceinline__ int chol8(float (&d)[32], float (&x)[8], int lane, int l0, float *gs, float *col, float *dinv) {
    if ((lane & ~7) == l0) {
        *reinterpret_cast<float4 *>(gs + (lane & 7) * 8) = make_float4(d[24], d[25], d[26], d[27]);
        *reinterpret_cast<float4 *>(gs + (lane & 7) * 8 + 4) = make_float4(d[28], d[29], d[30], d[31]);
    }
    __syncwarp();
    float g[8][8];                                   // (the upper triangle is used)
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float4 hi = *reinterpret_cast<const float4 *>(gs + 8 * i + 4);
        g[i][4] = hi.x; g[i][5] = hi.y; g[i][6] = hi.z; g[i][7] = hi.w;
        if (i < 4) {
            const float4 lo = *reinterpret_cast<const float4 *>(gs + 8 * i);
            g[i][0] = lo.x; g[i][1] = lo.y; g[i][2] = lo.z; g[i][3] = lo.w;
        }
    }
    int bad_col = -1;
#pragma unroll
    for (int k = 7; k >= 0; --k) {
        float piv = g[k][k], r;
        asm volatile("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(piv));
        const bool bad = !(piv >= 1.17549435e-38f) || !(piv < INFINITY);
        r = r * fmaf(-0.5f * piv, r * r, 1.5f);
        bad_col = (bad && bad_col < 0) ? k : bad_col;
        piv = bad ? 1.f : piv;
        r = bad ? 1.f : r;
#pragma unroll
        for (int i = k - 1; i >= 0; --i) {
            g[i][k] *= r;
#pragma unroll
            for (int j = i; j < k; ++j) g[i][j] = fmaf(-g[i][k], g[j][k], g[i][j]);
        }
        x[k] = d[24 + k] * r;
#pragma unroll
        for (int j = k - 1; j >= 0; --j) d[24 + j] = fmaf(-x[k], g[j][k], d[24 + j]);
        const float rk = lane == l0 + k ? piv * r : x[k];
        if (lane <= l0 + k) col[k * FP_LD + lane] = rk;
        if (lane == 0) dinv[k] = r;
    }
    return bad_col;
}

// ... the rows above: by substitution against the eight columns (R[j][k] at rt[k * FP_LD + j]); col[k * FP_LD + lane] receives
// the results.
__device__ __forceinline__ void solve8(float (&d)[32], float (&x)[8], int lane, const float *rt, const float *dinv, float *col) {
    const float4 r0 = *reinterpret_cast<const float4 *>(dinv), r1 = *reinterpret_cast<const float4 *>(dinv + 4);
    const float rv[8] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w};
    float c[8][8];
#pragma unroll
    for (int k = 1; k < 8; ++k) {
        const float4 lo = *reinterpret_cast<const float4 *>(rt + k * FP_LD);
        c[k][0] = lo.x; c[k][1] = lo.y; c[k][2] = lo.z; c[k][3] = lo.w;
        if (k > 4) {
            const float4 hi = *reinterpret_cast<const float4 *>(rt + k * FP_LD + 4);
            c[k][4] = hi.x; c[k][5] = hi.y; c[k][6] = hi.z; c[k][7] = hi.w;
        }
    }
#pragma unroll
    for (int k = 7; k >= 0; --k) {
        x[k] = d[24 + k] * rv[k];
#pragma unroll
        for (int j = k - 1; j >= 0; --j) d[24 + j] = fmaf(-x[k], c[k][j], d[24 + j]);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) col[k * FP_LD + lane] = x[k];
}

// d[J0 + j] -= sum over k of x[k] rt[k * FP_LD + j], j < 8
template <int J0>
__device__ __forceinline__ void rank8(float (&d)[32], const float (&x)[8], const float *rt) {
#pragma unroll
    for (int k = 7; k >= 0; --k)
#pragma unroll
        for (int j4 = 0; j4 < 2; ++j4) {
            const float4 r = *reinterpret_cast<const float4 *>(rt + k * FP_LD + 4 * j4);
            d[J0 + 4 * j4 + 0] = fmaf(-x[k], r.x, d[J0 + 4 * j4 + 0]); d[J0 + 4 * j4 + 1] = fmaf(-x[k], r.y, d[J0 + 4 * j4 + 1]);
            d[J0 + 4 * j4 + 2] = fmaf(-x[k], r.z, d[J0 + 4 * j4 + 2]); d[J0 + 4 * j4 + 3] = fmaf(-x[k], r.w, d[J0 + 4 * j4 + 3]);
        }
}

// Where the inverses of a block's four 32 x 32 diagonal sub-blocks lie: in the upper part of Rdiag, which R^T leaves free.  Row l
// (32 consecutive floats) of sub-block c: inv(R_cc)[j][l].
__device__ __forceinline__ int diag_inverse_at(int c, int l) { return ((c == 3 ? 32 : 0) + l) * NB + (c == 3 ? 64 : 32 * (c + 1)); }

// ---------------------------------------------------------------------------
// U_pp = R_pp^-1 onto the diagonal of H (strict lower part of the block zero), by one CTA: the starting point of U = R^-1.  The
// 32 x 32 diagonal sub-blocks come inverted from diag_factor_kernel; X12 = -X11 (R12 X22) for 32 -> 64 -> 128.  Bound by
// shared-memory reads: 4 x 4 outputs per thread.  A second CTA of the next block's diag_factor_kernel, which takes twice as long
// (as a CTA of panel_solve_kernel it held that up: a panel's rows 7 -> 11 us; as a kernel of its own behind the update, which
// inverted the sub-blocks itself, it took 11 us a panel and one stream operation more).  Block 1 has a launch of its own, beside block 0,
// which inverts itself.
// ---------------------------------------------------------------------------
constexpr int ID_THREADS = 256, ID_BAR = 15;
constexpr int ID_LD = FP_LD;
constexpr size_t ID_SMEM = (2 * NB * ID_LD + 64 * 68) * sizeof(float);

// C[i][j] = sign * sum_k A[i][k] B[k][j], S x S outputs, 4 x 4 per thread (rows ti + S / 4 e, four columns), all operands
// row-major in shared memory; `t` counts the (S / 4)^2 threads of one product.
template <int S>
__device__ __forceinline__ void tile_product(float *C, int ldc, const float *A, int lda, const float *B, int ldb, int t, float sign) {
    const int ti = t / (S / 4), tj = t % (S / 4);
    float acc[4][4];
#pragma unroll
    for (int e = 0; e < 4; ++e)
#pragma unroll
        for (int f = 0; f < 4; ++f) acc[e][f] = 0.f;
#pragma unroll 4
    for (int k = 0; k < S; k += 4) {
        float av[4][4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float4 v = *reinterpret_cast<const float4 *>(A + (ti + S / 4 * e) * lda + k);
            av[e][0] = v.x; av[e][1] = v.y; av[e][2] = v.z; av[e][3] = v.w;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float4 b = *reinterpret_cast<const float4 *>(B + (k + q) * ldb + 4 * tj);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                acc[e][0] = fmaf(av[e][q], b.x, acc[e][0]); acc[e][1] = fmaf(av[e][q], b.y, acc[e][1]);
                acc[e][2] = fmaf(av[e][q], b.z, acc[e][2]); acc[e][3] = fmaf(av[e][q], b.w, acc[e][3]);
            }
        }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e)
        *reinterpret_cast<float4 *>(C + (ti + S / 4 * e) * ldc + 4 * tj) =
            make_float4(sign * acc[e][0], sign * acc[e][1], sign * acc[e][2], sign * acc[e][3]);
}

// By the first ID_THREADS threads of a CTA, from R^T left of the sub-blocks on the diagonal (in S) and their inverses (in X, zeros
// elsewhere).
__device__ __forceinline__ void invert_products(float *S, float *X, float *T, float *H, int n, int b0) {
    const int tid = threadIdx.x;
    // R above the diagonal
    for (int idx = tid; idx < NB * NB; idx += ID_THREADS) {
        const int i = idx >> 7, j = idx & 127;
        if ((j >> 5) < (i >> 5)) S[j * ID_LD + i] = S[i * ID_LD + j];
    }
    named_bar_sync(ID_BAR, ID_THREADS);
    // X12 = -X11 (R12 X22), 32 -> 64 for both pairs, then 64 -> 128 (the triangular operands carry explicit zeros)
    const int pr = tid >> 6, o = 64 * pr;
    if (tid < 128) tile_product<32>(T + pr * 32 * 36, 36, S + o * ID_LD + o + 32, ID_LD, X + (o + 32) * ID_LD + o + 32, ID_LD, tid & 63, 1.f);
    named_bar_sync(ID_BAR, ID_THREADS);
    if (tid < 128) tile_product<32>(X + o * ID_LD + o + 32, ID_LD, X + o * ID_LD + o, ID_LD, T + pr * 32 * 36, 36, tid & 63, -1.f);
    named_bar_sync(ID_BAR, ID_THREADS);
    tile_product<64>(T, 68, S + 64, ID_LD, X + 64 * ID_LD + 64, ID_LD, tid, 1.f);
    named_bar_sync(ID_BAR, ID_THREADS);
    tile_product<64>(X + 64, ID_LD, X, ID_LD, T, 68, tid, -1.f);
    named_bar_sync(ID_BAR, ID_THREADS);
    const bool vec = (n & 3) == 0 && b0 + NB <= n;
#pragma unroll 4
    for (int it = 0; it < NB * NB / 4 / ID_THREADS; ++it) {
        const int i = (tid + it * ID_THREADS) >> 5, j = 4 * ((tid + it * ID_THREADS) & 31);
        const float4 x = *reinterpret_cast<const float4 *>(X + i * ID_LD + j);
        float *dst = H + (int64_t)(b0 + i) * n + b0 + j;
        if (vec) *reinterpret_cast<float4 *>(dst) = x;
        else if (b0 + i < n) {
            const float xe[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) if (b0 + j + e < n) dst[e] = xe[e];
        }
    }
}

// by the first ID_THREADS threads of a CTA
__device__ __forceinline__ void invert_diag_block(float *smem_f, float *H, int n, int b0, const float *Rdiag) {
    float *S = smem_f, *X = S + NB * ID_LD, *T = X + NB * ID_LD;
    const int tid = threadIdx.x;
    float4 v[NB * NB / 4 / ID_THREADS];
#pragma unroll
    for (int it = 0; it < NB * NB / 4 / ID_THREADS; ++it) v[it] = *reinterpret_cast<const float4 *>(Rdiag + 4 * (tid + it * ID_THREADS));
    float y[4 * 32 * 32 / ID_THREADS];
#pragma unroll
    for (int it = 0; it < 4 * 32 * 32 / ID_THREADS; ++it) {
        const int idx = tid + it * ID_THREADS;
        y[it] = Rdiag[diag_inverse_at(idx >> 10, (idx >> 5) & 31) + (idx & 31)];
    }
#pragma unroll
    for (int it = 0; it < NB * NB / 4 / ID_THREADS; ++it) {
        const int i = (tid + it * ID_THREADS) >> 5, j4 = (tid + it * ID_THREADS) & 31;
        // R^T as it comes, left of the sub-block on the diagonal
        if (j4 < (i >> 5) * 8) *reinterpret_cast<float4 *>(S + i * ID_LD + 4 * j4) = v[it];
        if ((j4 >> 3) != (i >> 5)) *reinterpret_cast<float4 *>(X + i * ID_LD + 4 * j4) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int it = 0; it < 4 * 32 * 32 / ID_THREADS; ++it) {
        const int idx = tid + it * ID_THREADS, c = idx >> 10, l = (idx >> 5) & 31, j = idx & 31;
        X[(32 * c + j) * ID_LD + 32 * c + l] = j <= l ? y[it] : 0.f;
    }
    named_bar_sync(ID_BAR, ID_THREADS);
    invert_products(S, X, T, H, n, b0);
}

__global__ void __launch_bounds__(ID_THREADS, 1) invert_diag_block_kernel(float *H, int n, int b0, const float *Rdiag) {
    extern __shared__ __align__(16) float smem_f[];
    invert_diag_block(smem_f, H, n, b0, Rdiag);
}

// ---------------------------------------------------------------------------
// The NB x NB diagonal block [b0, b0 + NB): R_pp^T in the lower part of Rdiag and the inverses of its four 32 x 32 diagonal
// sub-blocks in the upper part (diag_inverse_at; the rest is undefined).  Rows / columns beyond n are padded with the identity.
// Warps 0 - 3 hold the 128 rows, one per lane, and go through the 32-column sub-blocks from the right, eight columns at a time:
// the warp with the sub-block's own rows leads (chol8), those above it follow (solve8).  The helpers (warps 4 - 11) gather the
// products for the next sub-block's columns as the rows are solved, so that its leader starts soon after the sub-block before is
// done, and then update what lies further left.  Warp 12 inverts the sub-blocks, eight columns behind the leader; warp 13 runs
// the tensor-core product.
// What bounds it (clocks in a copy): eight columns take the leader 900 to 1400 cycles, of which 350 are dependent operations; the
// rest is the issue of LDS (a scheduler starts one 16-byte form in 8 cycles where all lanes read the same words, else in 16) and
// of code that a launch runs for the first time.  A warp for all 32 columns of a sub-block, one pivot at a time through shuffles,
// took 150 cycles a pivot, and the rows above waited for the sub-block's inverse.  Rows that keep the next sub-block's
// columns up to date by themselves (64 such reads per eight columns) fell 5k cycles behind the leader.
// ---------------------------------------------------------------------------
constexpr int DF_HELP = 8 * 32, DF_MAIN = 128 + DF_HELP, DF_THREADS = DF_MAIN + 64;
constexpr int DF_TILE_BYTES = NB * 64 * 2;           // 128 rows x 64 fp16
constexpr size_t DF_SMEM_BLOCK = 4 * DF_TILE_BYTES + (size_t)(NB * FP_LD + NB + 64 + 32) * sizeof(float) + 32 + 1024;
constexpr size_t DF_SMEM = DF_SMEM_BLOCK > ID_SMEM ? DF_SMEM_BLOCK : ID_SMEM;
constexpr size_t DF_SMEM_LAST = 4 * DF_TILE_BYTES + ID_SMEM + (NB + 64 + 32) * sizeof(float) + 32 + 1024;
static_assert(DF_SMEM_LAST <= 227 * 1024, "shared memory of one SM");
constexpr size_t DF_SMEM_WHOLE = ID_SMEM + (NB + 64 + 32) * sizeof(float) + 32 + 1024;
constexpr uint32_t DF_IDESC = (1u << 4) | ((NB >> 3) << 17) | ((NB >> 4) << 24);     // kind::f16, M = N = 128
// Named barriers.  COLS + q: eight columns (q = 0: the rightmost) of a sub-block are factored (its leader arrives; the warps above
// it and the inverter wait); ROWS + q: ... and solved in the rows above (these arrive, the helpers wait); NEXT: the next
// sub-block's columns are up to date (the helpers arrive, its rows wait); DONE: the last sub-block is factored.  Each is used
// again in the next sub-block, which nobody enters before all have passed it.
enum { DBAR_COLS = 1, DBAR_ROWS = 5, DBAR_NEXT = 9, DBAR_DONE = 10 };

struct DiagFactorArgs {
    const float *src; long long lds;     // element (0, 0) of the block and its row pitch; entries j >= i are used
    int n, b0;
    float *Rdiag;                        // [NB][NB]
    float *H; int inv_b0;                // a second CTA inverts the block at inv_b0 (onto the diagonal of H) from inv_Rdiag
    const float *inv_Rdiag;
    int syrk, pan_col0;                  // 1: subtract rows b0 .. of the panel at columns pan_col0 .. of the split copy times
                                         //    their transpose first (scale of the copy: tc_amax[AMAX_PAN])
    StateHeader *hd;
    // DF_WHOLE: the layer has one block, src is its sum H as it was accumulated
    float inv_tokens, damp;
    uint8_t *dead, *dead_working;
};

// DF_LAST (block 0): the block's inverse follows at once, from the factor as it lies in shared memory (as a kernel of its own it
// followed 2 us later and loaded it first).  DF_WHOLE (n <= NB): what diag_stats_kernel and scale_damp_kernel do for a wider layer happens here, too, with the same
// arithmetic: gptaq_factor at n = 128 36.6 us as four launches, 31.4 so, n = 100 39.2 and 31.7 (U bit-identical; with R_pp through
// global memory as between the launches 37.7 and 35.8).
enum { DF_BLOCK = 0, DF_LAST = 1, DF_WHOLE = 2 };
template <int MODE>
__global__ void __launch_bounds__(DF_THREADS, 1)
diag_factor_kernel(const __grid_constant__ CUtensorMap mapHi, const __grid_constant__ CUtensorMap mapLo, DiagFactorArgs a) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t *sm = smem_raw + (base - raw);
    constexpr bool WHOLE = MODE == DF_WHOLE, INVERT = MODE != DF_BLOCK;
    // (the inverse's other operands behind it)
    float (*S)[FP_LD] = reinterpret_cast<float (*)[FP_LD]>(sm + (WHOLE ? 0 : 4 * DF_TILE_BYTES));
    float *X = reinterpret_cast<float *>(S + NB), *T = X + NB * ID_LD;
    float *dinv = INVERT ? T + 64 * 68 : reinterpret_cast<float *>(S + NB);
    float *gs = dinv + NB;                           // 8 x 8: the diagonal block of the columns at hand
    float *rdiag = gs + 64;                          // 1 / R_kk of the sub-block that is being inverted
    uint8_t *tailp = reinterpret_cast<uint8_t *>(rdiag + 32);
    const uint32_t bar = smem_u32(tailp), bar_mma = bar + 8;
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(tailp + 16);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tailp + 20);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nv = min(NB, a.n - a.b0);
    pdl_launch_dependents();
    if (!WHOLE && blockIdx.x == 1) {
        pdl_wait();
        if (tid < ID_THREADS) invert_diag_block(reinterpret_cast<float *>(smem_raw), a.H, a.n, a.inv_b0, a.inv_Rdiag);
        return;
    }
    if (tid == 0) {
        mbar_init(bar, 1);
        mbar_init(bar_mma, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (!WHOLE && a.syrk && warp == 13) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(const_cast<uint32_t *>(tmem_slot))), "r"(128u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (INVERT)
        for (int idx = tid; idx < NB * NB; idx += DF_THREADS)
            if ((idx >> 12) != ((idx & 127) >> 5)) X[(idx >> 7) * ID_LD + (idx & 127)] = 0.f;
    pdl_wait();
    if constexpr (WHOLE) {
        double *sum = reinterpret_cast<double *>(T);
        float *top = reinterpret_cast<float *>(sum + NB);
        float d = tid < nv ? a.src[tid * a.lds + tid] : 0.f;
        const float raw = d;
        bool dd = false;
        constexpr int BATCH = 13, ROUNDS = (NB * NB + BATCH * DF_THREADS - 1) / (BATCH * DF_THREADS);      // (loads in flight)
#pragma unroll 1
        for (int r = 0; r < ROUNDS; ++r) {
            float v[BATCH];
#pragma unroll
            for (int e = 0; e < BATCH; ++e) {
                const int idx = tid + (r * BATCH + e) * DF_THREADS, i = idx >> 7, j = idx & 127;
                v[e] = i < nv && j < nv && j > i ? a.src[i * a.lds + j] : 0.f;
            }
#pragma unroll
            for (int e = 0; e < BATCH; ++e) {
                const int idx = tid + (r * BATCH + e) * DF_THREADS, i = idx >> 7, j = idx & 127;
                if (i < NB && (i != j || i >= nv)) S[i][j] = i == j ? 1.f : v[e] * a.inv_tokens;
            }
        }
        if (tid < NB) {
            if (tid < nv) {
                if (!isfinite(d)) record_status(a.hd, ST_NONFINITE, tid);
                dd = d == 0.f;
                a.dead[tid] = dd ? 1 : 0;
                if (a.dead_working) a.dead_working[tid] = dd ? 1 : 0;
                d = dd ? 1.f : d * a.inv_tokens;
                sum[tid] = dd ? 1.0 : (double)raw * (double)a.inv_tokens;
                top[tid] = d;
            } else { sum[tid] = 0.0; top[tid] = 0.f; }
        }
        for (int w = NB / 2; w > 0; w >>= 1) {
            __syncthreads();
            if (tid < w) { sum[tid] += sum[tid + w]; top[tid] = fmaxf(top[tid], top[tid + w]); }
        }
        __syncthreads();
        const float lambda = (float)((double)a.damp * sum[0] / (double)a.n);
        if (tid == 0) {
            a.hd->lambda = lambda;
            a.hd->inv_tokens = a.inv_tokens;
            a.hd->tc_amax[AMAX_PAN] = __float_as_uint(sqrtf(top[0] + lambda));
            a.hd->tc_amax[AMAX_INV] = lambda > 0.f ? __float_as_uint(rsqrtf(lambda)) : 0u;
        }
        if (tid < nv) S[tid][tid] = d + lambda;
    } else if (warp == 13) {
        if (a.syrk && lane == 0) {
            mbar_expect_tx(bar, 4 * DF_TILE_BYTES);
            for (int t = 0; t < 4; ++t) tma_load_2d(base + t * DF_TILE_BYTES, t < 2 ? &mapHi : &mapLo, a.pan_col0 + 64 * (t & 1), a.b0, bar);
            const uint32_t tmem = *tmem_slot;
            if (mbar_wait(bar, 0u, abort_flag)) {
                tc_fence_after();
                uint32_t acc = 0;
                for (int term = 0; term < 3; ++term)                 // lo hi, hi lo, hi hi
                    for (int kb = 0; kb < 2; ++kb) {
                        const uint64_t ad = make_kmajor_desc(base + ((term == 0 ? 2 : 0) + kb) * DF_TILE_BYTES);
                        const uint64_t bd = make_kmajor_desc(base + ((term == 1 ? 2 : 0) + kb) * DF_TILE_BYTES);
#pragma unroll
                        for (int k = 0; k < 4; ++k) { umma_f16(tmem, ad + (uint64_t)(k * 2), bd + (uint64_t)(k * 2), DF_IDESC, acc); acc = 1; }
                    }
                umma_commit(bar_mma);
            }
        }
        __syncwarp();
    } else if (warp < 12) {
        // the block (all loads in flight before the first store)
        constexpr int QUADS = NB * NB / 4, ITS = (QUADS + DF_MAIN - 1) / DF_MAIN;
        if (nv == NB && (a.lds & 3) == 0 && (reinterpret_cast<uintptr_t>(a.src) & 15) == 0) {
            float4 v[ITS];
#pragma unroll
            for (int it = 0; it < ITS; ++it) {
                const int idx = tid + it * DF_MAIN;
                if (idx < QUADS) v[it] = *reinterpret_cast<const float4 *>(a.src + (idx >> 5) * a.lds + 4 * (idx & 31));
            }
#pragma unroll
            for (int it = 0; it < ITS; ++it) {
                const int idx = tid + it * DF_MAIN;
                if (idx < QUADS) *reinterpret_cast<float4 *>(&S[idx >> 5][4 * (idx & 31)]) = v[it];
            }
        } else {
            for (int idx = tid; idx < NB * NB; idx += DF_MAIN) {
                const int i = idx >> 7, j = idx & 127;
                S[i][j] = (i < nv && j < nv && j >= i) ? a.src[i * a.lds + j] : (i == j ? 1.f : 0.f);
            }
        }
    }
    __syncthreads();
    if (!WHOLE && a.syrk) {
        const uint32_t tmem = *tmem_slot;
        // 32 x 32 pieces of the upper triangle, one or two per warp
        const int quarter = warp & 3, row = 32 * quarter + lane;
        const bool ok = warp < 12 && mbar_wait(bar_mma, 0u, abort_flag);
        __syncwarp();
        if (ok) {
            tc_fence_after();
            const float sc = split_scale(__uint_as_float(a.hd->tc_amax[AMAX_PAN]));
            const float inv = 1.f / (sc * sc);
            for (int cb = warp >> 2; cb < 4; cb += 3) {
                if (cb < quarter) continue;
                const int c0 = 32 * cb;
                uint32_t v[32];
                tmem_ld32(tmem + c0 + ((uint32_t)(quarter * 32) << 16), v);
                tmem_ld_wait();
#pragma unroll
                for (int c4 = 0; c4 < 8; ++c4) {
                    float4 x = *reinterpret_cast<float4 *>(&S[row][c0 + 4 * c4]);
                    x.x = fmaf(-inv, __uint_as_float(v[4 * c4]), x.x); x.y = fmaf(-inv, __uint_as_float(v[4 * c4 + 1]), x.y);
                    x.z = fmaf(-inv, __uint_as_float(v[4 * c4 + 2]), x.z); x.w = fmaf(-inv, __uint_as_float(v[4 * c4 + 3]), x.w);
                    *reinterpret_cast<float4 *>(&S[row][c0 + 4 * c4]) = x;
                }
            }
        }
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        if (warp == 13)
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(128u) : "memory");
    }

    // products of the solved rows, nk of them from row k0 of R^T on: acc[e][f] += X[i + e] . X[j + f]
    auto rows_dot = [&](int k0, int nk, int i, int j, float (&acc)[4][4]) {
#pragma unroll 4
        for (int k = k0 + nk - 1; k >= k0; --k) {
            const float4 ri = *reinterpret_cast<const float4 *>(&S[k][i]);
            const float4 rj = *reinterpret_cast<const float4 *>(&S[k][j]);
            const float av[4] = {ri.x, ri.y, ri.z, ri.w}, bv[4] = {rj.x, rj.y, rj.z, rj.w};
#pragma unroll
            for (int e = 0; e < 4; ++e)
#pragma unroll
                for (int f = 0; f < 4; ++f) acc[e][f] = fmaf(av[e], bv[f], acc[e][f]);
        }
    };
    auto subtract = [&](int i, int j, const float (&acc)[4][4]) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            float4 *cp = reinterpret_cast<float4 *>(&S[i + e][j]);
            float4 v = *cp;
            // (below the diagonal nothing is read before results are written there)
            v.x -= acc[e][0]; v.y -= acc[e][1]; v.z -= acc[e][2]; v.w -= acc[e][3];
            *cp = v;
        }
    };
    if (warp < 4) {
        const int row = 32 * warp + lane;
        float d[32], x[8];                           // the row in this sub-block's columns
#pragma unroll 1
        for (int sb = 3; sb >= warp; --sb) {
            const int o = 32 * sb;
            const bool leads = sb == warp;
            if (sb < 3) named_bar_sync(DBAR_NEXT, DF_HELP + 32 * (sb + 1));
#pragma unroll
            for (int j4 = 0; j4 < 8; ++j4) {
                const float4 v = *reinterpret_cast<const float4 *>(&S[row][o + 4 * j4]);       // (left of the diagonal: never used)
                d[4 * j4] = v.x; d[4 * j4 + 1] = v.y; d[4 * j4 + 2] = v.z; d[4 * j4 + 3] = v.w;
            }
#pragma unroll 1
            for (int q = 0; q < 4; ++q) {
                const int k0 = 24 - 8 * q;
                float *rt = &S[o + k0][0];           // rt[k * FP_LD + i]: R[i][o + k0 + k]
                if (leads) {
                    const int bad_col = chol8(d, x, lane, k0, gs, rt + o, dinv + o + k0);
                    named_bar_arrive(DBAR_COLS + q, 32 * (sb + 2));
                    if (bad_col >= 0 && lane == 0) record_status(a.hd, ST_NOT_SPD, a.b0 + o + k0 + bad_col);
                    __syncwarp();
                } else {
                    named_bar_sync(DBAR_COLS + q, 32 * (sb + 2));
                    solve8(d, x, lane, rt + o + k0, dinv + o + k0, rt + 32 * warp);
                    named_bar_arrive(DBAR_ROWS + q, DF_HELP + 32 * sb);
                }
                // the columns left of these
                if (k0 >= 8) rank8<16>(d, x, rt + o + k0 - 8);
                if (k0 >= 16) rank8<8>(d, x, rt + o + k0 - 16);
                if (k0 >= 24) rank8<0>(d, x, rt + o);
                move_up8(d);
            }
        }
        if (warp == 0) named_bar_arrive(DBAR_DONE, DF_HELP + 32);
    } else if (warp < 12) {
        const int t = tid - 128;
        // R^T of a sub-block's rows, up to the diagonal
        auto store_rows = [&](int sb) {
            for (int idx = t; idx < 32 * (NB / 4); idx += DF_HELP) {
                const int i = 32 * sb + (idx >> 5), j4 = idx & 31;
                if (!INVERT && j4 < 8 * (sb + 1)) *reinterpret_cast<float4 *>(a.Rdiag + i * NB + 4 * j4) = *reinterpret_cast<const float4 *>(&S[i][4 * j4]);
            }
        };
#pragma unroll 1
        for (int sb = 3; sb >= 1; --sb) {
            const int o = 32 * sb;
            float acc[4][4];
#pragma unroll
            for (int e = 0; e < 4; ++e)
#pragma unroll
                for (int f = 0; f < 4; ++f) acc[e][f] = 0.f;
            // the next sub-block's columns: S[i][j] -= X[i] . X[j], i < o, o - 32 <= j < o
            const int i = 4 * (t >> 3), j = o - 32 + 4 * (t & 7);
#pragma unroll 1
            for (int q = 0; q < 4; ++q) {
                named_bar_sync(DBAR_ROWS + q, DF_HELP + 32 * sb);
                if (i < o) rows_dot(o + 24 - 8 * q, 8, i, j, acc);
            }
            if (i < o) subtract(i, j, acc);
            named_bar_arrive(DBAR_NEXT, DF_HELP + 32 * sb);
            // ... and what lies left of them: i <= j < o - 32, the 4 x 4 tiles of the upper triangle numbered row by row
            const int q4 = (o - 32) / 4, ntile = q4 * (q4 + 1) / 2;
            if (t < ntile) {
                int ti = 0, left = t;
                while (left >= q4 - ti) { left -= q4 - ti; ++ti; }
#pragma unroll
                for (int e = 0; e < 4; ++e)
#pragma unroll
                    for (int f = 0; f < 4; ++f) acc[e][f] = 0.f;
                rows_dot(o, 32, 4 * ti, 4 * (ti + left), acc);
                subtract(4 * ti, 4 * (ti + left), acc);
            }
            store_rows(sb);
        }
        named_bar_sync(DBAR_DONE, DF_HELP + 32);
        store_rows(0);
    } else if (warp == 12) {
        // the inverses of the sub-blocks (lane = column), by the reciprocals of the diagonal as it was rounded (with the reciprocal
        // roots instead U was off by 3 to 5 % more)
#pragma unroll 1
        for (int sb = 3; sb >= 0; --sb) {
            const int o = 32 * sb;
            float y[32];
#pragma unroll
            for (int k = 0; k < 32; ++k) y[k] = (k == lane) ? 1.f : 0.f;
            float *dst = INVERT ? X + o * ID_LD + o + lane : a.Rdiag + diag_inverse_at(sb, lane);
            solve32(y, &S[o][o], rdiag,
                    [&](int k) {
                        named_bar_sync(DBAR_COLS + (31 - k) / 8, 32 * (sb + 2));
                        if (lane < 8) rdiag[k - lane] = 1.f / S[o + k - lane][o + k - lane];
                        __syncwarp();
                    },
                    [&](int k, float v) { dst[INVERT ? k * ID_LD : k] = !INVERT || k <= lane ? v : 0.f; });
        }
    }
    __syncthreads();
    if (*abort_flag && tid == 0) record_status(a.hd, ST_TIMEOUT, 4000000 + a.b0);
    if (INVERT && tid < ID_THREADS) invert_products(&S[0][0], X, T, a.H, a.n, a.b0);
}

// ---------------------------------------------------------------------------
// Rows above the block: R[0:b0, blk] = A[0:b0, blk] R_pp^-T, 32 columns at a time: a product with the inverse of the
// 32 x 32 diagonal sub-block, then a rank-32 update of the columns to the left.  In place and, if asked for, as split
// parts for the tensor-core rank update.
// A warp takes 2, 4 or 8 rows from end to end: lane = (one (two) rows, 2 or 4 columns of every 32), the rows live in registers, the 32
// values of a row that all its lanes need go through shared memory inside the warp, so that no barrier of the CTA is on
// the way (a CTA-wide form with two barriers per sub-block: n = 14336 17.3 against 15.9 ms in all).  What bounds it: the
// words of R that shared memory returns (8k cycles; fetching them 3k); with two rows per lane they serve twice as many
// products, with one a narrow panel has twice as many warps, and with two columns a lane instead of four twice as many again (n = 384 116
// -> 114 us in all, 1024 249.8 -> 247.7, 4096 1266 -> 1260).
// One more CTA copies the block that is next on the diagonal, for the diag_factor_kernel that runs beside the update.
// ---------------------------------------------------------------------------
constexpr int PS_WORKERS = 4;                        // warps that take rows, at most
constexpr int PS_THREADS = 256;                      // all fetch R; the workers are the first warps
constexpr size_t PS_SMEM = (size_t)(NB * FP_LD + 4 * 32 * FP_YLD + PS_WORKERS * 8 * FP_YLD) * sizeof(float);

struct PanelSolveArgs {
    float *H; int n; int b0;
    const float *Rdiag;        // as diag_factor_kernel leaves it
    __half *pan_hi, *pan_lo;   // nullptr, or fp16 parts of split_scale(tc_amax[AMAX_PAN]) * row: row pitch pan_ld, this panel
    int pan_ld, pan_col0;      //   at columns pan_col0 .. + NB (several panels side by side)
    int workers;               // warps of a CTA that take rows
    int early;                 // the panel is up to date before the diagonal block is: rows may be read before pdl_wait()
    float *next_diag;          // nullptr, or [NB][NB]: receives the block at b0 - NB (by the last CTA)
    StateHeader *hd;
};

// A lane has C columns of every 32 of RPT rows; a warp C * RPT rows.
template <int C> struct alignas(4 * C) Cols { float v[C]; };
template <int C, int RPT>
__global__ void __launch_bounds__(PS_THREADS) panel_solve_kernel(PanelSolveArgs a) {
    constexpr int ROWS = C * RPT;                        // rows per warp
    extern __shared__ __align__(16) float smem_f[];
    float (*S)[FP_LD] = reinterpret_cast<float (*)[FP_LD]>(smem_f);                       // R^T, below the 32 x 32 diagonal sub-blocks
    float *Yt = reinterpret_cast<float *>(S + NB);                                        // [4][32][FP_YLD]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = a.workers;
    const int n = a.n, b0 = a.b0;
    const int nv = min(NB, n - b0);
    const bool vec = (n & 3) == 0 && (reinterpret_cast<uintptr_t>(a.H) & 15) == 0 && nv == NB;
    const int slabs = gridDim.x - (a.next_diag ? 1 : 0);
    const int ngroups = b0 / ROWS;
    const int q = lane & (32 / C - 1), rp = lane / (32 / C);        // C columns of every 32; row (pair of rows)
    float x[RPT][4][C];                                    // [row][sub-block][column]
    auto load_rows = [&](int g) {
#pragma unroll
        for (int e = 0; e < RPT; ++e) {
            const float *src = a.H + (int64_t)(g * ROWS + RPT * rp + e) * n + b0 + C * q;
#pragma unroll
            for (int sb = 0; sb < 4; ++sb) {
                if (vec) {
                    const Cols<C> v = *reinterpret_cast<const Cols<C> *>(src + 32 * sb);
#pragma unroll
                    for (int f = 0; f < C; ++f) x[e][sb][f] = v.v[f];
                } else {
#pragma unroll
                    for (int f = 0; f < C; ++f) x[e][sb][f] = 32 * sb + C * q + f < nv ? src[32 * sb + f] : 0.f;
                }
            }
        }
    };
    pdl_launch_dependents();
    int g = warp < nwarps ? (int)blockIdx.x * nwarps + warp : ngroups;
    const bool worker = blockIdx.x < slabs;
    if (a.early && worker && g < ngroups) load_rows(g);
    pdl_wait();
    if (!worker) {
        // the next diagonal block (asked for only where its rows are 16-byte aligned)
        for (int idx = tid; idx < NB * NB / 4; idx += PS_THREADS)
            *reinterpret_cast<float4 *>(a.next_diag + 4 * idx) =
                *reinterpret_cast<const float4 *>(a.H + (int64_t)(b0 - NB + (idx >> 5)) * n + b0 - NB + 4 * (idx & 31));
        return;
    }
    for (int idx = tid; idx < NB * (NB / 4); idx += PS_THREADS) {
        const int i = idx >> 5, j4 = idx & 31;
        if (j4 < (i >> 5) * 8) sg_copy16(&S[i][4 * j4], a.Rdiag + 4 * idx);
    }
    for (int idx = tid; idx < 4 * 32 * 8; idx += PS_THREADS)
        sg_copy16(Yt + (idx >> 3) * FP_YLD + 4 * (idx & 7), a.Rdiag + diag_inverse_at(idx >> 8, (idx >> 3) & 31) + 4 * (idx & 7));
    if (!a.early && g < ngroups) load_rows(g);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if (warp >= nwarps) return;
    float *buf = Yt + 4 * 32 * FP_YLD + (warp * ROWS + RPT * rp) * FP_YLD;                          // this lane's rows, 32 values each
    const float sc = a.pan_hi ? split_scale(__uint_as_float(a.hd->tc_amax[AMAX_PAN])) : 1.f;
    bool first = true;
    for (; g < ngroups; g += slabs * nwarps) {
        if (!first) load_rows(g);
#pragma unroll
        for (int sb = 3; sb >= 0; --sb) {
            __syncwarp();
#pragma unroll
            for (int e = 0; e < RPT; ++e)
#pragma unroll
                for (int f = 0; f < C; ++f) buf[e * FP_YLD + C * q + f] = x[e][sb][f];
            __syncwarp();
            // X = (row) inv(R_ss)^T
            const float *Ys = Yt + sb * 32 * FP_YLD + C * q;
            float acc[RPT][C];
#pragma unroll
            for (int e = 0; e < RPT; ++e)
#pragma unroll
                for (int f = 0; f < C; ++f) acc[e][f] = 0.f;
#pragma unroll 2
            for (int l = 0; l < 32; l += 4) {
                float v[RPT][4];
#pragma unroll
                for (int e = 0; e < RPT; ++e) {
                    const float4 w = *reinterpret_cast<const float4 *>(buf + e * FP_YLD + l);
                    v[e][0] = w.x; v[e][1] = w.y; v[e][2] = w.z; v[e][3] = w.w;
                }
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    const Cols<C> y = *reinterpret_cast<const Cols<C> *>(Ys + (l + h) * FP_YLD);
#pragma unroll
                    for (int e = 0; e < RPT; ++e)
#pragma unroll
                        for (int f = 0; f < C; ++f) acc[e][f] = fmaf(v[e][h], y.v[f], acc[e][f]);
                }
            }
#pragma unroll
            for (int e = 0; e < RPT; ++e)
#pragma unroll
                for (int f = 0; f < C; ++f) x[e][sb][f] = acc[e][f];
            if (sb == 0) break;
            // columns to the left: x[s'] -= X[l] R[.][32 sb + l]
            __syncwarp();
#pragma unroll
            for (int e = 0; e < RPT; ++e)
#pragma unroll
                for (int f = 0; f < C; ++f) buf[e * FP_YLD + C * q + f] = acc[e][f];
            __syncwarp();
#pragma unroll 1
            for (int l = 0; l < 32; l += 4) {
                float v[RPT][4];
#pragma unroll
                for (int e = 0; e < RPT; ++e) {
                    const float4 w = *reinterpret_cast<const float4 *>(buf + e * FP_YLD + l);
                    v[e][0] = w.x; v[e][1] = w.y; v[e][2] = w.z; v[e][3] = w.w;
                }
#pragma unroll
                for (int h = 0; h < 4; ++h)
#pragma unroll
                    for (int t = 0; t < sb; ++t) {
                        const Cols<C> r = *reinterpret_cast<const Cols<C> *>(&S[32 * sb + l + h][32 * t + C * q]);
#pragma unroll
                        for (int e = 0; e < RPT; ++e)
#pragma unroll
                            for (int f = 0; f < C; ++f) x[e][t][f] = fmaf(-v[e][h], r.v[f], x[e][t][f]);
                    }
            }
        }
        first = false;
        // the rows (and their split parts)
#pragma unroll
        for (int e = 0; e < RPT; ++e) {
            const int64_t row = g * ROWS + RPT * rp + e;
#pragma unroll
            for (int sb = 0; sb < 4; ++sb) {
                const int c = 32 * sb + C * q;
                float *dst = a.H + row * n + b0 + c;
                Cols<C> v;
#pragma unroll
                for (int f = 0; f < C; ++f) v.v[f] = x[e][sb][f];
                if (vec) *reinterpret_cast<Cols<C> *>(dst) = v;
                else {
#pragma unroll
                    for (int f = 0; f < C; ++f) if (c + f < nv) dst[f] = v.v[f];
                }
                if (a.pan_hi) {
#pragma unroll
                    for (int f = 0; f < C; f += 2) {
                        const float s0 = sc * v.v[f], s1 = sc * v.v[f + 1];
                        const __half2 h = __floats2half2_rn(s0, s1);
                        const float2 hf = __half22float2(h);
                        const int64_t at = row * a.pan_ld + a.pan_col0 + c + f;
                        *reinterpret_cast<__half2 *>(a.pan_hi + at) = h;
                        *reinterpret_cast<__half2 *>(a.pan_lo + at) = __floats2half2_rn(s0 - hf.x, s1 - hf.y);
                    }
                }
            }
        }
    }
}

}  // namespace gptaq
