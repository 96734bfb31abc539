// The column loop of Algorithm 1 over several lazy-batch blocks of columns in ONE launch.
//
// Rows of W are independent, so a CTA that owns 32 rows (16 where there are few) can run the sequential part of the loop over many
// lazy-batch blocks without ever meeting another CTA.  Its slab of W (32 x 512 float32) stays in shared
// memory; what would be a launch per block and a product per block over the whole matrix is a pipeline of
// warp roles inside the CTA:
//
//   chain   (4 warps)  quantizes 32 columns at a time: a lane has a row, a warp 8 consecutive columns of all rows, which it
//                      publishes in shared memory four at a time for the warps with the columns behind them;
//   near    (8 warps)  applies a step's errors to the rest of its 128-column block (float32 FMA), 8 columns
//                      behind the chain, fetches the rows of U and P of the next step, makes the errors of every 64
//                      columns the tensor cores' operand, writes results out;
//   drain   (4 warps)  adds the products of the tensor cores to the later blocks of the slab;
//   load, mma (1 + 1)  stream U^T and P^T (fp16 hi / lo parts) and issue
//                      D[128 later columns][32 rows] = [U^T | P^T] [-Err | rho Wpre]^T   (tcgen05, M = 128)
//                      for every 64 quantized columns; hi*hi and the small terms hi*lo + lo*hi have a column each.
//
// What bounds it: the chain, and the near warps behind it.  A column is 7 dependent float32 operations (28 cycles); with its
// share of the updates, the codes and the hand-over to the next warp 8 columns take 750 cycles alone and 950 beside the near
// warps, which need 830 for them (a scheduler starts a 16-byte LDS in 8 cycles where lanes share words, in 16 where they do
// not).  A step of 32 columns ends 1500 to 2000 cycles after its last column (the near warps' last 8 columns, results), the products
// between two blocks take 4000 to 5000 (operand, streamed tiles, MMAs, adding them up).
// A launch of 512 columns of 4096 rows by itself (ncu; the second and the first of two: the first also writes the
// operand of the update beyond it) with a group grid per 128 columns and without: with 4-byte copies of U and P, the operand of a
// block's end behind the next step's rows and hi and lo parts in turn 69.6 / 74.9 and 67.6 / 71.6 us, now 64.1 / 69.0 and 62.1 / 67.5;
// of 512 rows, with 16 of them a CTA, 65.5 / 70.9 and 63.6 / 67.6, now 53.9 / 57.5 and 53.0 / 56.4.
// Spills (32 rows; 16): the tensor-core form has 96 registers and spills 64 bytes (44), static groups 60 (56); the near form has 80
// where two CTAs share an SM and spills 100 (static groups 132), with one to an SM up to 158 and spills nothing.
#pragma once
#include "simt_gemm.cuh"
#include "tc_gemm.cuh"

namespace gptaq {

// Rows of W per CTA, and where there are few of them (launch_quant_block): half the rows are half the work for the near and the
// drain warps, and the chain, which takes as long for 16 rows as for 32, has less of it beside itself (eight columns 700 to 900 cycles
// for 750 to 950, a launch of 512 columns 64 -> 57 us).
constexpr int QB_ROWS = 32, QB_ROWS_FEW = 16;
constexpr int QB_W = 128;               // columns per block (float32 updates inside, tensor cores beyond)
constexpr int QB_SUPER = 512;           // most columns per launch
constexpr int QB_CHAIN = 128, QB_NEAR = 256, QB_DRAIN = 128;
constexpr int QB_THREADS_NEAR = QB_CHAIN + QB_NEAR;                   // one block per launch, no tensor cores
constexpr int QB_THREADS_FAR = QB_THREADS_NEAR + QB_DRAIN + 64;
// rows of U and P of a step: boxes of 32 rows x 32 columns, the buffer of even steps has four of each matrix, that of odd ones three
constexpr int QB_BOX = 32 * 32, QB_BOXES0 = QB_W / 32, QB_BOXES1 = QB_BOXES0 - 1;
__host__ __device__ constexpr int qb_sld(int rows) { return rows + 4; }   // pitch of the published errors
// 128 x 64 fp16 tiles of U^T / P^T in flight: what shared memory holds (the grids per column take the room of one)
constexpr int QB_MAX_ASLOTS = 6;
__host__ __device__ constexpr int qb_aslots(bool percol, int rows) { return (rows == 32 ? 3 : QB_MAX_ASLOTS) - (percol ? 1 : 0); }
constexpr int QB_A_BYTES = 128 * 64 * 2;
__host__ __device__ constexpr int qb_e_bytes(int rows) { return rows * 64 * 2; }          // one K-block (64 columns) of one part of the errors
__host__ __device__ constexpr int qb_half_bytes(int rows) { return 4 * qb_e_bytes(rows); } // (hi, lo) x (-Err, Wpre) of 64 columns
// tensor memory: 2 halves x 3 blocks x 2 groups (hi hi; hi lo + lo hi) of a column per row, a power of two
__host__ __device__ constexpr int qb_tmem_cols(int rows) { return rows == 32 ? 512 : 256; }

struct QuantBlockArgs {
    float *W; int64_t ldw; int row_first, m, n;     // rows [row_first, m)
    // where the values come from: nullptr (W itself), or the caller's weights, float32 or bfloat16 (a launch that takes all columns)
    const void *src; int64_t lds; int src_bf16;
    const float *U, *P;        // n x n, ld n; entries below the diagonals are not used
    int up_tma;                // U and P qualify for tensor maps (16-byte rows)
    const uint8_t *dead;
    int i0, i1;                // columns of this launch: [i0, i1); i1 - i0 <= QB_SUPER (tensor-core form) or one block
    int bw;                    // columns per block: QB_W (tensor-core form); 32, 64 or 128
    int bits, group, sym;
    uint8_t *codes;            // m x n
    float *scales, *zeros;     // m x G
    int G;
    float *EW; int ew_ld, ew_pre;   // [-Err | rho * Wpre] of this launch, row pitch, offset of Wpre in a row
    // fp16 parts of [-Err | rho * Wpre] for the update beyond i1, one power-of-two scale per row (row_inv = 1 / scale),
    // or nullptr (nothing beyond); pitch ew_ld
    __half *EWS_hi, *EWS_lo;
    float *row_inv;
    const unsigned *amax_u, *amax_p;   // fp16-split handles: recorded maxima of U and P (rho = scale of U / scale of P)
    StateHeader *hd;
    float err_scale, asym_scale;   // 1 or 0: switches of the two terms of the weight update (ablation)
    const int *perm;               // nullptr, or: working column c is original column perm[c] (codes go there)
    int clip_steps; float clip_min;
};

static_assert(64 * qb_sld(QB_ROWS_FEW) >= 24 * qb_sld(QB_ROWS_FEW) + 8 * QB_ROWS_FEW + 2 * QB_NEAR, "scratch of the clipping search");
// Shared memory, in bytes from a 1024-byte boundary.  The tensor-core operands come first (alignment).
struct QuantBlockSmem {
    int a, e, w, up, st, grid, udinv, perm, inv, rmax, bars, total, wld;
};
__host__ __device__ constexpr QuantBlockSmem quant_block_smem(bool far_form, bool percol, int rows) {
    QuantBlockSmem s{};
    s.wld = (far_form ? QB_SUPER : QB_W) + 4;
    s.a = 0;
    s.e = s.a + (far_form ? qb_aslots(percol, rows) * QB_A_BYTES : 0);
    s.w = s.e + (far_form ? 2 * qb_half_bytes(rows) : 0);
    s.up = s.w + rows * s.wld * 4;
    s.st = s.up + 2 * (QB_BOXES0 + QB_BOXES1) * QB_BOX * 4;
    s.grid = s.st + 2 * 64 * qb_sld(rows) * 4;
    s.udinv = s.grid + (percol ? 3 * 32 * qb_sld(rows) * 4 : 0);
    s.perm = s.udinv + (s.wld - 4) * 4;
    s.inv = s.perm + (s.wld - 4) * 4;
    s.rmax = s.inv + 2 * rows * 4;
    s.bars = s.rmax + (far_form ? QB_NEAR * 4 : 0);
    s.total = s.bars + 384;
    return s;
}
constexpr size_t quant_block_smem_bytes(bool far_form, bool percol, int rows) {
    return (size_t)quant_block_smem(far_form, percol, rows).total + 1024;        // (alignment slack)
}
static_assert(quant_block_smem_bytes(true, false, QB_ROWS) <= 227 * 1024 && quant_block_smem_bytes(true, true, QB_ROWS) <= 227 * 1024 &&
              quant_block_smem_bytes(true, false, QB_ROWS_FEW) <= 227 * 1024 && quant_block_smem_bytes(true, true, QB_ROWS_FEW) <= 227 * 1024, "shared memory of one SM");

// kind::f16 instruction descriptor: fp16 A and B (K-major), fp32 D, M = 128, N = cols.
__host__ __device__ constexpr uint32_t qb_idesc(int cols) { return (1u << 4) | ((uint32_t)(cols >> 3) << 17) | ((128 >> 4) << 24); }

// Named barriers.  Chunk barriers are used once per step each; the step barrier keeps the chain from lapping them.
enum { QBAR_CHUNK = 1, QBAR_STEP = 5, QBAR_NEAR = 6, QBAR_DRAIN = 7, QBAR_CLIP = 8, QBAR_HAND = 9 /* .. 14 */, QBAR_CHAIN = 15 };

// Position of a row in a column of the published errors: the near warps' threads take rows ti, ti + 8, .. as
// one 16-byte read.
template <int ROWS>
__device__ __forceinline__ int qb_pos(int row) { return (row & 7) * (ROWS / 8) + (row >> 3); }

__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

// Two float32 FMAs in one instruction: the roles share their schedulers' issue slots, which the chain is short of.
__device__ __forceinline__ unsigned long long pack2(float x, float y) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ float lo2(unsigned long long v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ float hi2(unsigned long long v) { return __uint_as_float((uint32_t)(v >> 32)); }
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ float pick2(const unsigned long long (&v)[4], int j) { return (j & 1) ? hi2(v[j >> 1]) : lo2(v[j >> 1]); }

__device__ __forceinline__ void lds_pair2(const float *p, unsigned long long &x, unsigned long long &y) {
    const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(p);
    x = v.x; y = v.y;
}
__device__ __forceinline__ void lds_pair4(const float *p, unsigned long long (&x)[4]) {
    lds_pair2(p, x[0], x[1]);
    lds_pair2(p + 4, x[2], x[3]);
}

__device__ __forceinline__ float fma_sat(float a, float b, float c) {
    float r;
    asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Squared rounding errors of 2 NP candidates k, k + stride, .. over one row's group in one pass (`w`: n weights, n a multiple
// of 4, 16-byte aligned); keeps the least in (best, kbest).
template <int NP>
__device__ __forceinline__ void clip_pass(const float *w, int n, float lo, float hi, int bits, int sym, int steps, float clip_min,
                                          int k, int stride, float &best, int &kbest) {
    const float am = fmaxf(-lo, hi), maxq = (float)((1 << bits) - 1), magic = 12582912.f;
    const unsigned long long mg = pack2(magic, magic), mq = pack2(maxq, maxq), one = pack2(1.f, 1.f);
    float ta[2 * NP], tb[2 * NP];                   // (w / scale + zero) / maxq
    unsigned long long sc2[NP], nz[NP], err[NP];    // scale; -(1.5 * 2^23 + zero), exact
#pragma unroll
    for (int h = 0; h < NP; ++h) {
        float sc[2], z[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const float p = clip_ratio(min(k + (2 * h + e) * stride, steps - 1), steps, clip_min);
            make_grid(p * lo, p * hi, p * am, bits, sym, sc[e], z[e]);
            ta[2 * h + e] = 1.f / (sc[e] * maxq); tb[2 * h + e] = z[e] / maxq;
        }
        sc2[h] = pack2(sc[0], sc[1]); nz[h] = pack2(-(magic + z[0]), -(magic + z[1]));
        err[h] = 0ull;
    }
#pragma unroll 1
    for (int c = 0; c < n; c += 4) {
        const float4 v = *reinterpret_cast<const float4 *>(w + c);
        const float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            const unsigned long long nx2 = pack2(-x[f], -x[f]);
#pragma unroll
            for (int h = 0; h < NP; ++h) {
                // clamped to the grid by saturation (minimum and maximum are a pipe of their own, and it was the one that
                // bound the search), then rounded by adding and subtracting 1.5 * 2^23
                const unsigned long long t = pack2(fma_sat(x[f], ta[2 * h], tb[2 * h]), fma_sat(x[f], ta[2 * h + 1], tb[2 * h + 1]));
                const unsigned long long c = fma2(fma2(t, mq, mg), one, nz[h]);            // code - zero
                const unsigned long long d = fma2(sc2[h], c, nx2);
                err[h] = fma2(d, d, err[h]);
            }
        }
    }
#pragma unroll
    for (int e = 0; e < 2 * NP; ++e) {
        const float er = (e & 1) ? hi2(err[e >> 1]) : lo2(err[e >> 1]);
        if (k + e * stride < steps && er < best) { best = er; kbest = k + e * stride; }
    }
}

// Least squared rounding error of one row's group among candidates k0, k0 + stride, ..: ten per pass over the weights while
// more than four are left, else four (four throughout and clamped by minimum and maximum, 4096 x 4096 with 80 candidates:
// 1541 us a call, then 1419).  What bounds it is the number of its instructions, two cycles each on a scheduler whatever their pipe: an
// integer minimum in place of the two saturating FMAs of a pair, on codes rounded as subnormal numbers, took as long.  Four
// columns a round: unrolled further the registers ran out (4096 x 1024 251 us, now 242 with the range from the chain's own).
__device__ __forceinline__ void clip_search(const float *w, int n, float lo, float hi, int bits, int sym, int steps, float clip_min,
                                            int k0, int stride, float &best, int &kbest) {
    best = INFINITY; kbest = 0;
    int k = k0;
    for (; k + 4 * stride < steps; k += 10 * stride) clip_pass<5>(w, n, lo, hi, bits, sym, steps, clip_min, k, stride, best, kbest);
    if (k < steps) clip_pass<2>(w, n, lo, hi, bits, sym, steps, clip_min, k, stride, best, kbest);
}

// FAR: several blocks per launch, updates between them on the tensor cores.  PERCOL: static groups, a grid per column.
// CTAS: CTAs that share an SM (shared memory allows one of the tensor-core form).
template <bool FAR, bool PERCOL, int CTAS, int ROWS = QB_ROWS>
__global__ void __launch_bounds__(FAR ? QB_THREADS_FAR : QB_THREADS_NEAR, CTAS)
quant_block_kernel(const __grid_constant__ CUtensorMap mapUhi, const __grid_constant__ CUtensorMap mapUlo,
                   const __grid_constant__ CUtensorMap mapPhi, const __grid_constant__ CUtensorMap mapPlo,
                   const __grid_constant__ CUtensorMap mapU, const __grid_constant__ CUtensorMap mapP, QuantBlockArgs a) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t *sm = smem_raw + (base - raw);
    constexpr QuantBlockSmem L = quant_block_smem(FAR, PERCOL, ROWS);
    constexpr int SLD = qb_sld(ROWS), E_BYTES = qb_e_bytes(ROWS), HALF_BYTES = qb_half_bytes(ROWS), RPT = ROWS / 8;
    constexpr int ASLOTS = qb_aslots(PERCOL, ROWS);
    constexpr int WLD = L.wld;
    constexpr int NTHREADS = FAR ? QB_THREADS_FAR : QB_THREADS_NEAR;
    float *Ws = reinterpret_cast<float *>(sm + L.w);               // [32][WLD]: the slab
    float *UPs = reinterpret_cast<float *>(sm + L.up);             // rows of U and P of the current and the next step
    float *Sts = reinterpret_cast<float *>(sm + L.st);             // [2 steps][64][SLD]: -Err, then Wpre, of 32 columns
    float *grid_s = reinterpret_cast<float *>(sm + L.grid);        // PERCOL: scales, zero points, 1 / scales, [32 columns][SLD] each
    float *udinv_s = reinterpret_cast<float *>(sm + L.udinv);      // of every column of the launch: err_scale / U_kk
    int *perm_s = reinterpret_cast<int *>(sm + L.perm);            // ... and where its codes go
    float *inv_s = reinterpret_cast<float *>(sm + L.inv);          // [2 halves][32]: 1 / scale of a row's errors
    float *rmax_s = reinterpret_cast<float *>(sm + L.rmax);        // [8 near warps][32]: a row's largest error of 8 columns
    const uint32_t bar0 = base + L.bars;
    // mbarriers (8 bytes each): afull, aempty, efull[2], efree[2], tfull[6], tempty[6], upfull[2]; tmem slot, abort flag
    constexpr int EB = 2 * QB_MAX_ASLOTS;
    auto afull = [&](int s) { return bar0 + 8u * s; };
    auto aempty = [&](int s) { return bar0 + 8u * (QB_MAX_ASLOTS + s); };
    auto efull = [&](int s) { return bar0 + 8u * (EB + s); };
    auto efree = [&](int s) { return bar0 + 8u * (EB + 2 + s); };
    auto tfull = [&](int s) { return bar0 + 8u * (EB + 4 + s); };
    auto tempty = [&](int s) { return bar0 + 8u * (EB + 10 + s); };
    auto upfull = [&](int s) { return bar0 + 8u * (EB + 16 + s); };
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(sm + L.bars + 8 * (EB + 18));
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = a.n, i0 = a.i0, B = a.bw;
    const int row0 = a.row_first + blockIdx.x * ROWS;
    const int nrows = min(ROWS, a.m - row0);
    const int cols = a.i1 - i0;
    const int nblk = FAR ? (cols + QB_W - 1) / QB_W : 1;
    auto nsteps = [&](int b) { return min(B / 32, (cols - b * QB_W + 31) / 32); };     // 32-column steps of block b
    const float maxq = (float)((1 << a.bits) - 1);
    // U / P rows of step s of the block that starts at column cb, columns cb + 32 s ..: buffer s & 1, box by box; element (k, c) of
    // U at up_at(s, 0, k, c), of P at up_at(s, 1, k, c).  One thread asks the TMA unit for the boxes: as 16-byte
    // copies by all near warps a step's 32 KB took 1100 cycles of their time, in steps where the chain waits for them (4096 x 1024 with
    // groups 165 -> 161 us a call, 1024 x 1024 with static groups 163 -> 160).  Rows that are no multiple of 16 bytes come in asynchronous
    // copies of 4 (word by word through registers before: 777 x 777 217 -> 191, 4096 x 777 501 -> 486).
    // a step's error buffer, before its first column is quantized: the four quarters of the group's ranges
    auto range_at = [&](float *st) { return reinterpret_cast<float2 *>(st + 24 * SLD); };
    auto up_at = [&](int s, int q, int k, int c) {
        return UPs + ((s & 1) ? 2 * QB_BOXES0 * QB_BOX : 0) + (q * ((s & 1) ? QB_BOXES1 : QB_BOXES0) + (c >> 5)) * QB_BOX + k * 32 + (c & 31);
    };
    auto fetch_up = [&](int cb, int s, int t, int nthr) {
        const int r0 = cb + 32 * s;
        if (a.up_tma) {
            if (t == 0) {
                const int boxes = B / 32 - s;
                mbar_expect_tx(upfull(s & 1), (uint32_t)(2 * boxes * QB_BOX * 4));
                for (int x = 0; x < boxes; ++x) {
                    tma_load_2d(smem_u32(up_at(s, 0, 0, 32 * x)), &mapU, r0 + 32 * x, r0, upfull(s & 1));
                    tma_load_2d(smem_u32(up_at(s, 1, 0, 32 * x)), &mapP, r0 + 32 * x, r0, upfull(s & 1));
                }
            }
            return;
        }
        // (a warp per row, a lane per column)
        const int l = t & 31;
        for (int k = t >> 5; k < 32; k += nthr / 32)
            for (int x = 0; x < B / 32 - s; ++x) {
                const bool in = r0 + k < n && r0 + 32 * x + l < n;
                const int64_t off = in ? (int64_t)(r0 + k) * n + r0 + 32 * x + l : 0;
                sg_copy4(up_at(s, 0, k, 32 * x + l), a.U + off, in);
                sg_copy4(up_at(s, 1, k, 32 * x + l), a.P + off, in);
            }
    };
    auto load_perm = [&](int c) { return a.perm && c < n ? a.perm[c] : c; };
    // PERCOL: grids of four columns c .. c + 3 of a row
    auto load_grid = [&](int r, int c, float (&sc)[4], float (&zp)[4]) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            sc[e] = 1.f; zp[e] = 0.f;
            if (r < nrows && c + e < n) {
                const int64_t g = (int64_t)(row0 + r) * a.G + load_perm(c + e) / a.group;
                sc[e] = a.scales[g]; zp[e] = a.zeros[g];
            }
        }
    };
    auto store_grid = [&](int r, int c, const float (&sc)[4], const float (&zp)[4]) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            grid_s[(c + e) * SLD + r] = sc[e];
            grid_s[(32 + c + e) * SLD + r] = zp[e];
            grid_s[(64 + c + e) * SLD + r] = 1.f / sc[e];
        }
    };

    // ---------------------------------------------------------------- set-up: barriers, tensor memory, slab, first rows of U / P
    if (tid == 0) {
        for (int s = 0; s < 2; ++s) mbar_init(upfull(s), 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (FAR) {
        if (tid == 0) {
            for (int s = 0; s < ASLOTS; ++s) { mbar_init(afull(s), 1); mbar_init(aempty(s), 1); }
            for (int s = 0; s < 2; ++s) { mbar_init(efull(s), 8 * ROWS / 32); mbar_init(efree(s), QB_DRAIN / 32); }
            for (int s = 0; s < 6; ++s) { mbar_init(tfull(s), 1); mbar_init(tempty(s), QB_DRAIN / 32); }
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        if (warp == NTHREADS / 32 - 1) {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                         ::"r"(smem_u32(const_cast<uint32_t *>(tmem_slot))), "r"((uint32_t)qb_tmem_cols(ROWS)) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
    }
    // the slab and the first rows of U and P all in flight at once (8k cycles; in batches through registers twice that); U and P
    // without waiting for the launch before this one
    if (!FAR) pdl_launch_dependents();
    fetch_up(i0, 0, tid, NTHREADS);
    if (!FAR) pdl_wait();
    const int cq = FAR ? nblk * (QB_W / 4) : B / 4;                // quads per row, padded columns included
    // (i0 is a multiple of 32)
    const float *from = a.src ? static_cast<const float *>(a.src) : a.W;
    const int64_t ldf = a.src ? a.lds : a.ldw;
    const bool wvec = (ldf & 3) == 0 && (reinterpret_cast<uintptr_t>(from) & (a.src_bf16 ? 7 : 15)) == 0;
    // a thread: four columns of every RSTEP-th row
    constexpr int WQ = FAR ? QB_SUPER / 4 : QB_W / 4, RSTEP = NTHREADS / WQ;
    const int wq = tid % WQ, wr0 = tid / WQ, wc = 4 * wq;
    const bool fills = wr0 < RSTEP && wq < cq;
    if (fills) {
        const bool whole = wvec && wc + 3 < cols;
        const int64_t off = (int64_t)(row0 + wr0) * ldf + i0 + wc;
        const float *src = from + off;
        const __nv_bfloat16 *src16 = static_cast<const __nv_bfloat16 *>(a.src) + off;
        float *dst = Ws + wr0 * WLD + wc;
        if (a.src_bf16) {
#pragma unroll 4
            for (int r = wr0; r < ROWS; r += RSTEP, src16 += (int64_t)RSTEP * ldf, dst += RSTEP * WLD) {
                Quad<__nv_bfloat16> q;
                if (whole && r < nrows) q = *reinterpret_cast<const Quad<__nv_bfloat16> *>(src16);
                else {
#pragma unroll
                    for (int e = 0; e < 4; ++e) q.v[e] = r < nrows && wc + e < cols ? src16[e] : __float2bfloat16(0.f);
                }
                *reinterpret_cast<float4 *>(dst) = make_float4((float)q.v[0], (float)q.v[1], (float)q.v[2], (float)q.v[3]);
            }
        } else for (int r = wr0; r < ROWS; r += RSTEP) {
            if (whole && r < nrows) cp_async16(dst, src);
            else {
#pragma unroll
                for (int e = 0; e < 4; ++e) dst[e] = r < nrows && wc + e < cols ? src[e] : 0.f;
            }
            src += (int64_t)RSTEP * ldf; dst += RSTEP * WLD;
        }
    }
    // (dead inputs read as zero; the flags are 4-byte aligned and padded beyond n)
    const uint32_t dead4 = fills && wc < cols ? *reinterpret_cast<const uint32_t *>(a.dead + i0 + wc) : 0u;
    // (padded columns beyond n have no error: 0.  All at once here: with a step's 32 made by the near warps at the end of the step before,
    // the operand behind what the next step needs at a block's end and the minima eight columns at a time 512 x 1024 took 131 us, now
    // 130; 2369 x 1024 154.6 and 150.5, 4768 x 1024 231 and 226, 512 x 1024 without tensor cores 213 and 204)
    for (int c = tid; c < L.wld - 4; c += NTHREADS) {
        udinv_s[c] = i0 + c < n && c < cols ? a.err_scale * (1.f / a.U[(int64_t)(i0 + c) * n + i0 + c]) : 0.f;
        perm_s[c] = load_perm(i0 + c);
    }
    if (PERCOL && tid < 8 * ROWS) {
        float sc[4], zp[4];
        load_grid(tid >> 3, i0 + 4 * (tid & 7), sc, zp);
        store_grid(tid >> 3, 4 * (tid & 7), sc, zp);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (fills && dead4) {
        float4 *wp = reinterpret_cast<float4 *>(Ws + wr0 * WLD + wc);                  // (the words that this thread has copied)
        for (int r = wr0; r < ROWS; r += RSTEP, wp += RSTEP * WLD / 4) {
            float4 v = *wp;
            if (dead4 & 0xffu) v.x = 0.f;
            if (dead4 & 0xff00u) v.y = 0.f;
            if (dead4 & 0xff0000u) v.z = 0.f;
            if (dead4 & 0xff000000u) v.w = 0.f;
            *wp = v;
        }
    }
    if (FAR) tc_fence_before();
    __syncthreads();
    if (FAR) tc_fence_after();
    if (a.up_tma) mbar_wait(upfull(0), 0u, abort_flag);

    float rho = 1.f, su = 1.f;
    if (a.amax_u) {
        su = split_scale(__uint_as_float(*a.amax_u));
        const float ap = __uint_as_float(*a.amax_p);
        rho = ap > 0.f ? su / split_scale(ap) : 0.f;
    }
    const float inv_su = 1.f / su;
    const int last_groups = nblk - 1;                               // blocks 0 .. nblk - 2 have later blocks in this launch
    // a grid is made at column c (groups have 32, 64 or 128 columns)
    auto grid_starts = [&](int c) { return !PERCOL && a.group > 0 && (c & (a.group - 1)) == 0; };

    if (tid < QB_CHAIN) {
        // ================================================================ chain
        const int lrow = lane & (ROWS - 1), w8 = 8 * warp;          // (16 rows: the upper lanes do the same as the lower ones)
                             // this warp's columns of a step: w8 .. w8 + 7
        const int row = row0 + lrow;
        const bool live = lrow < nrows;
        float *wrow = Ws + lrow * WLD;
        const int pos = qb_pos<ROWS>(lrow);
        float scale = 1.f, zero = 0.f;
        if (!PERCOL && a.group <= 0 && live) { scale = a.scales[row]; zero = a.zeros[row]; }
        float inv_scale = 1.f / scale, qlo = -zero, qhi = maxq - zero;
#pragma unroll 1
        for (int b = 0; b < nblk; ++b) {
            const int nst = nsteps(b);
#pragma unroll 1
            for (int s = 0; s < nst; ++s) {
                const int co = b * QB_W + 32 * s;                   // first column of the step in the slab
                const int cg = i0 + co;                             // ... in W
                if (b + s > 0) named_bar_sync(QBAR_STEP, QB_THREADS_NEAR);
                if (FAR && s == 0 && b > 0) named_bar_sync(QBAR_DRAIN, QB_CHAIN + QB_DRAIN);
                float *St = Sts + (s & 1) * 64 * SLD;
                float scv[8], ivv[8], zv[8];
                if (PERCOL) {
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        scv[e] = grid_s[(w8 + e) * SLD + lrow];
                        zv[e] = grid_s[(32 + w8 + e) * SLD + lrow];
                        ivv[e] = grid_s[(64 + w8 + e) * SLD + lrow];
                    }
                } else if (grid_starts(cg)) {
                    // grid of the group that starts here, from the current values (columns of it beyond the layer are zeros):
                    // a quarter of the range per warp
                    float lo = 0.f, hi = 0.f;
                    const float *wq4 = wrow + co + warp * (a.group >> 2);
                    float4 v[8];                                    // (all loads in flight: 8, 16 or 32 columns)
#pragma unroll
                    for (int c = 0; c < 8; ++c)
                        v[c] = 4 * c < a.group >> 2 ? *reinterpret_cast<const float4 *>(wq4 + 4 * c) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        lo = fminf(lo, fminf(fminf(v[c].x, v[c].y), fminf(v[c].z, v[c].w)));
                        hi = fmaxf(hi, fmaxf(fmaxf(v[c].x, v[c].y), fmaxf(v[c].z, v[c].w)));
                    }
                    // (through the part of the step's error buffer that warp 3 publishes into, after all have read it)
                    float2 *range_s = range_at(St);
                    range_s[warp * ROWS + lrow] = make_float2(lo, hi);
                    named_bar_sync(QBAR_CHAIN, QB_CHAIN);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float2 v = range_s[q * ROWS + lrow];
                        lo = fminf(lo, v.x); hi = fmaxf(hi, v.y);
                    }
                    float p = 1.f;
                    if (a.clip_steps > 0) {
                        named_bar_sync(QBAR_CLIP, QB_THREADS_NEAR);          // the near warps search
                        named_bar_sync(QBAR_CLIP, QB_THREADS_NEAR);
                        p = clip_ratio(reinterpret_cast<int *>(St)[lrow], a.clip_steps, a.clip_min);
                    }
                    make_grid(p * lo, p * hi, p * fmaxf(-lo, hi), a.bits, a.sym, scale, zero);
                    if (live && warp == 3 && lane < ROWS) {          // (the warp that has most time)
                        const int g = cg >> (31 - __clz(a.group));
                        a.scales[(int64_t)row * a.G + g] = scale;
                        a.zeros[(int64_t)row * a.G + g] = zero;
                    }
                    if (a.clip_steps > 0) named_bar_sync(QBAR_CLIP, QB_THREADS_NEAR);   // the search's scratch is free again
                    inv_scale = 1.f / scale; qlo = -zero; qhi = maxq - zero;
                }
                constexpr int ld = 32;
                const float *Uw = up_at(s, 0, 0, w8), *Pw = up_at(s, 1, 0, w8);
                unsigned long long x[4];                            // this lane's 8 columns, in pairs
                {
                    const ulonglong2 v0 = *reinterpret_cast<const ulonglong2 *>(wrow + co + w8);
                    const ulonglong2 v1 = *reinterpret_cast<const ulonglong2 *>(wrow + co + w8 + 4);
                    x[0] = v0.x; x[1] = v0.y; x[2] = v1.x; x[3] = v1.y;
                }
                // the earlier columns of the step, four at a time as the warps before this one publish them; their rows of U
                // and P are fetched before the wait
#pragma unroll 1
                for (int h = 0; h < 2 * warp; ++h) {
                    unsigned long long u[4][4], pp[4][4];
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        lds_pair4(Uw + (4 * h + kk) * ld, u[kk]);
                        lds_pair4(Pw + (4 * h + kk) * ld, pp[kk]);
                    }
                    named_bar_sync(QBAR_HAND + h, 32 * (4 - (h >> 1)));
                    const float *Se = St + 4 * h * SLD + pos;
                    float er[4], wa[4];
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) { er[kk] = Se[kk * SLD]; wa[kk] = Se[(32 + kk) * SLD]; }
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        const unsigned long long ne2 = pack2(er[kk], er[kk]), wa2 = pack2(wa[kk], wa[kk]);
#pragma unroll
                        for (int j = 0; j < 4; ++j) x[j] = fma2(ne2, u[kk][j], fma2(wa2, pp[kk][j], x[j]));
                    }
                }
                // `c` is the chain: the current column's value.  Entries of x that belong to columns already done are garbage
                // (entries of U and P at or below the diagonal are applied to them) and never read again.
                const float *ud = udinv_s + co + w8;
                const float4 ud0 = *reinterpret_cast<const float4 *>(ud), ud1 = *reinterpret_cast<const float4 *>(ud + 4);
                const float udv[8] = {ud0.x, ud0.y, ud0.z, ud0.w, ud1.x, ud1.y, ud1.z, ud1.w};
                Uw += w8 * ld; Pw += w8 * ld;
                float *Sw = St + w8 * SLD + pos;
                float qv[8];
                uint32_t code[2] = {0u, 0u};
                float c = lo2(x[0]);
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    unsigned long long u[4][4], pp[4][4];           // (columns that no lane needs any more are not read)
                    float nerr[4], pre[4];
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        const int k = 4 * half + kk;
                        if (k < 3) { lds_pair2(Uw + k * ld, u[kk][0], u[kk][1]); lds_pair2(Pw + k * ld, pp[kk][0], pp[kk][1]); }
                        if (k < 7) { lds_pair2(Uw + k * ld + 4, u[kk][2], u[kk][3]); lds_pair2(Pw + k * ld + 4, pp[kk][2], pp[kk][3]); }
                    }
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        const int k = 4 * half + kk;
                        const float sc = PERCOL ? scv[k] : scale;
                        const float iv = PERCOL ? ivv[k] : inv_scale;
                        const float z = PERCOL ? zv[k] : zero;
                        const float w0 = c;
                        // round(w / scale), clamped to the grid, minus the zero point.  Adding 1.5 * 2^23 rounds to nearest even
                        // wherever |v| < 2^22 and leaves larger values large (the clamp decides those).
                        const float magic = 12582912.f;
                        const float r = __fsub_rn(__fadd_rn(__fmul_rn(w0, iv), magic), magic);
                        const float cz = fminf(fmaxf(r, PERCOL ? -z : qlo), PERCOL ? maxq - z : qhi);
                        const float d = __fmaf_rn(sc, cz, -w0);                  // -(w - q)
                        const float ne = d * udv[k];                             // ... / U_kk
                        const float wa = a.asym_scale * w0;
                        qv[k] = sc * cz; nerr[kk] = ne; pre[kk] = wa;
                        code[k >> 2] |= (__float_as_uint(cz + z + magic) & 0xffu) << (8 * (k & 3));
                        if (k == 7) continue;
                        // the next column from the error itself, the ones after it through x
                        c = fmaf(d, udv[k] * pick2(u[kk], k + 1), fmaf(wa, pick2(pp[kk], k + 1), pick2(x, k + 1)));
                        const unsigned long long ne2 = pack2(ne, ne), wa2 = pack2(wa, wa);
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            if (2 * j + 1 < k + 2) continue;
                            x[j] = fma2(ne2, u[kk][j], fma2(wa2, pp[kk][j], x[j]));
                        }
                    }
                    // publish these 4 columns: to the chain's other warps, then (8 columns) to the near warps
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        Sw[(4 * half + kk) * SLD] = nerr[kk];
                        Sw[(32 + 4 * half + kk) * SLD] = pre[kk];
                    }
                    if (warp < 3) named_bar_arrive(QBAR_HAND + 2 * warp + half, 32 * (4 - warp));
                }
                *reinterpret_cast<float4 *>(wrow + co + w8) = make_float4(qv[0], qv[1], qv[2], qv[3]);
                *reinterpret_cast<float4 *>(wrow + co + w8 + 4) = make_float4(qv[4], qv[5], qv[6], qv[7]);
                named_bar_arrive(QBAR_CHUNK + warp, 32 + QB_NEAR);
                if (live && lane < ROWS) {
                    uint8_t *crow = a.codes + (int64_t)row * n;
                    const int cc = cg + w8;
                    if (!a.perm && cc + 7 < n && (reinterpret_cast<uintptr_t>(crow + cc) & 7) == 0) {
                        *reinterpret_cast<uint2 *>(crow + cc) = make_uint2(code[0], code[1]);
                    } else {
#pragma unroll
                        for (int kk = 0; kk < 8; ++kk)
                            if (cc + kk < n) crow[perm_s[co + w8 + kk]] = (uint8_t)(code[kk >> 2] >> (8 * (kk & 3)));
                    }
                }
            }
        }
    } else if (tid < QB_THREADS_NEAR) {
        // ================================================================ near
        const int t = tid - QB_CHAIN;
        const int ti = t & 7, tj = t >> 3;                          // rows ti, ti + 8, ..; columns 4 tj .. of the rest
        int seq = 0;                                                // steps so far
        float row_max = 0.f;                                        // largest magnitude of row t % ROWS's errors in this launch
        for (int b = 0; b < nblk; ++b) {
            const int nst = nsteps(b);
            for (int s = 0; s < nst; ++s) {
                const int co = b * QB_W + 32 * s;
                named_bar_sync(QBAR_NEAR, QB_NEAR);                 // all near warps are done with the other buffer of U / P
                const bool last = b == nblk - 1 && s == nst - 1;
                const int nb = s + 1 < nst ? b : b + 1, ns = s + 1 < nst ? s + 1 : 0;       // the next step
                const int ncol = i0 + nb * QB_W + 32 * ns;
                float next_sc[4], next_zp[4];
                if (!last) {
                    fetch_up(i0 + nb * QB_W, ns, t, QB_NEAR);
                    if (PERCOL && t < 8 * ROWS) load_grid(t >> 3, ncol + 4 * (t & 7), next_sc, next_zp);
                }
                if (a.clip_steps > 0 && grid_starts(i0 + co)) {
                    // clipping-range search: thread = (row, a share of the candidates)
                    named_bar_sync(QBAR_CLIP, QB_THREADS_NEAR);     // the group's values are current
                    const int r = t & (ROWS - 1), cgi = t / ROWS;
                    const float *w = Ws + r * WLD + co;
                    float lo = 0.f, hi = 0.f, best;
                    int kb;
                    float *scratch = Sts + (s & 1) * 64 * SLD;      // (the chain writes there only after this search)
#pragma unroll
                    for (int q = 0; q < 4; ++q) {                   // the range, a quarter from each chain warp
                        const float2 v = range_at(scratch)[q * ROWS + r];
                        lo = fminf(lo, v.x); hi = fmaxf(hi, v.y);
                    }
                    clip_search(w, a.group, lo, hi, a.bits, a.sym, a.clip_steps, a.clip_min, cgi, QB_NEAR / ROWS, best, kb);
                    float *be = scratch + 24 * SLD + 8 * ROWS;      // (behind the ranges, which other warps still read)
                    int *bk = reinterpret_cast<int *>(be + QB_NEAR);
                    be[t] = best; bk[t] = kb;
                    named_bar_sync(QBAR_NEAR, QB_NEAR);
                    if (t < ROWS) {
                        for (int g = 1; g < QB_NEAR / ROWS; ++g) {
                            const float e = be[g * ROWS + t];
                            const int k = bk[g * ROWS + t];
                            if (e < best || (e == best && k < kb)) { best = e; kb = k; }
                        }
                        reinterpret_cast<int *>(scratch)[t] = kb;
                    }
                    named_bar_sync(QBAR_CLIP, QB_THREADS_NEAR);
                    named_bar_sync(QBAR_CLIP, QB_THREADS_NEAR);
                }
                constexpr int ld = 32;
                const float *Ub = up_at(s, 0, 0, 32 + 4 * tj), *Pb = up_at(s, 1, 0, 32 + 4 * tj);     // (columns beyond the step's own 32)
                const float *St = Sts + (s & 1) * 64 * SLD;
                const bool active = 32 + 4 * tj < B - 32 * s;
                unsigned long long acc[RPT][2];
#pragma unroll
                for (int e = 0; e < RPT; ++e) { acc[e][0] = 0ull; acc[e][1] = 0ull; }
                for (int ph = 0; ph < 4; ++ph) {
                    named_bar_sync(QBAR_CHUNK + ph, 32 + QB_NEAR);
                    if (!active) continue;
#pragma unroll
                    for (int kk = 0; kk < 16; ++kk) {
                        const int k = 8 * ph + (kk & 7);
                        const float *ap = St + (k + (kk < 8 ? 0 : 32)) * SLD + RPT * ti;
                        float ae[4];
                        if (RPT == 4) {
                            const float4 av = *reinterpret_cast<const float4 *>(ap);
                            ae[0] = av.x; ae[1] = av.y; ae[2] = av.z; ae[3] = av.w;
                        } else {
                            const float2 av = *reinterpret_cast<const float2 *>(ap);
                            ae[0] = av.x; ae[1] = av.y;
                        }
                        const ulonglong2 bv = *reinterpret_cast<const ulonglong2 *>((kk < 8 ? Ub : Pb) + k * ld);
#pragma unroll
                        for (int e = 0; e < RPT; ++e) {
                            const unsigned long long aa = pack2(ae[e], ae[e]);
                            acc[e][0] = fma2(aa, bv.x, acc[e][0]);
                            acc[e][1] = fma2(aa, bv.y, acc[e][1]);
                        }
                    }
                }
                if (active) {
#pragma unroll
                    for (int e = 0; e < RPT; ++e) {
                        float4 *cp = reinterpret_cast<float4 *>(Ws + (ti + 8 * e) * WLD + co + 32 + 4 * tj);
                        float4 v = *cp;
                        v.x += lo2(acc[e][0]); v.y += hi2(acc[e][0]); v.z += lo2(acc[e][1]); v.w += hi2(acc[e][1]);
                        *cp = v;
                    }
                }
                // 64 columns done: a thread takes eight of them in one row (before the chain goes on and overwrites the first 32)
                const int er = t & (ROWS - 1), ec = t / ROWS;
                float ev[2][8], mx = 0.f;
                if (FAR && (s & 1) && ec < 8) {
                    const float *S2 = Sts + ((ec >> 2) * 64 + 8 * (ec & 3)) * SLD + qb_pos<ROWS>(er);
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        ev[0][e] = S2[e * SLD];
                        ev[1][e] = rho * S2[(32 + e) * SLD];
                        mx = fmaxf(mx, fmaxf(fabsf(ev[0][e]), fabsf(ev[1][e])));
                    }
                    rmax_s[ec * ROWS + er] = mx;
                }
                ++seq;
                // the chain waits for the next step's rows, or, at the end of a block, for what the operand brings to the next one
                const bool operand_first = FAR && s == QB_W / 32 - 1 && !last;
#pragma unroll 1
                for (int turn = 0; turn < 2; ++turn) {
                    if ((turn == 0) != operand_first) {
                        if (last) continue;
                        if (a.up_tma) mbar_wait(upfull(ns & 1), (uint32_t)(seq >> 1) & 1u, abort_flag);
                        else asm volatile("cp.async.wait_all;" ::: "memory");
                        if (PERCOL && t < 8 * ROWS) store_grid(t >> 3, 4 * (t & 7), next_sc, next_zp);      // (the chain has read this step's)
                        named_bar_arrive(QBAR_STEP, QB_THREADS_NEAR);
                        continue;
                    }
                    if (!FAR || !(s & 1)) continue;
                    // ... as the tensor cores' operand, with one power-of-two scale per row
                    named_bar_sync(QBAR_NEAR, QB_NEAR);
#pragma unroll
                    for (int e = 0; e < 8; ++e) mx = fmaxf(mx, rmax_s[e * ROWS + er]);
                    row_max = fmaxf(row_max, mx);
                    if (b >= last_groups || ec >= 8) continue;
                    const int half = s >> 1;                        // buffer: even and odd halves alternate
                    // (the drain warps are done with this buffer's row scales, the MMAs with its operands)
                    if (b > 0) mbar_wait(efree(half), (uint32_t)(b - 1) & 1u, abort_flag);
                    const float sc = split_scale_bits(__float_as_uint(mx));
                    if (ec == 0) inv_s[half * ROWS + er] = pow2_inverse(sc) * inv_su;
                    uint8_t *eb = sm + L.e + half * HALF_BYTES + (er >> 3) * 1024 + (er & 7) * 128 + ((ec ^ (er & 7)) << 4);
#pragma unroll
                    for (int o = 0; o < 2; ++o) {
                        const float y0[4] = {sc * ev[o][0], sc * ev[o][1], sc * ev[o][2], sc * ev[o][3]};
                        const float y1[4] = {sc * ev[o][4], sc * ev[o][5], sc * ev[o][6], sc * ev[o][7]};
                        uint2 h0, l0, h1, l1;
                        split16_pack(y0, h0, l0);
                        split16_pack(y1, h1, l1);
                        *reinterpret_cast<uint4 *>(eb + 2 * o * E_BYTES) = make_uint4(h0.x, h0.y, h1.x, h1.y);
                        *reinterpret_cast<uint4 *>(eb + (2 * o + 1) * E_BYTES) = make_uint4(l0.x, l0.y, l1.x, l1.y);
                    }
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(efull(half));
                }
                // results of the step: dequantized columns, -Err and Wpre (a thread: four columns of a row)
                {
                    const int r = t >> 3, c4 = 4 * (t & 7);
                    const int cw = co + c4;                         // column in the slab
                    const float4 v = r < ROWS ? *reinterpret_cast<const float4 *>(Ws + r * WLD + cw) : make_float4(0.f, 0.f, 0.f, 0.f);
                    const int left = cols - cw;                     // columns that exist from here on
                    if (r < nrows && left > 0) {                    // (r < ROWS, too)
                        float *dst = a.W + (int64_t)(row0 + r) * a.ldw + i0 + cw;
                        if (left >= 4 && (reinterpret_cast<uintptr_t>(dst) & 15) == 0) *reinterpret_cast<float4 *>(dst) = v;
                        else {
                            dst[0] = v.x;
                            if (left > 1) dst[1] = v.y;
                            if (left > 2) dst[2] = v.z;
                            if (left > 3) dst[3] = v.w;
                        }
                    }
                    // Non-finite values are reported from every column's value before its rounding (and its error: a range that
                    // overflows, a pivot of zero).  Codes and dequantized weights come out finite (the clamp absorbs NaN and
                    // Inf), so the results do not show them, and values checked when the slab is filled miss what a later
                    // column receives through U and P inside the launch.
                    auto magnitude = [](float v) { return __float_as_uint(v) & 0x7fffffffu; };
                    if (!a.EW) {
                        const int k = t >> 3;                       // column k, rows ti, ti + 8, ..
                        const float *ep = St + k * SLD + RPT * ti, *pp = ep + 32 * SLD;
#pragma unroll
                        for (int f = 0; f < RPT; ++f) {
                            const uint32_t big = max(magnitude(ep[f]), magnitude(pp[f]));
                            if (big >= 0x7f800000u && ti + 8 * f < nrows) record_status(a.hd, ST_NONFINITE, row0 + ti + 8 * f);
                        }
                    } else if (r < nrows) {
                        const int pos = qb_pos<ROWS>(r);
                        float e4[4], p4[4];
                        uint32_t big = 0u;
#pragma unroll
                        for (int f = 0; f < 4; ++f) {
                            e4[f] = St[(c4 + f) * SLD + pos];
                            const float p = St[(32 + c4 + f) * SLD + pos];
                            big = max(big, max(magnitude(e4[f]), magnitude(p)));
                            p4[f] = rho * p;
                        }
                        if (big >= 0x7f800000u) record_status(a.hd, ST_NONFINITE, row0 + r);
                        float *ew = a.EW + (int64_t)(row0 + r) * a.ew_ld + cw;
                        *reinterpret_cast<float4 *>(ew) = make_float4(e4[0], e4[1], e4[2], e4[3]);
                        *reinterpret_cast<float4 *>(ew + a.ew_pre) = make_float4(p4[0], p4[1], p4[2], p4[3]);
                    }
                }
            }
        }
        if (FAR && a.EWS_hi && t < ROWS) {
            const float sc = t < nrows ? split_scale_bits(__float_as_uint(row_max)) : 1.f;
            udinv_s[t] = sc;                                        // (free since the first step; read after the barrier below)
            if (t < nrows) a.row_inv[row0 + t] = pow2_inverse(sc);
        }
    } else if (FAR && tid < QB_THREADS_NEAR + QB_DRAIN) {
        // ================================================================ drain: tensor memory -> later blocks of the slab
        const int quarter = warp & 3;                               // TMEM lanes 32 * quarter ..: columns of the block
        const uint32_t tmem_base = *tmem_slot;
        for (int b = 0; b < last_groups; ++b)
            for (int half = 0; half < 2; ++half) {
                mbar_wait(efull(half), (uint32_t)b & 1u, abort_flag);           // the row scales
                for (int j = b + 1; j < nblk; ++j) {
                    const int slot = half * 3 + (j - 1);            // (used once per earlier block: b = 0 .. j - 1)
                    mbar_wait(tfull(slot), (uint32_t)b & 1u, abort_flag);
                    tc_fence_after();
                    uint32_t v[ROWS], l[ROWS];                      // hi hi; hi lo + lo hi
                    const uint32_t taddr = tmem_base + slot * 2 * ROWS + ((uint32_t)(quarter * 32) << 16);
                    if constexpr (ROWS == 32) { tmem_ld32(taddr, v); tmem_ld32(taddr + ROWS, l); }
                    else { tmem_ld16(taddr, v); tmem_ld16(taddr + ROWS, l); }
                    tmem_ld_wait();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(tempty(slot));
                    float *wp = Ws + j * QB_W + quarter * 32 + lane;
#pragma unroll
                    for (int r4 = 0; r4 < ROWS / 4; ++r4) {
                        const float4 iv = *reinterpret_cast<const float4 *>(inv_s + half * ROWS + 4 * r4);
                        float *w4 = wp + 4 * r4 * WLD;
                        w4[0] = fmaf(__uint_as_float(v[4 * r4]) + __uint_as_float(l[4 * r4]), iv.x, w4[0]);
                        w4[WLD] = fmaf(__uint_as_float(v[4 * r4 + 1]) + __uint_as_float(l[4 * r4 + 1]), iv.y, w4[WLD]);
                        w4[2 * WLD] = fmaf(__uint_as_float(v[4 * r4 + 2]) + __uint_as_float(l[4 * r4 + 2]), iv.z, w4[2 * WLD]);
                        w4[3 * WLD] = fmaf(__uint_as_float(v[4 * r4 + 3]) + __uint_as_float(l[4 * r4 + 3]), iv.w, w4[3 * WLD]);
                    }
                    if (half == 1 && j == b + 1) named_bar_arrive(QBAR_DRAIN, QB_CHAIN + QB_DRAIN);
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(efree(half));
            }
    } else if (FAR && warp == (QB_THREADS_NEAR + QB_DRAIN) / 32) {
        // ================================================================ load: tiles of U^T and P^T
        if (lane == 0) {
            uint32_t slot = 0, phase = 0;
            int issued = 0;
            bool ok = true;
            for (int b = 0; ok && b < last_groups; ++b)
                for (int half = 0; ok && half < 2; ++half)
                    for (int j = b + 1; ok && j < nblk; ++j)
                        for (int t4 = 0; t4 < 4; ++t4) {            // U hi, U lo, P hi, P lo
                            if (!mbar_wait(aempty(slot), phase ^ 1u, abort_flag)) { ok = false; break; }
                            const CUtensorMap *map = t4 == 0 ? &mapUhi : (t4 == 1 ? &mapUlo : (t4 == 2 ? &mapPhi : &mapPlo));
                            mbar_expect_tx(afull(slot), QB_A_BYTES);
                            tma_load_2d(base + L.a + slot * QB_A_BYTES, map, i0 + b * QB_W + 64 * half, i0 + j * QB_W, afull(slot));
                            ++issued;
                            if (++slot == ASLOTS) { slot = 0; phase ^= 1u; }
                        }
            if (!ok) {
                // give copies that are still in flight time to land before the CTA exits
                const long long t0 = clock64();
                while (issued > 0 && clock64() - t0 < 4000000LL) {}
            }
        }
    } else if (FAR) {
        // ================================================================ mma
        if (lane == 0) {
            uint32_t slot = 0, phase = 0;
            const uint32_t tmem_base = *tmem_slot;
            bool ok = true;
            for (int b = 0; ok && b < last_groups; ++b)
                for (int half = 0; ok && half < 2; ++half) {
                    if (!mbar_wait(efull(half), (uint32_t)b & 1u, abort_flag)) { ok = false; break; }
                    const uint32_t eb = base + L.e + half * HALF_BYTES;
                    for (int j = b + 1; ok && j < nblk; ++j) {
                        const int acc = half * 3 + (j - 1);
                        if (b > 0 && !mbar_wait(tempty(acc), (uint32_t)(b - 1) & 1u, abort_flag)) { ok = false; break; }
                        tc_fence_after();
                        const uint32_t d = tmem_base + acc * 2 * ROWS;
                        for (int t4 = 0; t4 < 4; ++t4) {
                            if (!mbar_wait(afull(slot), phase, abort_flag)) { ok = false; break; }
                            tc_fence_after();
                            const uint64_t ad = make_kmajor_desc(base + L.a + slot * QB_A_BYTES);
                            // [hi | lo] of the errors are the rows of one operand: a tile of hi takes both in one pass (an MMA of
                            // 128 rows takes 95 cycles with 16 columns and 115 with 64): 16 MMAs for 24 where the chain waits for
                            // a block, 2300 -> 1820 cycles
                            const uint64_t bd = make_kmajor_desc(eb + (t4 >> 1) * 2 * E_BYTES);
                            if (t4 & 1) {
#pragma unroll
                                for (int k = 0; k < 4; ++k) umma_f16(d + ROWS, ad + (uint64_t)(k * 2), bd + (uint64_t)(k * 2), qb_idesc(ROWS), 1u);
                            } else {
#pragma unroll
                                for (int k = 0; k < 4; ++k)
                                    umma_f16(d, ad + (uint64_t)(k * 2), bd + (uint64_t)(k * 2), qb_idesc(2 * ROWS), (t4 | k) ? 1u : 0u);
                            }
                            umma_commit(aempty(slot));
                            if (++slot == ASLOTS) { slot = 0; phase ^= 1u; }
                        }
                        if (ok) umma_commit(tfull(acc));
                    }
                }
        }
    }

    if (!FAR) {
        if (a.up_tma) {
            __syncthreads();
            if (*abort_flag && tid == 0) record_status(a.hd, ST_TIMEOUT, 3000000 + blockIdx.x);
        }
        return;
    }
    tc_fence_before();
    __syncthreads();
    if (a.EWS_hi) {
        // fp16 parts of [-Err | rho Wpre] for everything beyond this launch's columns (the rows were written by this
        // CTA; one scale per row over the whole launch)
        // (columns [0, QB_SUPER) and [ew_pre, ew_pre + QB_SUPER) of a row; five loads in flight per thread)
        constexpr int Q = 2 * QB_SUPER / 4, BATCH = 5;
        const float *src = a.EW + (int64_t)row0 * (2 * QB_SUPER);
        __half *hi = a.EWS_hi + (int64_t)row0 * (2 * QB_SUPER), *lo = a.EWS_lo + (int64_t)row0 * (2 * QB_SUPER);
        for (int i0q = tid; i0q < nrows * Q; i0q += BATCH * NTHREADS) {
            float4 v[BATCH];
#pragma unroll
            for (int e = 0; e < BATCH; ++e)
                if (i0q + e * NTHREADS < nrows * Q) v[e] = *reinterpret_cast<const float4 *>(src + 4 * (i0q + e * NTHREADS));
#pragma unroll
            for (int e = 0; e < BATCH; ++e) {
                const int idx = i0q + e * NTHREADS;
                if (idx >= nrows * Q) break;
                const float sc = udinv_s[idx / Q];
                const float x[4] = {sc * v[e].x, sc * v[e].y, sc * v[e].z, sc * v[e].w};
                uint2 h2, l2;
                split16_pack(x, h2, l2);
                *reinterpret_cast<uint2 *>(hi + 4 * idx) = h2;
                *reinterpret_cast<uint2 *>(lo + 4 * idx) = l2;
            }
        }
    }
    if (*abort_flag && tid == 0) record_status(a.hd, ST_TIMEOUT, 3000000 + blockIdx.x);
    if (warp == NTHREADS / 32 - 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(*tmem_slot), "r"((uint32_t)qb_tmem_cols(ROWS)) : "memory");
    }
}

}  // namespace gptaq
