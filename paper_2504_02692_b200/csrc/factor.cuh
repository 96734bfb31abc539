// The reverse Cholesky factorisation H_d = R R^T (R upper), panel by panel of NB columns from the right:
//
//   diag_factor_kernel   one CTA: the NB x NB diagonal block (and the inverses of its 32 x 32 diagonal sub-blocks);
//   panel_solve_kernel   the rows above: R[0:b0, blk] = A[0:b0, blk] R_pp^-T, in place and as split parts;
//   the rank-NB update of the columns to the left (tc_gemm_kernel, simt kernels).
//
// The chain diagonal -> solve -> update -> next diagonal bounds narrow and ordinary layers, and of it the diagonal block
// (128 dependent pivots).  Where the next block belongs to the same super-panel its diagonal kernel does not wait for the
// update: it takes a copy of the block from before the update and subtracts this panel's contribution itself (one
// 128 x 128 x 128 product on the tensor cores), so that the update runs beside it on another stream.  A panel of a
// 1024-wide layer took 33 us (every CTA of one kernel factored the diagonal block first) + 12 us for the update, now
// about 20 us (diagonal) + 7 us (rows above).  Factorisation with the inversion that follows it, before and after (the
// inversion beside the panels included): n = 1024 404 -> 287 us, n = 2052 1118 -> 726 us, n = 4096 2036 -> 1500 to 1700 us,
// n = 14336 19.8 -> 16.6 ms.
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
// The same recurrence with a = unit vector e_l gives column l of R^-1.  ready(k) is called before columns k .. k - 3 are
// read (k = 31, 27, ..).
template <typename Ready, typename Emit>
__device__ __forceinline__ void solve32(float (&a)[32], const float *Rt, const float *dinv, Ready ready, Emit emit) {
#pragma unroll 1
    for (int k0 = 24; k0 >= 0; k0 -= 8) {
        // a[24 + e] is entry k0 + e
#pragma unroll
        for (int e = 7; e >= 0; --e) {
            const int k = k0 + e;
            if (e == 7 || e == 3) ready(k);
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

// 32 x 32 reverse Cholesky of a symmetric block held one full row per lane; R^T to the lower part of Sd (pitch FP_LD).
// Four columns at a time are signalled to a second warp at named barriers bar0, bar0 + 1, ..  The chain from pivot to
// pivot is the reciprocal root (hardware estimate plus one Newton step, to about one ulp), the scaling of the column, and
// two shuffles: the next pivot, and the entry that the next column's own update needs.  The rest of a column's rank-1
// update waits until the next step's root is under way: the column goes to shared memory (cv: two buffers of 64 floats)
// and comes back as broadcast float4s one step later.
// A pivot that is not a positive normal number counts as 1 (the estimate is taken from the pivot as it comes, the test
// runs beside it); returns the first such column (-1: none).
__device__ __forceinline__ int chol32(float (&d)[32], int lane, float *Sd, float *dinv, float *cv, int bar0) {
    int bad_col = -1;
    float piv = __shfl_sync(0xffffffffu, d[31], 31), cprev = 0.f;
    cv[lane] = 0.f; cv[32 + lane] = 0.f; cv[64 + lane] = 0.f; cv[96 + lane] = 0.f;
    __syncwarp();
#pragma unroll 1
    for (int k0 = 24; k0 >= 0; k0 -= 8) {
        // d[24 + e] is column k0 + e
#pragma unroll
        for (int e = 7; e >= 0; --e) {
            const int K = k0 + e;
            float r;
            asm volatile("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(piv));
            {
                // column K + 1 applied to the columns below K (its update of column K came by shuffle); columns below 0 read
                // what lies ahead in the buffers and are never used
                const uint32_t buf = (uint32_t)__cvta_generic_to_shared(cv + 64 * ((e + 1) & 1) + 32 + k0 - 24);
#pragma unroll
                for (int j4 = 5 + (e + 3) / 4; j4 >= 0; --j4) {
                    float4 cj;
                    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(cj.x), "=f"(cj.y), "=f"(cj.z), "=f"(cj.w) : "r"(buf + 16 * j4));
                    if (4 * j4 + 3 < 24 + e) d[4 * j4 + 3] = fmaf(-cprev, cj.w, d[4 * j4 + 3]);
                    if (4 * j4 + 2 < 24 + e) d[4 * j4 + 2] = fmaf(-cprev, cj.z, d[4 * j4 + 2]);
                    if (4 * j4 + 1 < 24 + e) d[4 * j4 + 1] = fmaf(-cprev, cj.y, d[4 * j4 + 1]);
                    if (4 * j4 + 0 < 24 + e) d[4 * j4 + 0] = fmaf(-cprev, cj.x, d[4 * j4 + 0]);
                }
            }
            const bool bad = !(piv >= 1.17549435e-38f) || !(piv < INFINITY);
            r = r * fmaf(-0.5f * piv, r * r, 1.5f);
            bad_col = (bad && bad_col < 0) ? K : bad_col;
            piv = bad ? 1.f : piv;
            r = bad ? 1.f : r;
            const float c = lane < K ? d[24 + e] * r : 0.f;
            // the next column (23 + e) receives its share of this one at once
            const int nx = K > 0 ? K - 1 : 0;
            const float ck = __shfl_sync(0xffffffffu, c, nx);
            const float next = __shfl_sync(0xffffffffu, fmaf(-c, c, d[23 + e]), nx);
            asm volatile("st.shared.f32 [%0], %1;" ::"r"((uint32_t)__cvta_generic_to_shared(cv + 64 * (e & 1) + 32 + lane)), "f"(c) : "memory");
            __syncwarp();
            d[23 + e] = fmaf(-c, ck, d[23 + e]);
            const float rk = lane == K ? piv * r : c;
            if (lane <= K) Sd[K * FP_LD + lane] = rk;
            if (lane == K) dinv[K] = r;
            piv = next;
            cprev = c;
            if (e == 4) named_bar_arrive(bar0 + (24 - k0) / 4, 64);
            if (e == 0) named_bar_arrive(bar0 + (24 - k0) / 4 + 1, 64);
        }
        move_up8(d);
    }
    return bad_col;
}

// ---------------------------------------------------------------------------
// The NB x NB diagonal block [b0, b0 + NB): R_pp^T in the lower part of Rdiag (the rest of Rdiag is undefined) and the
// inverses of its four 32 x 32 diagonal sub-blocks in Y.  Rows / columns beyond n are padded with the identity.
// Warp 0 factors the 32 x 32 sub-blocks in registers (lane = row); warps 12 - 15 invert them, four columns behind; the
// rows above are a product with that inverse (warps 0, 1 the 32 rows right above, whose contribution they then take off
// the next sub-block; warps 4 - 11 the rows further up, then the rest of the rank-32 update while the next sub-block is
// being factored).  Warp 16 runs the tensor-core product.
// What bounds it: the pivot chain (about 150 cycles a column, 5k per sub-block) and the words that shared memory returns
// (solving the rows 2.2k, the next sub-block 3.5k cycles): solving by substitution, a row per lane, reads R once per row and
// took as long as the factorisation itself.  The helpers start when the chain's rows are solved: beside that solve their
// reads delay it (n = 2052 761 -> 755 us in all), kept back until the chain factors again they slow the pivots more (45k
// against 38k cycles).  Two columns per pivot step (two roots and one round of shuffles for both) took longer, 321 -> 328
// us at n = 1024: the chain is short of issue slots and shared memory by then, not of latency.
// ---------------------------------------------------------------------------
constexpr int DF_MAIN = 512, DF_THREADS = DF_MAIN + 32;
constexpr int DF_CHAIN = 128, DF_HELP = 8 * 32;
constexpr int DF_TILE_BYTES = NB * 64 * 2;           // 128 rows x 64 fp16
constexpr size_t DF_SMEM = 4 * DF_TILE_BYTES + (size_t)(NB * FP_LD + 2 * 32 * FP_YLD + NB + 128) * sizeof(float) + 64 + 1024;
constexpr uint32_t DF_IDESC = (1u << 4) | ((NB >> 3) << 17) | ((NB >> 4) << 24);     // kind::f16, M = N = 128

struct DiagFactorArgs {
    const float *src; long long lds;     // element (0, 0) of the block and its row pitch; entries j >= i are used
    int n, b0;
    float *Rdiag;                        // [NB][NB]
    float *Y;                            // [4][32][FP_YLD]: Y[c][l][j] = inv(R_cc)[j][l]
    int syrk, pan_col0;                  // 1: subtract rows b0 .. of the panel at columns pan_col0 .. of the split copy times
                                         //    their transpose first (scale of the copy: tc_amax[AMAX_PAN])
    StateHeader *hd;
};

__global__ void __launch_bounds__(DF_THREADS, 1)
diag_factor_kernel(const __grid_constant__ CUtensorMap mapHi, const __grid_constant__ CUtensorMap mapLo, DiagFactorArgs a) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t *sm = smem_raw + (base - raw);
    float (*S)[FP_LD] = reinterpret_cast<float (*)[FP_LD]>(sm + 4 * DF_TILE_BYTES);
    // [2][32][FP_YLD]: inverses of the sub-blocks, Yc[s & 1][l][j] = inv(R_ss)[j][l] (the helpers still read one while the
    // next is being made)
    float *Yc = reinterpret_cast<float *>(S + NB);
    float *dinv = Yc + 2 * 32 * FP_YLD;
    float *cv = dinv + NB;                           // 2 x (32 words of padding, 32)
    uint8_t *tailp = reinterpret_cast<uint8_t *>(cv + 128);
    const uint32_t bar = smem_u32(tailp), bar_mma = bar + 8;
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(tailp + 16);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tailp + 20);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nv = min(NB, a.n - a.b0);
    pdl_launch_dependents();
    if (tid == 0) {
        mbar_init(bar, 1);
        mbar_init(bar_mma, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (a.syrk && warp == 16) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(const_cast<uint32_t *>(tmem_slot))), "r"(128u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_wait();
    if (warp == 16) {
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
    } else
    // the block (all loads in flight before the first store)
    if (nv == NB && (a.lds & 3) == 0 && (reinterpret_cast<uintptr_t>(a.src) & 15) == 0) {
        float4 v[NB * NB / 4 / DF_MAIN];
#pragma unroll
        for (int it = 0; it < NB * NB / 4 / DF_MAIN; ++it) {
            const int idx = tid + it * DF_MAIN;
            v[it] = *reinterpret_cast<const float4 *>(a.src + (idx >> 5) * a.lds + 4 * (idx & 31));
        }
#pragma unroll
        for (int it = 0; it < NB * NB / 4 / DF_MAIN; ++it) {
            const int idx = tid + it * DF_MAIN;
            *reinterpret_cast<float4 *>(&S[idx >> 5][4 * (idx & 31)]) = v[it];
        }
    } else {
        for (int idx = tid; idx < NB * NB; idx += DF_MAIN) {
            const int i = idx >> 7, j = idx & 127;
            S[i][j] = (i < nv && j < nv && j >= i) ? a.src[i * a.lds + j] : (i == j ? 1.f : 0.f);
        }
    }
    __syncthreads();
    if (a.syrk) {
        const uint32_t tmem = *tmem_slot;
        // 16 warps, 32 x 32 each
        const int quarter = warp & 3, c0 = 32 * (warp >> 2), row = 32 * quarter + lane;
        const bool ok = warp < 16 && mbar_wait(bar_mma, 0u, abort_flag);
        __syncwarp();
        if (ok && c0 + 31 >= 32 * quarter) {
            tc_fence_after();
            uint32_t v[32];
            tmem_ld32(tmem + c0 + ((uint32_t)(quarter * 32) << 16), v);
            tmem_ld_wait();
            const float sc = split_scale(__uint_as_float(a.hd->tc_amax[AMAX_PAN]));
            const float inv = 1.f / (sc * sc);
#pragma unroll
            for (int c4 = 0; c4 < 8; ++c4) {
                float4 x = *reinterpret_cast<float4 *>(&S[row][c0 + 4 * c4]);
                x.x = fmaf(-inv, __uint_as_float(v[4 * c4]), x.x); x.y = fmaf(-inv, __uint_as_float(v[4 * c4 + 1]), x.y);
                x.z = fmaf(-inv, __uint_as_float(v[4 * c4 + 2]), x.z); x.w = fmaf(-inv, __uint_as_float(v[4 * c4 + 3]), x.w);
                *reinterpret_cast<float4 *>(&S[row][c0 + 4 * c4]) = x;
            }
        }
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        if (warp == 16)
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(128u) : "memory");
    }

    // X = S[rows, sub] inv(R_ss)^T, 4 x 4 outputs per thread; into the lower part (transposed: S[o + j][i])
    auto solve_rows = [&](int o, int i0, int u) {
        const int i = i0 + 4 * (u >> 3), j = 4 * (u & 7);
        const float *Ys = Yc + ((o >> 5) & 1) * 32 * FP_YLD;
        float acc[4][4];
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int f = 0; f < 4; ++f) acc[e][f] = 0.f;
#pragma unroll 2
        for (int l = 0; l < 32; l += 4) {
            float av[4][4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float4 q = *reinterpret_cast<const float4 *>(&S[i + e][o + l]);
                av[e][0] = q.x; av[e][1] = q.y; av[e][2] = q.z; av[e][3] = q.w;
            }
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                const float4 y = *reinterpret_cast<const float4 *>(Ys + (l + g) * FP_YLD + j);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    acc[0][e] = fmaf(av[e][g], y.x, acc[0][e]); acc[1][e] = fmaf(av[e][g], y.y, acc[1][e]);
                    acc[2][e] = fmaf(av[e][g], y.z, acc[2][e]); acc[3][e] = fmaf(av[e][g], y.w, acc[3][e]);
                }
            }
        }
#pragma unroll
        for (int f = 0; f < 4; ++f)
            *reinterpret_cast<float4 *>(&S[o + j + f][i]) = make_float4(acc[f][0], acc[f][1], acc[f][2], acc[f][3]);
    };
    // products of the solved rows: acc[e][f] = X[i + e] . X[j + f]
    auto rows_dot = [&](int o, int i, int j, float (&acc)[4][4]) {
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int f = 0; f < 4; ++f) acc[e][f] = 0.f;
#pragma unroll 4
        for (int k = 0; k < 32; ++k) {
            const float4 ri = *reinterpret_cast<const float4 *>(&S[o + k][i]);
            const float4 rj = *reinterpret_cast<const float4 *>(&S[o + k][j]);
            const float av[4] = {ri.x, ri.y, ri.z, ri.w}, bv[4] = {rj.x, rj.y, rj.z, rj.w};
#pragma unroll
            for (int e = 0; e < 4; ++e)
#pragma unroll
                for (int f = 0; f < 4; ++f) acc[e][f] = fmaf(av[e], bv[f], acc[e][f]);
        }
    };
    // Named barriers: 1 -- a sub-block is factored and inverted and the helpers' last update is done (warps 0 - 15); 2 -- the
    // rows right above are solved (chain warps arrive, helpers wait); 3 -- the same, among the chain warps; 4 .. 11 -- four
    // columns of the sub-block are ready for its inverter; 12 -- the rows further up are solved, among the helpers.
    if (tid < DF_CHAIN) {
        float d[32];
        if (warp == 0) {
#pragma unroll
            for (int j = 0; j < 32; ++j) d[j] = (j >= lane) ? S[96 + lane][96 + j] : S[96 + j][96 + lane];
        }
#pragma unroll 1
        for (int sb = 3; sb >= 0; --sb) {
            const int o = 32 * sb, o1 = o - 32;
            if (warp == 0) {
                const int bad_col = chol32(d, lane, &S[o][o], dinv + o, cv, 4);
                if (bad_col >= 0 && lane == 0) record_status(a.hd, ST_NOT_SPD, a.b0 + o + bad_col);
            }
            if (sb == 0) break;
            named_bar_sync(1, DF_MAIN);
            if (tid < 64) solve_rows(o, o1, tid);
            named_bar_arrive(2, DF_CHAIN + DF_HELP);
            named_bar_sync(3, DF_CHAIN);
            // the next sub-block, less their contribution: 2 x 4 outputs of the upper triangle per thread, mirrored (4 x 4 in
            // 36 threads: 1 % more in all)
            {
                const int i = o1 + 2 * (tid >> 3), j = o1 + 4 * (tid & 7);
                if (j + 3 >= i) {
                    float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll 8
                    for (int k = 0; k < 32; ++k) {
                        const float2 ri = *reinterpret_cast<const float2 *>(&S[o + k][i]);
                        const float4 rj = *reinterpret_cast<const float4 *>(&S[o + k][j]);
                        acc[0][0] = fmaf(ri.x, rj.x, acc[0][0]); acc[0][1] = fmaf(ri.x, rj.y, acc[0][1]);
                        acc[0][2] = fmaf(ri.x, rj.z, acc[0][2]); acc[0][3] = fmaf(ri.x, rj.w, acc[0][3]);
                        acc[1][0] = fmaf(ri.y, rj.x, acc[1][0]); acc[1][1] = fmaf(ri.y, rj.y, acc[1][1]);
                        acc[1][2] = fmaf(ri.y, rj.z, acc[1][2]); acc[1][3] = fmaf(ri.y, rj.w, acc[1][3]);
                    }
#pragma unroll
                    for (int e = 0; e < 2; ++e)
#pragma unroll
                        for (int f = 0; f < 4; ++f)
                            if (j + f >= i + e) {
                                const float v = S[i + e][j + f] - acc[e][f];
                                S[i + e][j + f] = v;
                                if (j + f > i + e) S[j + f][i + e] = v;
                            }
                }
            }
            named_bar_sync(3, DF_CHAIN);
            if (warp == 0) {
#pragma unroll
                for (int j4 = 0; j4 < 8; ++j4) {
                    const float4 q = *reinterpret_cast<const float4 *>(&S[o1 + lane][o1 + 4 * j4]);
                    d[4 * j4] = q.x; d[4 * j4 + 1] = q.y; d[4 * j4 + 2] = q.z; d[4 * j4 + 3] = q.w;
                }
            }
        }
    } else if (tid < DF_CHAIN + DF_HELP) {
        const int t = tid - DF_CHAIN;
#pragma unroll 1
        for (int sb = 3; sb >= 1; --sb) {
            const int o = 32 * sb;
            named_bar_sync(1, DF_MAIN);
            named_bar_sync(2, DF_CHAIN + DF_HELP);
            if (t < 2 * (o - 32)) solve_rows(o, 0, t);
            named_bar_sync(12, DF_HELP);
            // leading part: S[i][j] -= X[i] . X[j] for i <= j < o, the tiles of the upper triangle numbered row by row; the
            // last 32 x 32 sub-block is the chain's own
            const int q = o / 4, ntile = q * (q + 1) / 2 - 36;
            for (int u = t; u < ntile; u += DF_HELP) {
                int ti = 0, left = u;
                while (left >= q - ti) { left -= q - ti; ++ti; }
                const int i = 4 * ti, j = 4 * (ti + left);
                float acc[4][4];
                rows_dot(o, i, j, acc);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    float4 *cp = reinterpret_cast<float4 *>(&S[i + e][j]);
                    float4 v = *cp;
                    v.x -= acc[e][0]; v.y -= acc[e][1]; v.z -= acc[e][2]; v.w -= acc[e][3];
                    *cp = v;
                }
            }
        }
    } else if (warp < 16) {
        // warp 12 + c inverts sub-block c (lane = column)
        const int c = warp - 12, o = 32 * c;
#pragma unroll 1
        for (int sb = 3; sb >= 0; --sb) {
            if (sb == c) {
                float y[32];
#pragma unroll
                for (int k = 0; k < 32; ++k) y[k] = (k == lane) ? 1.f : 0.f;
                float *dst = a.Y + (c * 32 + lane) * FP_YLD;
                solve32(y, &S[o][o], dinv + o, [&](int k) { named_bar_sync(4 + (31 - k) / 4, 64); },
                        [&](int k, float v) { Yc[(c & 1) * 32 * FP_YLD + lane * FP_YLD + k] = v; dst[k] = v; });
            }
            if (sb > 0) named_bar_sync(1, DF_MAIN);
        }
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < NB * NB / 4 / DF_MAIN; ++it) {
        const int idx = tid + it * DF_MAIN;
        if (warp < 16) *reinterpret_cast<float4 *>(a.Rdiag + 4 * idx) = *reinterpret_cast<const float4 *>(&S[idx >> 5][4 * (idx & 31)]);
    }
    if (*abort_flag && tid == 0) record_status(a.hd, ST_TIMEOUT, 4000000 + a.b0);
}

// ---------------------------------------------------------------------------
// Rows above the block: R[0:b0, blk] = A[0:b0, blk] R_pp^-T, 32 columns at a time: a product with the inverse of the
// 32 x 32 diagonal sub-block, then a rank-32 update of the columns to the left.  In place and, if asked for, as split
// parts for the tensor-core rank update.
// A warp takes 4 (8) rows from end to end: lane = (one (two) rows, 4 columns of every 32), the rows live in registers, the 32
// values of a row that all its lanes need go through shared memory inside the warp, so that no barrier of the CTA is on
// the way (a CTA-wide form with two barriers per sub-block: n = 14336 17.3 against 15.9 ms in all).  What bounds it: the
// words of R that shared memory returns (8k cycles; fetching them 3k); with two rows per lane they serve twice as many
// products, with one a narrow panel has twice as many warps.
// One more CTA copies the block that is next on the diagonal, for the diag_factor_kernel that runs beside the update.
// ---------------------------------------------------------------------------
constexpr int PS_WORKERS = 4;                        // warps that take rows, at most
constexpr int PS_THREADS = 256;                      // all fetch R; the workers are the first warps
constexpr size_t PS_SMEM = (size_t)(NB * FP_LD + 4 * 32 * FP_YLD + PS_WORKERS * 8 * FP_YLD) * sizeof(float);

struct PanelSolveArgs {
    float *H; int n; int b0;
    const float *Rdiag, *Y;    // as diag_factor_kernel leaves them (R_pp^T in the lower part)
    __half *pan_hi, *pan_lo;   // nullptr, or fp16 parts of split_scale(tc_amax[AMAX_PAN]) * row: row pitch pan_ld, this panel
    int pan_ld, pan_col0;      //   at columns pan_col0 .. + NB (several panels side by side)
    int workers;               // warps of a CTA that take rows
    int early;                 // the panel is up to date before the diagonal block is: rows may be read before pdl_wait()
    float *next_diag;          // nullptr, or [NB][NB]: receives the block at b0 - NB (by the last CTA)
    StateHeader *hd;
};

template <int RPT>
__global__ void __launch_bounds__(PS_THREADS) panel_solve_kernel(PanelSolveArgs a) {
    constexpr int ROWS = 4 * RPT;                        // rows per warp
    extern __shared__ __align__(16) float smem_f[];
    float (*S)[FP_LD] = reinterpret_cast<float (*)[FP_LD]>(smem_f);                       // R^T, below the 32 x 32 diagonal sub-blocks
    float *Yt = reinterpret_cast<float *>(S + NB);                                        // [4][32][FP_YLD]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = a.workers;
    const int n = a.n, b0 = a.b0;
    const int nv = min(NB, n - b0);
    const bool vec = (n & 3) == 0 && (reinterpret_cast<uintptr_t>(a.H) & 15) == 0 && nv == NB;
    const int slabs = gridDim.x - (a.next_diag ? 1 : 0);
    const int ngroups = b0 / ROWS;
    const int q = lane & 7, rp = lane >> 3;              // 4 columns of every 32; row (pair of rows)
    float x[RPT][4][4];                                    // [row][sub-block][column]
    auto load_rows = [&](int g) {
#pragma unroll
        for (int e = 0; e < RPT; ++e) {
            const float *src = a.H + (int64_t)(g * ROWS + RPT * rp + e) * n + b0 + 4 * q;
#pragma unroll
            for (int sb = 0; sb < 4; ++sb) {
                if (vec) {
                    const float4 v = *reinterpret_cast<const float4 *>(src + 32 * sb);
                    x[e][sb][0] = v.x; x[e][sb][1] = v.y; x[e][sb][2] = v.z; x[e][sb][3] = v.w;
                } else {
#pragma unroll
                    for (int f = 0; f < 4; ++f) x[e][sb][f] = 32 * sb + 4 * q + f < nv ? src[32 * sb + f] : 0.f;
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
    for (int idx = tid; idx < 4 * 32 * FP_YLD / 4; idx += PS_THREADS) sg_copy16(Yt + 4 * idx, a.Y + 4 * idx);
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
                *reinterpret_cast<float4 *>(buf + e * FP_YLD + 4 * q) = make_float4(x[e][sb][0], x[e][sb][1], x[e][sb][2], x[e][sb][3]);
            __syncwarp();
            // X = (row) inv(R_ss)^T
            const float *Ys = Yt + sb * 32 * FP_YLD + 4 * q;
            float acc[RPT][4];
#pragma unroll
            for (int e = 0; e < RPT; ++e)
#pragma unroll
                for (int f = 0; f < 4; ++f) acc[e][f] = 0.f;
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
                    const float4 y = *reinterpret_cast<const float4 *>(Ys + (l + h) * FP_YLD);
#pragma unroll
                    for (int e = 0; e < RPT; ++e) {
                        acc[e][0] = fmaf(v[e][h], y.x, acc[e][0]); acc[e][1] = fmaf(v[e][h], y.y, acc[e][1]);
                        acc[e][2] = fmaf(v[e][h], y.z, acc[e][2]); acc[e][3] = fmaf(v[e][h], y.w, acc[e][3]);
                    }
                }
            }
#pragma unroll
            for (int e = 0; e < RPT; ++e)
#pragma unroll
                for (int f = 0; f < 4; ++f) x[e][sb][f] = acc[e][f];
            if (sb == 0) break;
            // columns to the left: x[s'] -= X[l] R[.][32 sb + l]
            __syncwarp();
#pragma unroll
            for (int e = 0; e < RPT; ++e)
                *reinterpret_cast<float4 *>(buf + e * FP_YLD + 4 * q) = make_float4(acc[e][0], acc[e][1], acc[e][2], acc[e][3]);
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
                        const float4 r = *reinterpret_cast<const float4 *>(&S[32 * sb + l + h][32 * t + 4 * q]);
#pragma unroll
                        for (int e = 0; e < RPT; ++e) {
                            x[e][t][0] = fmaf(-v[e][h], r.x, x[e][t][0]); x[e][t][1] = fmaf(-v[e][h], r.y, x[e][t][1]);
                            x[e][t][2] = fmaf(-v[e][h], r.z, x[e][t][2]); x[e][t][3] = fmaf(-v[e][h], r.w, x[e][t][3]);
                        }
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
                const int c = 32 * sb + 4 * q;
                const float (&v)[4] = x[e][sb];
                float *dst = a.H + row * n + b0 + c;
                if (vec) *reinterpret_cast<float4 *>(dst) = make_float4(v[0], v[1], v[2], v[3]);
                else {
#pragma unroll
                    for (int f = 0; f < 4; ++f) if (c + f < nv) dst[f] = v[f];
                }
                if (a.pan_hi) {
                    const float s4[4] = {sc * v[0], sc * v[1], sc * v[2], sc * v[3]};
                    uint2 hi, lo;
                    split16_pack(s4, hi, lo);
                    *reinterpret_cast<uint2 *>(a.pan_hi + row * a.pan_ld + a.pan_col0 + c) = hi;
                    *reinterpret_cast<uint2 *>(a.pan_lo + row * a.pan_ld + a.pan_col0 + c) = lo;
                }
            }
        }
    }
}

// ---------------------------------------------------------------------------
// Inverts NB x NB diagonal factors R_pp from block `first` on (one CTA each) and stores the inverse on the
// diagonal of H (strict lower part of the block zero): the starting point of U = R^-1.  Bound by shared-memory
// reads: 4 x 4 outputs per thread (one output per thread, and divisions in the substitution, took 36 us; now 11).
// 32 x 32 diagonal sub-blocks by back substitution (one warp each, lane = column), then
// X12 = -X11 (R12 X22) for 32 -> 64 -> 128.
// ---------------------------------------------------------------------------
constexpr int ID_THREADS = 256;
constexpr int ID_LD = FP_LD;
constexpr size_t ID_SMEM = (32 + 2 * NB * ID_LD + 64 * 68 + NB) * sizeof(float);

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

__global__ void __launch_bounds__(ID_THREADS, 1) invert_diag_blocks_kernel(float *H, int n, const float *Rdiag, int first) {
    extern __shared__ __align__(16) float smem_f[];
    float *S = smem_f + 32, *X = S + NB * ID_LD,      // (padding: solve32 reads ahead of its block)
          *T = X + NB * ID_LD, *dinv = T + 64 * 68;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b0 = (first + blockIdx.x) * NB;
    const float *src = Rdiag + (int64_t)(first + blockIdx.x) * NB * NB;
    float4 v[NB * NB / 4 / ID_THREADS];
#pragma unroll
    for (int it = 0; it < NB * NB / 4 / ID_THREADS; ++it) v[it] = *reinterpret_cast<const float4 *>(src + 4 * (tid + it * ID_THREADS));
    if (tid < NB) dinv[tid] = 1.f / src[tid * NB + tid];
#pragma unroll
    for (int it = 0; it < NB * NB / 4 / ID_THREADS; ++it) {
        const int i = (tid + it * ID_THREADS) >> 5, j4 = (tid + it * ID_THREADS) & 31;
        // R^T as it comes (the substitution below reads it by rows), and R above the diagonal
        if (4 * j4 <= i) *reinterpret_cast<float4 *>(S + i * ID_LD + 4 * j4) = v[it];
        *reinterpret_cast<float4 *>(X + i * ID_LD + 4 * j4) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
    for (int idx = tid; idx < NB * NB; idx += ID_THREADS) {
        const int i = idx >> 7, j = idx & 127;
        if (j < i) S[j * ID_LD + i] = S[i * ID_LD + j];
    }
    __syncthreads();
    if (warp < NB / 32) {
        const int o = 32 * warp;
        float x[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) x[i] = (i == lane) ? 1.f : 0.f;
        solve32(x, S + o * ID_LD + o, dinv + o, [](int) {}, [&](int k, float v) { X[(o + k) * ID_LD + o + lane] = v; });
    }
    __syncthreads();
    // X12 = -X11 (R12 X22), 32 -> 64 for both pairs, then 64 -> 128 (the triangular operands carry explicit zeros)
    const int pr = tid >> 6, o = 64 * pr;
    if (tid < 128) tile_product<32>(T + pr * 32 * 36, 36, S + o * ID_LD + o + 32, ID_LD, X + (o + 32) * ID_LD + o + 32, ID_LD, tid & 63, 1.f);
    __syncthreads();
    if (tid < 128) tile_product<32>(X + o * ID_LD + o + 32, ID_LD, X + o * ID_LD + o, ID_LD, T + pr * 32 * 36, 36, tid & 63, -1.f);
    __syncthreads();
    tile_product<64>(T, 68, S + 64, ID_LD, X + 64 * ID_LD + 64, ID_LD, tid, 1.f);
    __syncthreads();
    tile_product<64>(X + 64, ID_LD, X, ID_LD, T, 68, tid, -1.f);
    __syncthreads();
    const bool vec = (n & 3) == 0 && b0 + NB <= n;
    for (int it = 0; it < NB * NB / 4 / ID_THREADS; ++it) {
        const int i = (tid + it * ID_THREADS) >> 5, j = 4 * ((tid + it * ID_THREADS) & 31);
        float x[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) x[e] = j + e >= i ? X[i * ID_LD + j + e] : 0.f;
        float *dst = H + (int64_t)(b0 + i) * n + b0 + j;
        if (vec) *reinterpret_cast<float4 *>(dst) = make_float4(x[0], x[1], x[2], x[3]);
        else if (b0 + i < n) {
#pragma unroll
            for (int e = 0; e < 4; ++e) if (b0 + j + e < n) dst[e] = x[e];
        }
    }
}

}  // namespace gptaq
