// Generic fp32 tile GEMM on the plain FMA pipes.
//
// C(M x N) = alpha * A(M x K) * B(K x N) + beta * C, 128 x 128 x 16 tiles, 256
// threads, 8 x 8 outputs per thread, double-buffered shared memory.  Operands
// are described by strides so that one kernel serves every shape the solve
// needs: token-major Gram products (both operands K-slow), A * B^T panels,
// triangular products with per-tile K ranges, and the stacked [Err | Wpre] *
// [U ; P] trailing update.  It is the exact-fp32 reference path of the
// library: the tensor-core kernels replace it where a product is large, and it
// stays in use for ragged or small shapes.  Products of few tiles take
// simt_small_kernel below.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace gptaq {

// element (r, k) of an operand = p[r * rs + k * ks]   (r: row of A / column of B)
// k >= k_split reads p2[r * rs + (k - k_split) * ks] instead (stacked operand).
// If sub != nullptr the value is sub[...] - p[...] (same strides): used for X~ - X.
struct Operand {
    const float *p;
    int64_t rs, ks;
    const float *p2;
    int k_split;
    const float *sub;
};

enum GemmMode {
    GEMM_FULL = 0,
    GEMM_UPPER_TILES = 1,   // skip tiles that lie entirely below the diagonal
    GEMM_O = 2,             // C[i][a] = sum_{k >= a} ..., kept only for a > i (else 0); lower tiles skipped
    GEMM_P = 3,             // C[i][j] = sum_{i < k <= j} ..., strictly upper; lower tiles zero-filled
    GEMM_TRI_RIGHT = 4,     // B upper triangular: k <= j
    GEMM_TRI_LEFT = 5       // A upper triangular: k >= i
};

struct GemmProblem {
    Operand A, B;
    float *C;
    int64_t ldc;
    int M, N, K;
    float alpha, beta;
    int mode;
    // batching along blockIdx.z: every pointer advances by these element counts
    int64_t batchA, batchB, batchC;
    int batchM_last, batchN_last, batchK_last;  // dims of the last batch entry (ragged tail), 0 = same
    int nbatch;
    // `paired` (32 x 32 tiles only, nbatch 2): entry 1 is the product (pair_sub - A) B into pair_C with its own mode
    int paired, pair_mode;
    const float *pair_sub;
    float *pair_C;
    // columns below this one are written without what C holds (beta counts for the others); the 32 x 32 form with K in one piece
    // knows it alone, the launch refuses it elsewhere
    int fresh;
};

constexpr int GBM = 128, GBN = 128, GBK = 16, GPAD = 4;

template <bool RC>   // RC: rows contiguous (rs == 1), else K contiguous (ks == 1)
__device__ __forceinline__ void gemm_load(const Operand &op, int row0, int k0, int R, int K,
                                          int tid, float (&v)[8]) {
    if (RC) {
        // thread: 4 consecutive rows at k = tid/32 and tid/32 + 8
        int r = row0 + (tid & 31) * 4;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            int k = k0 + (tid >> 5) + h * 8;
            const float *base = op.p;
            int kk = k;
            if (op.p2 && k >= op.k_split) { base = op.p2; kk = k - op.k_split; }
            int64_t off = (int64_t)kk * op.ks + r;
            bool kin = k < K;
            if (kin && r + 3 < R && ((reinterpret_cast<uintptr_t>(base + off) & 15) == 0) &&
                (!op.sub || (reinterpret_cast<uintptr_t>(op.sub + off) & 15) == 0)) {
                float4 t = *reinterpret_cast<const float4 *>(base + off);
                if (op.sub) {
                    float4 s = *reinterpret_cast<const float4 *>(op.sub + off);
                    t.x = s.x - t.x; t.y = s.y - t.y; t.z = s.z - t.z; t.w = s.w - t.w;
                }
                v[h * 4 + 0] = t.x; v[h * 4 + 1] = t.y; v[h * 4 + 2] = t.z; v[h * 4 + 3] = t.w;
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    float t = 0.f;
                    if (kin && r + e < R) {
                        t = base[off + e];
                        if (op.sub) t = op.sub[off + e] - t;
                    }
                    v[h * 4 + e] = t;
                }
            }
        }
    } else {
        // thread: 4 consecutive k at row = tid/4 and tid/4 + 64
        int k = k0 + (tid & 3) * 4;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            int r = row0 + (tid >> 2) + h * 64;
            const float *base = op.p;
            int kk = k;
            if (op.p2 && k >= op.k_split) { base = op.p2; kk = k - op.k_split; }
            int64_t off = (int64_t)r * op.rs + kk;
            bool rin = r < R;
            if (rin && k + 3 < K && ((reinterpret_cast<uintptr_t>(base + off) & 15) == 0) &&
                (!op.sub || (reinterpret_cast<uintptr_t>(op.sub + off) & 15) == 0)) {
                float4 t = *reinterpret_cast<const float4 *>(base + off);
                if (op.sub) {
                    float4 s = *reinterpret_cast<const float4 *>(op.sub + off);
                    t.x = s.x - t.x; t.y = s.y - t.y; t.z = s.z - t.z; t.w = s.w - t.w;
                }
                v[h * 4 + 0] = t.x; v[h * 4 + 1] = t.y; v[h * 4 + 2] = t.z; v[h * 4 + 3] = t.w;
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    float t = 0.f;
                    if (rin && k + e < K) {
                        t = base[off + e];
                        if (op.sub) t = op.sub[off + e] - t;
                    }
                    v[h * 4 + e] = t;
                }
            }
        }
    }
}

template <bool RC>
__device__ __forceinline__ void gemm_store(float (*S)[GBM + GPAD], int tid, const float (&v)[8]) {
    if (RC) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            int k = (tid >> 5) + h * 8;
            *reinterpret_cast<float4 *>(&S[k][(tid & 31) * 4]) =
                make_float4(v[h * 4], v[h * 4 + 1], v[h * 4 + 2], v[h * 4 + 3]);
        }
    } else {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            int r = (tid >> 2) + h * 64;
#pragma unroll
            for (int e = 0; e < 4; ++e) S[(tid & 3) * 4 + e][r] = v[h * 4 + e];
        }
    }
}

template <bool A_RC, bool B_RC>
__global__ void __launch_bounds__(256) simt_gemm_kernel(GemmProblem pr) {
    __shared__ __align__(16) float As[2][GBK][GBM + GPAD];
    __shared__ __align__(16) float Bs[2][GBK][GBN + GPAD];

    const int z = blockIdx.z;
    int M = pr.M, N = pr.N, K = pr.K;
    if (z == pr.nbatch - 1) {
        if (pr.batchM_last) M = pr.batchM_last;
        if (pr.batchN_last) N = pr.batchN_last;
        if (pr.batchK_last) K = pr.batchK_last;
    }
    Operand A = pr.A, B = pr.B;
    A.p += z * pr.batchA; if (A.p2) A.p2 += z * pr.batchA; if (A.sub) A.sub += z * pr.batchA;
    B.p += z * pr.batchB; if (B.p2) B.p2 += z * pr.batchB; if (B.sub) B.sub += z * pr.batchB;
    float *C = pr.C + z * pr.batchC;

    const int i0 = blockIdx.y * GBM, j0 = blockIdx.x * GBN;
    if (i0 >= M || j0 >= N) return;
    const int tid = threadIdx.x;
    const int tx = tid & 15, ty = tid >> 4;
    const int mode = pr.mode;

    bool skip = false;
    int kb = 0, ke = K;
    if (mode == GEMM_UPPER_TILES) skip = i0 >= j0 + GBN;
    else if (mode == GEMM_O) { skip = i0 >= j0 + GBN; kb = j0; }
    else if (mode == GEMM_P) { skip = i0 >= j0 + GBN; kb = i0; ke = min(K, j0 + GBN); }
    else if (mode == GEMM_TRI_RIGHT) ke = min(K, j0 + GBN);
    else if (mode == GEMM_TRI_LEFT) kb = i0;

    float acc[8][8];
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 8; ++b) acc[a][b] = 0.f;

    if (!skip && kb < ke) {
        float va[8], vb[8];
        gemm_load<A_RC>(A, i0, kb, M, ke, tid, va);
        gemm_load<B_RC>(B, j0, kb, N, ke, tid, vb);
        gemm_store<A_RC>(As[0], tid, va);
        gemm_store<B_RC>(Bs[0], tid, vb);
        __syncthreads();
        int buf = 0;
        for (int k0 = kb; k0 < ke; k0 += GBK) {
            bool more = k0 + GBK < ke;
            if (more) {
                gemm_load<A_RC>(A, i0, k0 + GBK, M, ke, tid, va);
                gemm_load<B_RC>(B, j0, k0 + GBK, N, ke, tid, vb);
            }
#pragma unroll
            for (int k = 0; k < GBK; ++k) {
                float4 a0 = *reinterpret_cast<const float4 *>(&As[buf][k][ty * 4]);
                float4 a1 = *reinterpret_cast<const float4 *>(&As[buf][k][64 + ty * 4]);
                float4 b0 = *reinterpret_cast<const float4 *>(&Bs[buf][k][tx * 4]);
                float4 b1 = *reinterpret_cast<const float4 *>(&Bs[buf][k][64 + tx * 4]);
                float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
                float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
                for (int x = 0; x < 8; ++x)
#pragma unroll
                    for (int y = 0; y < 8; ++y) acc[x][y] = fmaf(a[x], b[y], acc[x][y]);
            }
            if (more) {
                gemm_store<A_RC>(As[buf ^ 1], tid, va);
                gemm_store<B_RC>(Bs[buf ^ 1], tid, vb);
                __syncthreads();
                buf ^= 1;
            }
        }
    } else if (skip && mode != GEMM_P) {
        return;
    }

    const float alpha = pr.alpha, beta = pr.beta;
#pragma unroll
    for (int x = 0; x < 8; ++x) {
        int i = i0 + (x < 4 ? ty * 4 + x : 64 + ty * 4 + (x - 4));
        if (i >= M) continue;
#pragma unroll
        for (int yh = 0; yh < 2; ++yh) {
            int j = j0 + yh * 64 + tx * 4;
            float *cp = C + (int64_t)i * pr.ldc + j;
            float o[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                float val = alpha * acc[x][yh * 4 + e];
                if ((mode == GEMM_O || mode == GEMM_P) && (j + e) <= i) val = 0.f;
                o[e] = val;
            }
            bool masked = (mode == GEMM_O || mode == GEMM_P);
            if (j + 3 < N && ((reinterpret_cast<uintptr_t>(cp) & 15) == 0)) {
                float4 t = make_float4(o[0], o[1], o[2], o[3]);
                if (beta != 0.f && !masked) {
                    float4 c = *reinterpret_cast<const float4 *>(cp);
                    t.x += beta * c.x; t.y += beta * c.y; t.z += beta * c.z; t.w += beta * c.w;
                }
                *reinterpret_cast<float4 *>(cp) = t;
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (j + e < N) cp[e] = o[e] + ((beta != 0.f && !masked) ? beta * cp[e] : 0.f);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// The same products where 128 x 128 tiles are few: 32 x 32 tiles, 64 threads, 4 x 4 outputs per thread, operands
// through three 32-deep stages of asynchronous copies; the K range of a tile may be shared by a cluster of CTAs,
// whose partial sums meet in distributed shared memory in a fixed order (deterministic, no scratch).
// What bounds it: shared-memory reads (two 16-byte reads per 16 FMA: about half the FMA rate of the 128 x 128
// form), so it pays while those tiles leave the chip idle (simt_small_limit).  A rank-128 update of 384 columns: 30 us as 128 x 128
// tiles, 9 here; the statistics of 8192 tokens at n = 200: 2700 us there, 150 here.
// The 32 terms of a stage are summed by themselves: P of a float32 layer is 30 to 45 % closer to float64 so (n = 100 to 384), for 17
// to 32 registers more (128 at most, still eight CTAs to an SM; 4 bytes spilled where both operands have K contiguous) and up to 3 % of
// the time (gptaq_build_P at n = 256 26.8 -> 27.7 us, 777 94.2 -> 93.4).
// ---------------------------------------------------------------------------
constexpr int SGT = 32, SGK = 32, SG_LD = SGK + 4, SG_STAGES = 3, SG_THREADS = 64;
constexpr int SG_TILE = SGT * SG_LD;                  // floats of one operand tile

__device__ __forceinline__ void sg_copy16(float *dst, const float *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void sg_copy4(float *dst, const float *src, bool valid) {
    // (a source size of 0 writes a zero and reads nothing)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(valid ? 4 : 0) : "memory");
}

// Operand rows row0 .. + 31, contraction steps k0 .. + 31 into a tile.  RC: tile[k][row], else tile[row][k].
template <bool RC>
__device__ __forceinline__ void sg_fetch(float *tile, const float *p, const float *p2, int k_split, int64_t rs, int64_t ks,
                                         int row0, int R, int k0, int ke, int tid) {
    const bool second = p2 != nullptr && k0 >= k_split;               // (k_split is a multiple of 32)
    const float *base = second ? p2 : p;
    const int kk0 = second ? k0 - k_split : k0;
#pragma unroll
    for (int it = 0; it < SGT * SGK / 4 / SG_THREADS; ++it) {
        const int idx = tid + it * SG_THREADS, o = idx >> 3, c4 = (idx & 7) * 4;
        float *dst = tile + o * SG_LD + c4;
        const int row = RC ? row0 + c4 : row0 + o, k = RC ? o : c4;   // k: within the tile
        const float *src = base + (RC ? (int64_t)(kk0 + k) * ks + row : (int64_t)row * rs + kk0 + k);
        const int left = RC ? (k0 + k < ke ? R - row : 0) : (row < R ? ke - k0 - k : 0);      // valid elements of the four
        if (left >= 4 && (reinterpret_cast<uintptr_t>(src) & 15) == 0) sg_copy16(dst, src);
        else {
#pragma unroll
            for (int e = 0; e < 4; ++e) sg_copy4(dst + e, e < left ? src + e : base, e < left);
        }
    }
}

template <bool A_RC, bool B_RC>
__global__ void __launch_bounds__(SG_THREADS) simt_small_kernel(GemmProblem pr, int ksplit) {
    extern __shared__ __align__(16) float sg_smem[];
    const int tid = threadIdx.x;
    pdl_launch_dependents();
    pdl_wait();                                                       // (nothing before it: products may follow each other closely)
    const int z = blockIdx.z / ksplit, part = blockIdx.z - z * ksplit;
    int M = pr.M, N = pr.N, K = pr.K;
    if (z == pr.nbatch - 1) {
        if (pr.batchM_last) M = pr.batchM_last;
        if (pr.batchN_last) N = pr.batchN_last;
        if (pr.batchK_last) K = pr.batchK_last;
    }
    const int i0 = blockIdx.y * SGT, j0 = blockIdx.x * SGT;
    if (i0 >= M || j0 >= N) return;                                   // (the same for the CTAs of a cluster)
    const bool pair1 = pr.paired && z == 1;
    const int mode = pair1 ? pr.pair_mode : pr.mode;
    bool skip = false;
    int kb = 0, ke = K;
    if (mode == GEMM_UPPER_TILES) skip = i0 >= j0 + SGT;
    else if (mode == GEMM_O) { skip = i0 >= j0 + SGT; kb = j0; }
    else if (mode == GEMM_P) { skip = i0 >= j0 + SGT; kb = i0; ke = min(K, j0 + SGT); }
    else if (mode == GEMM_TRI_RIGHT) ke = min(K, j0 + SGT);
    else if (mode == GEMM_TRI_LEFT) kb = i0;
    if (skip && mode != GEMM_P) return;
    if (skip) ke = kb;
    if (ksplit > 1) {
        const int steps = max(0, (ke - kb + SGK - 1) / SGK);
        const int b = kb + steps * part / ksplit * SGK, e = kb + steps * (part + 1) / ksplit * SGK;
        kb = b; ke = min(ke, e);
    }

    const float *A = pr.A.p + z * pr.batchA, *B = pr.B.p + z * pr.batchB;
    const float *A2 = pr.A.p2 ? pr.A.p2 + z * pr.batchA : nullptr, *B2 = pr.B.p2 ? pr.B.p2 + z * pr.batchB : nullptr;
    const float *Asub = pair1 ? pr.pair_sub : (pr.A.sub ? pr.A.sub + z * pr.batchA : nullptr);
    const int stage_floats = (Asub ? 3 : 2) * SG_TILE;
    const int nk = max(0, (ke - kb + SGK - 1) / SGK);
    auto fetch = [&](int t) {
        if (t < nk) {
            float *st = sg_smem + (t % SG_STAGES) * stage_floats;
            const int k0 = kb + t * SGK;
            sg_fetch<A_RC>(st, A, A2, pr.A.k_split, pr.A.rs, pr.A.ks, i0, M, k0, ke, tid);
            sg_fetch<B_RC>(st + SG_TILE, B, B2, pr.B.k_split, pr.B.rs, pr.B.ks, j0, N, k0, ke, tid);
            if (Asub) sg_fetch<A_RC>(st + 2 * SG_TILE, Asub, nullptr, 0, pr.A.rs, pr.A.ks, i0, M, k0, ke, tid);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    const int tj = tid & 7, ti = tid >> 3;
    float acc[4][4];
#pragma unroll
    for (int e = 0; e < 4; ++e)
#pragma unroll
        for (int f = 0; f < 4; ++f) acc[e][f] = 0.f;
    // rows 4 ti + e (tile[k][row]) or ti + 8 e (tile[row][k]), columns likewise
    auto read4 = [&](const float *tile, bool rc, int t, int k, float (&v)[4][4]) {          // v[k][e]
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float4 x = *reinterpret_cast<const float4 *>(rc ? tile + (k + q) * SG_LD + 4 * t : tile + (t + 8 * q) * SG_LD + k);
            const float xx[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) { if (rc) v[q][e] = xx[e]; else v[e][q] = xx[e]; }
        }
    };
#pragma unroll
    for (int t = 0; t < SG_STAGES - 1; ++t) fetch(t);
    // what C holds arrives under the products (read at the end, each value would wait for its own round trip)
    float *C = pair1 ? pr.pair_C : pr.C + z * pr.batchC;
    const bool masked = mode == GEMM_O || mode == GEMM_P;
    const bool add_c = pr.beta != 0.f && !masked;
    float cv[4][4];
#pragma unroll
    for (int e = 0; e < 4; ++e)
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            const int i = i0 + (A_RC ? 4 * ti + e : ti + 8 * e), j = j0 + (B_RC ? 4 * tj + f : tj + 8 * f);
            cv[e][f] = (add_c && ksplit == 1 && i < M && j < N && j >= pr.fresh) ? C[(int64_t)i * pr.ldc + j] : 0.f;
        }
    for (int t = 0; t < nk; ++t) {
        asm volatile("cp.async.wait_group %0;" ::"n"(SG_STAGES - 2) : "memory");
        __syncthreads();
        fetch(t + SG_STAGES - 1);                                     // into the stage that was read last step
        const float *st = sg_smem + (t % SG_STAGES) * stage_floats;
        float sum[4][4];                                              // (a stage's 32 terms by themselves: shorter chains of roundings)
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int f = 0; f < 4; ++f) sum[e][f] = 0.f;
#pragma unroll 2
        for (int k = 0; k < SGK; k += 4) {
            float av[4][4], bv[4][4];
            read4(st, A_RC, ti, k, av);
            read4(st + SG_TILE, B_RC, tj, k, bv);
            if (Asub) {
                float sv[4][4];
                read4(st + 2 * SG_TILE, A_RC, ti, k, sv);
#pragma unroll
                for (int q = 0; q < 4; ++q)
#pragma unroll
                    for (int e = 0; e < 4; ++e) av[q][e] = sv[q][e] - av[q][e];
            }
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int e = 0; e < 4; ++e)
#pragma unroll
                    for (int f = 0; f < 4; ++f) sum[e][f] = fmaf(av[q][e], bv[q][f], sum[e][f]);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int f = 0; f < 4; ++f) acc[e][f] += sum[e][f];
    }
    asm volatile("cp.async.wait_all;" ::: "memory");

    auto store = [&](int i, int j, float v, float c) {
        if (i >= M || j >= N) return;
        v *= pr.alpha;
        if (masked && j <= i) v = 0.f;
        C[(int64_t)i * pr.ldc + j] = add_c ? fmaf(pr.beta, c, v) : v;
    };
    if (ksplit == 1) {
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int f = 0; f < 4; ++f)
                store(i0 + (A_RC ? 4 * ti + e : ti + 8 * e), j0 + (B_RC ? 4 * tj + f : tj + 8 * f), acc[e][f], cv[e][f]);
        return;
    }
    // partial sums meet: every CTA of the cluster adds up its share of the rows, in the order of the parts
    __syncthreads();
#pragma unroll
    for (int e = 0; e < 4; ++e)
#pragma unroll
        for (int f = 0; f < 4; ++f)
            sg_smem[(A_RC ? 4 * ti + e : ti + 8 * e) * SG_LD + (B_RC ? 4 * tj + f : tj + 8 * f)] = acc[e][f];
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    const int rows = SGT / ksplit;
    float own[SGT * SGT / 2 / SG_THREADS];               // (at least two parts)
#pragma unroll
    for (int q = 0; q < SGT * SGT / 2 / SG_THREADS; ++q) {
        const int idx = tid + q * SG_THREADS, i = i0 + part * rows + (idx >> 5), j = j0 + (idx & 31);
        own[q] = (add_c && idx < rows * SGT && i < M && j < N) ? C[(int64_t)i * pr.ldc + j] : 0.f;
    }
#pragma unroll
    for (int q = 0; q < SGT * SGT / 2 / SG_THREADS; ++q) {
        const int idx = tid + q * SG_THREADS;
        if (idx >= rows * SGT) break;
        const int i = part * rows + (idx >> 5), j = idx & 31;
        const uint32_t addr = (uint32_t)__cvta_generic_to_shared(sg_smem + i * SG_LD + j);
        float v = 0.f;
        for (int c = 0; c < ksplit; ++c) {
            uint32_t remote;
            float x;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(addr), "r"(c));
            asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(x) : "r"(remote) : "memory");
            v += x;
        }
        store(i0 + i, j0 + j, v, own[q]);
    }
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// 128 x 128 tiles of a product (all batch entries; the skipped ones of a triangular mode count, a factor of two at most)
inline int64_t simt_tiles(const GemmProblem &pr) {
    return (int64_t)pr.nbatch * ((pr.M + GBM - 1) / GBM) * ((pr.N + GBN - 1) / GBN);
}
// Two sums in one launch (the statistics of narrow layers): up to here.
constexpr int64_t SIMT_SMALL_TILES = 60;

// Rows of 16-byte multiples, so that the loads of the 128 x 128 form are float4?
inline bool simt_aligned(const Operand &o) {
    return ((o.rs == 1 ? o.ks : o.rs) & 3) == 0 &&
           ((reinterpret_cast<uintptr_t>(o.p) | reinterpret_cast<uintptr_t>(o.p2) | reinterpret_cast<uintptr_t>(o.sub)) & 15) == 0;
}
// 128 x 128 tiles up to which the 32 x 32 form is the faster one.  What it loses in reads of shared memory it gains in a chip that is
// full and in shorter last tiles of triangular products, whose K range the 128 x 128 form goes through on one SM; and its copies do
// not care for alignment, where the other form loads word by word into registers.  us a call, 128 x 128 beyond 60 tiles and by these limits:
//   unaligned  n = 1027 factor 707 / 434, P 620 / 132; 2049 2263 / 1116, 1308 / 384; 4097 (1089 tiles) 6287 / 3974, 3275 / 2270;
//              2500 tiles are 5 % slower (trailing updates of 16000 x 2597)
//   aligned    factor without damping n = 2052 1466 / 954, P 720 / 300, factor 4096 3204 / 2814 (up to 600 tiles 2876);
//              trailing updates of 1024 to 4096 x 1024 240 / 240, 303 / 277, 359 / 324, 488 / 451 (up to 300 tiles 462)
//   token sums 4096 tokens of n = 1024 605 / 431, 2832 of 1416 937 / 1018 with more than 100
inline int64_t simt_small_limit(const GemmProblem &pr, bool a_rc, bool b_rc) {
    if (!simt_aligned(pr.A) || !simt_aligned(pr.B)) return 1200;
    if (a_rc && b_rc) return 100;
    return pr.mode == GEMM_FULL ? 200 : 300;
}

template <bool A_RC, bool B_RC>
inline cudaError_t launch_simt_small(const GemmProblem &pr, cudaStream_t s, int early_ctas) {
    dim3 grid((pr.N + SGT - 1) / SGT, (pr.M + SGT - 1) / SGT, pr.nbatch);
    // long contractions of few tiles (the statistics of narrow layers) are shared by up to eight CTAs per tile
    int ksplit = 1;
    const int64_t tiles = (int64_t)grid.x * grid.y * grid.z;
    while (ksplit < 8 && tiles * ksplit <= 592 && pr.K / (2 * ksplit) >= 128) ksplit *= 2;      // 592: four CTAs per SM
    if (pr.fresh > 0 && ksplit > 1) return cudaErrorInvalidValue;
    grid.z *= ksplit;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = dim3(SG_THREADS); cfg.stream = s;
    cfg.dynamicSmemBytes = (size_t)SG_STAGES * (pr.A.sub || pr.paired ? 3 : 2) * SG_TILE * sizeof(float);
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = tiles * ksplit <= early_ctas ? 1 : 0;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 1; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = (unsigned)ksplit;
    cfg.attrs = attr; cfg.numAttrs = ksplit > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, simt_small_kernel<A_RC, B_RC>, pr, ksplit);
}

// early_ctas: the 32 x 32 form starts while the kernel before it drains where it has at most so many CTAs.  Those that are there
// before their turn hold the SMs that were free at that time, several to an SM, and it is there that the product runs.
inline cudaError_t launch_simt_gemm(const GemmProblem &pr, bool a_rc, bool b_rc, cudaStream_t s, int early_ctas = 0) {
    if (pr.M <= 0 || pr.N <= 0 || pr.nbatch <= 0) return cudaSuccess;
    if (simt_tiles(pr) <= simt_small_limit(pr, a_rc, b_rc) && !pr.B.sub) {
        if (a_rc && b_rc) return launch_simt_small<true, true>(pr, s, early_ctas);
        if (a_rc) return launch_simt_small<true, false>(pr, s, early_ctas);
        if (b_rc) return launch_simt_small<false, true>(pr, s, early_ctas);
        return launch_simt_small<false, false>(pr, s, early_ctas);
    }
    if (pr.fresh > 0) return cudaErrorInvalidValue;
    dim3 grid((pr.N + GBN - 1) / GBN, (pr.M + GBM - 1) / GBM, pr.nbatch);
    if (a_rc && b_rc) simt_gemm_kernel<true, true><<<grid, 256, 0, s>>>(pr);
    else if (a_rc && !b_rc) simt_gemm_kernel<true, false><<<grid, 256, 0, s>>>(pr);
    else if (!a_rc && b_rc) simt_gemm_kernel<false, true><<<grid, 256, 0, s>>>(pr);
    else simt_gemm_kernel<false, false><<<grid, 256, 0, s>>>(pr);
    return cudaGetLastError();
}

inline Operand make_operand(const float *p, int64_t rs, int64_t ks) {
    Operand o; o.p = p; o.rs = rs; o.ks = ks; o.p2 = nullptr; o.k_split = 0; o.sub = nullptr; return o;
}

inline GemmProblem make_problem(Operand A, Operand B, float *C, int64_t ldc, int M, int N, int K,
                                float alpha, float beta, int mode) {
    GemmProblem p; p.A = A; p.B = B; p.C = C; p.ldc = ldc; p.M = M; p.N = N; p.K = K;
    p.alpha = alpha; p.beta = beta; p.mode = mode; p.batchA = p.batchB = p.batchC = 0;
    p.batchM_last = p.batchN_last = p.batchK_last = 0; p.nbatch = 1;
    p.paired = p.pair_mode = 0; p.pair_sub = nullptr; p.pair_C = nullptr; p.fresh = 0; return p;
}

}  // namespace gptaq
