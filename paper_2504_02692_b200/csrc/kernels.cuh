// Small kernels of the GPTAQ layer solve: damping, grids, the column loop for groups of fewer than 32 columns, the row-by-row
// form of P, column orders and copies.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace gptaq {

// Device-resident header at the start of the caller's state buffer.
struct StateHeader {
    int status;          // first device-side condition (gptaq_status_t), 0 = none
    int pad0;
    long long info;      // index that goes with it
    float lambda;        // damp * mean(diag H / tokens)
    float inv_tokens;
    unsigned amax[2][2]; // per operand buffer: bit patterns of max|X| and max|X~ - X| of the batch converted into it
    unsigned tc_amax[8]; // largest magnitudes of FP16-split operands of the float32-grade GEMMs (see tc_gemm.cuh)
    unsigned sched_counter; // tile numbers drawn by the float32-grade GEMM launch that is running (0 between launches)
    unsigned stats_done;    // CTAs of the running statistics product that have finished
    unsigned sched_counter2; // as sched_counter, for launches that run beside those on the internal stream
    int pad1[11];
};
static_assert(sizeof(StateHeader) == 128, "header size");

constexpr int ST_NOT_SPD = 4, ST_NONFINITE = 5, ST_TIMEOUT = 6;

// Slots of StateHeader::tc_amax: factor panels (an a-priori bound), U, P, the blocks of the inverse factor while it is
// built (an a-priori bound), the intermediate product of one doubling level.
enum { AMAX_PAN = 0, AMAX_U = 1, AMAX_P = 2, AMAX_INV = 3, AMAX_T = 4 };

// Scale of an FP16-split operand: a power of two that puts the largest magnitude into [2^13, 2^14) (2^114 at most: it and
// its reciprocal are normal numbers).
__host__ __device__ __forceinline__ float split_scale(float amax) {
    if (!(amax > 0.f) || !isfinite(amax)) return 1.f;
    int e;
    frexpf(amax, &e);                 // amax = f * 2^e, f in [0.5, 1)
    return ldexpf(1.f, 14 - (e < -100 ? -100 : e));
}
// The same from the bit pattern, for threads that need several (in the factorisation's kernels, which need one, the code
// around it came out slower: n = 4096 1393 -> 1413 us).
__device__ __forceinline__ float split_scale_bits(unsigned amax) {
    if (amax == 0u || amax >= 0x7f800000u) return 1.f;
    return __uint_as_float(min(267u - (amax >> 23), 241u) << 23);       // biased exponents: 127 + 14 - (e - 126)
}

// 1 / s for a power of two s whose reciprocal is normal, too.
__device__ __forceinline__ float pow2_inverse(float s) { return __uint_as_float(0x7f000000u - __float_as_uint(s)); }

// Programmatic dependent launch: a kernel launched with the stream-serialization attribute may be
// scheduled while its predecessor in the stream drains; pdl_wait() returns once the predecessor has
// completed and its writes are visible (a no-op for a plain launch), pdl_launch_dependents() lets the
// successor be scheduled from here on.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ void record_status(StateHeader *hd, int code, long long info) {
    if (atomicCAS(&hd->status, 0, code) == 0) hd->info = info;
}

// ---------------------------------------------------------------------------
// lambda = damp * mean_q(H_qq / tokens, dead -> 1); dead flags.  One CTA, fixed
// reduction order (deterministic).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(1024) diag_stats_kernel(const float *H, int n, float inv_tokens,
                                                          float damp, StateHeader *hd,
                                                          uint8_t *dead, uint8_t *dead_working) {
    __shared__ double red[1024];
    __shared__ float redmax[1024];
    pdl_launch_dependents();
    double s = 0.0;
    float mx = 0.f;
    for (int q = threadIdx.x; q < n; q += 1024) {
        float d = H[(int64_t)q * n + q];
        if (!isfinite(d)) record_status(hd, ST_NONFINITE, q);
        bool dd = (d == 0.f);
        dead[q] = dd ? 1 : 0;
        if (dead_working) dead_working[q] = dd ? 1 : 0;
        const float v = dd ? 1.f : d * inv_tokens;
        s += dd ? 1.0 : (double)d * (double)inv_tokens;
        mx = fmaxf(mx, v);
    }
    red[threadIdx.x] = s;
    redmax[threadIdx.x] = mx;
    __syncthreads();
    for (int w = 512; w > 0; w >>= 1) {
        if (threadIdx.x < w) {
            red[threadIdx.x] += red[threadIdx.x + w];
            redmax[threadIdx.x] = fmaxf(redmax[threadIdx.x], redmax[threadIdx.x + w]);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const float lambda = (float)((double)damp * red[0] / (double)n);
        hd->lambda = lambda;
        hd->inv_tokens = inv_tokens;
        // every entry of row i of the factor R (H_d = R R^T) is at most sqrt(H_d,ii): the range of the
        // factor panels is known before they exist
        hd->tc_amax[AMAX_PAN] = __float_as_uint(sqrtf(redmax[0] + lambda));
        // ... and H_d >= lambda I bounds every entry of R^-1 (and of the inverse of any diagonal block of R)
        // by 1 / sqrt(lambda)
        hd->tc_amax[AMAX_INV] = lambda > 0.f ? __float_as_uint(rsqrtf(lambda)) : 0u;
    }
}

// Upper triangle: H <- H * inv_tokens (+ lambda on the diagonal, dead -> 1 + lambda);
// strict lower triangle <- 0.
// Tiles of 64 columns x 16 rows, four columns of a row per thread: one load in flight per thread everywhere
// (64 rows in a loop of dependent load-store pairs took 13 us at n = 1024).
// (src: H itself, or the matrix in sorted order.)
__global__ void __launch_bounds__(256) scale_damp_kernel(const float *src, float *H, int n, const StateHeader *hd,
                                                         const uint8_t *dead) {
    pdl_launch_dependents();
    pdl_wait();
    const int j = blockIdx.x * 64 + 4 * (threadIdx.x & 15), i = blockIdx.y * 16 + (threadIdx.x >> 4);
    if (j >= n || i >= n) return;
    const float inv = hd->inv_tokens, lam = hd->lambda;
    float *p = H + (int64_t)i * n + j;
    const float *sp = src + (int64_t)i * n + j;
    const bool vec = (n & 3) == 0 && ((reinterpret_cast<uintptr_t>(H) | reinterpret_cast<uintptr_t>(src)) & 15) == 0;
    float v[4] = {0.f, 0.f, 0.f, 0.f};
    if (j + 3 >= i) {
        if (vec) {
            const float4 q = *reinterpret_cast<const float4 *>(sp);
            v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) if (j + e < n) v[e] = sp[e];
        }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        if (j + e < i) v[e] = 0.f;
        else if (j + e == i) v[e] = (dead[i] ? 1.f : v[e] * inv) + lam;
        else v[e] *= inv;
    }
    if (vec) *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
    else {
#pragma unroll
        for (int e = 0; e < 4; ++e) if (j + e < n) p[e] = v[e];
    }
}

// ---------------------------------------------------------------------------
// quant(.)  -- min/max grid that contains zero, round half to even.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void make_grid(float lo, float hi, float amax, int bits, int sym,
                                          float &scale, float &zero) {
    if (sym) {
        float a = (amax == 0.f) ? 1.f : amax;
        scale = a / (float)((1 << (bits - 1)) - 1);
        zero = (float)(1 << (bits - 1));
    } else {
        lo = fminf(lo, 0.f);
        hi = fmaxf(hi, 0.f);
        if (hi == lo) { scale = 1.f; zero = 0.f; }
        else {
            scale = (hi - lo) / (float)((1 << bits) - 1);
            zero = rintf(-lo / scale);
        }
    }
}

// Clipping-range search of a grid by least squared rounding error (experimental setup of Section 5):
// candidate k of `steps` shrinks the min/max range by p_k = 1 - k (1 - min_ratio) / steps;
// the candidate with the least squared rounding error of the group's weights wins, the widest one on ties.
__device__ __forceinline__ float clip_ratio(int k, int steps, float min_ratio) {
    return 1.f - (float)k * ((1.f - min_ratio) / (float)steps);
}
__device__ __forceinline__ float rounding_error_sq(float w, float scale, float zero, float maxq) {
    const float cq = fminf(fmaxf(rintf(w * (1.f / scale)) + zero, 0.f), maxq);
    const float d = scale * (cq - zero) - w;
    return d * d;
}

template <typename T> struct alignas(4 * sizeof(T)) Quad { T v[4]; };

// Per-channel grids from the original rows (dead inputs count as zero weights), one warp per row; `copy`: also the rows
// themselves as float32 (the working copy of W, one pass and one launch less).  The clipping search takes four candidates
// per pass over the row.
template <typename T>
__global__ void __launch_bounds__(256) row_grid_kernel(const T *W, int64_t ldw, float *copy, int64_t ldc, int m, int n,
                                                       const uint8_t *dead, int bits, int sym,
                                                       float *scales, float *zeros, int clip_steps, float clip_min) {
    const int row = blockIdx.x * 8 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (row >= m) return;
    const T *w = W + (int64_t)row * ldw;
    float *cw = copy ? copy + (int64_t)row * ldc : nullptr;
    const bool vec = (n & 3) == 0 && (ldw & 3) == 0 && (reinterpret_cast<uintptr_t>(W) & (4 * sizeof(T) - 1)) == 0 &&
                     (!copy || ((ldc & 3) == 0 && (reinterpret_cast<uintptr_t>(copy) & 15) == 0));
    // four columns from c, dead ones as zero
    auto load4 = [&](int c, float (&v)[4], bool keep) {
        if (vec) {
            const Quad<T> q = *reinterpret_cast<const Quad<T> *>(w + c);
#pragma unroll
            for (int e = 0; e < 4; ++e) v[e] = (float)q.v[e];
            if (keep) *reinterpret_cast<float4 *>(cw + c) = make_float4(v[0], v[1], v[2], v[3]);
            const uint32_t dd = *reinterpret_cast<const uint32_t *>(dead + c);
            if (dd) {
#pragma unroll
                for (int e = 0; e < 4; ++e) if (dd >> (8 * e) & 0xffu) v[e] = 0.f;
            }
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                v[e] = c + e < n ? (float)w[c + e] : 0.f;
                if (keep && c + e < n) cw[c + e] = v[e];
                if (c + e < n && dead[c + e]) v[e] = 0.f;
            }
        }
    };
    float lo = 0.f, hi = 0.f, am = 0.f;
#pragma unroll 4
    for (int c = 4 * lane; c < n; c += 128) {
        float v[4];
        load4(c, v, copy != nullptr);
#pragma unroll
        for (int e = 0; e < 4; ++e) { lo = fminf(lo, v[e]); hi = fmaxf(hi, v[e]); am = fmaxf(am, fabsf(v[e])); }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        am = fmaxf(am, __shfl_xor_sync(0xffffffffu, am, o));
    }
    float s, z;
    make_grid(lo, hi, am, bits, sym, s, z);
    if (clip_steps > 0) {
        const float maxq = (float)((1 << bits) - 1);
        float best = INFINITY;
        for (int k = 0; k < clip_steps; k += 4) {
            float sk[4], zk[4], err[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const float p = clip_ratio(min(k + t, clip_steps - 1), clip_steps, clip_min);
                make_grid(p * lo, p * hi, p * am, bits, sym, sk[t], zk[t]);
            }
            for (int c = 4 * lane; c < n; c += 128) {
                float v[4];
                load4(c, v, false);
#pragma unroll
                for (int e = 0; e < 4; ++e)          // (columns beyond n are zeros: on every grid, no error)
#pragma unroll
                    for (int t = 0; t < 4; ++t) err[t] += rounding_error_sq(v[e], sk[t], zk[t], maxq);
            }
#pragma unroll
            for (int t = 0; t < 4; ++t) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) err[t] += __shfl_xor_sync(0xffffffffu, err[t], o);
                if (k + t < clip_steps && err[t] < best) { best = err[t]; s = sk[t]; z = zk[t]; }
            }
        }
    }
    if (lane == 0) { scales[row] = s; zeros[row] = z; }
}

// Static groups: one grid per output channel and per group of `group` consecutive columns of W in the
// caller's column order, from the original weights (dead inputs count as zero weights).  One warp per
// (row, group); W float32 or bf16.
template <typename T>
__global__ void __launch_bounds__(256) static_group_grid_kernel(const T *W, int64_t ldw, int m, int n, int group, int G,
                                                                const uint8_t *dead, int bits, int sym, float *scales,
                                                                float *zeros, int clip_steps, float clip_min) {
    const int64_t wid = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (wid >= (int64_t)m * G) return;
    const int row = (int)(wid / G), g = (int)(wid - (int64_t)row * G);
    const T *w = W + (int64_t)row * ldw;
    const int c0 = g * group, c1 = min(n, c0 + group);
    float lo = 0.f, hi = 0.f, am = 0.f;
    for (int c = c0 + lane; c < c1; c += 32) {
        const float v = dead[c] ? 0.f : (float)w[c];
        lo = fminf(lo, v); hi = fmaxf(hi, v); am = fmaxf(am, fabsf(v));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        am = fmaxf(am, __shfl_xor_sync(0xffffffffu, am, o));
    }
    float s, z;
    make_grid(lo, hi, am, bits, sym, s, z);
    if (clip_steps > 0) {
        const float maxq = (float)((1 << bits) - 1);
        float best = INFINITY;
        for (int k = 0; k < clip_steps; ++k) {
            const float p = clip_ratio(k, clip_steps, clip_min);
            float sk, zk;
            make_grid(p * lo, p * hi, p * am, bits, sym, sk, zk);
            float err = 0.f;
            for (int c = c0 + lane; c < c1; c += 32) err += rounding_error_sq(dead[c] ? 0.f : (float)w[c], sk, zk, maxq);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) err += __shfl_xor_sync(0xffffffffu, err, o);
            if (err < best) { best = err; s = sk; z = zk; }
        }
    }
    if (lane == 0) { scales[(int64_t)row * G + g] = s; zeros[(int64_t)row * G + g] = z; }
}

// ---------------------------------------------------------------------------
// Column loop over one lazy-batch block [i0, i0 + bw) (Algorithm 1, inner
// loop), for grids per group of fewer than 32 columns (quant_block_kernel takes all others).  One warp per weight row; the row's block lives in registers (lane
// owns columns lane, lane + 32, ...), the B x B diagonal tiles of U and P live
// in shared memory.  Outputs: codes, dequantized columns (in place in W),
// -Err and the pre-quantization columns (for the trailing update), group grids.
// ---------------------------------------------------------------------------
struct ColumnLoopArgs {
    float *W; int64_t ldw; int m, n;
    const float *U, *P;        // n x n, ld n
    const uint8_t *dead;
    int i0, bw;                // block start, valid width (<= 32 * T)
    int bits, group, sym;
    uint8_t *codes;            // m x n
    float *scales, *zeros;     // m x G
    int G;
    float *EW;                 // m x (2 * 32 * T): [-Err | Wpre]
    // fp16-split handles (else nullptr): Wpre is stored times rho = scale of U^T / scale of P^T (from the two recorded
    // maxima), which lets the two halves of the update's B operand keep scales of their own
    const unsigned *amax_u, *amax_p;
    StateHeader *hd;
    float err_scale, asym_scale;   // 1 or 0: switches of the two terms of the weight update (ablation)
    const int *perm;               // nullptr, or: working column c is original column perm[c] (codes go there)
    int clip_steps; float clip_min; // clipping-range search of the group grids (0: plain min/max)
};

template <int T>
__global__ void __launch_bounds__(1024) column_loop_kernel(ColumnLoopArgs a) {
    constexpr int BW = 32 * T;
    extern __shared__ float smem_f[];
    float (*Us)[BW] = reinterpret_cast<float (*)[BW]>(smem_f);
    float (*Ps)[BW] = reinterpret_cast<float (*)[BW]>(smem_f + BW * BW);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nwarps = blockDim.x >> 5;
    const int n = a.n, i0 = a.i0, bw = a.bw;

    for (int e = tid; e < BW * BW; e += blockDim.x) {
        int r = e / BW, c = e % BW;
        float u = 0.f, p = 0.f;
        if (r < bw && c < bw && c >= r) {
            int64_t off = (int64_t)(i0 + r) * n + (i0 + c);
            u = a.U[off];
            p = a.P[off];
        }
        Us[r][c] = u; Ps[r][c] = p;
    }
    __syncthreads();

    const int row = blockIdx.x * nwarps + warp;
    if (row >= a.m) return;
    float *wrow = a.W + (int64_t)row * a.ldw + i0;

    float w[T], nerr[T], pre[T];
    int code[T];
#pragma unroll
    for (int t = 0; t < T; ++t) {
        int c = lane + 32 * t;
        float v = 0.f;
        if (c < bw && !a.dead[i0 + c]) v = wrow[c];
        w[t] = v; nerr[t] = 0.f; pre[t] = 0.f; code[t] = 0;
        // reported from the value that was read: the clamp of the quantizer would absorb a NaN or Inf
        if (!isfinite(v)) record_status(a.hd, ST_NONFINITE, row);
    }

    const float maxq = (float)((1 << a.bits) - 1);
    float scale = 1.f, zero = 0.f;
    if (a.group <= 0) { scale = a.scales[row]; zero = a.zeros[row]; }

#pragma unroll
    for (int t = 0; t < T; ++t) {
        for (int jj = 0; jj < 32; ++jj) {
            const int j = t * 32 + jj;
            if (j >= bw) break;
            if (a.group > 0 && ((i0 + j) % a.group) == 0) {
                // grid of the group that starts here, from the current values
                const int gend = min(j + a.group, bw);
                float lo = 0.f, hi = 0.f, am = 0.f;
#pragma unroll
                for (int t2 = 0; t2 < T; ++t2) {
                    int c = lane + 32 * t2;
                    if (c >= j && c < gend) {
                        lo = fminf(lo, w[t2]); hi = fmaxf(hi, w[t2]); am = fmaxf(am, fabsf(w[t2]));
                    }
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
                    hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
                    am = fmaxf(am, __shfl_xor_sync(0xffffffffu, am, o));
                }
                make_grid(lo, hi, am, a.bits, a.sym, scale, zero);
                if (a.clip_steps > 0) {
                    float best = INFINITY;
                    for (int k = 0; k < a.clip_steps; ++k) {
                        const float p = clip_ratio(k, a.clip_steps, a.clip_min);
                        float sk, zk;
                        make_grid(p * lo, p * hi, p * am, a.bits, a.sym, sk, zk);
                        float err = 0.f;
#pragma unroll
                        for (int t2 = 0; t2 < T; ++t2) {
                            int c = lane + 32 * t2;
                            if (c >= j && c < gend) err += rounding_error_sq(w[t2], sk, zk, maxq);
                        }
#pragma unroll
                        for (int o = 16; o > 0; o >>= 1) err += __shfl_xor_sync(0xffffffffu, err, o);
                        if (err < best) { best = err; scale = sk; zero = zk; }
                    }
                }
                if (lane == 0) {
                    int g = (i0 + j) / a.group;
                    a.scales[(int64_t)row * a.G + g] = scale;
                    a.zeros[(int64_t)row * a.G + g] = zero;
                }
            }
            const float wj = __shfl_sync(0xffffffffu, w[t], jj);
            float cq = fminf(fmaxf(rintf(wj * (1.f / scale)) + zero, 0.f), maxq);
            const float q = scale * (cq - zero);
            const float ne = a.err_scale * ((q - wj) * (1.f / Us[j][j]));   // -(w - q) / U_jj
            const float wp = a.asym_scale * wj;
            if (lane == jj) { w[t] = q; nerr[t] = ne; pre[t] = wp; code[t] = (int)cq; }
#pragma unroll
            for (int t2 = 0; t2 < T; ++t2) {
                if (t2 < t) continue;
                int c = lane + 32 * t2;
                if (c > j) w[t2] = fmaf(wp, Ps[j][c], fmaf(ne, Us[j][c], w[t2]));
            }
        }
    }

    bool bad = false;
    float rho = 1.f;
    if (a.amax_u) {
        const float ap = __uint_as_float(*a.amax_p);
        rho = ap > 0.f ? split_scale(__uint_as_float(*a.amax_u)) / split_scale(ap) : 0.f;
    }
    float *ew = a.EW + (int64_t)row * (2 * BW);
    uint8_t *crow = a.codes + (int64_t)row * n + i0;
#pragma unroll
    for (int t = 0; t < T; ++t) {
        int c = lane + 32 * t;
        ew[c] = nerr[t];
        ew[BW + c] = rho * pre[t];
        if (c < bw) {
            wrow[c] = w[t];
            if (a.perm) a.codes[(int64_t)row * n + a.perm[i0 + c]] = (uint8_t)code[t];
            else crow[c] = (uint8_t)code[t];
            // (of the value before the rounding and of the error: the rounded weight is finite whatever came in)
            bad |= !isfinite(w[t]) || !isfinite(nerr[t]) || !isfinite(pre[t]);
        }
    }
    if (bad) record_status(a.hd, ST_NONFINITE, row);
}

// ---------------------------------------------------------------------------
// Row-by-row form of P (Eq. "unparallel"):  P[q, f] = scale * (D[q, f] U[f, f]^T) U[f, f],  f = q + 1 .. n - 1
// (L[f, f] of the paper is U[f, f]^T).  One CTA per row q, two passes over the trailing triangle of U:
//   v_a     = sum_{k >= a} D[q, k] U[a, k]      a in f   (a warp per a, along row a of U)
//   P[q, j] = sum_{q < a <= j} v_a U[a, j]      j in f   (a thread per j, coalesced across j)
// This is the form that Theorem 4.2 replaces by two matrix products; it is kept as the comparison of the
// latency discussion of Section 5, not as a path of the solve.  In place: row q of P overwrites row q of D.
// ---------------------------------------------------------------------------
constexpr int PR_THREADS = 1024;
__global__ void __launch_bounds__(PR_THREADS) p_rowwise_kernel(float *D, const float *U, int n, float scale) {
    extern __shared__ float pr_smem[];
    float *d = pr_smem, *v = pr_smem + n;
    const int q = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float *row = D + (int64_t)q * n;
    for (int c = tid; c < n; c += PR_THREADS) d[c] = c > q ? row[c] : 0.f;
    __syncthreads();
    for (int a = q + 1 + warp; a < n; a += PR_THREADS / 32) {
        const float *ur = U + (int64_t)a * n;
        float s = 0.f;
        for (int k = a + lane; k < n; k += 32) s = fmaf(d[k], ur[k], s);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) v[a] = s;
    }
    __syncthreads();
    for (int j = tid; j < n; j += PR_THREADS) {
        float s0 = 0.f, s1 = 0.f;
        int a = q + 1;
        for (; a + 1 <= j; a += 2) {
            s0 = fmaf(v[a], U[(int64_t)a * n + j], s0);
            s1 = fmaf(v[a + 1], U[(int64_t)(a + 1) * n + j], s1);
        }
        if (a <= j) s0 = fmaf(v[a], U[(int64_t)a * n + j], s0);
        row[j] = j > q ? scale * (s0 + s1) : 0.f;
    }
}

// ---------------------------------------------------------------------------
// act_order: columns sorted by decreasing diag(H).
// ---------------------------------------------------------------------------
// perm[rank] = q, rank = number of inputs that sort before q: larger value v (v = 1 for dead
// inputs, else H_qq / tokens), ties by smaller index (a stable descending sort).  O(n^2) compares, RANK_COLS inputs
// per CTA against all of them, in shared memory in chunks (a thread per input kept n / 256 CTAs busy: 63 us at n = 4096,
// now 15).
constexpr int RANK_COLS = 32, RANK_CHUNK = 4096;
__global__ void __launch_bounds__(256) rank_desc_kernel(const float *H, int n, float inv_tokens, const uint8_t *dead,
                                                        int *perm, uint8_t *dead_perm) {
    __shared__ float v[RANK_CHUNK];
    const int lane = threadIdx.x & 31, q0 = blockIdx.x * RANK_COLS + (threadIdx.x >> 5) * (RANK_COLS / 8);
    auto value = [&](int j) { return dead[j] ? 1.f : H[(int64_t)j * n + j] * inv_tokens; };
    float vq[RANK_COLS / 8];
    int rank[RANK_COLS / 8];
#pragma unroll
    for (int e = 0; e < RANK_COLS / 8; ++e) { vq[e] = q0 + e < n ? value(q0 + e) : 0.f; rank[e] = 0; }
    for (int j0 = 0; j0 < n; j0 += RANK_CHUNK) {
        const int lim = min(RANK_CHUNK, n - j0);
        for (int t = threadIdx.x; t < lim; t += 256) v[t] = value(j0 + t);
        __syncthreads();
        for (int t = lane; t < lim; t += 32) {
            const float x = v[t];
#pragma unroll
            for (int e = 0; e < RANK_COLS / 8; ++e) rank[e] += (x > vq[e]) || (x == vq[e] && j0 + t < q0 + e);
        }
        __syncthreads();
    }
#pragma unroll
    for (int e = 0; e < RANK_COLS / 8; ++e) {
        const int r = __reduce_add_sync(0xffffffffu, rank[e]);
        if (lane == 0 && q0 + e < n) { perm[r] = q0 + e; dead_perm[r] = dead[q0 + e]; }
    }
}

// dst[i][j] = src[perm[i]][perm[j]], j >= i only, of a symmetric matrix given by its upper triangle (element (a, b) is read
// at (min, max)).
__global__ void __launch_bounds__(256) permute_symmetric_kernel(const float *src, float *dst, int n, const int *perm) {
    const int j = blockIdx.x * 256 + threadIdx.x;
    const int i = blockIdx.y;
    if (j >= n || j < i) return;
    const int a = perm[i], b = perm[j];
    dst[(int64_t)i * n + j] = src[(int64_t)min(a, b) * n + max(a, b)];
}

// Rows in the two kernels below: as many as PERM_ROWS per CTA at a time, so that the order is read once for all of them;
// staged in shared memory, so that device memory sees whole rows only.
constexpr int PERM_ROWS = 4;

// dst[r][c] = src[r][perm[c]] as float32 (src float32 or bf16), or src[row_perm[r]][perm[c]]: the working copy of W, and
// dXX^T, in sorted order.  Bound by device
// memory (4096 x 4096 bf16: 30 us; gathered from device memory element by element 51).
template <typename T>
__global__ void __launch_bounds__(256) gather_cols_kernel(const T *src, int64_t lds, float *dst, int64_t ldd, int m, int n,
                                                          const int *perm, const int *row_perm, int rows) {
    extern __shared__ __align__(16) float row_s[];
    T *rs = reinterpret_cast<T *>(row_s);
    for (int r0 = blockIdx.x * rows; r0 < m; r0 += gridDim.x * rows) {
        const int nr = min(rows, m - r0);
        for (int r = 0; r < nr; ++r) {
            const T *sp = src + (int64_t)(row_perm ? row_perm[r0 + r] : r0 + r) * lds;
#pragma unroll 8
            for (int c = threadIdx.x; c < n; c += 256) rs[(size_t)r * n + c] = sp[c];
        }
        __syncthreads();
#pragma unroll 4
        for (int c = threadIdx.x; c < n; c += 256) {
            const int p = perm[c];
#pragma unroll
            for (int r = 0; r < PERM_ROWS; ++r)
                if (r < nr) dst[(int64_t)(r0 + r) * ldd + c] = (float)rs[(size_t)r * n + p];
        }
        __syncthreads();
    }
}

// In place: W[r][perm[c]] <- W[r][c] (back to the original column order).  Bound by device memory (4096 x 4096: 43 us;
// scattered to device memory 81).
__global__ void __launch_bounds__(256) unpermute_rows_kernel(float *W, int64_t ldw, int m, int n, const int *perm, int rows) {
    extern __shared__ __align__(16) float row_s[];
    for (int r0 = blockIdx.x * rows; r0 < m; r0 += gridDim.x * rows) {
        const int nr = min(rows, m - r0);
#pragma unroll 4
        for (int c = threadIdx.x; c < n; c += 256) {
            const int p = perm[c];
            float v[PERM_ROWS];
#pragma unroll
            for (int r = 0; r < PERM_ROWS; ++r) if (r < nr) v[r] = W[(int64_t)(r0 + r) * ldw + c];
#pragma unroll
            for (int r = 0; r < PERM_ROWS; ++r) if (r < nr) row_s[(size_t)r * n + p] = v[r];
        }
        __syncthreads();
        for (int r = 0; r < nr; ++r)
#pragma unroll 8
            for (int c = threadIdx.x; c < n; c += 256) W[(int64_t)(r0 + r) * ldw + c] = row_s[(size_t)r * n + c];
        __syncthreads();
    }
}

// dst[r][c] = src[r][c] as float32: the working copy of W.  A thread takes 4 columns of WIDEN_ROWS rows, all loads before the
// first store.  Bound by device memory (16384 x 4096 bf16 58 us, one element at a time 160; 4096 x 4096 float32 18, 43).
constexpr int WIDEN_ROWS = 8;
template <typename T>
__global__ void __launch_bounds__(256) widen_kernel(const T *src, int64_t lds, float *dst, int64_t ldd, int m, int n) {
    const int c = (blockIdx.x * 256 + threadIdx.x) * 4;
    if (c >= n) return;
    const bool vec = c + 3 < n && (lds & 3) == 0 && (ldd & 3) == 0 && (reinterpret_cast<uintptr_t>(src) & (4 * sizeof(T) - 1)) == 0 &&
                     (reinterpret_cast<uintptr_t>(dst) & 15) == 0;
    for (int r0 = blockIdx.y * WIDEN_ROWS; r0 < m; r0 += gridDim.y * WIDEN_ROWS) {
        if (vec) {
            Quad<T> q[WIDEN_ROWS];
#pragma unroll
            for (int i = 0; i < WIDEN_ROWS; ++i)
                if (r0 + i < m) q[i] = *reinterpret_cast<const Quad<T> *>(src + (int64_t)(r0 + i) * lds + c);
#pragma unroll
            for (int i = 0; i < WIDEN_ROWS; ++i)
                if (r0 + i < m)
                    *reinterpret_cast<float4 *>(dst + (int64_t)(r0 + i) * ldd + c) =
                        make_float4((float)q[i].v[0], (float)q[i].v[1], (float)q[i].v[2], (float)q[i].v[3]);
        } else {
            for (int i = 0; i < WIDEN_ROWS && r0 + i < m; ++i)
                for (int e = 0; e < 4 && c + e < n; ++e) dst[(int64_t)(r0 + i) * ldd + c + e] = (float)src[(int64_t)(r0 + i) * lds + c + e];
        }
    }
}

}  // namespace gptaq
