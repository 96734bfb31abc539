// The correction matrix of narrow layers in one launch: P = alpha ((D U^T) .* M_U) U in plain float32.
//
// Rows of P need rows of D and all of U, and row a of U serves both products: it makes column a of O = (D U^T) .* M_U, and that
// column times the row is what it adds to P.  So a CTA takes four rows and goes through U once, 32 rows at a time: a warp has two of
// them and sums their products with the rows of D, the lanes side by side, through a butterfly of shuffles; then a thread has two
// columns of P and every other row of the tile.
// What bounds it: a tile is two barriers, a chain of five shuffles and 16 dependent pairs of reads and FMAs, 0.8 us, and the launch is 6.
// us as two products of 32 x 32 tiles and so: n = 40 15.4 / 9.7, 128 19.5 / 12.2, 256 27.3 / 18.4, 320 28.7 / 24.6, 400 34.8 / 32.8,
// odd n = 99 20.9 / 13.4, 255 32.8 / 20.5, 449 40.9 / 46.8, hence NP_MAX_N.  (With 256 threads 256 22.5; copied ahead by two or more tiles, by
// bulk copies of rows or read from global memory twice, 22.5 to 28.7.)  P from the device's own U and dXX^T is 20 to 30 % closer to
// float64 (n = 128 1.22e-7 / 0.85e-7, 384 1.36e-7 / 1.06e-7): its sums are shorter.
#pragma once
#include "simt_gemm.cuh"

namespace gptaq {

constexpr int NP_ROWS = 4, NP_THREADS = 512, NP_TILE = 32, NP_MAX_N = 384;
__host__ __device__ inline int np_pitch(int n) { return (n + 3) / 4 * 4 + 4; }
inline size_t np_smem(int n) {
    const size_t tiles = (size_t)(2 * NP_TILE + NP_ROWS) * np_pitch(n) * sizeof(float), sums = NP_ROWS * 256 * 2 * sizeof(float);
    return tiles > sums ? tiles : sums;
}

__global__ void __launch_bounds__(NP_THREADS) p_narrow_kernel(float *D, const float *U, int n, float alpha) {
    extern __shared__ __align__(16) float np_tiles[];                 // [2][NP_TILE][pitch], then the rows of D [NP_ROWS][pitch]
    __shared__ __align__(16) float Os[NP_TILE][NP_ROWS];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int i0 = blockIdx.x * NP_ROWS, ld = np_pitch(n), n4 = (n + 3) / 4 * 4;
    float *Ds = np_tiles + 2 * NP_TILE * ld;
    const bool vec = (n & 3) == 0;                                    // (bases are 256-byte aligned)
    pdl_launch_dependents();
    pdl_wait();
    // rows a0 .. + 31 of U from column a0 on, zeros beyond n
    auto fetch = [&](int tile) {
        const int a0 = tile * NP_TILE;
        if (a0 < n) {
            float *dst = np_tiles + (tile & 1) * NP_TILE * ld;
#pragma unroll 1
            for (int a = warp; a < NP_TILE; a += NP_THREADS / 32) {
                const float *src = U + (int64_t)(a0 + a) * n;
                if (vec) {
                    for (int c = a0 + 4 * lane; c < n; c += 128)
                        if (a0 + a < n) sg_copy16(dst + a * ld + c, src + c);
                        else *reinterpret_cast<float4 *>(dst + a * ld + c) = make_float4(0.f, 0.f, 0.f, 0.f);
                } else {
                    for (int c = a0 + lane; c < n4; c += 32) {
                        const bool in = a0 + a < n && c < n;
                        sg_copy4(dst + a * ld + c, in ? src + c : U, in);
                    }
                }
            }
        }
        };
    int tile = (i0 + 1) / NP_TILE;                                    // (column a of O is kept for a > i)
    fetch(tile);
    // D right of the diagonal
#pragma unroll 1
    for (int r = warp; r < NP_ROWS; r += NP_THREADS / 32)
#pragma unroll 4
        for (int c = lane; c < n4; c += 32) Ds[r * ld + c] = i0 + r < n && c < n && c > i0 + r ? D[(int64_t)(i0 + r) * n + c] : 0.f;
    // this thread's columns of P: j, j + 1; rows part, part + 2, .. of a tile (two threads meet at the end)
    const int part = tid >> 8, j = 2 * (tid & 255);
    float p[NP_ROWS][2];
#pragma unroll
    for (int r = 0; r < NP_ROWS; ++r) p[r][0] = p[r][1] = 0.f;
    for (; tile * NP_TILE < n; ++tile) {
        const int a0 = tile * NP_TILE;
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();                                              // (all have left the tile before, and its products of O)
        fetch(tile + 1);
        const float *Ut = np_tiles + (tile & 1) * NP_TILE * ld;
        // O: rows a0 + 4 warp + e of U against the rows of D
        float s[8];
#pragma unroll
        for (int v = 0; v < 8; ++v) s[v] = 0.f;
#pragma unroll 1
        for (int c = a0 / 128 * 128 + 4 * lane; c < n; c += 128) {
            if (c < a0) continue;
            float4 d[NP_ROWS];
#pragma unroll
            for (int r = 0; r < NP_ROWS; ++r) d[r] = *reinterpret_cast<const float4 *>(Ds + r * ld + c);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float4 u = *reinterpret_cast<const float4 *>(Ut + (2 * warp + e) * ld + c);
#pragma unroll
                for (int r = 0; r < NP_ROWS; ++r) {
                    float x = s[4 * e + r];
                    x = fmaf(d[r].x, u.x, x); x = fmaf(d[r].y, u.y, x); x = fmaf(d[r].z, u.z, x); x = fmaf(d[r].w, u.w, x);
                    s[4 * e + r] = x;
                }
            }
        }
        __syncwarp();
        // eight sums over the lanes: three steps halve the values that a lane carries; value v ends in the lanes 4 v .. 4 v + 3
#pragma unroll
        for (int w = 4; w >= 1; w >>= 1) {
            const bool up = (lane & (4 * w)) != 0;
#pragma unroll
            for (int v = 0; v < w; ++v) {
                const float other = __shfl_xor_sync(0xffffffffu, up ? s[v] : s[v + w], 4 * w);
                s[v] = (up ? s[v + w] : s[v]) + other;
            }
        }
        s[0] += __shfl_xor_sync(0xffffffffu, s[0], 2);
        s[0] += __shfl_xor_sync(0xffffffffu, s[0], 1);
        if ((lane & 3) == 0) {
            const int v = lane >> 2, a = a0 + 2 * warp + (v >> 2);
            Os[2 * warp + (v >> 2)][v & 3] = a > i0 + (v & 3) && a < n ? s[0] : 0.f;
        }
        __syncthreads();
        // P += O U, a tile's 32 terms by themselves
        if (j + 1 >= a0 && j < n) {
            float t[NP_ROWS][2];
#pragma unroll
            for (int r = 0; r < NP_ROWS; ++r) t[r][0] = t[r][1] = 0.f;
#pragma unroll 4
            for (int a = part; a < NP_TILE; a += 2) {
                const float4 o = *reinterpret_cast<const float4 *>(&Os[a][0]);
                const float2 u = *reinterpret_cast<const float2 *>(Ut + a * ld + j);
                const float ov[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
                for (int r = 0; r < NP_ROWS; ++r) { t[r][0] = fmaf(ov[r], u.x, t[r][0]); t[r][1] = fmaf(ov[r], u.y, t[r][1]); }
            }
#pragma unroll
            for (int r = 0; r < NP_ROWS; ++r) { p[r][0] += t[r][0]; p[r][1] += t[r][1]; }
        }
    }
    __syncthreads();
    float2 *other = reinterpret_cast<float2 *>(np_tiles);             // [NP_ROWS][256]
    if (part == 1) {
#pragma unroll
        for (int r = 0; r < NP_ROWS; ++r) other[r * 256 + (tid & 255)] = make_float2(p[r][0], p[r][1]);
    }
    __syncthreads();
    if (part == 1) return;
#pragma unroll
    for (int r = 0; r < NP_ROWS; ++r) { p[r][0] += other[r * 256 + tid].x; p[r][1] += other[r * 256 + tid].y; }
#pragma unroll
    for (int r = 0; r < NP_ROWS; ++r) {
        const int i = i0 + r;
        if (i >= n) continue;
#pragma unroll
        for (int e = 0; e < 2; ++e)
            if (j + e < n) D[(int64_t)i * n + j + e] = j + e > i ? alpha * p[r][e] : 0.f;
    }
}

}  // namespace gptaq
