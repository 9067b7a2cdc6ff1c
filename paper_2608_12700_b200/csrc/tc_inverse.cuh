// fp32 blocked inversion of a unit lower triangular 64 x 64 matrix in shared memory (T = (I + A)^-1 of the chunk-local
// solve, Section 4.2), shared by every kernel family.  The first 256 threads of the calling CTA work; all of them have to
// call, because the steps are separated by the caller's CTA-wide barrier.
#pragma once
#include "gdn_internal.cuh"

namespace gdn {
namespace {

// Rows of kLdi floats: 16-byte aligned, eight consecutive rows on distinct banks.
constexpr int kLdi = 68;

// A chain of dependent steps on one small matrix: what bounds it is latency (barriers, shared-memory loads, FMA chains) and the
// shared-memory pipe, hence few steps and register tiles.  The inverse doubles its block size twice:
//   1  the four 16 x 16 diagonal blocks, one per warp, a column per lane, forward substitution in registers
//   2  X = A10 T00, 3  T10 = -T11 X                 for the two pairs of 16 x 16 blocks
//   4  Y = A10 T00, 5  T10 = -T11 Y                 for the pair of 32 x 32 blocks
// X and Y lie in the upper right 32 x 32 quadrant of T and Y is left there (consumers take that quadrant as zero); the other
// blocks above the block diagonal are zeroed.
// In steps 2 to 5 a thread multiplies a 4 x 4 tile over a quarter of the contraction; the four partial tiles are added by two
// exchanges that also leave every lane with one row of four results.
// (Against 8 x 8 diagonal blocks, six barriers and rows of four outputs per thread, whole calls: backward of 16 heads of 16384
// tokens 643 -> 626 us, of 4 x 16 heads of 2048 tokens 281 -> 277 us, forward and backward of 6 x 16 x 1500 380 -> 374 us.)
__device__ __forceinline__ void inv_diag16(const float* A, float* T) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp < 4 && lane < 16) {   // t_i = [i == j] - sum_{m<i} A_im t_m
        const float* a = A + (warp * 16) * kLdi + warp * 16;
        float t[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            float s0 = (i == lane) ? 1.f : 0.f, s1 = 0.f;
#pragma unroll
            for (int m = 0; m < i; m += 4) {
                const float4 v = *reinterpret_cast<const float4*>(a + i * kLdi + m);
                s0 = fmaf(-v.x, t[m], s0);
                if (m + 1 < i) s1 = fmaf(-v.y, t[m + 1], s1);
                if (m + 2 < i) s0 = fmaf(-v.z, t[m + 2], s0);
                if (m + 3 < i) s1 = fmaf(-v.w, t[m + 3], s1);
            }
            t[i] = s0 + s1;
            T[(warp * 16 + i) * kLdi + warp * 16 + lane] = t[i];
        }
    } else if (warp == 0 || warp == 2) {   // lanes 16..31: the block right of the diagonal block
#pragma unroll
        for (int i = 0; i < 16; ++i) T[(warp * 16 + i) * kLdi + warp * 16 + lane] = 0.f;
    }
}
// D = (NEG ? -1 : 1) * A B, [4 rows of this lane's group x 4 columns] over 4 * STEPS indices from this lane's k0 on, summed
// over the four lanes that differ in the bits KS and 2 KS of the lane index (q: this lane's two bits); lane q stores row q.
template <int STEPS, int KS, bool NEG>
__device__ __forceinline__ void inv_tile(const float* A, const float* B, float* D, int k0, int q) {
    float acc[4][4] = {};
#pragma unroll
    for (int s = 0; s < STEPS; ++s) {
        const int k = k0 + 4 * s;
        float4 a[4], b[4];
#pragma unroll
        for (int z = 0; z < 4; ++z) {
            a[z] = *reinterpret_cast<const float4*>(A + z * kLdi + k);
            b[z] = *reinterpret_cast<const float4*>(B + (k + z) * kLdi);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const float w[4] = {a[r].x, a[r].y, a[r].z, a[r].w};
#pragma unroll
            for (int z = 0; z < 4; ++z) {
                acc[r][0] = fmaf(w[z], b[z].x, acc[r][0]);
                acc[r][1] = fmaf(w[z], b[z].y, acc[r][1]);
                acc[r][2] = fmaf(w[z], b[z].z, acc[r][2]);
                acc[r][3] = fmaf(w[z], b[z].w, acc[r][3]);
            }
        }
    }
    // rows 0, 1 go to the lanes with bit 2 KS clear, rows 2, 3 to the others; then one row each
    const bool hi = (q & 2) != 0, odd = (q & 1) != 0;
    float h[2][4], r4[4];
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int y = 0; y < 4; ++y) {
            const float send = hi ? acc[r][y] : acc[r + 2][y], keep = hi ? acc[r + 2][y] : acc[r][y];
            h[r][y] = keep + __shfl_xor_sync(0xffffffffu, send, 2 * KS);
        }
#pragma unroll
    for (int y = 0; y < 4; ++y) {
        const float send = odd ? h[0][y] : h[1][y], keep = odd ? h[1][y] : h[0][y];
        r4[y] = keep + __shfl_xor_sync(0xffffffffu, send, KS);
        if (NEG) r4[y] = -r4[y];
    }
    *reinterpret_cast<float4*>(D + q * kLdi) = make_float4(r4[0], r4[1], r4[2], r4[3]);
}
template <class Sync>
__device__ __forceinline__ void invert64(const float* A, float* T, Sync sync) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    inv_diag16(A, T);
    sync();
    // pairs of 16 x 16 blocks: warps 0, 1 the first, warps 2, 3 the second; eight rows a warp, lane = (row group, quarter, columns)
    const int pr = warp >> 1, p0 = pr * 32, r16 = (warp & 1) * 8 + (lane >> 4) * 4, q16 = (lane >> 2) & 3, c16 = (lane & 3) * 4;
    float* X = T + (pr * 16) * kLdi + 32 + pr * 16;
    if (warp < 4) inv_tile<1, 4, false>(A + (p0 + 16 + r16) * kLdi + p0, T + p0 * kLdi + p0 + c16, X + r16 * kLdi + c16, q16 * 4, q16);
    sync();
    if (warp < 4) inv_tile<1, 4, true>(T + (p0 + 16 + r16) * kLdi + p0 + 16, X + c16, T + (p0 + 16 + r16) * kLdi + p0 + c16, q16 * 4, q16);
    sync();
    // the pair of 32 x 32 blocks: four rows a warp, lane = (quarter, columns)
    const int r32 = warp * 4, q32 = lane >> 3, c32 = (lane & 7) * 4;
    if (warp < 8) inv_tile<2, 8, false>(A + (32 + r32) * kLdi, T + c32, T + r32 * kLdi + 32 + c32, q32 * 8, q32);
    sync();
    if (warp < 8) inv_tile<2, 8, true>(T + (32 + r32) * kLdi + 32, T + 32 + c32, T + (32 + r32) * kLdi + c32, q32 * 8, q32);
    sync();
}

}  // namespace
}  // namespace gdn
