// Register-tiled fp32 products on CUDA cores for the FFMA kernel families: operands staged in shared memory, 256 threads.
//
// What bounds such a product is the shared-memory pipe, not the FMAs: on this GPU a 16-byte load costs a warp four cycles,
// or two when groups of at least four neighbouring lanes read the same address, against one issue cycle per FFMA and
// scheduler (measured: 245 fp32 FMAs per ns and SM, 217 from an outer-product loop; packed fma.f32x2 has the same rate).
// A thread therefore owns (4 * HALVES) rows x 4 columns: per contraction index eight cycles of loads feed 32 FFMAs of a
// warp with HALVES = 2, six feed 16 with HALVES = 1.  Lanes 0..7 of a group of eight share the rows (broadcast loads), the
// four groups share the columns.
//
// Thread -> output, warp = threadIdx.x / 32, lane = threadIdx.x % 32:
//   narrow form (64 columns):  rows 4 rg .. 4 rg + 3 with rg = wr * 4 + lane / 8, columns (warp / 4) * 32 + lane % 8 + 8 y;
//                              wr = warp or 7 - warp, so that the two warps of a scheduler share the work of a triangle evenly
//   wide form (128 columns):   rows 4 rg ..          with rg = (warp % 2) * 4 + lane / 8, columns (warp / 2) * 32 + lane % 8 + 8 y
// y = 0..3.  The second half of the rows (HALVES = 2) comes from a base pointer of its own: rows 32 .. 63 of the same tile
// (wide form) or the same rows of another tile with the same second operand (narrow form: two products in one pass).
// The columns of a thread are eight apart, so that an operand read by columns (B[k][j]) and one read by rows (B[j][k]) both
// give conflict-free loads: tile pitches are 64 + 4 or 128 + 4 floats.
#pragma once
#include "chunk_geom.cuh"
#include "tc_inverse.cuh"

namespace gdn {
namespace {
namespace ffma {

constexpr int kThreads = 256;
constexpr int kPc = kC + 4;   // pitch of a [64][64] tile
__host__ __device__ constexpr int pitch(int cols) { return cols + 4; }

__device__ __forceinline__ float ldf(const float* p) { return *p; }
__device__ __forceinline__ float ldf(const __nv_bfloat16* p) { return __bfloat162float(*p); }
__device__ __forceinline__ void stf(float* p, float x) { *p = x; }
__device__ __forceinline__ void stf(__nv_bfloat16* p, float x) { *p = __float2bfloat16_rn(x); }
__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 ld4(const __nv_bfloat16* p) {
    const uint2 u = *reinterpret_cast<const uint2*>(p);
    return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xFFFF0000u), __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xFFFF0000u));
}

struct Thread {
    int rn, rw, cn, cw;   // first row / first column of this thread in the narrow and in the wide form
    __device__ __forceinline__ Thread() {
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 3, c = lane & 7;
        rn = ((warp < 4 ? warp : 7 - warp) * 4 + g) * 4;
        cn = (warp >> 2) * 32 + c;
        rw = ((warp & 1) * 4 + g) * 4;
        cw = (warp >> 1) * 32 + c;
    }
};

// Unrolling of the products of the per-channel kernels (and of dU0) at DK key features.  At 128 such a kernel is 100 KB of code that a CTA runs
// once, and with a CTA on most SMs two steps side by side cost more in instruction fetches than they give: 8 heads of 1024 tokens
// 216 -> 206 us, and dU0 with E alone 3 us less.  (The line is drawn by DK alone: with fewer CTAs there is nothing to gain, 6 heads of 800 tokens, on
// half of the SMs, 175 -> 176; at d = 64 the code is short enough for two steps, 87.3 us against 90.2.)
template <int DK>
constexpr int kU = DK == 128 ? 1 : 2;

enum AForm { A_ROW, A_COL };   // A(i, k) = A[i * pa + k] / A[k * pa + i]
enum BForm { B_ROW, B_COL };   // B(k, j) = B[j * pb + k] / B[k * pb + j]

// acc[R0 + 4 h + x][y] += sum over k in [k0, k1) of A_h(i + x, k) B(k, j + 8 y);  i, j: first row and column of this thread;
// (k0, k1 multiples of 4; pointers at row / column 0)
// (CS: distance of a thread's columns; U: how far the loop is unrolled)
template <int HALVES, AForm AF, BForm BF, int R0 = 0, int CS = 8, int U = 2, int R>
__device__ __forceinline__ void mac(float (&acc)[R][4], const float* A0, const float* A1, int pa, int i, const float* B,
                                    int pb, int j, int k0, int k1) {
    static_assert(R0 + 4 * HALVES <= R, "rows of the accumulator");
    const float* a0 = AF == A_ROW ? A0 + i * pa : A0 + i;
    const float* a1 = HALVES == 2 ? (AF == A_ROW ? A1 + i * pa : A1 + i) : nullptr;
    const float* b0 = BF == B_ROW ? B + j * pb : B + j;
#pragma unroll U
    for (int k = k0; k < k1; k += 4) {
        float a[4 * HALVES][4], b[4][4];   // a[row][k], b[k][column]
#pragma unroll
        for (int h = 0; h < HALVES; ++h) {
            const float* ap = h ? a1 : a0;
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                const float4 v = *reinterpret_cast<const float4*>(AF == A_ROW ? ap + x * pa + k : ap + (k + x) * pa);
                const float w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int z = 0; z < 4; ++z) {
                    if (AF == A_ROW) a[4 * h + x][z] = w[z]; else a[4 * h + z][x] = w[z];
                }
            }
        }
#pragma unroll
        for (int y = 0; y < 4; ++y) {
            if (BF == B_ROW) {
                const float4 v = *reinterpret_cast<const float4*>(b0 + CS * y * pb + k);
                b[0][y] = v.x; b[1][y] = v.y; b[2][y] = v.z; b[3][y] = v.w;
            } else {
#pragma unroll
                for (int z = 0; z < 4; ++z) b[z][y] = b0[(k + z) * pb + CS * y];
            }
        }
#pragma unroll
        for (int z = 0; z < 4; ++z)
#pragma unroll
            for (int x = 0; x < 4 * HALVES; ++x)
#pragma unroll
                for (int y = 0; y < 4; ++y) acc[R0 + x][y] = fmaf(a[x][z], b[z][y], acc[R0 + x][y]);
    }
}

template <int R>
__device__ __forceinline__ void zero(float (&acc)[R][4]) {
#pragma unroll
    for (int x = 0; x < R; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y) acc[x][y] = 0.f;
}

// Rows of a thread in a [64 x N] result (N = 64: narrow, 128: wide form), their index and its first column.
template <int N>
struct Out {
    static constexpr int R = N == 128 ? 8 : 4;
    int r0, c;
    __device__ __forceinline__ Out(const Thread& t) : r0(N == 128 ? t.rw : t.rn), c(N == 128 ? t.cw : t.cn) {}
    __device__ __forceinline__ int row(int x) const { return r0 + (x & 3) + 32 * (x >> 2); }
};

// acc = A [64 x 64] (zero above, A_LOWER, or below the diagonal) times B [64 x N].  In the wide form the half of the
// contraction in which one half of the rows meets only zeros is left out for those rows, in the narrow form the 16-row
// blocks that a warp's rows do not reach.
enum Tri { A_LOWER, A_UPPER };
template <int N, AForm AF, Tri TRI, int U = 2>
__device__ __forceinline__ void tri_product(const Thread& t, const float* A, const float* B, int pb, float (&acc)[N == 128 ? 8 : 4][4]) {
    const Out<N> o(t);
    zero(acc);
    if constexpr (N == 128) {
        const float* A1 = AF == A_ROW ? A + 32 * kPc : A + 32;
        constexpr bool low = TRI == A_LOWER;
        mac<2, AF, B_COL, 0, 8, U>(acc, A, A1, kPc, o.r0, B, pb, o.c, low ? 0 : 32, low ? 32 : kC);
        if constexpr (low) mac<1, AF, B_COL, 4, 8, U>(acc, A1, nullptr, kPc, o.r0, B, pb, o.c, 32, kC);
        else mac<1, AF, B_COL, 0, 8, U>(acc, A, nullptr, kPc, o.r0, B, pb, o.c, 0, 32);
    } else {
        const int w16 = (o.r0 >> 4) * 16;
        mac<1, AF, B_COL, 0, 8, U>(acc, A, nullptr, kPc, o.r0, B, pb, o.c, TRI == A_LOWER ? 0 : w16, TRI == A_LOWER ? w16 + 16 : kC);
    }
}

// Rows [0, 64) of a [T, H, COLS] tensor into a tile of pitch COLS + 4; rows beyond `len` become zero.  fp32 rows travel by
// cp.async (the caller commits and waits), bf16 rows are widened on the way.
template <int COLS>
__device__ __forceinline__ void load_rows(float* tile, const float* src, size_t row_pitch, int len) {
    for (int t = threadIdx.x; t < kC * (COLS / 4); t += kThreads) {
        const int i = t / (COLS / 4), c = (t % (COLS / 4)) * 4;
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(tile + i * pitch(COLS) + c);
        const bool live = i < len;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src + (live ? (size_t)i * row_pitch + c : 0)), "r"(live ? 16 : 0) : "memory");
    }
}
template <int COLS>
__device__ __forceinline__ void load_rows(float* tile, const __nv_bfloat16* src, size_t row_pitch, int len) {
#pragma unroll 4
    for (int t = threadIdx.x; t < kC * (COLS / 4); t += kThreads) {
        const int i = t / (COLS / 4), c = (t % (COLS / 4)) * 4;
        *reinterpret_cast<float4*>(tile + i * pitch(COLS) + c) = i < len ? ld4(src + (size_t)i * row_pitch + c) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
}
// A contiguous [ROWS][COLS] fp32 block of the workspace into a tile of pitch COLS + 4.
template <int ROWS, int COLS>
__device__ __forceinline__ void load_block(float* tile, const float* src) {
    for (int t = threadIdx.x; t < ROWS * (COLS / 4); t += kThreads) {
        const int i = t / (COLS / 4), c = (t % (COLS / 4)) * 4;
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(tile + i * pitch(COLS) + c);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src + (size_t)t * 4) : "memory");
    }
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <typename IO>
__device__ __forceinline__ const IO* rows_of(const void* base, const ChunkInfo& x, int H, int d) {
    return reinterpret_cast<const IO*>(base) + ((size_t)x.tok0 * H + x.hd) * d;
}
template <typename IO>
__device__ __forceinline__ IO* rows_of(void* base, const ChunkInfo& x, int H, int d) {
    return reinterpret_cast<IO*>(base) + ((size_t)x.tok0 * H + x.hd) * d;
}
__device__ __forceinline__ float* block_of(const Problem& p, size_t region, int ch, int floats) {
    return reinterpret_cast<float*>(p.ws + region) + (size_t)ch * floats;
}

// T = (I + A)^-1 with a clean upper right quadrant.  Everybody takes part; the caller synchronises afterwards.
__device__ __forceinline__ void invert(const float* A, float* T) {
    static_assert(kPc == kLdi, "the inversion works on the tiles of this family");
    invert64(A, T, [] { __syncthreads(); });
    for (int e = threadIdx.x; e < 32 * 32; e += kThreads) T[(e >> 5) * kPc + 32 + (e & 31)] = 0.f;
}

// Which part of the preparation a launch makes: the forward's, that and the backward's, the backward's alone.
enum PrepMode { PREP_FWD = 0, PREP_FWD_BWD = 1, PREP_BWD = 2 };
// CTAs per chunk-head of the scalar-gate preparation: two as long as every one of them finds an SM of its own (2 heads of 128 tokens, d = 64,
// closed backward: 23.7 -> 16.8 us).  With per-channel gates both chains need the decay within the blocks, and two CTAs gain nothing.
inline int prep_parts(const Problem& p, PrepMode mode) { return mode != PREP_BWD && 2 * p.L.max_chunks * p.d.H <= tc_sm_count() ? 2 : 1; }

// Sum over the eight lanes that share a row (fixed order).
__device__ __forceinline__ float row_sum8(float v) {
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    v += __shfl_xor_sync(0xffffffffu, v, 4);
    return v;
}
__device__ __forceinline__ float warp_total(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

}  // namespace ffma
}  // namespace
}  // namespace gdn
