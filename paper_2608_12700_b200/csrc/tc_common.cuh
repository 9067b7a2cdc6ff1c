// Device helpers shared by the tcgen05 kernel families: tile chunk access, fixed-order reductions, staged output
// stores, chunk bookkeeping and the bounded MMA wait.
#pragma once
#include "chunk_geom.cuh"
#include "tc_ptx.cuh"
#include "tc_tmap.cuh"

namespace gdn {
namespace {

using namespace tc;

constexpr float kLog2e = 1.4426950408889634f;

__device__ __forceinline__ void report_timeout(char* ws, int where) {
    WsHeader* h = reinterpret_cast<WsHeader*>(ws);
    h->status = GDN_ERR_DEVICE_TIMEOUT;
    h->detail = where;
}

__device__ __forceinline__ unsigned char* align1024(unsigned char* p) {
    return p + ((1024u - (smem_u32(p) & 1023u)) & 1023u);
}

// 8 fp32 <-> one 16-byte chunk of bf16
__device__ __forceinline__ uint4 pack8(const float* v) {
    return make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
}
__device__ __forceinline__ void unpack8(const uint4& u, float* v) {
    v[0] = bf16_lo(u.x); v[1] = bf16_hi(u.x); v[2] = bf16_lo(u.y); v[3] = bf16_hi(u.y);
    v[4] = bf16_lo(u.z); v[5] = bf16_hi(u.z); v[6] = bf16_lo(u.w); v[7] = bf16_hi(u.w);
}
// Chunk `ch` (columns 8 ch .. 8 ch + 7) of row r of a tile with R rows.
__device__ __forceinline__ void chunk_store(unsigned char* tile, int R, int r, int ch, const float* v) {
    *reinterpret_cast<uint4*>(tile + tile_chunk_off(R, r, ch)) = pack8(v);
}
__device__ __forceinline__ void chunk_load(const unsigned char* tile, int R, int r, int ch, float* v) {
    unpack8(*reinterpret_cast<const uint4*>(tile + tile_chunk_off(R, r, ch)), v);
}
// Eight consecutive floats from a 16-byte aligned shared array (two vector loads instead of eight scalar ones).
__device__ __forceinline__ void ld8s(const float* p, float* v) {
    *reinterpret_cast<float4*>(v) = *reinterpret_cast<const float4*>(p);
    *reinterpret_cast<float4*>(v + 4) = *reinterpret_cast<const float4*>(p + 4);
}

// Zero rows [row0 + len, row0 + 64) of a tile with R rows and 128 columns (threads 0 .. nthr-1 of the CTA take part).
__device__ __forceinline__ void zero_tail_rows(unsigned char* tile, int R, int row0, int len, int nthr) {
    for (int t = threadIdx.x; t < (kC - len) * 16; t += nthr) {
        const int r = row0 + len + t / 16, ch = t % 16;
        *reinterpret_cast<uint4*>(tile + tile_chunk_off(R, r, ch)) = make_uint4(0, 0, 0, 0);
    }
}
__device__ __forceinline__ void zero_tail_rows(unsigned char* tile, int R, int row0, int len) {
    zero_tail_rows(tile, R, row0, len, (int)blockDim.x);
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Copy the first `d` features of a staged [64 tokens][128 features] bf16 tile (rows row0 .. of one of R rows) to a [T, H, d] tensor with
// 16-byte stores (rows < len only).
__device__ __forceinline__ void flush_rows(const unsigned char* tile, void* base, const ChunkInfo& x, int H, int d, int nthr, int R = 64, int row0 = 0) {
    __nv_bfloat16* g = reinterpret_cast<__nv_bfloat16*>(base) + ((size_t)x.tok0 * H + x.hd) * d;
    for (int t = threadIdx.x; t < kC * 16; t += nthr) {
        const int i = t >> 4, chk = t & 15;
        if (i < x.len && chk * 8 < d) *reinterpret_cast<uint4*>(g + (size_t)i * H * d + chk * 8) = *reinterpret_cast<const uint4*>(tile + tile_chunk_off(R, row0 + i, chk));
    }
}

// dg_j = sum_{i >= j} dgam_i inside a chunk (gam_i = sum_{j <= i} g_j), by one warp: lane l owns tokens l and l + 32.
// v0 + v1 (two partial arrays, v1 may be null) are the 64 values of dgam; `last_extra` is added to the last one.
__device__ __forceinline__ void write_dg_suffix(const float* v0, const float* v1, float last_extra, float* dg, size_t stride,
                                                int len, int lane) {
    float a = v0[lane] + (v1 ? v1[lane] : 0.f);
    float b = v0[lane + 32] + (v1 ? v1[lane + 32] : 0.f) + (lane == 31 ? last_extra : 0.f);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float ta = __shfl_down_sync(0xffffffffu, a, o), tb = __shfl_down_sync(0xffffffffu, b, o);
        if (lane + o < 32) { a += ta; b += tb; }
    }
    a += __shfl_sync(0xffffffffu, b, 0);
    if (lane < len) dg[(size_t)lane * stride] = a;
    if (lane + 32 < len) dg[(size_t)(lane + 32) * stride] = b;
}

// Warps judge by their own clocks whether a wait has run out, so the warps of a CTA may disagree about one that ends close to the limit.  A warp
// that gives up reports it, does nothing more and stands by: it takes part in the barriers that are left, so that those that go on are not held
// up at one and tear nothing down beside it; what depends on its share runs out in turn.  (Going through all steps without work instead: the
// operator-form carries 2 % slower, the d = 64 passes 1.6 %.)  The low-rank carries leave together on a word in shared memory (`gave_up`): a warp that
// gives up sets it and takes part in every barrier up to the place where all look at it, with a barrier between the last write and the
// first look.  Kernels that meet at barrier 0 only need neither: a warp at its teardown there releases those that go on, which find nothing issued.
template <class Sync>
__device__ __forceinline__ void stand_by(int left, Sync sync) {
#pragma unroll 1
    for (; left > 0; --left) sync();
}
// ... at the end of item `item`, in a kernel that walks over items blockIdx.x, blockIdx.x + gridDim.x, ... with N barriers each
template <int N, class Sync>
__device__ __forceinline__ void stand_by_items(int item, int n_items, Sync sync) {
#pragma unroll 1
    for (int it = item + (int)gridDim.x; it < n_items; it += gridDim.x) stand_by(N, sync);
}

// After a wait gave up in step `s` of a chain: waits (bounded) for the loads of the ring that are in flight, so that the CTA does
// not retire under them.  By one thread.  (Without a time-out s = nsteps and there is nothing to wait for; at most one of the
// waits is for a load that was never issued.)
template <int STAGES>
__device__ __forceinline__ void drain_ring(uint64_t* bar_full, int s, int nsteps) {
#pragma unroll 1
    for (int k = s; k < nsteps && k < s + STAGES; ++k) (void)mbar_wait(&bar_full[k % STAGES], (k / STAGES) & 1);
}

// Wait for the MMAs committed to `bar`; on a timeout record it once.
#define GDN_WAIT_MMA(where)                                                    \
    if (ok) {                                                                  \
        ok = mbar_wait(&bar_mma, mma_phase);                                   \
        mma_phase ^= 1;                                                        \
        if (!ok && (threadIdx.x & 31) == 0) report_timeout(p.ws, where);       \
    }                                                                          \
    tc_fence_after();

}  // namespace
}  // namespace gdn
