// Inter-chunk carries of the FFMA families in low-rank form (fp32), for scalar and for per-channel gates:
//     forward   U = U~ - W h (stored),          h' = Ge h + Kb^T U            (h stored per chunk)
//     reverse   Y = Kb dh', dU += Y (stored),   dh = Ge dh' + E - W^T Y        (dh' stored per chunk; the paper's K#1)
// with Kb the keys scaled to the chunk end (made by the preparation kernel), Ge the decay of the state over the chunk (one
// factor, or one per state row) and dU preset to scale P^T dO.  U and dU are what the gradient stage needs, so it repeats
// neither product.
//
// The chain of chunks is serial, so a step is made short: the state columns evolve independently and a CTA carries 16 of
// them; with so few columns the products are split over the contraction (eight warps; an 8 x 4 tile per thread keeps the
// loads of shared memory below the FMAs) and the partial sums are added in a fixed order.  W and Kb of the next step arrive by
// cp.async under the current one.  Measured on 8 chains of 16 chunks, d_k = d_v = 128: 3.6 us a step; with one CTA per chain
// reading its operands from global memory and a 4 x 4 tile per thread it was 38 us (forward) and 103 us (reverse).
#pragma once
#include "ffma_tile.cuh"

namespace gdn {
namespace {
namespace ffma {

constexpr int kScanCols = 16, kScanPitch = kScanCols + 4;
template <int DK>
constexpr size_t scan_smem() {
    return sizeof(float) * (4 * kC * pitch(DK) + 8192 + DK * kScanPitch + kC * kScanPitch);
}

// acc[x][y] = sum over k in [k0, k1) of A(row x, k) B[k][4 cg + y]: rows rg + 8 x (row form) or 4 rg + x % 4 + 32 (x / 4)
template <AForm AF>
__device__ __forceinline__ void mac_slice(float (&acc)[8][4], const float* A, int pa, int rg, const float* B, int cg, int k0, int k1) {
#pragma unroll 1
    for (int k = k0; k < k1; k += 4) {
        float a[8][4];
        float4 b[4];
        if (AF == A_ROW) {
#pragma unroll
            for (int x = 0; x < 8; ++x) {
                const float4 v = *reinterpret_cast<const float4*>(A + (rg + 8 * x) * pa + k);
                a[x][0] = v.x; a[x][1] = v.y; a[x][2] = v.z; a[x][3] = v.w;
            }
        } else {
#pragma unroll
            for (int z = 0; z < 4; ++z)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float4 v = *reinterpret_cast<const float4*>(A + (k + z) * pa + 4 * rg + 32 * h);
                    a[4 * h][z] = v.x; a[4 * h + 1][z] = v.y; a[4 * h + 2][z] = v.z; a[4 * h + 3][z] = v.w;
                }
        }
#pragma unroll
        for (int z = 0; z < 4; ++z) b[z] = *reinterpret_cast<const float4*>(B + (k + z) * kScanPitch + 4 * cg);
#pragma unroll
        for (int z = 0; z < 4; ++z)
#pragma unroll
            for (int x = 0; x < 8; ++x) {
                acc[x][0] = fmaf(a[x][z], b[z].x, acc[x][0]);
                acc[x][1] = fmaf(a[x][z], b[z].y, acc[x][1]);
                acc[x][2] = fmaf(a[x][z], b[z].z, acc[x][2]);
                acc[x][3] = fmaf(a[x][z], b[z].w, acc[x][3]);
            }
    }
}

// One direction of one chain, columns [part * 16, part * 16 + 16) of the state.  VEC: per-channel gates.
template <int DK, int DV, bool REVERSE, bool VEC>
__device__ __forceinline__ void scan_chain(const Problem& p, int chain, int part, float* sm) {
    constexpr int PK = pitch(DK), TILE = kC * PK, NS = DK * kScanCols / 4 / kThreads;   // float4 pieces of the state per thread
    float* red = sm + 4 * TILE;          // partial sums, 8192 floats
    float* hs = red + 8192;              // state slice [DK][16]
    float* ys = hs + DK * kScanPitch;    // U or Y [64][16]
    const int H = p.d.H, n = chain / H, hd = chain % H;
    const SeqGeom sg = seq_geom(p, n);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, rg = lane >> 2, cg = lane & 3;
    const float* wsW = reinterpret_cast<const float*>(p.ws + p.L.W);
    const float* wsKb = reinterpret_cast<const float*>(p.ws + p.L.Kb);
    const float* wsG = reinterpret_cast<const float*>(p.ws + p.L.gamma);
    auto chunk_head = [&](int s) { return (size_t)(REVERSE ? sg.c0 + sg.n_chunks - 1 - s : sg.c0 + s) * H + hd; };
    auto fill = [&](int s) {   // W and Kb of step s into stage s % 2
        float* st = sm + (s & 1) * 2 * TILE;
        load_block<kC, DK>(st, wsW + chunk_head(s) * kC * DK);
        load_block<kC, DK>(st + TILE, wsKb + chunk_head(s) * kC * DK);
        cp_commit();
    };
    if (sg.n_chunks > 0) fill(0);
    float4 state[NS];
    const float* init = REVERSE ? p.dhT : p.h0;
    const size_t soff = (size_t)chain * DK * DV + part * kScanCols;
#pragma unroll
    for (int m = 0; m < NS; ++m) {
        const int e = tid + m * kThreads, r = e >> 2, c = (e & 3) * 4;
        state[m] = init ? *reinterpret_cast<const float4*>(init + soff + (size_t)r * DV + c) : make_float4(0.f, 0.f, 0.f, 0.f);
        *reinterpret_cast<float4*>(hs + r * kScanPitch + c) = state[m];
    }
#pragma unroll 1
    for (int s = 0; s < sg.n_chunks; ++s) {
        const size_t ch = chunk_head(s);
        const float* W = sm + (s & 1) * 2 * TILE;
        const float* Kb = W + TILE;
        // this thread's pieces of the additive terms, and the state that enters the chunk -> workspace
        float* keep = reinterpret_cast<float*>(p.ws + (REVERSE ? p.L.dhn : p.L.hc)) + ch * DK * DV + part * kScanCols;
        const size_t yoff = ch * kC * DV + (size_t)(tid >> 2) * DV + part * kScanCols + (tid & 3) * 4;
        float* ydst = reinterpret_cast<float*>(p.ws + (REVERSE ? p.L.dU : p.L.U)) + yoff;
        const float4 yadd = *reinterpret_cast<const float4*>(REVERSE ? ydst : reinterpret_cast<const float*>(p.ws + p.L.Ut) + yoff);
        float4 add[NS];
        float ge[NS];
#pragma unroll
        for (int m = 0; m < NS; ++m) {
            const int e = tid + m * kThreads, r = e >> 2, c = (e & 3) * 4;
            *reinterpret_cast<float4*>(keep + (size_t)r * DV + c) = state[m];
            if (REVERSE) add[m] = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(p.ws + p.L.E) + ch * DK * DV + part * kScanCols + (size_t)r * DV + c);
            ge[m] = VEC ? wsG[(ch * kC + kC - 1) * DK + r] : wsG[ch * kC + kC - 1];
        }
        cp_wait<0>();
        __syncthreads();   // the step's W, Kb and the state are in shared memory; everybody has left the step before
        if (s + 1 < sg.n_chunks) fill(s + 1);
        {   // W h or Kb dh': [64 x 16], the contraction over DK cut into eight
            float acc[8][4];
            zero(acc);
            mac_slice<A_ROW>(acc, REVERSE ? Kb : W, PK, rg, hs, cg, warp * (DK / 8), (warp + 1) * (DK / 8));
#pragma unroll
            for (int x = 0; x < 8; ++x) *reinterpret_cast<float4*>(red + warp * 1024 + (rg + 8 * x) * 16 + 4 * cg) = make_float4(acc[x][0], acc[x][1], acc[x][2], acc[x][3]);
        }
        __syncthreads();
        {
            float4 y = *reinterpret_cast<const float4*>(red + tid * 4);
#pragma unroll
            for (int w = 1; w < 8; ++w) {
                const float4 v = *reinterpret_cast<const float4*>(red + w * 1024 + tid * 4);
                y.x += v.x; y.y += v.y; y.z += v.z; y.w += v.w;
            }
            float4 out;
            if (REVERSE) { out = make_float4(yadd.x + y.x, yadd.y + y.y, yadd.z + y.z, yadd.w + y.w); }
            else { out = make_float4(yadd.x - y.x, yadd.y - y.y, yadd.z - y.z, yadd.w - y.w); y = out; }
            *reinterpret_cast<float4*>(ydst) = out;
            *reinterpret_cast<float4*>(ys + (tid >> 2) * kScanPitch + (tid & 3) * 4) = y;
        }
        __syncthreads();
        {   // Kb^T U or W^T Y: [DK x 16], row blocks of 64, the contraction over the 64 tokens cut into 512 / DK
            constexpr int RB = DK / 64, SPLIT = 8 / RB, KS = kC / SPLIT;
            const int rb = warp % RB, ks = warp / RB;
            float acc[8][4];
            zero(acc);
            mac_slice<A_COL>(acc, (REVERSE ? W : Kb) + rb * 64, PK, rg, ys, cg, ks * KS, (ks + 1) * KS);
#pragma unroll
            for (int x = 0; x < 8; ++x)
                *reinterpret_cast<float4*>(red + ks * DK * 16 + (rb * 64 + 4 * rg + (x & 3) + 32 * (x >> 2)) * 16 + 4 * cg) = make_float4(acc[x][0], acc[x][1], acc[x][2], acc[x][3]);
        }
        __syncthreads();
#pragma unroll
        for (int m = 0; m < NS; ++m) {
            constexpr int SPLIT = 8 / (DK / 64);
            const int e = tid + m * kThreads, r = e >> 2, c = (e & 3) * 4;
            float4 d = *reinterpret_cast<const float4*>(red + e * 4);
#pragma unroll
            for (int w = 1; w < SPLIT; ++w) {
                const float4 v = *reinterpret_cast<const float4*>(red + w * DK * 16 + e * 4);
                d.x += v.x; d.y += v.y; d.z += v.z; d.w += v.w;
            }
            const float G = expf(ge[m]);
            if (REVERSE) d = make_float4(add[m].x - d.x, add[m].y - d.y, add[m].z - d.z, add[m].w - d.w);
            state[m] = make_float4(fmaf(G, state[m].x, d.x), fmaf(G, state[m].y, d.y), fmaf(G, state[m].z, d.z), fmaf(G, state[m].w, d.w));
            *reinterpret_cast<float4*>(hs + r * kScanPitch + c) = state[m];
        }
    }
    float* fin = REVERSE ? p.dh0 : p.hT;
    if (fin) {
#pragma unroll
        for (int m = 0; m < NS; ++m) {
            const int e = tid + m * kThreads, r = e >> 2, c = (e & 3) * 4;
            *reinterpret_cast<float4*>(fin + soff + (size_t)r * DV + c) = state[m];
        }
    }
}

// Block index -> (chain, direction, column slice).  dirs: 0 forward, 1 reverse, 2 both in one launch.
template <int DK, int DV, bool VEC>
__device__ __forceinline__ void scan_block(const Problem& p, int dirs, float* sm, int b) {
    constexpr int PARTS = DV / kScanCols;
    const int part = b % PARTS;
    b /= PARTS;
    const bool reverse = dirs == 2 ? (b & 1) != 0 : dirs == 1;
    const int chain = dirs == 2 ? b >> 1 : b;
    if (reverse) scan_chain<DK, DV, true, VEC>(p, chain, part, sm);
    else scan_chain<DK, DV, false, VEC>(p, chain, part, sm);
}

}  // namespace ffma
}  // namespace
}  // namespace gdn
