// Inter-chunk carries of the FFMA families in low-rank form (fp32), for scalar and for per-channel gates:
//     forward   U = U~ - W h (stored),          h' = Ge h + Kb^T U            (h stored per chunk)
//     reverse   dU = scale P^T dO + Kb dh' (stored),   dh = Ge dh' + E - W^T dU   (dh' stored per chunk; the paper's K#1)
// with Kb the keys scaled to the chunk end (made by the preparation kernel), Ge the decay of the state over the chunk (one
// factor, or one per state row), E = scale (Gam . Q)^T dO, and dU preset to scale P^T dO.  U and dU are what the gradient stage
// needs, so it repeats neither product; and because W^T meets the whole of dU here, E needs neither P nor W.
//
// The chain of chunks is serial, so a step is made short.  The state columns evolve independently and a CTA carries CS of them, in
// passes of at most eight.  A warp owns eight tokens of the chunk: it makes their rows of U or dU (a contraction over the features, split
// over eight lanes and summed by exchanges) and multiplies them into the state at once (over its own eight tokens), so only the sum
// of the eight warps' shares crosses the CTA: two barriers a step.  W and Kb come straight into the registers of the threads
// that use them, each as soon as the step before has used its predecessor; no element of them is wanted twice.
// What bounds a step: the load/store pipe (each element of W and Kb feeds only CS FMAs; 75 % busy at CS = 8) and some 2000 cycles of
// dependent latency.  d_k = 128: 1.6, 2.15 and 3.25 us a step at CS = 4, 8 and 16; with W and Kb staged in shared memory, partial sums
// of both products exchanged there and four barriers 3.6 us at CS = 16 and 2.6 at 8.  2 x 4 heads of 1000 tokens, one direction
// 63.9 -> 38.4 us; 2 heads of 600 tokens, both 42.1 -> 22.4; 64 chains (CS = 16, several waves) 406 -> 396.
#pragma once
#include "ffma_tile.cuh"

namespace gdn {
namespace {
namespace ffma {

__device__ __forceinline__ float lane_of(const float4& v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }
__device__ __forceinline__ void fma4(float4& acc, float a, const float4& b) {
    acc.x = fmaf(a, b.x, acc.x); acc.y = fmaf(a, b.y, acc.y); acc.z = fmaf(a, b.z, acc.z); acc.w = fmaf(a, b.w, acc.w);
}
// N consecutive columns
template <int N>
__device__ __forceinline__ void ld_cols(float (&v)[N], const float* p) {
    if constexpr (N == 4) { const float4 u = *reinterpret_cast<const float4*>(p); v[0] = u.x; v[1] = u.y; v[2] = u.z; v[3] = u.w; }
    else if constexpr (N == 2) { const float2 u = *reinterpret_cast<const float2*>(p); v[0] = u.x; v[1] = u.y; }
    else v[0] = *p;
}
template <int N>
__device__ __forceinline__ void st_cols(float* p, const float (&v)[N]) {
    if constexpr (N == 4) *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    else if constexpr (N == 2) *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
    else *p = v[0];
}

// A [DK x CB] slice of the state, or of a sum that goes into it, in shared memory: [row % 4][row / 4][quad of columns][4], the quads
// of a row permuted so that eight consecutive row / 4 at one quad lie on distinct banks.
template <int DK, int CB>
struct Slice {
    static constexpr int NQ = CB / 4, FLOATS = DK * CB;
    static __device__ __forceinline__ int perm(int l) { return (l * NQ / 8) & (NQ - 1); }
    static __device__ __forceinline__ int at(int x, int l, int q) { return ((x * (DK / 4) + l) * NQ + (q ^ perm(l))) * 4; }
};
template <int DK, int CS>
struct ScanShape {
    static constexpr int CB = CS < 8 ? CS : 8, NP = CS / CB;   // columns of a pass, passes
    static constexpr int GB = 128 / DK;                        // token groups of a warp in the second product: DK / 4 lanes cover a row
    static constexpr int SLICES = kThreads / 32 * GB;          // partial sums of the state's increment
    static constexpr size_t BYTES = sizeof(float) * (NP * (SLICES + 1) * Slice<DK, CB>::FLOATS + kC * CB);
};

// One direction of one chain, columns [part * CS, part * CS + CS) of the state.  VEC: per-channel gates.
template <int DK, int DV, int CS, bool REVERSE, bool VEC>
__device__ __forceinline__ void scan_chain(const Problem& p, int chain, int part, float* sm) {
    using Sh = ScanShape<DK, CS>;
    constexpr int CB = Sh::CB, NP = Sh::NP, GB = Sh::GB, NQ = CB / 4, TB = 8 / GB;
    using Sl = Slice<DK, CB>;
    constexpr int MA = DK / 32;                       // 16-byte pieces of a row per lane in the first product
    constexpr int PW = DK * CB / kThreads;            // consecutive columns of the state that a thread keeps, per pass
    constexpr int YW = CB / 4;                        // ... and of U or dU that a lane sums up
    float* red = sm;                                  // [NP][SLICES] slices
    float* hs = red + NP * Sh::SLICES * Sl::FLOATS;   // [NP] slices: the state
    float* ys = hs + NP * Sl::FLOATS;                 // [64][CB]: U or dU, every warp its own eight rows
    const int H = p.d.H, n = chain / H, hd = chain % H;
    const SeqGeom sg = seq_geom(p, n);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const float* wsW = reinterpret_cast<const float*>(p.ws + p.L.W);
    const float* wsKb = reinterpret_cast<const float*>(p.ws + p.L.Kb);
    const float* wsG = reinterpret_cast<const float*>(p.ws + p.L.gamma);
    const float* wsE = reinterpret_cast<const float*>(p.ws + p.L.E);
    float* wsY = reinterpret_cast<float*>(p.ws + (REVERSE ? p.L.dU : p.L.U));
    const float* wsY0 = REVERSE ? wsY : reinterpret_cast<const float*>(p.ws + p.L.Ut);
    float* wsS = reinterpret_cast<float*>(p.ws + (REVERSE ? p.L.dhn : p.L.hc));
    auto chunk_head = [&](int s) { return (size_t)(REVERSE ? sg.c0 + sg.n_chunks - 1 - s : sg.c0 + s) * H + hd; };

    // first product: lane = (piece kk, token pair g); features 4 (kk + 8 m) .., tokens 8 warp + 2 g and the next
    const int kk = lane >> 2, g = lane & 3;
    float4 a[2][MA];
    auto load_a = [&](int s) {
        const float* src = (REVERSE ? wsKb : wsW) + (chunk_head(s) * kC + warp * 8 + 2 * g) * DK + 4 * kk;
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int m = 0; m < MA; ++m) a[r][m] = ld4(src + r * DK + 32 * m);
    };
    // second product: lane = (token group gb, features 4 lb ..)
    const int lb = lane % (DK / 4), gb = lane / (DK / 4);
    float4 b[TB];
    auto load_b = [&](int s) {
        const float* src = (REVERSE ? wsW : wsKb) + (chunk_head(s) * kC + warp * 8 + gb * TB) * DK + 4 * lb;
#pragma unroll
        for (int t = 0; t < TB; ++t) b[t] = ld4(src + t * DK);
    };
    // after the exchanges of the first product this lane holds YW columns of one token
    const int yrow = warp * 8 + 2 * g + (kk >> 2), ycol = (kk & 3) * YW;
    float yadd[NP][YW];
    // this thread's PW entries of the state's slice: row 4 sl + sx, columns scol ..
    const int slot = tid * PW / 4, sx = slot / (NQ * (DK / 4)), sl = slot / NQ % (DK / 4);
    const int srow = 4 * sl + sx, scol = 4 * ((slot % NQ) ^ Sl::perm(sl)) + tid * PW % 4;
    float state[NP][PW], add[NP][PW], ge = 0.f;
    auto load_yadd = [&](int s, int u) { ld_cols(yadd[u], wsY0 + (chunk_head(s) * kC + yrow) * DV + part * CS + u * CB + ycol); };
    auto load_add = [&](int s) {
        const size_t ch = chunk_head(s);
        ge = VEC ? wsG[(ch * kC + kC - 1) * DK + srow] : wsG[ch * kC + kC - 1];
        if (REVERSE)
#pragma unroll
            for (int u = 0; u < NP; ++u) ld_cols(add[u], wsE + (ch * DK + srow) * DV + part * CS + u * CB + scol);
    };
    if (sg.n_chunks > 0) {
        load_a(0); load_b(0); load_add(0);
#pragma unroll
        for (int u = 0; u < NP; ++u) load_yadd(0, u);
    }
    const float* init = REVERSE ? p.dhT : p.h0;
    const size_t soff = ((size_t)chain * DK + srow) * DV + part * CS + scol;
#pragma unroll
    for (int u = 0; u < NP; ++u) {
        if (init) ld_cols(state[u], init + soff + u * CB);
        else
#pragma unroll
            for (int c = 0; c < PW; ++c) state[u][c] = 0.f;
        st_cols(hs + u * Sl::FLOATS + tid * PW, state[u]);
    }
    __syncthreads();
#pragma unroll 1
    for (int s = 0; s < sg.n_chunks; ++s) {
        const size_t ch = chunk_head(s);
        const bool more = s + 1 < sg.n_chunks;
#pragma unroll
        for (int u = 0; u < NP; ++u) st_cols(wsS + (ch * DK + srow) * DV + part * CS + u * CB + scol, state[u]);   // the state that enters the chunk
#pragma unroll
        for (int u = 0; u < NP; ++u) {
            {   // W h or Kb dh'
                float acc[2 * CB] = {};
                const float* hsu = hs + u * Sl::FLOATS;
                constexpr bool AHEAD = DK == 128;   // the next piece's rows of the state arrive under the current one's products (d_k = 64: 3 % slower)
                float4 h[2][4][NQ];
                auto load_h = [&](int m) {
#pragma unroll
                    for (int z = 0; z < 4; ++z)
#pragma unroll
                        for (int q = 0; q < NQ; ++q) h[m & 1][z][q] = *reinterpret_cast<const float4*>(hsu + Sl::at(z, kk + 8 * m, q));
                };
                if (AHEAD) load_h(0);
#pragma unroll
                for (int m = 0; m < MA; ++m) {
                    if (!AHEAD) load_h(m);
                    else if (m + 1 < MA) load_h(m + 1);
#pragma unroll
                    for (int z = 0; z < 4; ++z)
#pragma unroll
                        for (int r = 0; r < 2; ++r) {
                            const float w = lane_of(a[r][m], z);
#pragma unroll
                            for (int q = 0; q < NQ; ++q) {
                                const float4 v = h[m & 1][z][q];
                                float* c = acc + r * CB + 4 * q;
                                c[0] = fmaf(w, v.x, c[0]); c[1] = fmaf(w, v.y, c[1]); c[2] = fmaf(w, v.z, c[2]); c[3] = fmaf(w, v.w, c[3]);
                            }
                        }
                }
                // sum over kk: at each exchange a lane keeps the half of the values that its bit of kk selects
#pragma unroll
                for (int half = CB; half >= YW; half /= 2) {
                    const int o = 16 * half / CB;   // 16, 8, 4: bits 2, 1, 0 of kk
                    const bool hi = lane & o;
#pragma unroll
                    for (int i = 0; i < half; ++i) {
                        const float send = hi ? acc[i] : acc[half + i], keep = hi ? acc[half + i] : acc[i];
                        acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                    }
                }
                float y[YW];
#pragma unroll
                for (int c = 0; c < YW; ++c) y[c] = REVERSE ? yadd[u][c] + acc[c] : yadd[u][c] - acc[c];
                st_cols(wsY + (ch * kC + yrow) * DV + part * CS + u * CB + ycol, y);
                st_cols(ys + yrow * CB + ycol, y);
            }
            if (more) load_yadd(s + 1, u);
            if (more && u == NP - 1) load_a(s + 1);
            __syncwarp();
            {   // Kb^T U or W^T dU
                float4 acc[4][NQ] = {};
#pragma unroll
                for (int t = 0; t < TB; ++t)
#pragma unroll
                    for (int q = 0; q < NQ; ++q) {
                        const float4 v = *reinterpret_cast<const float4*>(ys + (warp * 8 + gb * TB + t) * CB + 4 * q);
#pragma unroll
                        for (int x = 0; x < 4; ++x) fma4(acc[x][q], lane_of(b[t], x), v);
                    }
                float* dst = red + (u * Sh::SLICES + warp * GB + gb) * Sl::FLOATS;
#pragma unroll
                for (int x = 0; x < 4; ++x)
#pragma unroll
                    for (int q = 0; q < NQ; ++q) *reinterpret_cast<float4*>(dst + Sl::at(x, lb, q)) = acc[x][q];
            }
            __syncwarp();   // (the next pass rewrites this warp's rows of ys)
        }
        if (more) load_b(s + 1);
        const float G = expf(ge);
        __syncthreads();
#pragma unroll
        for (int u = 0; u < NP; ++u) {
            const float* src = red + u * Sh::SLICES * Sl::FLOATS + tid * PW;
            float v[Sh::SLICES][PW];   // summed in pairs
#pragma unroll
            for (int w = 0; w < Sh::SLICES; ++w) ld_cols(v[w], src + w * Sl::FLOATS);
#pragma unroll
            for (int h = Sh::SLICES / 2; h > 0; h /= 2)
#pragma unroll
                for (int w = 0; w < h; ++w)
#pragma unroll
                    for (int c = 0; c < PW; ++c) v[w][c] += v[w + h][c];
            const float (&d)[PW] = v[0];
#pragma unroll
            for (int c = 0; c < PW; ++c) state[u][c] = fmaf(G, state[u][c], REVERSE ? add[u][c] - d[c] : d[c]);
            st_cols(hs + u * Sl::FLOATS + tid * PW, state[u]);
        }
        if (more) load_add(s + 1);
        __syncthreads();
    }
    float* fin = REVERSE ? p.dh0 : p.hT;
    if (fin)
#pragma unroll
        for (int u = 0; u < NP; ++u) st_cols(fin + soff + u * CB, state[u]);
}

// Block index -> (chain, direction, column slice).  dirs: 0 forward, 1 reverse, 2 both in one launch.
template <int DK, int DV, int CS, bool VEC>
__device__ __forceinline__ void scan_block(const Problem& p, int dirs, float* sm, int b) {
    constexpr int PARTS = DV / CS;
    const int part = b % PARTS;
    b /= PARTS;
    const bool reverse = dirs == 2 ? (b & 1) != 0 : dirs == 1;
    const int chain = dirs == 2 ? b >> 1 : b;
    if (reverse) scan_chain<DK, DV, CS, true, VEC>(p, chain, part, sm);
    else scan_chain<DK, DV, CS, false, VEC>(p, chain, part, sm);
}

// Columns per CTA: as few as fit the SMs at one CTA each (a step costs 2000 cycles and 270 a column, so narrow slices pay as long as they
// run side by side, and no longer: 2 x 8 heads of 1000 tokens, d_k = d_v = 128, forward 57 us at 16 (128 CTAs), 70 at 8 (256 CTAs)).
__host__ __device__ inline int scan_blocks(const Problem& p, int dirs, int cs) { return p.d.N * p.d.H * (dirs == 2 ? 2 : 1) * (p.d.d_v / cs); }
inline int scan_columns(const Problem& p, int dirs) {
    for (int cs = 4; cs < 16; cs *= 2)
        if (scan_blocks(p, dirs, cs) <= tc_sm_count()) return cs;
    return 16;
}

}  // namespace ffma
}  // namespace
}  // namespace gdn
