// fp32 FFMA kernels for the GDN backward: the arithmetic path of the fp32 dtype (tolerance 1e-4 rules
// out tf32/bf16 operands) and a plain-CUDA-core statement of every stage of the chunked method.
//
// Stage map (Section 4.2 of the paper; names follow the library header):
//   table  : chunk table from cu_seqlens (packed sequences only)
//   prep   : gamma = cumsum(g); A = stril(Diag(b)(K K^T . D)); P = tril(Q K^T . D); T = (I + A)^-1; W = T Diag(b Gam) K;
//            Ut = T Diag(w) V; Kb = Diag(exp(gam_e - gam)) K; and for the backward
//            dU0 = scale P^T dO, E = scale (Diag(Gam) Q)^T dO (alone on a workspace fresh from the forward)
//   scan   : h' = Gam_e h + Kb^T U with U = Ut - W h, and dh = Gam_e dh' + E - W^T dU with dU = dU0 + Kb dh' (the paper's
//            K#1), both directions in one launch when both are wanted (ffma_scan.cuh)
//   intra  : all token gradients of a chunk, including the VJP of the triangular solve (the paper's K#2)
//   out    : forward output
// One CTA handles one (chunk, head) in the parallel stages.  Operands are staged in shared memory, products are register
// tiles (ffma_tile.cuh).  Every reduction has a fixed order: results are bit-identical from run to run.
// At d = 128 the gradient stage of a chunk-head is 5.6 M FMAs, 23 us at the rate of one SM; measured 58 us (forward preparation
// 27 us, the backward's share of it 22 us): eight warps on an SM issue in half of the cycles, between barriers.  With the operands of every FMA read from
// global memory, and the solve and the sums over a chunk done by single threads, the same stages took 907, 165 and 102 us
// (2 x 4 heads of 1000 tokens); the smallest call, 2 heads of 128 tokens at d = 64, went from 370 to 35 us.
#include <cooperative_groups.h>

#include "ffma_scan.cuh"

namespace gdn {
namespace {

namespace cg = cooperative_groups;
using namespace ffma;

// ------------------------------------------------------------------------------------------------
// Chunk table.  One block.  Validates cu_seqlens; on failure records the status and leaves no work.  In a backward on the
// forward's workspace (fresh) an error that the forward left stands: nothing is to be computed from what it left.
// ------------------------------------------------------------------------------------------------
__global__ void table_kernel(Problem p, int fresh) {
    wait_prerequisites();
    WsHeader* hdr = reinterpret_cast<WsHeader*>(p.ws);
    int32_t* seq_first = reinterpret_cast<int32_t*>(p.ws + p.L.seq_first);
    int32_t* seq_tok0 = reinterpret_cast<int32_t*>(p.ws + p.L.seq_tok0);
    int32_t* chunk_tok0 = reinterpret_cast<int32_t*>(p.ws + p.L.chunk_tok0);
    int32_t* chunk_len = reinterpret_cast<int32_t*>(p.ws + p.L.chunk_len);
    const int N = p.d.N;
    __shared__ int ok;
    auto cu = [&](int n) -> long long { return p.cu ? (long long)p.cu[n] : (long long)n * p.d.T; };
    // (all threads: the loads of the one that goes through the sequences below then find them in the cache)
    if (p.Ttot > 0)
        for (int n = threadIdx.x; n <= N; n += blockDim.x) seq_tok0[n] = (int)cu(n);
    if (threadIdx.x == 0 && fresh && hdr->status != GDN_OK && !status_from_fresh(hdr)) {
        ok = 0;
    } else if (threadIdx.x == 0) {
        int good = 1, bad_at = -1;
        if (cu(0) != 0) { good = 0; bad_at = 0; }
        int acc = 0;
        for (int n = 0; n < N && good; ++n) {
            const long long a = cu(n), e = cu(n + 1);
            if (e < a || e > p.Ttot) { good = 0; bad_at = n + 1; break; }
            seq_first[n] = acc;
            acc += (int)((e - a + kC - 1) / kC);
        }
        if (good && cu(N) != p.Ttot) { good = 0; bad_at = N; }
        if (!fresh) hdr->cw_fallback = 0;
        if (!fresh) hdr->seqlens_ok = good;
        if (good) {
            seq_first[N] = acc;
            hdr->status = GDN_OK;
            hdr->n_chunks = acc;
            hdr->detail = 0;
        } else {
            for (int n = 0; n <= N; ++n) seq_first[n] = 0;
            hdr->status = GDN_ERR_BAD_SEQLENS;
            hdr->n_chunks = 0;
            hdr->detail = bad_at;
        }
        ok = good;
    }
    __syncthreads();
    if (!ok) return;
    const int nch = seq_first[N];
    for (int c = threadIdx.x; c < nch; c += blockDim.x) {
        int lo = 0, hi = N - 1;  // last n with seq_first[n] <= c and a non-empty chunk range
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (seq_first[mid] <= c) lo = mid; else hi = mid - 1;
        }
        const int n = lo;
        const long long a = cu(n), e = cu(n + 1);
        const long long t0 = a + (long long)(c - seq_first[n]) * kC;
        chunk_tok0[c] = (int)t0;
        chunk_len[c] = (int)((e - t0) < kC ? (e - t0) : kC);
    }
}

// One (chunk, head) of the grid; false when there is none or an earlier stage has failed.
__device__ __forceinline__ bool chunk_head(const Problem& p, ChunkInfo& x) {
    return reinterpret_cast<const WsHeader*>(p.ws)->status == GDN_OK && chunk_info(p, x);
}

// Gate arrays of a chunk in shared memory, made by warp 0: lane l owns tokens l and l + 32.
struct Gates {
    float gam[kC], Gam[kC], ee[kC];   // cumulative log decay, its exponential, exp(gam_e - gam)
    float bb[kC], ww[kC];             // erase and write gate (0 beyond the sequence)
};
__device__ __forceinline__ void finish_gates(Gates& s, int lane, float a, float b, float gend) {
    s.gam[lane] = a; s.gam[lane + 32] = b;
    s.Gam[lane] = expf(a); s.Gam[lane + 32] = expf(b);
    s.ee[lane] = expf(gend - a); s.ee[lane + 32] = expf(gend - b);
}
__device__ __forceinline__ void load_erase_write(const Problem& p, const ChunkInfo& x, Gates& s, int lane) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int i = lane + 32 * h;
        const bool live = i < x.len;
        const float beta = live && p.d.delta_rule ? p.beta[(size_t)(x.tok0 + i) * p.d.H + x.hd] : 0.f;
        s.bb[i] = beta;
        s.ww[i] = p.d.delta_rule ? beta : (live ? 1.f : 0.f);
    }
}
// ... from the log decays: inclusive sums over the chunk; gam goes to the workspace for the other stages.
__device__ __forceinline__ void make_gates(const Problem& p, const ChunkInfo& x, Gates& s, float* wsG) {
    const int lane = threadIdx.x;
    auto g = [&](int i) { return i < x.len ? p.g[(size_t)(x.tok0 + i) * p.d.H + x.hd] : 0.f; };
    float a = g(lane), b = g(lane + 32);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float ua = __shfl_up_sync(0xffffffffu, a, o), ub = __shfl_up_sync(0xffffffffu, b, o);
        if (lane >= o) { a += ua; b += ub; }
    }
    b += __shfl_sync(0xffffffffu, a, 31);
    const float gend = __shfl_sync(0xffffffffu, b, 31);
    if (wsG) { wsG[lane] = a; wsG[lane + 32] = b; }
    finish_gates(s, lane, a, b, gend);
    load_erase_write(p, x, s, lane);
}
// ... from the stored gam.
__device__ __forceinline__ void load_gates(const Problem& p, const ChunkInfo& x, Gates& s, const float* wsG) {
    finish_gates(s, threadIdx.x, wsG[threadIdx.x], wsG[threadIdx.x + 32], wsG[kC - 1]);
    load_erase_write(p, x, s, threadIdx.x);
}

// ------------------------------------------------------------------------------------------------
// prep
//
// Two chains of steps that share only Q, K and the gates: A -> T -> W, U~, and P -> dU0, E.  One CTA takes both (Q K^T and K K^T in one
// pass over K), or, when that leaves half of the SMs idle, two CTAs one each (prep_parts).
// ------------------------------------------------------------------------------------------------
template <int DK, int DV>
constexpr size_t prep_smem() { return sizeof(float) * (kC * (2 * pitch(DK) + 2 * pitch(DV)) + 4 * kC * kPc); }

template <typename IO, int DK, int DV>
__global__ void __launch_bounds__(kThreads, 1) prep_kernel(Problem p, int mode, int parts) {
    wait_prerequisites();
    const int item = parts == 2 ? blockIdx.x >> 1 : blockIdx.x;
    const bool fwd = mode != PREP_BWD;
    const bool solve = fwd && (parts == 1 || (blockIdx.x & 1) == 0);           // A, T, W, U~
    const bool readout = parts == 1 || (blockIdx.x & 1) == 1;                  // P, Kb; with a backward dU0, E
    const bool bwd = mode != PREP_FWD && readout;
    if (fwd) init_header_if_untabled(p); else check_fresh_seqlens(p);   // (the backward's part alone: the status word is the forward's)
    ChunkInfo x;
    if (!chunk_info(p, x, item)) return;   // (no chunk at all when the table was refused)
    constexpr int PK = pitch(DK), PV = pitch(DV);
    extern __shared__ __align__(16) float sm[];
    float* sK = sm;                  // K
    float* sQ = sK + kC * PK;        // Q, then Diag(Gam) Q
    float* sV = sQ + kC * PK;        // V
    float* sO = sV + kC * PV;        // dO
    float* A = sO + kC * PV;         // A, then T Diag(w)
    float* T = A + kC * kPc;
    float* S = T + kC * kPc;         // T Diag(b Gam)
    float* Pm = S + kC * kPc;
    __shared__ Gates gs;
    const int H = p.d.H, tid = threadIdx.x;
    const Thread t;
    const Out<DK> ok(t);
    const Out<DV> ov(t);
    const size_t rk = (size_t)H * DK, rv = (size_t)H * DV;
    float* wsG = block_of(p, p.L.gamma, x.ch, kC);
    float* wsP = block_of(p, p.L.Pm, x.ch, kC * kC);
    const float sc = p.d.scale;

    if (readout) load_rows<DK>(sQ, rows_of<IO>(p.q, x, H, DK), rk, x.len);
    if (fwd) load_rows<DK>(sK, rows_of<IO>(p.k, x, H, DK), rk, x.len);
    cp_commit();
    if (solve) load_rows<DV>(sV, rows_of<IO>(p.v, x, H, DV), rv, x.len);
    if (!fwd) load_block<kC, kC>(Pm, wsP);
    if (bwd) load_rows<DV>(sO, rows_of<IO>(p.dO, x, H, DV), rv, x.len);
    cp_commit();
    if (tid < 32) { if (fwd) make_gates(p, x, gs, readout ? wsG : nullptr); else load_gates(p, x, gs, wsG); }
    if (fwd) {
        cp_wait<1>();
        __syncthreads();
        // P = tril(Q K^T . D) and A = stril(Diag(b)(K K^T . D)); the decay exponent is only evaluated where j <= i (non-positive)
        {
            float acc[8][4];
            zero(acc);
            if (parts == 1) mac<2, A_ROW, B_ROW>(acc, sQ, sK, PK, t.rn, sK, PK, t.cn, 0, DK);
            else if ((tid >> 7) * 32 <= (t.rn >> 4) * 16 + 15) {   // (warps whose block lies above the diagonal have nothing to add up)
                float one[4][4];
                zero(one);
                mac<1, A_ROW, B_ROW>(one, solve ? sK : sQ, nullptr, PK, t.rn, sK, PK, t.cn, 0, DK);
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int y = 0; y < 4; ++y) acc[r][y] = acc[4 + r][y] = one[r][y];
            }
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int y = 0; y < 4; ++y) {
                    const int i = t.rn + r, j = t.cn + 8 * y;
                    const float D = j <= i ? expf(gs.gam[i] - gs.gam[j]) : 0.f;
                    if (readout) {
                        const float P_ = j <= i ? acc[r][y] * D : 0.f;
                        Pm[i * kPc + j] = P_;
                        wsP[i * kC + j] = P_;
                    }
                    if (solve) A[i * kPc + j] = j < i ? gs.bb[i] * acc[4 + r][y] * D : 0.f;
                }
        }
        if (readout) {   // Kb = Diag(exp(gam_e - gam)) K, for the carries
            float* wsKb = block_of(p, p.L.Kb, x.ch, kC * DK);
            for (int e = tid; e < kC * DK / 4; e += kThreads) {
                const int i = e / (DK / 4), c = (e % (DK / 4)) * 4;
                float4 k = ld4(sK + i * PK + c);
                const float w = gs.ee[i];
                *reinterpret_cast<float4*>(wsKb + (size_t)e * 4) = make_float4(w * k.x, w * k.y, w * k.z, w * k.w);
            }
        }
        __syncthreads();
    }
    if (solve) {
        invert(A, T);
        cp_wait<0>();
        __syncthreads();
        float* wsT = block_of(p, p.L.Tm, x.ch, kC * kC);
        for (int e = tid; e < kC * kC; e += kThreads) {
            const int i = e / kC, j = e % kC;
            const float v = T[i * kPc + j];
            wsT[e] = v;
            S[i * kPc + j] = v * gs.bb[j] * gs.Gam[j];
            A[i * kPc + j] = v * gs.ww[j];
        }
        __syncthreads();
        // Ut = T Diag(w) V, W = T Diag(b Gam) K
        float* wsU = block_of(p, p.L.Ut, x.ch, kC * DV);
        {
            float acc[Out<DV>::R][4];
            tri_product<DV, A_ROW, A_LOWER>(t, A, sV, PV, acc);
#pragma unroll
            for (int r = 0; r < Out<DV>::R; ++r)
#pragma unroll
                for (int y = 0; y < 4; ++y) wsU[ov.row(r) * DV + ov.c + 8 * y] = acc[r][y];
        }
        float* wsW = block_of(p, p.L.W, x.ch, kC * DK);
        {
            float acc[Out<DK>::R][4];
            tri_product<DK, A_ROW, A_LOWER>(t, S, sK, PK, acc);
#pragma unroll
            for (int r = 0; r < Out<DK>::R; ++r)
#pragma unroll
                for (int y = 0; y < 4; ++y) wsW[ok.row(r) * DK + ok.c + 8 * y] = acc[r][y];
        }
    }
    if (!bwd) return;
    if (!solve) {
        cp_wait<0>();
        __syncthreads();
    }
    for (int e = tid; e < kC * DK / 4; e += kThreads) {   // Diag(Gam) Q, in place
        const int i = e / (DK / 4);
        float4* q = reinterpret_cast<float4*>(sQ + i * PK + (e % (DK / 4)) * 4);
        const float4 v = *q;
        const float G = gs.Gam[i];
        *q = make_float4(G * v.x, G * v.y, G * v.z, G * v.w);
    }
    // dU0 = scale P^T dO
    float* wsD = block_of(p, p.L.dU, x.ch, kC * DV);
    {
        float acc[Out<DV>::R][4];
        tri_product<DV, A_COL, A_UPPER, kU<DK>>(t, Pm, sO, PV, acc);
#pragma unroll
        for (int r = 0; r < Out<DV>::R; ++r)
#pragma unroll
            for (int y = 0; y < 4; ++y) wsD[ov.row(r) * DV + ov.c + 8 * y] = sc * acc[r][y];
    }
    __syncthreads();
    // E = scale (Diag(Gam) Q)^T dO, 64 rows at a time
    float* wsE = block_of(p, p.L.E, x.ch, DK * DV);
#pragma unroll 1
    for (int r0 = 0; r0 < DK; r0 += 64) {
        float acc[Out<DV>::R][4];
        zero(acc);
        mac<Out<DV>::R / 4, A_COL, B_COL>(acc, sQ + r0, sQ + r0 + 32, PK, ov.r0, sO, PV, ov.c, 0, kC);
#pragma unroll
        for (int r = 0; r < Out<DV>::R; ++r)
#pragma unroll
            for (int y = 0; y < 4; ++y) wsE[(r0 + ov.row(r)) * DV + ov.c + 8 * y] = sc * acc[r][y];
    }
}

// ------------------------------------------------------------------------------------------------
// Forward and reverse carries (ffma_scan.cuh).
// ------------------------------------------------------------------------------------------------
template <int DK, int DV, int CS>
__global__ void __launch_bounds__(kThreads, DK == 64 ? 2 : 1) scan_kernel(const __grid_constant__ Problem p, int dirs) {
    wait_prerequisites();
    extern __shared__ __align__(16) float sm[];
    if (reinterpret_cast<const WsHeader*>(p.ws)->status != GDN_OK) return;
    scan_block<DK, DV, CS, false>(p, dirs, sm, (int)blockIdx.x);
}

// ------------------------------------------------------------------------------------------------
// Forward output (optional): o = scale (Diag(Gam) Q h + P U)
// ------------------------------------------------------------------------------------------------
template <int DK, int DV>
constexpr size_t out_smem() { return sizeof(float) * (kC * pitch(DK) + DK * pitch(DV) + kC * pitch(DV) + kC * kPc); }

template <typename IO, int DK, int DV>
__global__ void __launch_bounds__(kThreads, 1) out_kernel(Problem p) {
    wait_prerequisites();
    ChunkInfo x;
    if (!chunk_head(p, x)) return;
    constexpr int PK = pitch(DK), PV = pitch(DV);
    extern __shared__ __align__(16) float sm[];
    float* sQ = sm;
    float* sH = sQ + kC * PK;
    float* sU = sH + DK * PV;
    float* Pm = sU + kC * PV;
    const int H = p.d.H;
    const Thread t;
    load_rows<DK>(sQ, rows_of<IO>(p.q, x, H, DK), (size_t)H * DK, x.len);
    load_block<DK, DV>(sH, block_of(p, p.L.hc, x.ch, DK * DV));
    cp_commit();
    load_block<kC, DV>(sU, block_of(p, p.L.U, x.ch, kC * DV));
    load_block<kC, kC>(Pm, block_of(p, p.L.Pm, x.ch, kC * kC));
    cp_commit();
    const float* wsG = block_of(p, p.L.gamma, x.ch, kC);
    IO* op = rows_of<IO>(p.o, x, H, DV);
    const size_t rv = (size_t)H * DV;
    const float sc = p.d.scale;
    cp_wait<1>();
    __syncthreads();
    const Out<DV> o(t);
    constexpr int R = Out<DV>::R;
    float acc[R][4];
    zero(acc);
    mac<R / 4, A_ROW, B_COL>(acc, sQ, sQ + 32 * PK, PK, o.r0, sH, PV, o.c, 0, DK);
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const float G = expf(wsG[o.row(r)]);
#pragma unroll
        for (int y = 0; y < 4; ++y) acc[r][y] *= G;
    }
    cp_wait<0>();
    __syncthreads();
    mac<R / 4, A_ROW, B_COL>(acc, Pm, Pm + 32 * kPc, kPc, o.r0, sU, PV, o.c, 0, kC);
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (o.row(r) < x.len)
#pragma unroll
            for (int y = 0; y < 4; ++y) stf(op + o.row(r) * rv + o.c + 8 * y, sc * acc[r][y]);
}

// ------------------------------------------------------------------------------------------------
// intra: token gradients of one (chunk, head).
//
// The solve's VJP (K#2) in its short form: dXv = T^T dU, dXk = -dXv h^T, dA = -stril(dXv U^T).  With dPD = scale
// tril(dO U^T) . D and G = dA . D:
//     dq = scale Gam (dO h^T) + dPD K        dk^row = G K + Gam dXk       dv = w dXv
//     dk = b dk^row + dk^col                 dk^col = e (U dh'^T) + dPD^T Q + (b G)^T K
//     dgam_i = <q, dq> + b <k, dk^row> - <k, dk^col>, and the last row adds sum_j e_j <k_j, (U dh'^T)_j> + Gam_e <dh', h>
// dPD, G and dXv are made once; dq and dk then in passes of 64 channels over the slices of h, dh', K and Q that these need (at d_v = 128
// dh' comes over h, for the tiles do not fit beside each other).  The passes are a rolled loop: a CTA goes through the code once, and at
// d = 128 what it waits for most is instructions.
// ------------------------------------------------------------------------------------------------
template <int DK, int DV>
struct IntraTiles {
    static constexpr int PV = pitch(DV);
    static constexpr int O = 0;                  // dO
    static constexpr int X = O + kC * PV;        // dU, then dXv
    static constexpr int U = X + kC * PV;
    static constexpr int T = U + kC * PV;        // T, then G
    static constexpr int B = T + kC * kPc;       // Diag(b) G
    static constexpr int P = B + kC * kPc;       // dPD
    static constexpr int K = P + kC * kPc;       // slices of 64 channels
    static constexpr int Q = K + kC * kPc;
    static constexpr int H = Q + kC * kPc;       // h
    static constexpr bool OWN = DV == 64;        // dh' has a tile of its own
    static constexpr int D = OWN ? H + 64 * PV : H;
    static constexpr size_t BYTES = sizeof(float) * (D + 64 * PV);
};

// dg_j = sum_{i >= j} dgam_i, by warp 0: lane l owns tokens l and l + 32; `end` is the chunk-end term.
__device__ __forceinline__ void write_dg(const Problem& p, const ChunkInfo& x, const float* dgam, float end) {
    const int lane = threadIdx.x;
    float a = dgam[lane], b = dgam[lane + 32] + (lane == 31 ? end : 0.f);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float ta = __shfl_down_sync(0xffffffffu, a, o), tb = __shfl_down_sync(0xffffffffu, b, o);
        if (lane + o < 32) { a += ta; b += tb; }
    }
    a += __shfl_sync(0xffffffffu, b, 0);
    float* dg = p.dg + (size_t)x.tok0 * p.d.H + x.hd;
    if (lane < x.len) dg[(size_t)lane * p.d.H] = a;
    if (lane + 32 < x.len) dg[(size_t)(lane + 32) * p.d.H] = b;
}

// dPD, G and Diag(b) G, dXv (and with it, if `values`, dv and <v, dXv>), from the first two groups of loads; two more groups are under way behind them.
template <typename IO, int DV>
__device__ __forceinline__ void intra_factors(const Problem& p, const ChunkInfo& x, const Thread& t, const Gates& gs, const float* sO, float* sX,
                                              const float* sU, float* sT, float* sB, float* sP, float (*dot_v)[kC], bool values) {
    constexpr int PV = pitch(DV);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const size_t rv = (size_t)p.d.H * DV;
    const float sc = p.d.scale;
    cp_wait<3>();
    __syncthreads();
    // 64 x 64 matrices: warps whose 16 x 32 block lies above the diagonal have nothing to add up
    const bool below = (warp >> 2) * 32 <= (t.rn >> 4) * 16 + 15;
    {   // dPD = scale tril(dO U^T) . D; the decay exponent is only evaluated where it is non-positive
        float acc[4][4];
        zero(acc);
        if (below) mac<1, A_ROW, B_ROW>(acc, sO, nullptr, PV, t.rn, sU, PV, t.cn, 0, DV);
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int y = 0; y < 4; ++y) {
                const int i = t.rn + r, j = t.cn + 8 * y;
                sP[i * kPc + j] = j <= i ? sc * acc[r][y] * expf(gs.gam[i] - gs.gam[j]) : 0.f;
            }
    }
    cp_wait<2>();
    __syncthreads();
    {   // dXv = T^T dU, in place; dv = w dXv; <v, dXv>
        const Out<DV> o(t);
        constexpr int R = Out<DV>::R;
        float acc[R][4], vv[R][4];
        const IO* vp = rows_of<IO>(p.v, x, p.d.H, DV);
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int y = 0; y < 4; ++y) vv[r][y] = values && o.row(r) < x.len ? ldf(vp + o.row(r) * rv + o.c + 8 * y) : 0.f;
        tri_product<DV, A_COL, A_UPPER>(t, sT, sX, PV, acc);
        __syncthreads();
        IO* dvp = rows_of<IO>(p.dv, x, p.d.H, DV);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int i = o.row(r);
            const float w = gs.ww[i];
            float dot = 0.f;
#pragma unroll
            for (int y = 0; y < 4; ++y) {
                sX[i * PV + o.c + 8 * y] = acc[r][y];
                dot = fmaf(vv[r][y], acc[r][y], dot);
                if (values && i < x.len) stf(dvp + i * rv + o.c + 8 * y, w * acc[r][y]);
            }
            dot = row_sum8(dot);
            if ((lane & 7) == 0) dot_v[DV == 128 ? warp >> 1 : warp >> 2][i] = dot;
        }
    }
    __syncthreads();
    {   // G = -stril(dXv U^T) . D and Diag(b) G (over T)
        float acc[4][4];
        zero(acc);
        if (below) mac<1, A_ROW, B_ROW>(acc, sX, nullptr, PV, t.rn, sU, PV, t.cn, 0, DV);
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int y = 0; y < 4; ++y) {
                const int i = t.rn + r, j = t.cn + 8 * y;
                const float g = j < i ? -acc[r][y] * expf(gs.gam[i] - gs.gam[j]) : 0.f;
                sT[i * kPc + j] = g;
                sB[i * kPc + j] = gs.bb[i] * g;
            }
    }
}

template <typename IO, int DK, int DV>
__global__ void __launch_bounds__(kThreads, 1) intra_kernel(Problem p) {
    wait_prerequisites();
    ChunkInfo x;
    if (!chunk_head(p, x)) return;
    using L = IntraTiles<DK, DV>;
    constexpr int PV = pitch(DV), NH = DK / 64;
    extern __shared__ __align__(16) float sm[];
    float *sO = sm + L::O, *sX = sm + L::X, *sU = sm + L::U, *sT = sm + L::T, *sB = sm + L::B, *sP = sm + L::P, *sK = sm + L::K, *sQ = sm + L::Q,
          *sH = sm + L::H, *sD = sm + L::D;
    __shared__ Gates gs;
    __shared__ float red[4][4][kC];  // row dots <q, dq>, <k, dk^row>, <k, dk^col>, <v, dXv>: [which][column block][row]
    __shared__ float dgam[kC], part[2][kThreads / 32];
    const int H = p.d.H, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const Thread t;
    const size_t rk = (size_t)H * DK, rv = (size_t)H * DV;
    const float sc = p.d.scale;
    const float* wsH = block_of(p, p.L.hc, x.ch, DK * DV);
    const float* wsD = block_of(p, p.L.dhn, x.ch, DK * DV);
    const IO* qp = rows_of<IO>(p.q, x, H, DK);
    const IO* kp = rows_of<IO>(p.k, x, H, DK);

    load_rows<DV>(sO, rows_of<IO>(p.dO, x, H, DV), rv, x.len);
    load_block<kC, DV>(sU, block_of(p, p.L.U, x.ch, kC * DV));
    cp_commit();
    load_block<kC, DV>(sX, block_of(p, p.L.dU, x.ch, kC * DV));
    load_block<kC, kC>(sT, block_of(p, p.L.Tm, x.ch, kC * kC));
    cp_commit();
    load_block<64, DV>(sH, wsH);
    cp_commit();
    load_rows<64>(sK, kp, rk, x.len);
    load_rows<64>(sQ, qp, rk, x.len);
    if (L::OWN) load_block<64, DV>(sD, wsD);
    cp_commit();
    if (tid < 32) load_gates(p, x, gs, block_of(p, p.L.gamma, x.ch, kC));
    intra_factors<IO, DV>(p, x, t, gs, sO, sX, sU, sT, sB, sP, red[3], true);
    const int w16 = (t.rn >> 4) * 16;
    float rsum = 0.f, hh = 0.f, dqq[4] = {}, drow[4] = {}, dcol[4] = {};
#pragma unroll 1
    for (int n = 0; n < NH; ++n) {
        // [dO; dXv] h^T: rows 0..3 become dq, rows 4..7 dk^row
        float acc[8][4], col[4][4];
        zero(acc);
        zero(col);
        if (n || !L::OWN) cp_wait<0>(); else cp_wait<1>();   // (the first slice of K and Q may still be under way; see below)
        __syncthreads();
        mac<2, A_ROW, B_ROW>(acc, sO, sX, PV, t.rn, sH, PV, t.cn, 0, DV);
        float4 h4[64 * DV / 4 / kThreads];
#pragma unroll
        for (int m = 0; m < 64 * DV / 4 / kThreads; ++m) h4[m] = ld4(wsH + (size_t)n * 64 * DV + (tid + m * kThreads) * 4);
        if (!L::OWN) {
            __syncthreads();
            load_block<64, DV>(sD, wsD + (size_t)n * 64 * DV);
            cp_commit();
        } else {
            cp_wait<0>();
            __syncthreads();
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const float a = sc * gs.Gam[t.rn + r], b = -gs.Gam[t.rn + r];
#pragma unroll
            for (int y = 0; y < 4; ++y) { acc[r][y] *= a; acc[4 + r][y] *= b; }
        }
        // += [dPD; G] K
        mac<2, A_ROW, B_COL>(acc, sP, sT, kPc, t.rn, sK, kPc, t.cn, 0, w16 + 16);
        if (!L::OWN) {
            cp_wait<0>();
            __syncthreads();
        }
        // dk^col = e (U dh'^T) + dPD^T Q + (b G)^T K, then everything is written
        mac<1, A_ROW, B_ROW>(col, sU, nullptr, PV, t.rn, sD, PV, t.cn, 0, DV);
#pragma unroll
        for (int m = 0; m < 64 * DV / 4 / kThreads; ++m) {   // <dh', h> (h from the workspace: its tile may have been overwritten)
            const int e = tid + m * kThreads;
            const float4 b = ld4(sD + (e / (DV / 4)) * PV + (e % (DV / 4)) * 4);
            hh = fmaf(h4[m].x, b.x, fmaf(h4[m].y, b.y, fmaf(h4[m].z, b.z, fmaf(h4[m].w, b.w, hh))));
        }
        if (n + 1 < NH) {   // the next slice of the states
            __syncthreads();
            load_block<64, DV>(sH, wsH + (size_t)(n + 1) * 64 * DV);
            if (L::OWN) load_block<64, DV>(sD, wsD + (size_t)(n + 1) * 64 * DV);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const float e = gs.ee[t.rn + r];
#pragma unroll
            for (int y = 0; y < 4; ++y) {
                col[r][y] *= e;
                rsum = fmaf(sK[(t.rn + r) * kPc + t.cn + 8 * y], col[r][y], rsum);
            }
        }
        mac<1, A_COL, B_COL>(col, sP, nullptr, kPc, t.rn, sQ, kPc, t.cn, w16, kC);
        mac<1, A_COL, B_COL>(col, sB, nullptr, kPc, t.rn, sK, kPc, t.cn, w16, kC);
        IO* dqp = rows_of<IO>(p.dq, x, H, DK) + n * 64;
        IO* dkp = rows_of<IO>(p.dk, x, H, DK) + n * 64;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int i = t.rn + r;
            const float b = gs.bb[i];
#pragma unroll
            for (int y = 0; y < 4; ++y) {
                const int c = t.cn + 8 * y;
                const float q = sQ[i * kPc + c], k = sK[i * kPc + c];
                dqq[r] = fmaf(q, acc[r][y], dqq[r]);
                drow[r] = fmaf(k, acc[4 + r][y], drow[r]);
                dcol[r] = fmaf(k, col[r][y], dcol[r]);
                if (i < x.len) {
                    stf(dqp + i * rk + c, acc[r][y]);
                    stf(dkp + i * rk + c, fmaf(b, acc[4 + r][y], col[r][y]));
                }
            }
        }
        if (n + 1 < NH) {
            __syncthreads();
            load_rows<64>(sK, kp + (n + 1) * 64, rk, x.len);
            load_rows<64>(sQ, qp + (n + 1) * 64, rk, x.len);
            cp_commit();
        }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        dqq[r] = row_sum8(dqq[r]); drow[r] = row_sum8(drow[r]); dcol[r] = row_sum8(dcol[r]);
        if ((lane & 7) == 0) {
            const int cb = warp >> 2, i = t.rn + r;
            red[0][cb][i] = dqq[r]; red[1][cb][i] = drow[r]; red[2][cb][i] = dcol[r];
        }
    }
    rsum = warp_total(rsum);
    hh = warp_total(hh);
    if (lane == 0) { part[0][warp] = rsum; part[1][warp] = hh; }
    __syncthreads();
    if (tid < kC) {
        const int i = tid;
        const float db = red[1][0][i] + red[1][1][i];
        float dw = red[3][0][i] + red[3][1][i];
        if (DV == 128) dw += red[3][2][i] + red[3][3][i];
        if (p.d.delta_rule && i < x.len) p.dbeta[(size_t)(x.tok0 + i) * H + x.hd] = db + dw;
        dgam[i] = (red[0][0][i] + red[0][1][i]) + gs.bb[i] * db - (red[2][0][i] + red[2][1][i]);
    }
    __syncthreads();
    if (warp == 0) {
        float rs = 0.f, hs = 0.f;
#pragma unroll
        for (int w = 0; w < kThreads / 32; ++w) { rs += part[0][w]; hs += part[1][w]; }
        write_dg(p, x, dgam, rs + gs.Gam[kC - 1] * hs);
    }
}

// The same by a cluster of DK / 32 CTAs, each of which makes 32 channels of dq and dk (and all of the factors, the first of them dv): for calls
// of so few chunk-heads that most SMs would idle.  Of a [64 x 32] result a half of the warps takes dq, the other the row role of k; dk^col
// is U dh'^T by the first half and the rest by the second.  The row sums behind dbeta and dg meet in the first CTA's hands.
// What bounds it: latency, as every kernel of one chunk-head per SM, and the factors, which every CTA makes for itself.  Gradient stage of 4
// chunk-heads at d = 64 27.0 -> 25.0 us; backward of 2 heads of 1024 tokens at d = 128 (four CTAs each) 102 -> 77 us.
template <int DV>
struct IntraSplitTiles {
    static constexpr int PV = pitch(DV), NC = 32, PC = pitch(NC);
    static constexpr int O = 0, X = O + kC * PV, U = X + kC * PV, T = U + kC * PV, B = T + kC * kPc, P = B + kC * kPc;   // as above
    static constexpr int K = P + kC * kPc, Q = K + kC * PC, C = Q + kC * PC;   // slices of 32 channels; C: e (U dh'^T)
    static constexpr int H = C + kC * PC, D = H + NC * PV;
    static constexpr size_t BYTES = sizeof(float) * (D + NC * PV);
};

template <typename IO, int DK, int DV>
__global__ void __launch_bounds__(kThreads, 1) intra_split_kernel(Problem p) {
    wait_prerequisites();
    using L = IntraSplitTiles<DV>;
    constexpr int PV = pitch(DV), PC = L::PC, NC = L::NC, S = DK / NC;
    const int rank = blockIdx.x % S;
    ChunkInfo x;
    if (reinterpret_cast<const WsHeader*>(p.ws)->status != GDN_OK || !chunk_info(p, x, (int)blockIdx.x / S)) return;   // (the whole cluster)
    extern __shared__ __align__(16) float sm[];
    float *sO = sm + L::O, *sX = sm + L::X, *sU = sm + L::U, *sT = sm + L::T, *sB = sm + L::B, *sP = sm + L::P, *sK = sm + L::K, *sQ = sm + L::Q,
          *sC = sm + L::C, *sH = sm + L::H, *sD = sm + L::D;
    __shared__ Gates gs;
    __shared__ float dot_v[4][kC], red[3][kC];   // <v, dXv> by column block; <q, dq>, <k, dk^row>, <k, dk^col> of this CTA's channels
    __shared__ float dgam[kC], part[2][kThreads / 32];
    const int H = p.d.H, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const Thread t;
    const size_t rk = (size_t)H * DK, rv = (size_t)H * DV;
    const float sc = p.d.scale;

    load_rows<DV>(sO, rows_of<IO>(p.dO, x, H, DV), rv, x.len);
    load_block<kC, DV>(sU, block_of(p, p.L.U, x.ch, kC * DV));
    cp_commit();
    load_block<kC, DV>(sX, block_of(p, p.L.dU, x.ch, kC * DV));
    load_block<kC, kC>(sT, block_of(p, p.L.Tm, x.ch, kC * kC));
    cp_commit();
    load_block<NC, DV>(sH, block_of(p, p.L.hc, x.ch, DK * DV) + rank * NC * DV);
    cp_commit();
    load_rows<NC>(sK, rows_of<IO>(p.k, x, H, DK) + rank * NC, rk, x.len);
    load_rows<NC>(sQ, rows_of<IO>(p.q, x, H, DK) + rank * NC, rk, x.len);
    load_block<NC, DV>(sD, block_of(p, p.L.dhn, x.ch, DK * DV) + rank * NC * DV);
    cp_commit();
    if (tid < 32) load_gates(p, x, gs, block_of(p, p.L.gamma, x.ch, kC));
    intra_factors<IO, DV>(p, x, t, gs, sO, sX, sU, sT, sB, sP, dot_v, rank == 0);
    cp_wait<0>();
    __syncthreads();
    const bool row = warp >= 4;              // dO and dPD, or dXv and G
    const int w16 = (t.rn >> 4) * 16, c = lane & 7;
    float rsum = 0.f, hh = 0.f, acc[4][4], col[4][4];
    zero(acc);
    zero(col);
    mac<1, A_ROW, B_ROW>(acc, row ? sX : sO, nullptr, PV, t.rn, sH, PV, c, 0, DV);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const float a = row ? -gs.Gam[t.rn + r] : sc * gs.Gam[t.rn + r];
#pragma unroll
        for (int y = 0; y < 4; ++y) acc[r][y] *= a;
    }
    mac<1, A_ROW, B_COL>(acc, row ? sT : sP, nullptr, kPc, t.rn, sK, PC, c, 0, w16 + 16);
    if (!row) {
        mac<1, A_ROW, B_ROW>(col, sU, nullptr, PV, t.rn, sD, PV, c, 0, DV);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const float e = gs.ee[t.rn + r];
#pragma unroll
            for (int y = 0; y < 4; ++y) {
                const int o = (t.rn + r) * PC + c + 8 * y;
                col[r][y] *= e;
                rsum = fmaf(sK[o], col[r][y], rsum);
                sC[o] = col[r][y];
            }
        }
    } else {
#pragma unroll 1
        for (int m = 0; m < 2; ++m) mac<1, A_COL, B_COL>(col, m ? sB : sP, nullptr, kPc, t.rn, m ? sK : sQ, PC, c, w16, kC);
    }
    for (int e = tid; e < NC * DV / 4; e += kThreads) {   // <dh', h>
        const int o = e / (DV / 4) * PV + e % (DV / 4) * 4;
        const float4 a = ld4(sH + o), b = ld4(sD + o);
        hh = fmaf(a.x, b.x, fmaf(a.y, b.y, fmaf(a.z, b.z, fmaf(a.w, b.w, hh))));
    }
    __syncthreads();
    IO* out = rows_of<IO>(row ? p.dk : p.dq, x, H, DK) + rank * NC;
    float d0[4] = {}, d1[4] = {};   // <q, dq>; or <k, dk^row> and <k, dk^col>
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int i = t.rn + r;
        const float b = gs.bb[i];
#pragma unroll
        for (int y = 0; y < 4; ++y) {
            const int o = i * PC + c + 8 * y;
            const float f = row ? sK[o] : sQ[o], v = acc[r][y];
            d0[r] = fmaf(f, v, d0[r]);
            float res = v;
            if (row) {
                const float cl = sC[o] + col[r][y];
                d1[r] = fmaf(f, cl, d1[r]);
                res = fmaf(b, v, cl);
            }
            if (i < x.len) stf(out + i * rk + c + 8 * y, res);
        }
        d0[r] = row_sum8(d0[r]);
        d1[r] = row_sum8(d1[r]);
        if (c == 0) {
            red[row ? 1 : 0][i] = d0[r];
            if (row) red[2][i] = d1[r];
        }
    }
    rsum = warp_total(rsum);
    hh = warp_total(hh);
    if (lane == 0) { part[0][warp] = rsum; part[1][warp] = hh; }
    cg::cluster_group cluster = cg::this_cluster();
    cluster.sync();
    if (rank == 0) {   // (in the order of the CTAs)
        if (tid < kC) {
            float v[3] = {};
#pragma unroll
            for (int q = 0; q < S; ++q)
#pragma unroll
                for (int w = 0; w < 3; ++w) v[w] += cluster.map_shared_rank(&red[0][0], q)[w * kC + tid];
            float dw = dot_v[0][tid] + dot_v[1][tid];
            if (DV == 128) dw += dot_v[2][tid] + dot_v[3][tid];
            if (p.d.delta_rule && tid < x.len) p.dbeta[(size_t)(x.tok0 + tid) * H + x.hd] = v[1] + dw;
            dgam[tid] = v[0] + gs.bb[tid] * v[1] - v[2];
        }
        __syncthreads();
        if (warp == 0) {
            float rs = 0.f, hs = 0.f;
            for (int q = 0; q < S; ++q) {
                const float* o = cluster.map_shared_rank(&part[0][0], q);
                for (int w = 0; w < kThreads / 32; ++w) { rs += o[w]; hs += o[kThreads / 32 + w]; }
            }
            write_dg(p, x, dgam, rs + gs.Gam[kC - 1] * hs);
        }
    }
    cluster.sync();   // the sums have been read: the CTAs may leave
}

template <int DK, int DV, int CS>
cudaError_t launch_scan_cs(const Problem& p, int dirs, cudaStream_t st) {
    static SmemLimitOnce once;
    const cudaError_t e = once.ensure(scan_kernel<DK, DV, CS>, (uint32_t)ScanShape<DK, CS>::BYTES);
    if (e != cudaSuccess) return e;
    { StageScope t(dirs == 2 ? ST_SCANS : dirs == 1 ? ST_RSCAN : ST_FSCAN, st); launch_kernel(scan_kernel<DK, DV, CS>, scan_blocks(p, dirs, CS), kThreads, ScanShape<DK, CS>::BYTES, st, p, dirs); }
    return cudaGetLastError();
}
template <int DK, int DV>
cudaError_t launch_scan_t(const Problem& p, int dirs, cudaStream_t st) {
    switch (scan_columns(p, dirs)) {
        case 4: return launch_scan_cs<DK, DV, 4>(p, dirs, st);
        case 8: return launch_scan_cs<DK, DV, 8>(p, dirs, st);
        default: return launch_scan_cs<DK, DV, 16>(p, dirs, st);
    }
}

template <typename IO, int DK, int DV>
cudaError_t launch_prep_t(const Problem& p, PrepMode mode, cudaStream_t st) {
    static SmemLimitOnce once;
    const cudaError_t e = once.ensure(prep_kernel<IO, DK, DV>, (uint32_t)prep_smem<DK, DV>());
    if (e != cudaSuccess) return e;
    const int parts = prep_parts(p, mode);
    { StageScope t(mode == PREP_BWD ? ST_EPREP : ST_PREP, st); launch_kernel(prep_kernel<IO, DK, DV>, p.L.max_chunks * p.d.H * parts, kThreads, prep_smem<DK, DV>(), st, p, (int)mode, parts); }
    return cudaGetLastError();
}

template <typename IO, int DK, int DV>
cudaError_t launch_fwd_t(const Problem& p, cudaStream_t st) {
    cudaError_t e;
    if (p.cu && (e = launch_table(p, st)) != cudaSuccess) return e;
    if ((e = launch_prep_t<IO, DK, DV>(p, PREP_FWD, st)) != cudaSuccess) return e;
    if ((e = launch_scan_t<DK, DV>(p, 0, st)) != cudaSuccess || !p.o) return e;
    static SmemLimitOnce once;
    if ((e = once.ensure(out_kernel<IO, DK, DV>, (uint32_t)out_smem<DK, DV>())) != cudaSuccess) return e;
    { StageScope t(ST_OUT, st); launch_kernel(out_kernel<IO, DK, DV>, p.L.max_chunks * p.d.H, kThreads, out_smem<DK, DV>(), st, p); }
    return cudaGetLastError();
}

template <typename IO, int DK, int DV>
cudaError_t launch_bwd_t(const Problem& p, bool skip_recompute, cudaStream_t st) {
    cudaError_t e;
    if (p.cu && !skip_recompute && (e = launch_table(p, st)) != cudaSuccess) return e;
    if ((e = launch_prep_t<IO, DK, DV>(p, skip_recompute ? PREP_BWD : PREP_FWD_BWD, st)) != cudaSuccess) return e;
    if ((e = launch_scan_t<DK, DV>(p, skip_recompute ? 1 : 2, st)) != cudaSuccess) return e;
    static SmemLimitOnce once, once_split;
    constexpr int S = DK / IntraSplitTiles<DV>::NC;
    if (S * p.L.max_chunks * p.d.H <= tc_sm_count()) {   // every CTA of a cluster on an SM of its own
        if ((e = once_split.ensure(intra_split_kernel<IO, DK, DV>, (uint32_t)IntraSplitTiles<DV>::BYTES)) != cudaSuccess) return e;
        { StageScope t(ST_INTRA, st); launch_kernel_cluster(intra_split_kernel<IO, DK, DV>, S * p.L.max_chunks * p.d.H, kThreads, IntraSplitTiles<DV>::BYTES, st, S, p); }
        return cudaGetLastError();
    }
    if ((e = once.ensure(intra_kernel<IO, DK, DV>, (uint32_t)IntraTiles<DK, DV>::BYTES)) != cudaSuccess) return e;
    { StageScope t(ST_INTRA, st); launch_kernel(intra_kernel<IO, DK, DV>, p.L.max_chunks * p.d.H, kThreads, IntraTiles<DK, DV>::BYTES, st, p); }
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_table(const Problem& p, cudaStream_t st, bool fresh) {
    StageScope t(ST_TABLE, st);
    launch_kernel(table_kernel, 1, 256, 0, st, p, fresh ? 1 : 0);
    return cudaGetLastError();
}

#define GDN_DISPATCH(FN, ...)                                                                       \
    do {                                                                                            \
        const bool bf = p.d.dtype == GDN_BF16;                                                      \
        if (p.d.d_k == 64 && p.d.d_v == 64)                                                         \
            return bf ? FN<__nv_bfloat16, 64, 64>(__VA_ARGS__) : FN<float, 64, 64>(__VA_ARGS__);    \
        if (p.d.d_k == 128 && p.d.d_v == 128)                                                       \
            return bf ? FN<__nv_bfloat16, 128, 128>(__VA_ARGS__) : FN<float, 128, 128>(__VA_ARGS__); \
        if (p.d.d_k == 128 && p.d.d_v == 64)                                                        \
            return bf ? FN<__nv_bfloat16, 128, 64>(__VA_ARGS__) : FN<float, 128, 64>(__VA_ARGS__);  \
        if (p.d.d_k == 64 && p.d.d_v == 128)                                                        \
            return bf ? FN<__nv_bfloat16, 64, 128>(__VA_ARGS__) : FN<float, 64, 128>(__VA_ARGS__);  \
        return cudaErrorInvalidValue;                                                               \
    } while (0)

cudaError_t simt_launch_fwd(const Problem& p, cudaStream_t st) { GDN_DISPATCH(launch_fwd_t, p, st); }
cudaError_t simt_launch_bwd(const Problem& p, bool skip_recompute, cudaStream_t st) { GDN_DISPATCH(launch_bwd_t, p, skip_recompute, st); }

}  // namespace gdn
