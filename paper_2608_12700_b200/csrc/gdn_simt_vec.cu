// fp32 FFMA kernels for the general recurrence with PER-CHANNEL gates (Eq. 1 of the paper as printed: log-decay
// g_t and erase gate b_t in R^{d_k}, write gate w_t in R^{d_v}; Table 2: KDA, GLA and the full GDN are gate settings).
//
// The channel-wise decay does not factor out of the chunk-local contractions as a token-token matrix; it folds inside
// them (Appendix A, last paragraph): every token-token quantity is a sum over the channel r that carries the factor
// exp(gam_i[r] - gam_j[r]), j <= i, so that no exponent is ever positive.  The chunk is cut into four blocks of 16 tokens.
// Between two blocks J < I the factor splits at the start of the later one, ref_I = gam at the last token before block I:
//     exp(gam_i - gam_j) = exp(gam_i - ref_I) exp(ref_I - gam_j)      (both exponents non-positive)
// so rows are scaled once (q, b k by exp(gam_i - ref)), the columns once per later block (k by exp(ref_I - gam_j)), and the
// off-diagonal blocks are plain products; only the pairs inside a block, a quarter of all, are summed with the exponential
// in place.  Stages (arithmetic in fp32 whatever the I/O dtype):
//   table  : chunk table from cu_seqlens (shared with the scalar-gate family)
//   vprep  : gam = cumsum(g) per channel;  A_ij = sum_r b_i k_i k_j e^{gam_i - gam_j} (j < i);  P_ij = sum_r q_i k_j
//            e^{gam_i - gam_j} (j <= i);  T = (I + A)^-1;  W = T (Gam . b . K);  Ut = T (w . V);  Kb_j = e^{gam_e - gam_j} . k_j;
//            and for the backward dU0 = scale P^T dO, E = scale (Gam . Q)^T dO
//   vscan  : the carries (ffma_scan.cuh; the state decays by one factor per row)
//   vintra : every token gradient, including the VJP of the triangular solve from the stored T (K#2), the gate
//            gradients per channel, and dg by a reverse cumulative sum inside the chunk
//   vout   : forward output
// One CTA handles one (chunk, head) in the parallel stages.  Every reduction has a fixed order: results are bit-identical
// from run to run.  Measured against the plain statement (decay evaluated for every pair and channel, operands read from global
// memory, one CTA per chain in the carries): 8 heads of 1024 tokens at d = 128, bf16 I/O, decay beyond the tensor-core route:
// 4.4 ms -> 0.21 ms; a step of 2 x 4 heads of 500 tokens at d = 64, fp32: 1.01 -> 0.088 ms.  With bf16 I/O at d_k = d_v = 128 the path runs on the tensor cores instead (gdn_tc_cw.cu), with these
// kernels enqueued behind it for gates that leave its range.
#include "ffma_scan.cuh"

namespace gdn {
namespace {

using namespace ffma;

constexpr int kB = 16, kNB = kC / kB;   // tokens of a block, blocks of a chunk

// Whether this launch has work: no earlier stage has reported an error, and, for a launch of the fall-back sequence, the
// tensor-core route has refused the gates of this call (decided on the device, no host round trip).
__device__ __forceinline__ bool vec_go(const Problem& p) {
    const WsHeader* hdr = reinterpret_cast<const WsHeader*>(p.ws);
    return hdr->status == GDN_OK && (!p.fallback || hdr->cw_fallback);
}

// The (chunk, head) items of a block.
template <class Body>
__device__ __forceinline__ void for_chunks(const Problem& p, Body body) {
    ChunkInfo x;
    for (int item = blockIdx.x; chunk_info(p, x, item); item += gridDim.x) {
        body(x);
        __syncthreads();
    }
}

// References of the four blocks and their exponentials: ref_0 = 0 (the chunk start), ref_I = gam of token 16 I - 1.
template <int DK>
struct __align__(16) Refs { float ref[kNB][DK], eref[kNB][DK]; };
template <int DK>
__device__ __forceinline__ void make_refs(Refs<DK>& s, const float* G) {
    for (int t = threadIdx.x; t < kNB * DK; t += kThreads) {
        const int I = t / DK, r = t % DK;
        const float v = I ? G[(I * kB - 1) * pitch(DK) + r] : 0.f;
        s.ref[I][r] = v;
        s.eref[I][r] = expf(v);
    }
}
// The elementwise passes go over four channels of a token at a time; what they read from global memory is fetched ahead of the pass,
// all of it at once: with a load per element between the stores a pass of a chunk waited out 32 latencies, one behind the other.
__device__ __forceinline__ float4 exp4(const float4& a, const float4& b) { return make_float4(expf(a.x - b.x), expf(a.y - b.y), expf(a.z - b.z), expf(a.w - b.w)); }
__device__ __forceinline__ float4 mul4(const float4& a, const float4& b) { return make_float4(a.x * b.x, a.y * b.y, a.z * b.z, a.w * b.w); }
__device__ __forceinline__ void st4(float* p, const float4& v) { *reinterpret_cast<float4*>(p) = v; }
// v[i4 + y], i4 a multiple of four that is not known at compile time
__device__ __forceinline__ float pick(const float (&v)[kB], int i4, int y) { return (i4 & 8) ? (i4 & 4 ? v[12 + y] : v[8 + y]) : (i4 & 4 ? v[4 + y] : v[y]); }
template <int D>
struct Quads {   // the quads of a [64 x D] tile, N per thread
    static constexpr int N = kC * D / 4 / kThreads;
    static __device__ __forceinline__ int row(int n) { return (threadIdx.x + n * kThreads) / (D / 4); }
    static __device__ __forceinline__ int col(int n) { return (threadIdx.x + n * kThreads) % (D / 4) * 4; }
};
// Rows [0, 64) of a [T, H, D] tensor, this thread's quads; zero beyond `len`.
template <int D, typename IO>
__device__ __forceinline__ void fetch_quads(float4 (&v)[Quads<D>::N], const IO* src, size_t row_pitch, int len) {
    using Qd = Quads<D>;
#pragma unroll
    for (int n = 0; n < Qd::N; ++n) v[n] = Qd::row(n) < len ? ld4(src + Qd::row(n) * row_pitch + Qd::col(n)) : make_float4(0.f, 0.f, 0.f, 0.f);
}
// Rows of a tile times exp(gam - ref of their block), in place.
template <int DK>
__device__ __forceinline__ void scale_rows(float* X, const float* G, const Refs<DK>& s) {
    using Qd = Quads<DK>;
#pragma unroll 2
    for (int n = 0; n < Qd::N; ++n) {
        const int i = Qd::row(n), c = Qd::col(n), o = i * pitch(DK) + c;
        st4(X + o, mul4(ld4(X + o), exp4(ld4(G + o), ld4(s.ref[i / kB] + c))));
    }
}
// The scaled copies of the keys, k_j exp(ref_I - gam_j) for j < 16 I, I = 1 .. 3, one behind the other (96 rows).
__host__ __device__ constexpr int copy_row(int I) { return kB * (I * (I - 1) / 2); }   // first row of copy I
template <int DK>
__device__ __forceinline__ void make_copies(float* C, int j, int c, const float4& k, const float4& g, const Refs<DK>& s) {
#pragma unroll 1
    for (int I = j / kB + 1; I < kNB; ++I) st4(C + (copy_row(I) + j) * pitch(DK) + c, mul4(k, exp4(ld4(s.ref[I] + c), g)));
}

// ------------------------------------------------------------------------------------------------
// vprep
// ------------------------------------------------------------------------------------------------
template <int DK, int DV>
struct PrepTiles {
    static constexpr int PM = pitch(DK > DV ? DK : DV), COPY = 96 * pitch(DK);
    static constexpr int G = 0;                       // gam, then dO
    static constexpr int Q = G + kC * PM;             // q, scaled, then Gam . Q
    static constexpr int K = Q + kC * pitch(DK);      // k, then Gam . b . K
    static constexpr int R = K + kC * pitch(DK);      // b . k, scaled, then w . V
    static constexpr int C = R + kC * PM;             // scaled copies of the keys, then T
    static constexpr int A = C + COPY;
    static constexpr int P = A + kC * kPc;
    static constexpr size_t BYTES = sizeof(float) * (P + kC * kPc);
    static_assert(BYTES + sizeof(Refs<DK>) <= 227 * 1024, "shared memory budget");
};

template <typename IO, int DK, int DV>
__device__ __forceinline__ void vprep_chunk(const Problem& p, int mode, const ChunkInfo& x) {
    using L = PrepTiles<DK, DV>;
    constexpr int PK = pitch(DK), PV = pitch(DV);
    extern __shared__ __align__(16) float sm[];
    float *G = sm + L::G, *Q = sm + L::Q, *K = sm + L::K, *R = sm + L::R, *C = sm + L::C, *A = sm + L::A, *Pm = sm + L::P;
    float *T = C, *O = G;
    __shared__ Refs<DK> refs;
    const bool fwd = mode != PREP_BWD, bwd = mode != PREP_FWD;
    const int H = p.d.H, tid = threadIdx.x;
    const Thread t;
    const Out<DK> ok(t);
    const Out<DV> ov(t);
    const size_t rk = (size_t)H * DK, rv = (size_t)H * DV, base_k = ((size_t)x.tok0 * H + x.hd) * DK, base_v = ((size_t)x.tok0 * H + x.hd) * DV;
    float* wsG = block_of(p, p.L.gamma, x.ch, kC * DK);
    float* wsP = block_of(p, p.L.Pm, x.ch, kC * kC);
    const float sc = p.d.scale;

    load_rows<DK>(Q, rows_of<IO>(p.q, x, H, DK), rk, x.len);
    if (fwd) {
        load_rows<DK>(K, rows_of<IO>(p.k, x, H, DK), rk, x.len);
        cp_commit();
        // chunk-local cumulative log decay per channel; rows beyond the sequence repeat the last valid one
        using Qd = Quads<DK>;
        load_rows<DK>(R, p.bv + base_k, rk, x.len);
        cp_commit();
        if (tid < DK) {
            float s = 0.f;
#pragma unroll 1
            for (int i0 = 0; i0 < kC; i0 += 32) {   // 32 loads in flight, then their running sum in token order
                float g[32];
#pragma unroll
                for (int k = 0; k < 32; ++k) g[k] = i0 + k < x.len ? p.gv[base_k + (size_t)(i0 + k) * rk + tid] : 0.f;
#pragma unroll
                for (int k = 0; k < 32; ++k) { s += g[k]; G[(i0 + k) * PK + tid] = s; }
            }
        }
        for (int e = tid; e < 2 * kC * kPc / 4; e += kThreads) st4(A + 4 * e, make_float4(0.f, 0.f, 0.f, 0.f));   // (A and P lie behind each other)
        cp_wait<0>();
        __syncthreads();
        make_refs(refs, G);
        float* wsKb = block_of(p, p.L.Kb, x.ch, kC * DK);
#pragma unroll 2
        for (int n = 0; n < Qd::N; ++n) {
            const int o = Qd::row(n) * PK + Qd::col(n), e = (tid + n * kThreads) * 4;
            const float4 k = ld4(K + o), g = ld4(G + o);
            st4(R + o, mul4(ld4(R + o), k));
            st4(wsG + e, g);
            st4(wsKb + e, mul4(k, exp4(ld4(G + (kC - 1) * PK + Qd::col(n)), g)));
        }
        __syncthreads();
        // pairs inside a block, in pieces of 2 x 2: the 36 of a block that reach the diagonal; four lanes share one, a quarter of the channels each
        const int z4 = tid & 3;
#pragma unroll 1
        for (int piece = tid >> 2; piece < kNB * 36; piece += kThreads / 4) {   // (a multiple of the eight pieces of a warp)
            const int I = piece / 36;
            int n = piece % 36, a = 0;
            while (n > a) { n -= a + 1; ++a; }   // piece (a, n), n <= a
            const int i = I * kB + 2 * a, j = I * kB + 2 * n;
            float aa[2][2] = {}, pp[2][2] = {};
#pragma unroll 1
            for (int r = 4 * z4; r < DK; r += 16) {
                float gi[2][4], gj[2][4], q[2][4], b[2][4], k[2][4];
#pragma unroll
                for (int y = 0; y < 2; ++y) {
                    *reinterpret_cast<float4*>(gi[y]) = ld4(G + (i + y) * PK + r);
                    *reinterpret_cast<float4*>(gj[y]) = ld4(G + (j + y) * PK + r);
                    *reinterpret_cast<float4*>(q[y]) = ld4(Q + (i + y) * PK + r);
                    *reinterpret_cast<float4*>(b[y]) = ld4(R + (i + y) * PK + r);
                    *reinterpret_cast<float4*>(k[y]) = ld4(K + (j + y) * PK + r);
                }
#pragma unroll
                for (int z = 0; z < 4; ++z)
#pragma unroll
                    for (int y = 0; y < 2; ++y)
#pragma unroll
                        for (int w = 0; w < 2; ++w) {
                            const float ke = k[w][z] * expf(i + y >= j + w ? gi[y][z] - gj[w][z] : 0.f);   // (above the diagonal: not used)
                            aa[y][w] = fmaf(b[y][z], ke, aa[y][w]);
                            pp[y][w] = fmaf(q[y][z], ke, pp[y][w]);
                        }
            }
#pragma unroll
            for (int y = 0; y < 2; ++y)
#pragma unroll
                for (int w = 0; w < 2; ++w) {
#pragma unroll
                    for (int o = 1; o < 4; o <<= 1) {
                        aa[y][w] += __shfl_xor_sync(0xffffffffu, aa[y][w], o);
                        pp[y][w] += __shfl_xor_sync(0xffffffffu, pp[y][w], o);
                    }
                    if (z4 != 2 * y + w) continue;
                    if (j + w < i + y) A[(i + y) * kPc + j + w] = aa[y][w];
                    if (j + w <= i + y) Pm[(i + y) * kPc + j + w] = pp[y][w];
                }
        }
        __syncthreads();
#pragma unroll 2
        for (int n = 0; n < Qd::N; ++n) {
            const int i = Qd::row(n), c = Qd::col(n), o = i * PK + c;
            const float4 g = ld4(G + o), e = exp4(g, ld4(refs.ref[i / kB] + c));
            make_copies<DK>(C, i, c, ld4(K + o), g, refs);
            st4(Q + o, mul4(ld4(Q + o), e));
            st4(R + o, mul4(ld4(R + o), e));
        }
        __syncthreads();
        // pairs of blocks J < I: A and P, 16 threads a 16 x 16 block, 4 x 4 each
        if (tid < 192) {
            const int which = tid / 96, o = tid % 96, blk = o / 16, ti = ((o % 16) >> 2) * 4, tj = o & 3;
            const int I = blk == 0 ? 1 : blk < 3 ? 2 : 3, J = blk == 0 ? 0 : blk < 3 ? blk - 1 : blk - 3;
            float acc[4][4];
            zero(acc);
            mac<1, A_ROW, B_ROW, 0, 4, kU<DK>>(acc, which ? Q : R, nullptr, PK, I * kB + ti, C + (copy_row(I) + J * kB) * PK, PK, tj, 0, DK);
            float* dst = (which ? Pm : A) + (I * kB + ti) * kPc + J * kB + tj;
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int y = 0; y < 4; ++y) dst[r * kPc + 4 * y] = acc[r][y];
        }
#pragma unroll 2
        for (int n = 0; n < Qd::N; ++n) {   // Gam . b . K, the right-hand side of W
            const int i = Qd::row(n), c = Qd::col(n), o = i * PK + c;
            st4(K + o, mul4(ld4(R + o), ld4(refs.eref[i / kB] + c)));
        }
        using Qv = Quads<DV>;
        float4 wq[Qv::N];
        fetch_quads<DV>(wq, p.wv + base_v, rv, x.len);
        __syncthreads();
        load_rows<DV>(R, rows_of<IO>(p.v, x, H, DV), rv, x.len);
        cp_commit();
        if (bwd) load_rows<DV>(O, rows_of<IO>(p.dO, x, H, DV), rv, x.len);
        cp_commit();
        for (int e = 4 * tid; e < kC * kC; e += 4 * kThreads) st4(wsP + e, ld4(Pm + (e / kC) * kPc + e % kC));
        invert(A, T);
        cp_wait<1>();
        __syncthreads();
        float* wsT = block_of(p, p.L.Tm, x.ch, kC * kC);
        for (int e = 4 * tid; e < kC * kC; e += 4 * kThreads) st4(wsT + e, ld4(T + (e / kC) * kPc + e % kC));
#pragma unroll
        for (int n = 0; n < Qv::N; ++n) {
            float* v = R + Qv::row(n) * PV + Qv::col(n);
            st4(v, mul4(ld4(v), wq[n]));
        }
        __syncthreads();
        float* wsU = block_of(p, p.L.Ut, x.ch, kC * DV);
        {
            float acc[Out<DV>::R][4];
            tri_product<DV, A_ROW, A_LOWER, kU<DK>>(t, T, R, PV, acc);
#pragma unroll
            for (int r = 0; r < Out<DV>::R; ++r)
#pragma unroll
                for (int y = 0; y < 4; ++y) wsU[ov.row(r) * DV + ov.c + 8 * y] = acc[r][y];
        }
        float* wsW = block_of(p, p.L.W, x.ch, kC * DK);
        {
            float acc[Out<DK>::R][4];
            tri_product<DK, A_ROW, A_LOWER, kU<DK>>(t, T, K, PK, acc);
#pragma unroll
            for (int r = 0; r < Out<DK>::R; ++r)
#pragma unroll
                for (int y = 0; y < 4; ++y) wsW[ok.row(r) * DK + ok.c + 8 * y] = acc[r][y];
        }
        if (!bwd) return;
    } else {
        load_block<kC, DK>(G, wsG);
        load_block<kC, kC>(Pm, wsP);
        cp_commit();
        cp_wait<0>();
        __syncthreads();
        make_refs(refs, G);
        __syncthreads();
        scale_rows<DK>(Q, G, refs);
        __syncthreads();
        load_rows<DV>(O, rows_of<IO>(p.dO, x, H, DV), rv, x.len);
        cp_commit();
    }
    cp_wait<0>();
    __syncthreads();
    using Qd = Quads<DK>;
#pragma unroll 2
    for (int n = 0; n < Qd::N; ++n) {   // Gam . Q, in place
        const int i = Qd::row(n), c = Qd::col(n), o = i * PK + c;
        st4(Q + o, mul4(ld4(Q + o), ld4(refs.eref[i / kB] + c)));
    }
    // dU0 = scale P^T dO
    float* wsD = block_of(p, p.L.dU, x.ch, kC * DV);
    {
        float acc[Out<DV>::R][4];
        tri_product<DV, A_COL, A_UPPER, kU<DK>>(t, Pm, O, PV, acc);
#pragma unroll
        for (int r = 0; r < Out<DV>::R; ++r)
#pragma unroll
            for (int y = 0; y < 4; ++y) wsD[ov.row(r) * DV + ov.c + 8 * y] = sc * acc[r][y];
    }
    __syncthreads();
    // E = scale (Gam . Q)^T dO, 64 rows at a time
    float* wsE = block_of(p, p.L.E, x.ch, DK * DV);
#pragma unroll 1
    for (int r0 = 0; r0 < DK; r0 += 64) {
        float acc[Out<DV>::R][4];
        zero(acc);
        mac<Out<DV>::R / 4, A_COL, B_COL>(acc, Q + r0, Q + r0 + 32, PK, ov.r0, O, PV, ov.c, 0, kC);
#pragma unroll
        for (int r = 0; r < Out<DV>::R; ++r)
#pragma unroll
            for (int y = 0; y < 4; ++y) wsE[(r0 + ov.row(r)) * DV + ov.c + 8 * y] = sc * acc[r][y];
    }
}

template <typename IO, int DK, int DV>
__global__ void __launch_bounds__(kThreads, 1) vprep_kernel(Problem p, int mode) {
    wait_prerequisites();
    if (p.fallback) { if (!vec_go(p)) return; }
    else if (mode != PREP_BWD) init_header_if_untabled(p);
    else check_fresh_seqlens(p);   // (the backward's part alone: the status word is the forward's)
    for_chunks(p, [&](const ChunkInfo& x) { vprep_chunk<IO, DK, DV>(p, mode, x); });
}

// ------------------------------------------------------------------------------------------------
// vscan: forward and reverse carries (ffma_scan.cuh).
// ------------------------------------------------------------------------------------------------
// (WALK: a block goes over the items, as the fall-back launches do; the loop costs 60 registers, hence an instance of its own.)
template <int DK, int DV, int CS, bool WALK>
__global__ void __launch_bounds__(kThreads, DK == 64 ? 2 : 1) vscan_kernel(const __grid_constant__ Problem p, int dirs) {
    wait_prerequisites();
    extern __shared__ __align__(16) float sm[];
    if (!vec_go(p)) return;
    if constexpr (!WALK) {
        scan_block<DK, DV, CS, true>(p, dirs, sm, blockIdx.x);
    } else {
        for (int b = blockIdx.x; b < scan_blocks(p, dirs, CS); b += gridDim.x) {
            scan_block<DK, DV, CS, true>(p, dirs, sm, b);
            __syncthreads();
        }
    }
}

// ------------------------------------------------------------------------------------------------
// vout, forward output (optional): o = scale ((Gam . Q) h + P U)
// ------------------------------------------------------------------------------------------------
template <int DK, int DV>
constexpr size_t vout_smem() { return sizeof(float) * (kC * pitch(DK) + DK * pitch(DV) + kC * pitch(DV) + kC * kPc); }

template <typename IO, int DK, int DV>
__device__ __forceinline__ void vout_chunk(const Problem& p, const ChunkInfo& x) {
    constexpr int PK = pitch(DK), PV = pitch(DV), R = Out<DV>::R;
    extern __shared__ __align__(16) float sm[];
    float* sQ = sm;
    float* sH = sQ + kC * PK;
    float* sU = sH + DK * PV;
    float* Pm = sU + kC * PV;
    const int H = p.d.H;
    const Thread t;
    const Out<DV> o(t);
    load_rows<DK>(sQ, rows_of<IO>(p.q, x, H, DK), (size_t)H * DK, x.len);
    load_block<DK, DV>(sH, block_of(p, p.L.hc, x.ch, DK * DV));
    load_block<kC, DV>(sU, block_of(p, p.L.U, x.ch, kC * DV));
    load_block<kC, kC>(Pm, block_of(p, p.L.Pm, x.ch, kC * kC));
    cp_commit();
    float4 gq[Quads<DK>::N];
    fetch_quads<DK>(gq, block_of(p, p.L.gamma, x.ch, kC * DK), DK, kC);
    cp_wait<0>();
    __syncthreads();
    using Qd = Quads<DK>;
#pragma unroll
    for (int n = 0; n < Qd::N; ++n) {
        float* q = sQ + Qd::row(n) * PK + Qd::col(n);
        st4(q, mul4(ld4(q), exp4(gq[n], make_float4(0.f, 0.f, 0.f, 0.f))));
    }
    __syncthreads();
    float acc[R][4];
    zero(acc);
    mac<R / 4, A_ROW, B_COL, 0, 8, kU<DK>>(acc, sQ, sQ + 32 * PK, PK, o.r0, sH, PV, o.c, 0, DK);
    mac<R / 4, A_ROW, B_COL, 0, 8, kU<DK>>(acc, Pm, Pm + 32 * kPc, kPc, o.r0, sU, PV, o.c, 0, kC);
    IO* op = rows_of<IO>(p.o, x, H, DV);
    const size_t rv = (size_t)H * DV;
    const float sc = p.d.scale;
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (o.row(r) < x.len)
#pragma unroll
            for (int y = 0; y < 4; ++y) stf(op + o.row(r) * rv + o.c + 8 * y, sc * acc[r][y]);
}

template <typename IO, int DK, int DV>
__global__ void __launch_bounds__(kThreads, 1) vout_kernel(Problem p) {
    wait_prerequisites();
    if (!vec_go(p)) return;
    for_chunks(p, [&](const ChunkInfo& x) { vout_chunk<IO, DK, DV>(p, x); });
}

// ------------------------------------------------------------------------------------------------
// vintra: token gradients of one (chunk, head).  K#2 in its short form: dXv = T^T dU, dXk = -dXv h^T, dA = -stril(dXv U^T).
//     dq_i = scale Gam_i (dO h^T)_i + sum_{j <= i} dP_ij e^{gam_i - gam_j} k_j
//     row_i = -Gam_i (dXv h^T)_i + sum_{j < i} dA_ij e^{gam_i - gam_j} k_j
//     col_j = e_j (U dh'^T)_j + sum_{i >= j} e^{gam_i - gam_j} (dP_ij q_i + dA_ij b_i k_i)
//     dk = b row + col,  db = k row,  dgam = q dq + b k row - k col,  and the last row adds
//     sum_j k_j e_j (U dh'^T)_j + Gam_e rowdot(dh', h)
// First the products with the states (results in registers), then, with their tiles gone, the pairs of blocks from the scaled
// tiles; a last pass in which a thread owns a channel of a block adds the pairs inside the block and writes everything.
// ------------------------------------------------------------------------------------------------
template <int DK, int DV>
struct IntraTiles {
    static constexpr int PM = pitch(DK > DV ? DK : DV), PK = pitch(DK), PV = pitch(DV);
    static constexpr int S0 = 0;                  // dO
    static constexpr int S1 = S0 + kC * PM;       // dU, then dXv
    static constexpr int U = S1 + kC * PM;
    static constexpr int H = U + kC * PV;         // h, then dh'
    static constexpr int END1 = H + DK * PV;
    static constexpr int G = 0;                   // gam                        (over dO)
    static constexpr int Q = G + kC * PK;         // q, scaled; then row        (over dXv)
    static constexpr int R = Q + kC * PK;         // b . k, scaled; then col
    static constexpr int C = R + kC * PK;         // scaled copies of the keys; then dq, then dgam
    static constexpr int END2 = C + 96 * PK;
    static constexpr int T = END1 > END2 ? END1 : END2;   // T, then dA
    static constexpr int P = T + kC * kPc;        // scale tril(dO U^T)
    static constexpr size_t BYTES = sizeof(float) * (P + kC * kPc);
    static_assert(Q + kC * PK <= U, "gam and q arrive while U and dh' are in use");
    static_assert(BYTES + sizeof(Refs<DK>) + 4 * (kNB + 1) * DK <= 227 * 1024, "shared memory budget");
};

template <typename IO, int DK, int DV>
__device__ __forceinline__ void vintra_chunk(const Problem& p, const ChunkInfo& x) {
    using L = IntraTiles<DK, DV>;
    constexpr int PK = pitch(DK), PV = pitch(DV), NH = DK / 64;
    extern __shared__ __align__(16) float sm[];
    float *s0 = sm + L::S0, *s1 = sm + L::S1, *sU = sm + L::U, *sH = sm + L::H, *sT = sm + L::T, *sP = sm + L::P;
    float *G = sm + L::G, *Q = sm + L::Q, *R = sm + L::R, *C = sm + L::C;
    __shared__ Refs<DK> refs;
    __shared__ __align__(16) float ends[DK], blk[kNB][DK];   // chunk-end term of dg; first: its parts by row blocks; later: block sums of dgam
    const int H = p.d.H, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const Thread t;
    const size_t rk = (size_t)H * DK, rv = (size_t)H * DV;
    const size_t base_k = ((size_t)x.tok0 * H + x.hd) * DK, base_v = ((size_t)x.tok0 * H + x.hd) * DV;
    const IO* qp = reinterpret_cast<const IO*>(p.q) + base_k;
    const IO* kp = reinterpret_cast<const IO*>(p.k) + base_k;
    const float* wsH = block_of(p, p.L.hc, x.ch, DK * DV);
    const float* wsG = block_of(p, p.L.gamma, x.ch, kC * DK);
    const float sc = p.d.scale;

    load_rows<DV>(s0, rows_of<IO>(p.dO, x, H, DV), rv, x.len);
    load_block<kC, DV>(sU, block_of(p, p.L.U, x.ch, kC * DV));
    cp_commit();
    load_block<kC, DV>(s1, block_of(p, p.L.dU, x.ch, kC * DV));
    load_block<kC, kC>(sT, block_of(p, p.L.Tm, x.ch, kC * kC));
    cp_commit();
    load_block<DK, DV>(sH, wsH);
    cp_commit();
    cp_wait<2>();
    __syncthreads();
    const int I = t.rn / kB;                      // the rows of a warp are one block of tokens
    const bool below = (warp >> 2) * 32 <= I * kB + kB - 1;
    {   // dP = scale tril(dO U^T)
        float acc[4][4];
        zero(acc);
        if (below) mac<1, A_ROW, B_ROW, 0, 8, kU<DK>>(acc, s0, nullptr, PV, t.rn, sU, PV, t.cn, 0, DV);
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int y = 0; y < 4; ++y) sP[(t.rn + r) * kPc + t.cn + 8 * y] = t.cn + 8 * y <= t.rn + r ? sc * acc[r][y] : 0.f;
    }
    cp_wait<1>();
    __syncthreads();
    {   // dXv = T^T dU, in place; dv = w . dXv, dw = v . dXv
        const Out<DV> o(t);
        float acc[Out<DV>::R][4], vv[Out<DV>::R][4], ww[Out<DV>::R][4];
        const IO* vp = reinterpret_cast<const IO*>(p.v) + base_v;
        IO* dvp = reinterpret_cast<IO*>(p.dv) + base_v;
#pragma unroll
        for (int r = 0; r < Out<DV>::R; ++r)
#pragma unroll
            for (int y = 0; y < 4; ++y) {
                const bool live = o.row(r) < x.len;
                vv[r][y] = live ? ldf(vp + o.row(r) * rv + o.c + 8 * y) : 0.f;
                ww[r][y] = live ? p.wv[base_v + o.row(r) * rv + o.c + 8 * y] : 0.f;
            }
        tri_product<DV, A_COL, A_UPPER, kU<DK>>(t, sT, s1, PV, acc);
        __syncthreads();
#pragma unroll
        for (int r = 0; r < Out<DV>::R; ++r)
#pragma unroll
            for (int y = 0; y < 4; ++y) {
                const int i = o.row(r), c = o.c + 8 * y;
                s1[i * PV + c] = acc[r][y];
                if (i < x.len) {
                    stf(dvp + i * rv + c, ww[r][y] * acc[r][y]);
                    p.dwv[base_v + i * rv + c] = vv[r][y] * acc[r][y];
                }
            }
    }
    cp_wait<0>();
    __syncthreads();
    {   // dA = -stril(dXv U^T), over T
        float acc[4][4];
        zero(acc);
        if (below) mac<1, A_ROW, B_ROW, 0, 8, kU<DK>>(acc, s1, nullptr, PV, t.rn, sU, PV, t.cn, 0, DV);
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int y = 0; y < 4; ++y) sT[(t.rn + r) * kPc + t.cn + 8 * y] = t.cn + 8 * y < t.rn + r ? -acc[r][y] : 0.f;
    }
    // [dO; dXv] h^T: rows 0..3 become dq, rows 4..7 the row role of k
    float acc[NH][8][4];
#pragma unroll
    for (int n = 0; n < NH; ++n) {
        zero(acc[n]);
        mac<2, A_ROW, B_ROW, 0, 8, kU<DK>>(acc[n], s0, s1, PV, t.rn, sH + n * 64 * PV, PV, t.cn, 0, DV);
    }
    __syncthreads();
    load_block<DK, DV>(sH, block_of(p, p.L.dhn, x.ch, DK * DV));
    load_block<kC, DK>(G, wsG);
    load_rows<DK>(Q, qp, rk, x.len);
    cp_commit();
    cp_wait<0>();
    __syncthreads();
    make_refs(refs, G);
    // col = e . (U dh'^T); its dot with k over the tokens, per channel, goes to the chunk end
    float col[NH][4][4];
#pragma unroll
    for (int n = 0; n < NH; ++n) {
        float kr[4][4];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int y = 0; y < 4; ++y) kr[r][y] = t.rn + r < x.len ? ldf(kp + (t.rn + r) * rk + n * 64 + t.cn + 8 * y) : 0.f;
        zero(col[n]);
        mac<1, A_ROW, B_ROW, 0, 8, kU<DK>>(col[n], sU, nullptr, PV, t.rn, sH + n * 64 * PV, PV, t.cn, 0, DV);
#pragma unroll
        for (int y = 0; y < 4; ++y) {
            const int c = n * 64 + t.cn + 8 * y;
            float s = 0.f;
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int i = t.rn + r;
                const float g = G[i * PK + c], Gi = expf(g);
                col[n][r][y] *= expf(G[(kC - 1) * PK + c] - g);
                acc[n][r][y] *= sc * Gi;
                acc[n][4 + r][y] *= -Gi;
                s = fmaf(kr[r][y], col[n][r][y], s);
            }
            s += __shfl_xor_sync(0xffffffffu, s, 8);
            s += __shfl_xor_sync(0xffffffffu, s, 16);
            if (lane < 8) blk[I][c] = s;
        }
    }
    // Gam_e rowdot(dh', h): one warp per state row (h from the workspace: its tile has been overwritten)
    constexpr int HB = 8;   // rows whose loads are in flight at a time
#pragma unroll 1
    for (int r0 = warp * (DK / 8); r0 < (warp + 1) * (DK / 8); r0 += HB) {
        float4 h4[HB];
#pragma unroll
        for (int k = 0; k < HB; ++k) h4[k] = lane * 4 < DV ? ld4(wsH + (size_t)(r0 + k) * DV + lane * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int k = 0; k < HB; ++k) {
            float s = 0.f;
            if (lane * 4 < DV) {
                const float4 a = h4[k], b = ld4(sH + (r0 + k) * PV + lane * 4);
                s = fmaf(a.x, b.x, fmaf(a.y, b.y, fmaf(a.z, b.z, a.w * b.w)));
            }
            s = warp_total(s);
            if (lane == 0) ends[r0 + k] = expf(G[(kC - 1) * PK + r0 + k]) * s;
        }
    }
    using Qd = Quads<DK>;
    float4 kq[Qd::N], bq[Qd::N];
    fetch_quads<DK>(kq, kp, rk, x.len);
    fetch_quads<DK>(bq, p.bv + base_k, rk, x.len);
    __syncthreads();
    if (tid < DK) ends[tid] += (blk[0][tid] + blk[1][tid]) + (blk[2][tid] + blk[3][tid]);
#pragma unroll
    for (int n = 0; n < Qd::N; ++n) {
        const int i = Qd::row(n), c = Qd::col(n), o = i * PK + c;
        const float4 g = ld4(G + o), e = exp4(g, ld4(refs.ref[i / kB] + c));
        make_copies<DK>(C, i, c, kq[n], g, refs);
        st4(R + o, mul4(mul4(bq[n], kq[n]), e));
        st4(Q + o, mul4(ld4(Q + o), e));
    }
    __syncthreads();
    // pairs of blocks J < I
#pragma unroll
    for (int n = 0; n < NH; ++n) {
        float tmp[8][4];
        zero(tmp);
        mac<2, A_ROW, B_COL, 0, 8, kU<DK>>(tmp, sP, sT, kPc, t.rn, C + copy_row(I) * PK + n * 64, PK, t.cn, 0, I * kB);
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int y = 0; y < 4; ++y) {
                const int c = n * 64 + t.cn + 8 * y;
                const float e = expf(G[(t.rn + r) * PK + c] - refs.ref[I][c]);
                acc[n][r][y] = fmaf(e, tmp[r][y], acc[n][r][y]);
                acc[n][4 + r][y] = fmaf(e, tmp[4 + r][y], acc[n][4 + r][y]);
            }
#pragma unroll 1
        for (int I2 = I + 1; I2 < kNB; ++I2) {
            float tc[4][4];
            zero(tc);
            mac<1, A_COL, B_COL, 0, 8, kU<DK>>(tc, sP, nullptr, kPc, t.rn, Q + n * 64, PK, t.cn, I2 * kB, I2 * kB + kB);
            mac<1, A_COL, B_COL, 0, 8, kU<DK>>(tc, sT, nullptr, kPc, t.rn, R + n * 64, PK, t.cn, I2 * kB, I2 * kB + kB);
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int y = 0; y < 4; ++y) {
                    const int c = n * 64 + t.cn + 8 * y;
                    col[n][r][y] = fmaf(expf(refs.ref[I2][c] - G[(t.rn + r) * PK + c]), tc[r][y], col[n][r][y]);
                }
        }
    }
    __syncthreads();
    // hand the sums so far to the owners of the channels: row over Q, col over R, dq over the copies
#pragma unroll
    for (int n = 0; n < NH; ++n)
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int y = 0; y < 4; ++y) {
                const int o = (t.rn + r) * PK + n * 64 + t.cn + 8 * y;
                C[o] = acc[n][r][y];
                Q[o] = acc[n][4 + r][y];
                R[o] = col[n][r][y];
            }
    __syncthreads();
    IO* dqp = reinterpret_cast<IO*>(p.dq) + base_k;
    IO* dkp = reinterpret_cast<IO*>(p.dk) + base_k;
#pragma unroll 1
    for (int task = tid; task < kNB * DK; task += kThreads) {   // one channel of one block of tokens
        const int B = task / DK, r = task % DK, i0 = B * kB;
        float k[kB], b[kB], g[kB], dc[kB];
        float qn[4];   // q of four rows, fetched a group ahead
        auto fetch_q = [&](int i4) {
#pragma unroll
            for (int y = 0; y < 4; ++y) qn[y] = i4 < kB && i0 + i4 + y < x.len ? ldf(qp + (i0 + i4 + y) * rk + r) : 0.f;
        };
        fetch_q(0);
#pragma unroll
        for (int i = 0; i < kB; ++i) {
            const bool live = i0 + i < x.len;
            k[i] = live ? ldf(kp + (i0 + i) * rk + r) : 0.f;
            b[i] = live ? p.bv[base_k + (i0 + i) * rk + r] : 0.f;
            g[i] = G[(i0 + i) * PK + r];
            dc[i] = R[(i0 + i) * PK + r];
        }
        // four rows at a time (a rolled loop: the code of all 136 pairs is 30 KB, which a CTA would fetch for two passes): their dq and row
        // role are complete at once, the column roles collect
#pragma unroll 1
        for (int i4 = 0; i4 < kB; i4 += 4) {
            float gi[4], q[4], bk[4], ki[4], dq[4], row[4];
#pragma unroll
            for (int y = 0; y < 4; ++y) {
                gi[y] = G[(i0 + i4 + y) * PK + r]; q[y] = qn[y]; ki[y] = pick(k, i4, y); bk[y] = pick(b, i4, y) * ki[y];
                dq[y] = C[(i0 + i4 + y) * PK + r]; row[y] = Q[(i0 + i4 + y) * PK + r];
            }
            fetch_q(i4 + 4);
#pragma unroll
            for (int j4 = 0; j4 < kB; j4 += 4) {
                if (j4 > i4) break;
#pragma unroll
                for (int y = 0; y < 4; ++y) {
                    const float4 P4 = ld4(sP + (i0 + i4 + y) * kPc + i0 + j4), A4 = ld4(sT + (i0 + i4 + y) * kPc + i0 + j4);   // (zero above the diagonal, dA on it too)
                    const float P_[4] = {P4.x, P4.y, P4.z, P4.w}, A_[4] = {A4.x, A4.y, A4.z, A4.w};
#pragma unroll
                    for (int z = 0; z < 4; ++z) {
                        const float e = expf(j4 + z < i4 + y ? gi[y] - g[j4 + z] : 0.f), pe = P_[z] * e, ae = A_[z] * e;
                        dq[y] = fmaf(pe, k[j4 + z], dq[y]);
                        row[y] = fmaf(ae, k[j4 + z], row[y]);
                        dc[j4 + z] = fmaf(pe, q[y], fmaf(ae, bk[y], dc[j4 + z]));
                    }
                }
            }
#pragma unroll
            for (int y = 0; y < 4; ++y) {
                const int i = i0 + i4 + y;
                if (i < x.len) {
                    stf(dqp + i * rk + r, dq[y]);
                    p.dbv[base_k + i * rk + r] = ki[y] * row[y];
                }
                Q[i * PK + r] = row[y];
                C[i * PK + r] = fmaf(q[y], dq[y], bk[y] * row[y]);
            }
        }
        float run = 0.f;   // dgam, summed from the end of the block
#pragma unroll
        for (int i = kB - 1; i >= 0; --i) {
            if (i0 + i < x.len) stf(dkp + (i0 + i) * rk + r, fmaf(b[i], Q[(i0 + i) * PK + r], dc[i]));
            run += fmaf(-k[i], dc[i], C[(i0 + i) * PK + r]);
            C[(i0 + i) * PK + r] = run;
        }
        blk[B][r] = run;
    }
    __syncthreads();
    // dg_j = sum_{i >= j} dgam_i: the sum inside the block, the blocks behind it and the chunk end
#pragma unroll 2
    for (int n = 0; n < Qd::N; ++n) {
        const int i = Qd::row(n), c = Qd::col(n);
        float4 s = ld4(ends + c);
#pragma unroll
        for (int B = kNB - 1; B > 0; --B)
            if (B > i / kB) { const float4 v = ld4(blk[B] + c); s = make_float4(s.x + v.x, s.y + v.y, s.z + v.z, s.w + v.w); }
        const float4 v = ld4(C + i * PK + c);
        if (i < x.len) st4(p.dgv + base_k + i * rk + c, make_float4(s.x + v.x, s.y + v.y, s.z + v.z, s.w + v.w));
    }
}

template <typename IO, int DK, int DV>
__global__ void __launch_bounds__(kThreads, 1) vintra_kernel(Problem p) {
    wait_prerequisites();
    if (!vec_go(p)) return;
    for_chunks(p, [&](const ChunkInfo& x) { vintra_chunk<IO, DK, DV>(p, x); });
}

// Blocks of a launch over `items`: one each, or, for the fall-back sequence, one per SM (it rarely has work, and a grid of
// thousands of blocks that return at once takes microseconds: three launches behind a call of 2112 chunk-heads, see launch).
int grid_of(const Problem& p, int items) { return p.fallback && items > tc_sm_count() ? tc_sm_count() : items; }

template <int DK, int DV, int CS, bool WALK>
cudaError_t launch_vscan_cs(const Problem& p, int dirs, cudaStream_t st) {
    static SmemLimitOnce once;
    const auto kernel = vscan_kernel<DK, DV, CS, WALK>;
    const cudaError_t e = once.ensure(kernel, (uint32_t)ScanShape<DK, CS>::BYTES);
    if (e != cudaSuccess) return e;
    { StageScope t(p.fallback ? ST_FALLBACK : dirs == 2 ? ST_SCANS : dirs == 1 ? ST_RSCAN : ST_FSCAN, st); launch_kernel(kernel, grid_of(p, scan_blocks(p, dirs, CS)), kThreads, ScanShape<DK, CS>::BYTES, st, p, dirs); }
    return cudaGetLastError();
}
template <int DK, int DV>
cudaError_t launch_vscan(const Problem& p, int dirs, cudaStream_t st) {
    const int cs = scan_columns(p, dirs);
    if constexpr (DK == 128 && DV == 128)
        if (p.fallback && scan_blocks(p, dirs, cs) > tc_sm_count()) return launch_vscan_cs<DK, DV, 16, true>(p, dirs, st);
    return cs == 4 ? launch_vscan_cs<DK, DV, 4, false>(p, dirs, st) : cs == 8 ? launch_vscan_cs<DK, DV, 8, false>(p, dirs, st) : launch_vscan_cs<DK, DV, 16, false>(p, dirs, st);
}
template <typename IO, int DK, int DV>
cudaError_t launch_vprep(const Problem& p, PrepMode mode, cudaStream_t st) {
    static SmemLimitOnce once;
    constexpr size_t sm = PrepTiles<DK, DV>::BYTES;
    const cudaError_t e = once.ensure(vprep_kernel<IO, DK, DV>, (uint32_t)sm);
    if (e != cudaSuccess) return e;
    { StageScope t(p.fallback ? ST_FALLBACK : mode == PREP_BWD ? ST_EPREP : ST_PREP, st); launch_kernel(vprep_kernel<IO, DK, DV>, grid_of(p, p.L.max_chunks * p.d.H), kThreads, sm, st, p, mode); }
    return cudaGetLastError();
}

// The FFMA sequences.  `q` is the problem as these kernels see it (fp32 factors and states); with q.fallback set the chunk
// table is not rebuilt (the tensor-core route has built it, and rebuilding would reset the status word the launches look at).
template <typename IO, int DK, int DV>
cudaError_t ffma_fwd(const Problem& q, cudaStream_t st) {
    cudaError_t e;
    if (q.cu && !q.fallback && (e = launch_table(q, st)) != cudaSuccess) return e;
    if ((e = launch_vprep<IO, DK, DV>(q, PREP_FWD, st)) != cudaSuccess) return e;
    if ((e = launch_vscan<DK, DV>(q, 0, st)) != cudaSuccess || !q.o) return e;
    static SmemLimitOnce once;
    if ((e = once.ensure(vout_kernel<IO, DK, DV>, (uint32_t)vout_smem<DK, DV>())) != cudaSuccess) return e;
    { StageScope t(q.fallback ? ST_FALLBACK : ST_OUT, st); launch_kernel(vout_kernel<IO, DK, DV>, grid_of(q, q.L.max_chunks * q.d.H), kThreads, vout_smem<DK, DV>(), st, q); }
    return cudaGetLastError();
}

template <typename IO, int DK, int DV>
cudaError_t ffma_bwd(const Problem& q, bool skip_recompute, cudaStream_t st) {
    cudaError_t e;
    if (q.cu && !q.fallback && !skip_recompute && (e = launch_table(q, st)) != cudaSuccess) return e;
    if ((e = launch_vprep<IO, DK, DV>(q, skip_recompute ? PREP_BWD : PREP_FWD_BWD, st)) != cudaSuccess) return e;
    if ((e = launch_vscan<DK, DV>(q, skip_recompute ? 1 : 2, st)) != cudaSuccess) return e;
    static SmemLimitOnce once;
    constexpr size_t sm = IntraTiles<DK, DV>::BYTES;
    if ((e = once.ensure(vintra_kernel<IO, DK, DV>, (uint32_t)sm)) != cudaSuccess) return e;
    { StageScope t(q.fallback ? ST_FALLBACK : ST_INTRA, st); launch_kernel(vintra_kernel<IO, DK, DV>, grid_of(q, q.L.max_chunks * q.d.H), kThreads, sm, st, q); }
    return cudaGetLastError();
}

// bf16 I/O at d = 128 runs on the tensor cores (gdn_tc_cw.cu).  That route refuses gates whose chunk-cumulative log decay
// leaves its range, through the workspace header; the FFMA sequence is therefore enqueued behind it in fall-back mode: its
// launches return at once unless the header says so, in which case they compute the call (with the decay inside the
// contractions there is no range limit).  No host round trip, the same launches every call.
template <typename IO, int DK, int DV>
cudaError_t ffma_fallback(const Problem& p, bool bwd, bool skip_recompute, cudaStream_t st) {
    Problem q = p;
    q.fallback = 1;
    q.L.tc_scans = 0;
    return bwd ? ffma_bwd<IO, DK, DV>(q, skip_recompute, st) : ffma_fwd<IO, DK, DV>(q, st);
}

template <typename IO, int DK, int DV>
cudaError_t vlaunch_fwd_t(const Problem& p, cudaStream_t st) {
    if (!p.L.tc_scans) return ffma_fwd<IO, DK, DV>(p, st);
    const int CH = p.L.max_chunks * p.d.H;
    cudaError_t e = cw_tc_launch(p, /*bwd=*/false, false, st);
    if (e != cudaSuccess) return e;
    if (p.o && CH > 0 && (e = tc_launch_out_channelwise(p, st)) != cudaSuccess) return e;
    return ffma_fallback<IO, DK, DV>(p, false, false, st);
}

template <typename IO, int DK, int DV>
cudaError_t vlaunch_bwd_t(const Problem& p, bool skip_recompute, cudaStream_t st) {
    if (!p.L.tc_scans) return ffma_bwd<IO, DK, DV>(p, skip_recompute, st);
    const cudaError_t e = cw_tc_launch(p, /*bwd=*/true, skip_recompute, st);
    return e != cudaSuccess ? e : ffma_fallback<IO, DK, DV>(p, true, skip_recompute, st);
}

}  // namespace

#define GDN_VDISPATCH(FN, ...)                                                                      \
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

cudaError_t vec_launch_fwd(const Problem& p, cudaStream_t st) { GDN_VDISPATCH(vlaunch_fwd_t, p, st); }
cudaError_t vec_launch_bwd(const Problem& p, bool skip_recompute, cudaStream_t st) { GDN_VDISPATCH(vlaunch_bwd_t, p, skip_recompute, st); }

}  // namespace gdn
