// tcgen05 / TMEM kernels of the channel-wise path (per-channel gates, Eq. 1 of the paper as printed) for bf16 I/O and
// d_k = d_v = 128.
//
// "The channel-wise path folds the per-channel decay Diag(e^{g_t}) inside those contractions" (Appendix A): with the
// chunk-local cumulative log decay gam_i in R^{d_k}, Gam_i = exp(gam_i), and a reference S in R^{d_k} of the chunk, every factor
// exp(gam_i - gam_j) of a token pair splits into a row part and a column part, and the keys and queries are scaled once, element by
// element, before any product.  With G_i = Gam_i / S:
//     q~_i = G_i . q_i        k+_i = G_i . b_i . k_i   (row role)        k-_j = k_j / G_j   (column role)
//     v~_i = w_i . v_i                                                    dO'  = scale dO (the factor is applied to fp32 accumulators)
// In these variables, and with the states h~ = Diag(S) h and dh'' = Diag(G_e) dh' (e: the chunk's end), the chunk is a decay-free
// delta rule whose token-token matrices carry plain triangular masks:
//     A = stril(K+ K-^T)   P = tril(Q~ K-^T)   T = (I + A)^-1   W = T K+   U~ = T V~   E = (Q~ - P W)^T dO'
//     U = U~ - W h~   dU = P^T dO' + K- dh''
//     dP = tril(dO' U^T)   dW = -dU h~^T   dXk = T^T dW   dXv = T^T dU   dA = -stril(dXk W^T + dXv U~^T)
//     dQ~ = dO' h~^T + dP K-    dK+ = dXk + dA K-     dK- = U dh''^T + dP^T Q~ + dA^T K+
//     h' = Gam_e . h + G_e . (K-^T U)        dh = Gam_e . dh' + S . (E - W^T (K- dh''))                (the carries)
// and the gradients of the caller's tensors follow element by element.  S = 2^ref, per channel, lies in the middle of the range
// that gam and the chunk start (gam = 0) span: a chunk that decays by e^-80 then scales its operands and states by factors
// between e^-40 and e^40.  With S = 1, K- reached e^80 and dh'' e^-80 of the values: an increment K-^T U beyond fp32 for values
// of 1e5, a subnormal dh'' for gradients of 1e-6.  A power of two, because every operand is then the same number
// with another exponent, and no rounding depends on S.  Beside the carries (tc_scan_cw in gdn_tc.cu):
//   cw_scale  scaled operand tiles as bf16 tile images, gam, ref; checks that gam stays in range (beyond it the split would
//             need reference points inside the chunk): otherwise it sets the fall-back word of the workspace header, the kernels below
//             stand down, and the FFMA sequence enqueued behind them computes the call (gdn_simt_vec.cu)
//   cw_prep   [Q~;K+] K-^T, fp32 blocked inversion, W^T, U~^T, (P^T dO')^T, E               (tcgen05)
//   cw_intra  the thirteen products of the gradient stage in four dependent steps (K#2 reuses T), and from them dq, dk, dv,
//             db, dw, and dg by a reverse cumulative sum per channel                                  (tcgen05)
// The tensor-core kernels are written straight-line (a CTA walks over chunk-heads; one thread issues every product and
// copy; CTA-wide barriers between the steps).  Accumulators live in one TMEM reservation at fixed column offsets; every wait
// is bounded.
#include "tc_common.cuh"
#include "tc_inverse.cuh"

namespace gdn {
namespace {

using namespace tc;

constexpr int D = 128;
constexpr int kT = 256;               // 8 warps: TMEM lane quadrant = warp % 4, column half = warp / 4
constexpr float kMaxDecay = 80.f;     // bound on |gam| inside a chunk, hence |log2 S| <= 58
constexpr float kMaxSwing = 92.f;     // ... and on the range of gam and 0, hence |log2 G| <= 67: G, 1 / G and the factors of the carries (G_e
                                      // times another chunk's S) are normal numbers.  Gates that only decay never come near it.

// (chunk, head) of an elementwise CTA, from the chunk table (which these calls always build)
struct ChunkCtx { int hd, ch, tok0, len; };
__device__ __forceinline__ bool chunk_ctx(const Problem& p, ChunkCtx& x) {
    const WsHeader* hdr = reinterpret_cast<const WsHeader*>(p.ws);
    const int c = blockIdx.x / p.d.H;
    if (c >= hdr->n_chunks) return false;
    x.hd = blockIdx.x % p.d.H;
    x.ch = blockIdx.x;
    x.tok0 = reinterpret_cast<const int32_t*>(p.ws + p.L.chunk_tok0)[c];
    x.len = reinterpret_cast<const int32_t*>(p.ws + p.L.chunk_len)[c];
    return true;
}

// ------------------------------------------------------------------------------------------------
// cw_scale
// ------------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kT) cw_scale_kernel(Problem p) {
    wait_prerequisites();
    ChunkCtx x;
    if (!chunk_ctx(p, x)) return;
    extern __shared__ __align__(16) float gam[];   // [64][D + 1]
    __shared__ int bad;
    __shared__ int ref[D];
    const int H = p.d.H;
    const size_t base = ((size_t)x.tok0 * H + x.hd) * D, rs = (size_t)H * D;
    const __nv_bfloat16* qp = reinterpret_cast<const __nv_bfloat16*>(p.q) + base;
    const __nv_bfloat16* kp = reinterpret_cast<const __nv_bfloat16*>(p.k) + base;
    const __nv_bfloat16* vp = reinterpret_cast<const __nv_bfloat16*>(p.v) + base;
    if (threadIdx.x == 0) bad = 0;
    __syncthreads();
    if (threadIdx.x < D) {
        const int r = threadIdx.x;
        float s = 0.f, lo = 0.f, hi = 0.f;   // (the chunk start counts: the states enter there)
#pragma unroll 1
        for (int i0 = 0; i0 < kC; i0 += 16) {   // sixteen loads in flight, then their running sum in token order
            float g16[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) g16[k] = (i0 + k < x.len) ? p.gv[base + (size_t)(i0 + k) * rs + r] : 0.f;
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                s += g16[k];
                gam[(i0 + k) * (D + 1) + r] = s;
                lo = fminf(lo, s);
                hi = fmaxf(hi, s);
            }
        }
        if (lo < -kMaxDecay || hi > kMaxDecay || hi - lo > kMaxSwing) bad = 1;   // (a NaN gate passes and comes out as NaN)
        ref[r] = __float2int_rn(0.5f * kLog2e * (lo + hi));
    }
    __syncthreads();
    if (bad) {
        if (threadIdx.x == 0) {
            WsHeader* hdr = reinterpret_cast<WsHeader*>(p.ws);
            hdr->cw_fallback = 1;
        }
        return;
    }
    float* wsG = reinterpret_cast<float*>(p.ws + p.L.gamma) + (size_t)x.ch * kC * D;
    for (int t = threadIdx.x; t < kC * D; t += kT) wsG[t] = gam[(t / D) * (D + 1) + t % D];
    if (threadIdx.x < D) reinterpret_cast<int32_t*>(p.ws + p.L.ref)[(size_t)x.ch * D + threadIdx.x] = ref[threadIdx.x];
    char* iQKp = p.ws + p.L.img_QKp + (size_t)x.ch * 32768;
    char* iKm = p.ws + p.L.img_Km + (size_t)x.ch * 16384;
    char* iVt = p.ws + p.L.img_Vt + (size_t)x.ch * 16384;
    for (int t = threadIdx.x; t < kC * 16; t += kT) {   // one 16-byte piece (8 features) of one token row
        const int i = t >> 4, ch = t & 15;
        float q8[8], k8[8], v8[8], a[8], b[8], c[8], b8[8], w8[8];
        const bool live = i < x.len;
#pragma unroll
        for (int j = 0; j < 8; ++j) { q8[j] = k8[j] = v8[j] = b8[j] = w8[j] = 0.f; }
        if (live) {
            unpack8(*reinterpret_cast<const uint4*>(qp + i * rs + ch * 8), q8);
            unpack8(*reinterpret_cast<const uint4*>(kp + i * rs + ch * 8), k8);
            unpack8(*reinterpret_cast<const uint4*>(vp + i * rs + ch * 8), v8);
            const float4* bp = reinterpret_cast<const float4*>(p.bv + base + i * rs + ch * 8);
            const float4* wp = reinterpret_cast<const float4*>(p.wv + base + i * rs + ch * 8);
            const float4 b0 = bp[0], b1 = bp[1], w0 = wp[0], w1 = wp[1];
            b8[0] = b0.x; b8[1] = b0.y; b8[2] = b0.z; b8[3] = b0.w; b8[4] = b1.x; b8[5] = b1.y; b8[6] = b1.z; b8[7] = b1.w;
            w8[0] = w0.x; w8[1] = w0.y; w8[2] = w0.z; w8[3] = w0.w; w8[4] = w1.x; w8[5] = w1.y; w8[6] = w1.z; w8[7] = w1.w;
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int r = ch * 8 + j;
            const float g = gam[i * (D + 1) + r];
            const float G = expf(g) * pow2(-ref[r]);
            const float bb = b8[j], ww = w8[j];
            a[j] = G * q8[j];                 // q~
            b[j] = G * bb * k8[j];            // k+
            c[j] = expf(-g) * pow2(ref[r]) * k8[j];   // k-
            v8[j] *= ww;                      // v~
        }
        *reinterpret_cast<uint4*>(iQKp + tile_chunk_off(128, i, ch)) = pack8(a);
        *reinterpret_cast<uint4*>(iQKp + tile_chunk_off(128, 64 + i, ch)) = pack8(b);
        *reinterpret_cast<uint4*>(iKm + tile_chunk_off(64, i, ch)) = pack8(c);
        *reinterpret_cast<uint4*>(iVt + tile_chunk_off(64, i, ch)) = pack8(v8);
    }
}

// Whether the tensor-core kernels of the call have work: no error so far, and no gates beyond their range (then the FFMA
// sequence enqueued behind them computes the call).
__device__ __forceinline__ bool cw_go(const WsHeader* hdr) { return hdr->status == GDN_OK && !hdr->cw_fallback; }

struct CwParams {
    Problem p;
    CUtensorMap tm_do;   // [T_total, H, 128] bf16, boxes of 64 tokens x 64 features of a head
    int with_bwd;        // prep: also produce E
};

// ------------------------------------------------------------------------------------------------
// cw_prep: P, T, W^T, U~^T and, for a backward, E = scale (Q~ - P W)^T dO.  Two CTAs per SM, as tc_prep_lr: a chain of four
// dependent phases, whose waits the neighbour fills: 95 -> 70 us on 4 x 16 heads of 2048 tokens against one CTA with look-ahead.
// K- is needed by the first product only and shares its place with the fp32
// blocks of the inversion and the staged E, so it is loaded at the top of its trip.
// ------------------------------------------------------------------------------------------------
namespace prepcw {
constexpr uint32_t QKP = 0;                 // [Q~ rows 0..63 ; K+ rows 64..127] x 128                              32 KB
constexpr uint32_t VO = 32768;              // [V~ ; dO] x 128                                                      32 KB
constexpr uint32_t XA = VO + 32768;         // K- [64][128]; then fp32 A [64][kLdi]; then T and W^T; finally the E image
constexpr uint32_t XT = XA + 17408;         // fp32 T [64][kLdi]
constexpr uint32_t PT = XT + 17408;         // P = tril(Q~ K-^T)                                                     8 KB
constexpr uint32_t KM = XA, TT = XA, WT = XA + 8192, ES = XA;
// U~^T [128][64] over V~ and (P^T dO)^T [128][64] over K+: two pieces of 64 rows each, 16 KB apart
constexpr uint32_t UTT = VO, PDOT = QKP + 8192;
constexpr uint32_t SMEM_BYTES = PT + 8192 + 1024 /* alignment slack */;
constexpr uint32_t C_S1 = 0, C_PDO = 64, C_W = 128, C_U = 192, C_E = 0;   // TMEM columns (256 allocated; E over S1 and P^T dO)
static_assert(ES + 32768 <= PT && PT % 1024 == 0, "T, W^T and the E image fit over the fp32 blocks");
static_assert(2 * (SMEM_BYTES + 4096) <= 228 * 1024, "two CTAs per SM");
}  // namespace prepcw

__global__ void __launch_bounds__(kT, 2) cw_prep_kernel(const __grid_constant__ CwParams P) {
    wait_prerequisites();
    using namespace prepcw;
    const Problem& p = P.p;
    const int H = p.d.H;
    const WsHeader* hdr = reinterpret_cast<const WsHeader*>(p.ws);
    if (!cw_go(hdr)) return;
    const int n_items = hdr->n_chunks * H;
    if ((int)blockIdx.x >= n_items) return;
    const bool bwd = P.with_bwd != 0;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* sm = align1024(smem_raw);
    __shared__ uint64_t bar_in, bar_k, bar_mma;
    __shared__ uint32_t tmem_slot;
    const int warp = warp_id(), lane = threadIdx.x & 31;
    const int q4 = warp & 3, grp = warp >> 2;
    const uint32_t lane_base = (uint32_t)(q4 * 32) << 16;
    if (threadIdx.x == 0) { mbar_init(&bar_in, 1); mbar_init(&bar_k, 1); mbar_init(&bar_mma, 1); fence_mbar_init(); }
    if (warp == 0) { tmem_alloc(&tmem_slot, 256); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    float* Af = reinterpret_cast<float*>(sm + XA);
    float* Tf = reinterpret_cast<float*>(sm + XT);
    const float sc = p.d.scale;
    bool ok = true, pending = false;
    uint32_t mma_phase = 0, in_phase = 0;
    // [Q~; K+], V~ and dO of a trip are dead once its last product is done: the next trip's are loaded right then, under the
    // readout of E and its store.
    auto issue_loads = [&](const ChunkInfo& c) {   // thread 0
        mbar_expect_tx(&bar_in, 49152 + (bwd ? 16384 : 0));
        bulk_load(sm + QKP, p.ws + p.L.img_QKp + (size_t)c.ch * 32768, 32768, &bar_in);
        for (int cb = 0; cb < 2; ++cb) {
            bulk_load(sm + VO + cb * 16384, p.ws + p.L.img_Vt + (size_t)c.ch * 16384 + cb * 8192, 8192, &bar_in);
            if (bwd) tma_load_3d(sm + VO + cb * 16384 + 8192, &P.tm_do, cb * 64, c.hd, c.tok0, &bar_in);
        }
        prefetch_l2_bulk(p.ws + p.L.img_Km + (size_t)c.ch * 16384, 16384);
        pending = true;
    };
    ChunkInfo x;
    chunk_entry_tab(p, x, blockIdx.x);
    if (threadIdx.x == 0) issue_loads(x);
#pragma unroll 1
    for (int item = blockIdx.x; item < n_items; item += gridDim.x, in_phase ^= 1) {
        const bool has_next = item + (int)gridDim.x < n_items;
        ChunkInfo xn = x;
        if (has_next) chunk_entry_tab(p, xn, item + gridDim.x);
        if (warp == 0 && elect_one()) {
            bulk_wait_read<0>();   // the previous trip's stores have read P and the E image: rewritten from here on
            mbar_expect_tx(&bar_k, 16384);
            bulk_load(sm + KM, p.ws + p.L.img_Km + (size_t)x.ch * 16384, 16384, &bar_k);
        }
        if (ok) {
            ok = mbar_wait(&bar_in, in_phase);
            if (ok && threadIdx.x == 0) pending = false;
        }
        {   // (waited for in any case: it is in flight)
            const bool okk = mbar_wait(&bar_k, in_phase);
            ok = ok && okk;
            if (!ok && lane == 0) report_timeout(p.ws, 40);
        }
        if (ok && bwd && x.len < kC) {   // rows beyond the sequence belong to somebody else (the images have zeros there)
            zero_tail_rows(sm + VO, 128, 64, x.len, kT);
            fence_async_smem();
        }
        __syncthreads();
        // ---- phase 1: S1 = [Q~; K+] K-^T  (rows 0..63: P before masking, rows 64..127: A)
        if (warp == 0 && elect_one() && ok) {
            tc_fence_after();
            mma_tile<128, 64, 128>(tmem + C_S1, op_k_major(sm + QKP, 128, 0), op_k_major(sm + KM, 64), false);
            mma_commit(&bar_mma);
        }
        GDN_WAIT_MMA(41)
        if (ok) {
            const int i = (q4 & 1) * 32 + lane, j0 = grp * 32;
#pragma unroll 2
            for (int part = 0; part < 4; ++part) {
                float v[8];
                const int jb = j0 + part * 8;
                tmem_ld8(tmem + lane_base + C_S1 + jb, v);
                tmem_wait_ld();
                if (q4 < 2) {   // P = tril(.), diagonal included
#pragma unroll
                    for (int j = 0; j < 8; ++j) v[j] = (jb + j <= i) ? v[j] : 0.f;
                    chunk_store(sm + PT, 64, i, jb >> 3, v);
                } else {        // A = stril(.)
#pragma unroll
                    for (int j = 0; j < 8; ++j) v[j] = (jb + j < i) ? v[j] : 0.f;
                    *reinterpret_cast<float4*>(Af + i * kLdi + jb) = make_float4(v[0], v[1], v[2], v[3]);
                    *reinterpret_cast<float4*>(Af + i * kLdi + jb + 4) = make_float4(v[4], v[5], v[6], v[7]);
                }
            }
        }
        tc_fence_before();
        fence_async_smem();
        __syncthreads();
        // (P^T dO)^T needs nothing of the inversion: it runs under it, covered by the next commit
        if (warp == 0 && elect_one() && ok) {
            tc_fence_after();
            if (bwd) mma_tile<128, 64, 64>(tmem + C_PDO, op_mn_major(sm + VO, 128, 64), op_mn_major(sm + PT, 64), false);
            bulk_store(p.ws + p.L.Pm + (size_t)x.ch * 8192, sm + PT, 8192);
            bulk_commit();
        }
        invert64(Af, Tf, [] { __syncthreads(); });
        {   // T -> bf16 tile over A: every row is in registers before the first one is written
            const int cch = threadIdx.x & 7;
            float a[2][8];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int i = (threadIdx.x >> 3) + 32 * h;
                if ((cch >> 1) <= (i >> 4)) {   // (beyond the block diagonal: zero)
                    ld8s(Tf + i * kLdi + cch * 8, a[h]);
                } else {
#pragma unroll
                    for (int k = 0; k < 8; ++k) a[h][k] = 0.f;
                }
            }
            __syncthreads();
#pragma unroll
            for (int h = 0; h < 2; ++h) chunk_store(sm + TT, 64, (threadIdx.x >> 3) + 32 * h, cch, a[h]);
        }
        fence_async_smem();
        __syncthreads();
        // ---- phase 2: W^T = K+^T T^T ; U~^T = V~^T T^T
        if (warp == 0 && elect_one() && ok) {
            tc_fence_after();
            mma_tile<128, 64, 64>(tmem + C_W, op_mn_major(sm + QKP, 128, 64), op_k_major(sm + TT, 64), false);
            mma_tile<128, 64, 64>(tmem + C_U, op_mn_major(sm + VO, 128, 0), op_k_major(sm + TT, 64), false);
            mma_commit(&bar_mma);
            bulk_store(p.ws + p.L.Tm + (size_t)x.ch * 8192, sm + TT, 8192);
            bulk_commit();
        }
        GDN_WAIT_MMA(42)
        if (ok) {
            const int f = q4 * 32 + lane, i0 = grp * 32;
            unsigned char* ut = sm + UTT + (f >> 6) * 16384;      // this feature's half of the two-piece tiles
            unsigned char* pd = sm + PDOT + (f >> 6) * 16384;
#pragma unroll 1
            for (int part = 0; part < 4; ++part) {
                const int ib = i0 + part * 8;
                float a[8], b[8], c[8];
                tmem_ld8(tmem + lane_base + C_W + ib, a);
                tmem_ld8(tmem + lane_base + C_U + ib, b);
                tmem_ld8(tmem + lane_base + C_PDO + ib, c);
                tmem_wait_ld();
                chunk_store(sm + WT, 128, f, ib >> 3, a);
                chunk_store(ut, 64, f & 63, ib >> 3, b);
                if (bwd) chunk_store(pd, 64, f & 63, ib >> 3, c);
            }
        }
        tc_fence_before();
        fence_async_smem();
        __syncthreads();
        // ---- phase 3: E = Q~^T dO - W^T (P^T dO)   (the second operand of the second product in two pieces: 64 columns each)
        if (warp == 0 && elect_one() && ok) {
            tc_fence_after();
            if (bwd) {
                mma_tile<128, 128, 64>(tmem + C_E, op_mn_major(sm + QKP, 128, 0), op_mn_major(sm + VO, 128, 64), false);
                mma_tile<128, 64, 64>(tmem + C_E, op_k_major(sm + WT, 128), op_k_major(sm + PDOT, 64), true, /*neg_a=*/true);
                mma_tile<128, 64, 64>(tmem + C_E + 64, op_k_major(sm + WT, 128), op_k_major(sm + PDOT + 16384, 64), true, /*neg_a=*/true);
            }
            bulk_store(p.ws + p.L.img_W + (size_t)x.ch * 16384, sm + WT, 16384);
            bulk_store(p.ws + p.L.img_U + (size_t)x.ch * 16384, sm + UTT, 8192);
            bulk_store(p.ws + p.L.img_U + (size_t)x.ch * 16384 + 8192, sm + UTT + 16384, 8192);
            bulk_commit();
            bulk_wait_read<0>();   // T, W^T and U~^T have left: the E image and the next inputs go over them
            mma_commit(&bar_mma);
        }
        GDN_WAIT_MMA(43)
        if (ok && has_next && threadIdx.x == 0) issue_loads(xn);   // every input tile has been read for the last time
        if (ok && bwd) {   // E -> bf16 tile image
            const int rr = q4 * 32 + lane, c0 = grp * 64;
#pragma unroll 2
            for (int part = 0; part < 8; ++part) {
                const int cb = c0 + part * 8;
                float v[8];
                tmem_ld8(tmem + lane_base + C_E + cb, v);
                tmem_wait_ld();
#pragma unroll
                for (int k = 0; k < 8; ++k) v[k] *= sc;
                chunk_store(sm + ES, 128, rr, cb >> 3, v);
            }
        }
        tc_fence_before();
        fence_async_smem();
        __syncthreads();
        if (warp == 0 && elect_one() && ok && bwd) {
            bulk_store(p.ws + p.L.img_E + (size_t)x.ch * 32768, sm + ES, 32768);
            bulk_commit();
        }
        if (!ok) break;
        x = xn;
    }
    if (warp == 0) bulk_wait_read<0>();
    if (threadIdx.x == 0 && pending) (void)mbar_wait(&bar_in, in_phase);   // after a timeout a load may still be in flight
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 256);
}

// ------------------------------------------------------------------------------------------------
// cw_eprep: E alone, from the stored P and W^T (backward on a workspace fresh from the forward).  Two CTAs per SM.
// ------------------------------------------------------------------------------------------------
namespace eprepcw {
constexpr uint32_t QT = 0;                  // Q~ [64][128]                                  16 KB
constexpr uint32_t DOT = 16384;             // dO [64][128]                                  16 KB
constexpr uint32_t WT = 32768;              // W^T [128][64]                                 16 KB
constexpr uint32_t PT = 49152;              // P [64][64]                                     8 KB
constexpr uint32_t PDOT = PT + 8192;        // (P^T dO)^T [128][64]                          16 KB
constexpr uint32_t ES = PDOT + 16384;       // staged E image [128][128]                     32 KB
constexpr uint32_t SMEM_BYTES = ES + 32768 + 1024 /* alignment slack */;
constexpr uint32_t C_PDO = 0, C_E = 128;    // TMEM columns (256 allocated)
static_assert(2 * (SMEM_BYTES + 4096) <= 228 * 1024, "two CTAs per SM");
}  // namespace eprepcw

__global__ void __launch_bounds__(kT, 2) cw_eprep_kernel(const __grid_constant__ CwParams P) {
    wait_prerequisites();
    using namespace eprepcw;
    const Problem& p = P.p;
    const int H = p.d.H;
    const WsHeader* hdr = reinterpret_cast<const WsHeader*>(p.ws);
    check_fresh_seqlens(p);
    // (its verdict may come at any moment and concerns the kernels behind this one: either status is a go here, for every thread)
    const int32_t status = hdr->status;
    if (!(status == GDN_OK || (status == GDN_ERR_BAD_SEQLENS && hdr->seqlens_ok)) || hdr->cw_fallback) return;
    const int n_items = hdr->n_chunks * H;
    if ((int)blockIdx.x >= n_items) return;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* sm = align1024(smem_raw);
    __shared__ uint64_t bar_in, bar_mma;
    __shared__ uint32_t tmem_slot;
    const int warp = warp_id(), lane = threadIdx.x & 31;
    const int q4 = warp & 3, grp = warp >> 2;
    const uint32_t lane_base = (uint32_t)(q4 * 32) << 16;
    if (threadIdx.x == 0) { mbar_init(&bar_in, 1); mbar_init(&bar_mma, 1); fence_mbar_init(); }
    if (warp == 0) { tmem_alloc(&tmem_slot, 256); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    const float sc = p.d.scale;
    bool ok = true, pending = false;
    uint32_t mma_phase = 0, in_phase = 0;
    auto issue_loads = [&](const ChunkInfo& c) {   // thread 0: every tile of a trip is dead once its last product is done
        mbar_expect_tx(&bar_in, 57344);
        for (int cb = 0; cb < 2; ++cb) {
            bulk_load(sm + QT + cb * 8192, p.ws + p.L.img_QKp + (size_t)c.ch * 32768 + cb * 16384, 8192, &bar_in);
            tma_load_3d(sm + DOT + cb * 8192, &P.tm_do, cb * 64, c.hd, c.tok0, &bar_in);
        }
        bulk_load(sm + PT, p.ws + p.L.Pm + (size_t)c.ch * 8192, 8192, &bar_in);
        bulk_load(sm + WT, p.ws + p.L.img_W + (size_t)c.ch * 16384, 16384, &bar_in);
        pending = true;
    };
    ChunkInfo x;
    chunk_entry_tab(p, x, blockIdx.x);
    if (threadIdx.x == 0) issue_loads(x);
#pragma unroll 1
    for (int item = blockIdx.x; item < n_items; item += gridDim.x, in_phase ^= 1) {
        const bool has_next = item + (int)gridDim.x < n_items;
        ChunkInfo xn = x;
        if (has_next) chunk_entry_tab(p, xn, item + gridDim.x);
        if (ok) {
            ok = mbar_wait(&bar_in, in_phase);
            if (!ok && lane == 0) report_timeout(p.ws, 46);
            if (ok && threadIdx.x == 0) pending = false;
        }
        if (ok && x.len < kC) {
            zero_tail_rows(sm + DOT, 64, 0, x.len, kT);
            fence_async_smem();
        }
        __syncthreads();
        if (warp == 0 && elect_one() && ok) {   // (P^T dO)^T ; Q~^T dO
            tc_fence_after();
            mma_tile<128, 64, 64>(tmem + C_PDO, op_mn_major(sm + DOT, 64), op_mn_major(sm + PT, 64), false);
            mma_commit(&bar_mma);
            mma_tile<128, 128, 64>(tmem + C_E, op_mn_major(sm + QT, 64), op_mn_major(sm + DOT, 64), false);
        }
        GDN_WAIT_MMA(47)
        if (ok) {
            const int f = q4 * 32 + lane, i0 = grp * 32;
#pragma unroll 2
            for (int part = 0; part < 4; ++part) {
                float v[8];
                tmem_ld8(tmem + lane_base + C_PDO + i0 + part * 8, v);
                tmem_wait_ld();
                chunk_store(sm + PDOT, 128, f, (i0 >> 3) + part, v);
            }
        }
        tc_fence_before();
        fence_async_smem();
        __syncthreads();
        if (warp == 0 && elect_one() && ok) {   // E -= W^T (P^T dO)
            tc_fence_after();
            mma_tile<128, 128, 64>(tmem + C_E, op_k_major(sm + WT, 128), op_k_major(sm + PDOT, 128), true, /*neg_a=*/true);
            bulk_wait_read<0>();   // the previous trip's store has read the E image
            mma_commit(&bar_mma);
        }
        GDN_WAIT_MMA(48)
        if (ok && has_next && threadIdx.x == 0) issue_loads(xn);
        if (ok) {
            const int rr = q4 * 32 + lane, c0 = grp * 64;
#pragma unroll 2
            for (int part = 0; part < 8; ++part) {
                const int cb = c0 + part * 8;
                float v[8];
                tmem_ld8(tmem + lane_base + C_E + cb, v);
                tmem_wait_ld();
#pragma unroll
                for (int k = 0; k < 8; ++k) v[k] *= sc;
                chunk_store(sm + ES, 128, rr, cb >> 3, v);
            }
        }
        tc_fence_before();
        fence_async_smem();
        __syncthreads();
        if (warp == 0 && elect_one() && ok) {
            bulk_store(p.ws + p.L.img_E + (size_t)x.ch * 32768, sm + ES, 32768);
            bulk_commit();
        }
        if (!ok) break;
        x = xn;
    }
    if (warp == 0) bulk_wait_read<0>();
    if (threadIdx.x == 0 && pending) (void)mbar_wait(&bar_in, in_phase);   // after a timeout a load may still be in flight
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 256);
}

// ------------------------------------------------------------------------------------------------
// cw_intra: every gradient of one (chunk, head).
//
// Four dependent steps (products; [readout] what the threads make of them):
// (h and Gam stand for h~ and G of the head of this file.)
//   1  (W h)^T ; (K- dh'')^T ; (P^T dO)^T             [U = U~ - W h ; dU = scale P^T dO + K- dh'']
//   2  dP = dO U^T ; dXv^T = dU^T T ; under the readout h dO^T ; dK-^T = dh'' U^T        [scale tril ; dv, dw]
//   3  dA = dXv U^T (K#2) ; under the readout dK+^T = -h dXv^T ; K-^T dP^T ; Q~^T dP               [-stril]
//   4  dK+^T += K-^T dA^T ; (Q~^T dP) += K+^T dA                                                   [dq, dk, db, dg]
// What bounds it is HBM: 176 KB of operands, 144 KB of gates, inputs and gammas, 144 KB of gradients per chunk-head.  The
// gradients are made with features on the TMEM lanes and tokens on the columns: a warp's accesses to the gate vectors and
// gradients are then whole 128-byte lines, all lanes work (a 64-row accumulator fills half of them), and the sums of dg
// over the tokens of a chunk run along a thread's own columns.  So nothing passes through HBM between the products and the
// elementwise part: with fp32 scratch and a kernel of its own (256 KB more traffic per chunk-head) the two took 300 us on
// 4 x 16 heads of 2048 tokens, this kernel 211 us.
// (L2 prefetches of what the elementwise part reads, a trip ahead, made it slower: 481 -> 495 us for the call.)
// ------------------------------------------------------------------------------------------------
namespace intracw {
constexpr uint32_t QKM = 0;                 // [Q~ rows 0..63 ; K- rows 64..127] x 128         32 KB
constexpr uint32_t KP = 32768;              // K+ [64][128]                                     16 KB
constexpr uint32_t DOT = KP + 16384;        // dO  [64][128]                                    16 KB
constexpr uint32_t WT = DOT + 16384;        // W^T  [128][64]                                   16 KB
constexpr uint32_t UTT = WT + 16384;        // U~^T [128][64]                                   16 KB
constexpr uint32_t TT = UTT + 16384;        // T [64][64]; later dA                              8 KB
constexpr uint32_t PT = TT + 8192;          // P [64][64]; later dP                              8 KB
constexpr uint32_t HH = PT + 8192;          // h~ [128][128]                                    32 KB
constexpr uint32_t DH = HH + 32768;         // dh'' [128][128]                                  32 KB
constexpr uint32_t UT = DH + 32768;         // U^T  [128][64]                                   16 KB
constexpr uint32_t DUT = UT + 16384;        // dU^T [128][64]; later dXv^T [128][64]            16 KB
constexpr uint32_t SMEM_BYTES = DUT + 16384 + 1024;
constexpr uint32_t DA = TT, DP = PT, DXVT = DUT;   // (dA over T, dP over P, dXv^T over dU^T, each after its last reader)
// TMEM columns (512 allocated, fixed offsets): eight accumulators of 64 columns, features on the lanes except dP and dA
// (token rows on lanes 0..15 of each quadrant).
constexpr uint32_t C_A = 0, C_B = 64, C_PDO = 128, C_PP = 192, C_DQ = 256, C_KM = 320, C_KP = 384, C_KM2 = 448;
constexpr uint32_t C_DQ2 = C_B;             // (K-^T dP^T, over an accumulator of step 1)
constexpr int kWorkers = 512;               // 16 readout warps: lane quadrant = warp % 4, tokens 16 (warp / 4) ..
                                            // (a seventeenth warp would cost every thread 32 of its 128 registers; warp 0 issues
                                            // the products, warp 1 the loads)
constexpr int kTok = 16;                    // tokens of a thread
static_assert(SMEM_BYTES <= 220 * 1024, "shared memory budget");
}  // namespace intracw

__global__ void __launch_bounds__(intracw::kWorkers, 1) cw_intra_kernel(const __grid_constant__ CwParams P) {
    wait_prerequisites();
    using namespace intracw;
    const Problem& p = P.p;
    const int H = p.d.H;
    const WsHeader* hdr = reinterpret_cast<const WsHeader*>(p.ws);
    if (!cw_go(hdr)) return;
    const int n_items = hdr->n_chunks * H;
    if ((int)blockIdx.x >= n_items) return;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* sm = align1024(smem_raw);
    __shared__ uint64_t bar_s, bar_a, bar_b, bar_k, bar_mma;
    __shared__ uint32_t tmem_slot;
    __shared__ float tot[4][D], end_part[4][D];   // per token group and channel: sum of dgam, part of the chunk-end term
    const int warp = warp_id(), lane = threadIdx.x & 31;
    const int q4 = warp & 3, grp = warp >> 2;
    const uint32_t lane_base = (uint32_t)(q4 * 32) << 16;
    if (threadIdx.x == 0) {
        mbar_init(&bar_s, 1); mbar_init(&bar_a, 1); mbar_init(&bar_b, 1); mbar_init(&bar_k, 1); mbar_init(&bar_mma, 1);
        fence_mbar_init();
    }
    if (warp == 0) { tmem_alloc(&tmem_slot, 512); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    const int f = q4 * 32 + lane;             // feature row of the M = 128 accumulators
    const int tr = q4 * 16 + (lane & 15);     // token row of the M = 64 accumulators (lanes 0..15 of the quadrant)
    const int i0 = grp * kTok;                // first of this thread's 16 tokens
    const float sc = p.d.scale;
    const bool ga = lane < 16;
    bool ok = true;
    uint32_t mma_phase = 0, in_phase = 0;
    // The tiles of a trip arrive in groups, each loaded during the previous trip as soon as the last product that reads its
    // region is done (look-ahead without a second buffer):
    //   b  W^T, U~^T     after the first readout          a  dO after step 2, P after step 4
    //   s  dh'' after step 2, h after step 4              k  Q~, K-, K+, T after step 4
    bool pend_s = false, pend_a = false, pend_b = false, pend_k = false;   // the elected lane of warp 1
    auto load_s1 = [&](size_t c) {
        mbar_expect_tx(&bar_s, 65536);
        bulk_load(sm + DH, p.ws + p.L.dhn + c * 32768, 32768, &bar_s);
        pend_s = true;
    };
    auto load_s2 = [&](size_t c) { bulk_load(sm + HH, p.ws + p.L.hc + c * 32768, 32768, &bar_s); };
    auto load_a1 = [&](int c) {
        ChunkInfo y;
        chunk_entry_tab(p, y, c);
        mbar_expect_tx(&bar_a, 24576);
        for (int cb = 0; cb < 2; ++cb) tma_load_3d(sm + DOT + cb * 8192, &P.tm_do, cb * 64, y.hd, y.tok0, &bar_a);
        pend_a = true;
    };
    auto load_a2 = [&](size_t c) { bulk_load(sm + PT, p.ws + p.L.Pm + c * 8192, 8192, &bar_a); };
    auto load_b = [&](size_t c) {
        mbar_expect_tx(&bar_b, 32768);
        bulk_load(sm + WT, p.ws + p.L.img_W + c * 16384, 16384, &bar_b);
        bulk_load(sm + UTT, p.ws + p.L.img_U + c * 16384, 16384, &bar_b);
        pend_b = true;
    };
    auto load_k = [&](size_t c) {
        const char* iQKp = p.ws + p.L.img_QKp + c * 32768;
        const char* iKm = p.ws + p.L.img_Km + c * 16384;
        mbar_expect_tx(&bar_k, 57344);
        for (int cb = 0; cb < 2; ++cb) {
            bulk_load(sm + QKM + cb * 16384 + 8192, iKm + cb * 8192, 8192, &bar_k);             // K-
            bulk_load(sm + QKM + cb * 16384, iQKp + cb * 16384, 8192, &bar_k);                  // Q~
            bulk_load(sm + KP + cb * 8192, iQKp + cb * 16384 + 8192, 8192, &bar_k);             // K+
        }
        bulk_load(sm + TT, p.ws + p.L.Tm + c * 8192, 8192, &bar_k);
        pend_k = true;
    };
    if (warp == 1 && elect_one()) {
        const size_t c = blockIdx.x;
        load_s1(c); load_s2(c); load_k(c); load_b(c); load_a1((int)c); load_a2(c);
    }
#pragma unroll 1
    for (int item = blockIdx.x; item < n_items; item += gridDim.x, in_phase ^= 1) {
        const size_t ch = (size_t)item;
        const bool has_next = item + (int)gridDim.x < n_items;
        const size_t chn = ch + gridDim.x;
        ChunkInfo x;
        chunk_entry_tab(p, x, item);
        const size_t rs = (size_t)H * D, base = ((size_t)x.tok0 * H + x.hd) * D + (size_t)i0 * rs + f;   // this thread's channel of its first token
        const int live = x.len - i0;          // tokens of this thread inside the sequence (may be negative)
        const bool whole = live >= kTok;      // (two copies of the accesses: a condition at each of them costs more than it skips)
        if (ok) {   // everything step 1 reads (the carries left h~ and dh'', the forms used here)
            ok = mbar_wait(&bar_s, in_phase) && mbar_wait(&bar_k, in_phase) && mbar_wait(&bar_b, in_phase) && mbar_wait(&bar_a, in_phase);
            if (!ok && lane == 0) report_timeout(p.ws, 44);
            if (ok) pend_s = pend_k = pend_a = pend_b = false;
        }
        if (ok && x.len < kC) {   // rows beyond the sequence belong to somebody else (the images have zeros there)
            zero_tail_rows(sm + DOT, 64, 0, x.len, kWorkers);
            fence_async_smem();
        }
        __syncthreads();
        // ---- step 1
        if (warp == 0 && elect_one() && ok) {
            tc_fence_after();
            mma_tile<128, 64, 128>(tmem + C_A, op_mn_major(sm + HH, 128), op_mn_major(sm + WT, 128), false);
            mma_tile<128, 64, 128>(tmem + C_B, op_mn_major(sm + DH, 128), op_k_major(sm + QKM, 128, 64), false);
            mma_tile<128, 64, 64>(tmem + C_PDO, op_mn_major(sm + DOT, 64), op_mn_major(sm + PT, 64), false);
            mma_commit(&bar_mma);
        }
        float end = 0.f;   // chunk-end term of the decay gradient: rowdot(dh'', h), and below sum_j k-_j (U dh''^T)_j
        {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                float a[8], b[8];
                chunk_load(sm + DH, 128, f, grp * 4 + k, a);
                chunk_load(sm + HH, 128, f, grp * 4 + k, b);
#pragma unroll
                for (int j = 0; j < 8; ++j) end = fmaf(a[j], b[j], end);
            }
        }
        GDN_WAIT_MMA(45)
        if (ok) {   // U^T = U~^T - (W h)^T ; dU^T = scale (P^T dO)^T + (K- dh'')^T
#pragma unroll
            for (int part = 0; part < 2; ++part) {
                const int ib = i0 + part * 8;
                float t[8], kb[8], pd[8], u[8];
                tmem_ld8(tmem + lane_base + C_A + ib, t);
                tmem_ld8(tmem + lane_base + C_B + ib, kb);
                tmem_ld8(tmem + lane_base + C_PDO + ib, pd);
                chunk_load(sm + UTT, 128, f, ib >> 3, u);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 8; ++j) { u[j] -= t[j]; pd[j] = fmaf(sc, pd[j], kb[j]); }
                chunk_store(sm + UT, 128, f, ib >> 3, u);
                chunk_store(sm + DUT, 128, f, ib >> 3, pd);
            }
        }
        tc_fence_before();
        fence_async_smem();
        __syncthreads();
        // ---- step 2
        if (warp == 0 && elect_one() && ok) {
            tc_fence_after();
            mma_tile<64, 64, 128>(tmem + C_PP, op_k_major(sm + DOT, 64), op_mn_major(sm + UT, 128), false);
            mma_tile<128, 64, 64>(tmem + C_A, op_k_major(sm + DUT, 128), op_mn_major(sm + TT, 64), false);
            mma_commit(&bar_mma);
            mma_tile<128, 64, 128>(tmem + C_DQ, op_k_major(sm + HH, 128), op_k_major(sm + DOT, 64), false);
            mma_tile<128, 64, 128>(tmem + C_KM, op_k_major(sm + DH, 128), op_mn_major(sm + UT, 128), false);
        }
        if (warp == 1 && elect_one() && ok && has_next) load_b(chn);   // W^T (step 1) and U~^T (the readout) have been read for the last time
        float wv[kTok];
        uint32_t vraw[kTok];
        {   // v and w of this thread's channel, while the products run
            const uint16_t* vp = reinterpret_cast<const uint16_t*>(p.v) + base;
            const float* wp = p.wv + base;
            if (whole) {
#pragma unroll
                for (int i = 0; i < kTok; ++i) { wv[i] = wp[i * rs]; vraw[i] = vp[i * rs]; }
            } else {
#pragma unroll
                for (int i = 0; i < kTok; ++i) { wv[i] = i < live ? wp[i * rs] : 0.f; vraw[i] = i < live ? vp[i * rs] : 0u; }
            }
        }
        GDN_WAIT_MMA(46)
        if (ok) {
            float x8[2][8], v[8];
#pragma unroll
            for (int part = 0; part < 2; ++part) tmem_ld8(tmem + lane_base + C_A + i0 + part * 8, x8[part]);   // dXv^T, all lanes
            tmem_wait_ld();
            __nv_bfloat16* dvp = reinterpret_cast<__nv_bfloat16*>(p.dv) + base;
            float* dwp = p.dwv + base;
#pragma unroll
            for (int part = 0; part < 2; ++part) {   // dXv^T: operand tile (over dU^T, which its product has read); dv = w . dXv, dw = v . dXv
                chunk_store(sm + DXVT, 128, f, (i0 >> 3) + part, x8[part]);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int i = part * 8 + j;
                    if (whole || i < live) {
                        dvp[i * rs] = __float2bfloat16_rn(wv[i] * x8[part][j]);
                        dwp[i * rs] = __uint_as_float(vraw[i] << 16) * x8[part][j];
                    }
                }
            }
#pragma unroll
            for (int part = 0; part < 2; ++part) {   // dP = scale tril(dO U^T), rows on lanes 0..15
                const int jb = i0 + part * 8;
                tmem_ld8(tmem + lane_base + C_PP + jb, v);
                tmem_wait_ld();
                if (ga) {
#pragma unroll
                    for (int j = 0; j < 8; ++j) v[j] = (jb + j <= tr) ? sc * v[j] : 0.f;
                    chunk_store(sm + DP, 64, tr, jb >> 3, v);
                }
            }
        }
        tc_fence_before();
        fence_async_smem();
        __syncthreads();
        // ---- step 3 (K#2): dA = -stril(dXv U^T) (= -stril(dXk W^T + dXv U~^T): dXk = T^T dW = -dXv h^T, U = U~ - W h)
        if (warp == 0 && elect_one() && ok) {
            tc_fence_after();
            mma_tile<64, 64, 128>(tmem + C_PP, op_mn_major(sm + DXVT, 128), op_mn_major(sm + UT, 128), false);
            mma_commit(&bar_mma);
            mma_tile<128, 64, 128>(tmem + C_KP, op_k_major(sm + HH, 128), op_mn_major(sm + DXVT, 128), false, /*neg_a=*/true);
            mma_tile<128, 64, 64>(tmem + C_DQ2, op_mn_major(sm + QKM, 128, 64), op_k_major(sm + DP, 64), false);
            mma_tile<128, 64, 64>(tmem + C_KM2, op_mn_major(sm + QKM, 128, 0), op_mn_major(sm + DP, 64), false);
        }
        GDN_WAIT_MMA(47)
        if (warp == 1 && elect_one() && ok && has_next) { load_a1((int)chn); load_s1(chn); }   // dO and dh'' have been read for the last time
        if (ok) {   // dA = -stril(.)  (over T, which step 2 has read)
#pragma unroll
            for (int part = 0; part < 2; ++part) {
                float v[8];
                const int jb = i0 + part * 8;
                tmem_ld8(tmem + lane_base + C_PP + jb, v);
                tmem_wait_ld();
                if (ga) {
#pragma unroll
                    for (int j = 0; j < 8; ++j) v[j] = (jb + j < tr) ? -v[j] : 0.f;
                    chunk_store(sm + DA, 64, tr, jb >> 3, v);
                }
            }
        }
        tc_fence_before();
        fence_async_smem();
        __syncthreads();
        // ---- step 4
        if (warp == 0 && elect_one() && ok) {
            tc_fence_after();
            mma_tile<128, 64, 64>(tmem + C_KP, op_mn_major(sm + QKM, 128, 64), op_k_major(sm + DA, 64), true);
            mma_tile<128, 64, 64>(tmem + C_KM2, op_mn_major(sm + KP, 64), op_mn_major(sm + DA, 64), true);
            mma_commit(&bar_mma);
        }
        const float* gp = reinterpret_cast<const float*>(p.ws + p.L.gamma) + ch * (kC * D) + i0 * D + f;
        const uint16_t* qp = reinterpret_cast<const uint16_t*>(p.q) + base;
        const uint16_t* kp = reinterpret_cast<const uint16_t*>(p.k) + base;
        const float* bp = p.bv + base;
        const int ref = reinterpret_cast<const int32_t*>(p.ws + p.L.ref)[ch * D + f];
        float g8[8], b8[8];
        uint32_t q8[8], k8[8];
        auto fetch = [&](int i1) {   // eight tokens' gates and inputs of this channel
            if (whole) {
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int i = i1 + j;
                    g8[j] = gp[i * D]; b8[j] = bp[i * rs]; q8[j] = qp[i * rs]; k8[j] = kp[i * rs];
                }
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int i = i1 + j;
                    g8[j] = gp[i * D];
                    b8[j] = i < live ? bp[i * rs] : 0.f;
                    q8[j] = i < live ? qp[i * rs] : 0u;
                    k8[j] = i < live ? kp[i * rs] : 0u;
                }
            }
        };
        fetch(0);   // while the products run
        const float S = pow2(ref), iS = pow2(-ref);
        GDN_WAIT_MMA(49)
        if (warp == 1 && elect_one() && ok && has_next) { load_k(chn); load_s2(chn); load_a2(chn); }   // every tile has been read for the last time
        float dgm[kTok];
        if (ok) {
            __nv_bfloat16* dqp = reinterpret_cast<__nv_bfloat16*>(p.dq) + base;
            __nv_bfloat16* dkp = reinterpret_cast<__nv_bfloat16*>(p.dk) + base;
            float* dbp = p.dbv + base;
#pragma unroll
            for (int part = 0; part < 2; ++part) {
                float dq[8], dq2[8], kr[8], km[8], km2[8];
                tmem_ld8(tmem + lane_base + C_DQ + i0 + part * 8, dq);
                tmem_ld8(tmem + lane_base + C_DQ2 + i0 + part * 8, dq2);
                tmem_ld8(tmem + lane_base + C_KP + i0 + part * 8, kr);
                tmem_ld8(tmem + lane_base + C_KM + i0 + part * 8, km);
                tmem_ld8(tmem + lane_base + C_KM2 + i0 + part * 8, km2);
                tmem_wait_ld();
                float dk[8], db[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float G = expf(g8[j]) * iS, iG = expf(-g8[j]) * S;
                    const float q = __uint_as_float(q8[j] << 16), k = __uint_as_float(k8[j] << 16);
                    dq[j] = G * fmaf(sc, dq[j], dq2[j]);             // dq = Gam . dQ~
                    const float row = G * kr[j];                     // what multiplies b . k in the row role
                    const float ucol = iG * km[j];
                    const float col = fmaf(iG, km2[j], ucol);        // column role
                    end = fmaf(k, ucol, end);
                    dk[j] = fmaf(b8[j], row, col);
                    db[j] = k * row;
                    dgm[part * 8 + j] = q * dq[j] + k * b8[j] * row - k * col;
                }
                if (part == 0) fetch(8);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int i = part * 8 + j;
                    if (whole || i < live) {
                        dqp[i * rs] = __float2bfloat16_rn(dq[j]);
                        dkp[i * rs] = __float2bfloat16_rn(dk[j]);
                        dbp[i * rs] = db[j];
                    }
                }
            }
#pragma unroll
            for (int i = kTok - 2; i >= 0; --i) dgm[i] += dgm[i + 1];   // sums from the end of this thread's tokens
            tot[grp][f] = dgm[0];
            end_part[grp][f] = end;
        }
        tc_fence_before();
        __syncthreads();   // every reader of this trip's tiles and accumulators is done; the sums are visible
        if (ok) {   // dg_j = sum_{i >= j} dgam_i + the chunk end
            float run = (end_part[0][f] + end_part[1][f]) + (end_part[2][f] + end_part[3][f]);
#pragma unroll
            for (int k = 3; k > 0; --k)
                if (k > grp) run += tot[k][f];
            float* dgp = p.dgv + base;
#pragma unroll
            for (int i = 0; i < kTok; ++i)
                if (whole || i < live) dgp[i * rs] = run + dgm[i];
        }
        if (!ok) break;
    }
    if (warp == 1 && elect_one() && !ok) {   // after a timeout a load may still be in flight: wait for it (bounded) before the CTA retires
        // a group issued during the trip that gave up belongs to the next phase of its barrier; one pending since the top of
        // that trip to the current one.  Both parities are tried; the wrong one returns at once or after the bound.
        uint64_t* bars[4] = {&bar_s, &bar_a, &bar_b, &bar_k};
        const bool pend[4] = {pend_s, pend_a, pend_b, pend_k};
        for (int i = 0; i < 4; ++i)
            if (pend[i]) { (void)mbar_wait(bars[i], in_phase); (void)mbar_wait(bars[i], in_phase ^ 1); }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 512);
}

}  // namespace

#undef GDN_WAIT_MMA

// Host side: the channel-wise calls on this route (bf16 I/O, d_k = d_v = 128).
cudaError_t cw_tc_launch(const Problem& p, bool bwd, bool skip_recompute, cudaStream_t st) {
    static SmemLimitOnce once_scale, once_prep, once_eprep, once_intra;
    const int CH = p.L.max_chunks * p.d.H, chains = p.d.N * p.d.H;
    cudaError_t e;
    const bool fresh = bwd && skip_recompute;   // the chunk table, the images, gam and the factors are still there
    if ((!fresh || p.Ttot == 0) && (e = launch_table(p, st, fresh)) != cudaSuccess) return e;
    const int sms = tc_sm_count(), grid = CH < sms ? CH : sms, grid2 = CH < 2 * sms ? CH : 2 * sms;
    CwParams P;
    P.p = p;
    P.with_bwd = bwd ? 1 : 0;
    if (p.Ttot > 0) {
        if (!make_tmap_bf16_heads(&P.tm_do, bwd ? p.dO : p.v, p.Ttot, p.d.H, D)) return cudaErrorUnknown;
        if (fresh) {
            if ((e = once_eprep.ensure(cw_eprep_kernel, eprepcw::SMEM_BYTES)) != cudaSuccess) return e;
            StageScope t(ST_EPREP, st);
            e = launch_kernel(cw_eprep_kernel, grid2, kT, eprepcw::SMEM_BYTES, st, P);
        } else {
            const uint32_t sm_scale = sizeof(float) * kC * (D + 1);
            if ((e = once_scale.ensure(cw_scale_kernel, sm_scale)) != cudaSuccess) return e;
            if ((e = once_prep.ensure(cw_prep_kernel, prepcw::SMEM_BYTES)) != cudaSuccess) return e;
            { StageScope t(ST_SCALE, st); launch_kernel(cw_scale_kernel, CH, kT, sm_scale, st, p); }
            { StageScope t(ST_PREP, st); e = launch_kernel(cw_prep_kernel, grid2, kT, prepcw::SMEM_BYTES, st, P); }
        }
        if (e != cudaSuccess) return e;
    }
    if (chains > 0 && (e = tc_launch_scan_channelwise(p, bwd ? (skip_recompute ? 1 : 2) : 0, st)) != cudaSuccess) return e;
    if (bwd && p.Ttot > 0) {
        if ((e = once_intra.ensure(cw_intra_kernel, intracw::SMEM_BYTES)) != cudaSuccess) return e;
        { StageScope t(ST_INTRA, st); launch_kernel(cw_intra_kernel, grid, intracw::kWorkers, intracw::SMEM_BYTES, st, P); }
    }
    return cudaGetLastError();
}

}  // namespace gdn
