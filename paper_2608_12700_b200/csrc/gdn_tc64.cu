// tcgen05 kernels for the scalar-gate linear recurrence (delta rule off: erase gate 0, write gate 1; the SSD-like
// row of Table 2 of the paper), bf16 I/O, d_k = d_v = 64, chunk 64.
//
// With the erase gate at zero the triangular solve vanishes (M = 0, T = I, W = 0, U~ = V; Section 4.1), so the
// carries lose their matrix operator:   h' = Gam_e h + Kb^T V,   dh = Gam_e dh' + scale (Diag(Gam) Q)^T dO.
// A chain step then costs one small product, and the whole backward fits two sequential passes per chain that
// move little more than the inputs and outputs themselves:
//   tc64_fwd  (one CTA per chain, chunks ascending)   h per chunk -> workspace (8 KB bf16 tile image per chunk)
//   tc64_bwd  (one CTA per chain, chunks descending)  dh' carried in registers; per chunk all of
//             P = tril(Q K^T . D), dP = scale tril(dO V^T), dv = scale P^T dO + Diag(e) K dh',
//             dq = scale Gam (dO h^T) + (dP.D) K,  dk = (dP.D)^T Q + Diag(e) V dh'^T,
//             dgamma_i = <q_i,dq_i> - <k_i,dk_i>,  dgamma_63 += sum_j r_j + Gam_e <dh',h>,  dg = reverse cumsum.
// Accumulators are 64 x 64 (M = 64: row i on TMEM lane i % 16 + 32 (i / 16)), token rows on lanes, so a thread owns
// a token row: row dots are thread-local and gradient rows leave with 16-byte stores.  Two CTAs share an SM.
// A 64-row accumulator occupies lanes 0..15 of each quadrant ("group A"), a second one lanes 16..31 of the same columns
// ("group B", address + 16 lanes).  What bounds a step is the issue of the readouts, so both groups run one instruction
// stream: either they hold two accumulators that are treated alike (Q K^T and dO V^T; K dh' and V dh'^T; P^T dO and
// (dP.D)^T Q), or the two column halves of one, which is then issued as two N = 32 products.
#define GDN_INLINE_WAIT   // small kernels: the polling loops sit at the wait sites (see tc_ptx.cuh)
#include "tc_common.cuh"

namespace gdn {

namespace {

constexpr int D6 = 64;
constexpr int kThreads64 = 256;   // 8 warps: lane quadrant = warp % 4 (rows 16 q .. 16 q + 15 on lanes 0..15), column half = warp / 4

struct Tc64Params {
    Problem p;
    CUtensorMap tm_q, tm_k, tm_v, tm_do;   // [T_total, H * 64] bf16, boxes of 64 rows x 64 columns
    CUtensorMap tm_dq, tm_dk, tm_dv;       // same geometry, for the gradient stores of full chunks
};

// Chunk-local cumulative log decay.  A block takes one chunk and 32 heads: the [64 tokens][32 heads] patch of g is
// read token by token (128 contiguous bytes each), then each warp scans the tokens of four heads (lane l owns
// tokens l and l + 32).  First kernel of a call.
__global__ void __launch_bounds__(256) tc64_gamma_kernel(Problem p) {
    wait_prerequisites();
    init_header_if_untabled(p);
    __shared__ float gs[kC][33];
    const int c = blockIdx.x, h0 = blockIdx.y * 32, H = p.d.H;
    if (c >= n_chunks_of(p)) return;
    const ChunkGeom cg = chunk_geom(p);
    const int tok0 = cg.chunk_tok0(c), len = cg.chunk_len(c);
    const int warp = warp_id(), lane = threadIdx.x & 31;
    for (int i = warp; i < kC; i += 8)
        gs[i][lane] = (i < len && h0 + lane < H) ? p.g[(size_t)(tok0 + i) * H + h0 + lane] : 0.f;
    __syncthreads();
    for (int hh = warp; hh < 32 && h0 + hh < H; hh += 8) {
        float a = gs[lane][hh], b = gs[lane + 32][hh];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const float ua = __shfl_up_sync(0xffffffffu, a, o), ub = __shfl_up_sync(0xffffffffu, b, o);
            if (lane >= o) { a += ua; b += ub; }
        }
        b += __shfl_sync(0xffffffffu, a, 31);
        float* out = reinterpret_cast<float*>(p.ws + p.L.gamma) + ((size_t)c * H + h0 + hh) * kC;
        out[lane] = a;
        out[lane + 32] = b;
    }
}

__device__ __forceinline__ void zero_tail_rows64(unsigned char* tile, int len) {   // [64][64] tile; threads 0 .. kThreads64-1
    for (int t = threadIdx.x; t < (kC - len) * 8; t += kThreads64)
        *reinterpret_cast<uint4*>(tile + tile_chunk_off(64, len + t / 8, t % 8)) = make_uint4(0, 0, 0, 0);
}

// ------------------------------------------------------------------------------------------------
// forward pass
// ------------------------------------------------------------------------------------------------
namespace f64 {
// The ring is what feeds a chain (a step is shorter than the latency of HBM), so it takes the shared memory that two CTAs per
// SM leave: with two slots a step waited for its tiles (256 chains of 64 chunks: 97 us with two slots, three barriers a step and the
// state on half of the lanes; 75 us now, 5.3 TB/s).
template <bool O> struct Cfg {   // O: the forward output is wanted
    static constexpr int STAGES = O ? 3 : 5;
    static constexpr uint32_t KT = 0, VT = 8192, QT = 16384, STAGE_BYTES = O ? 24576 : 16384;   // per slot: K, V (and Q)
    static constexpr uint32_t VE = STAGES * STAGE_BYTES;   // Diag(e) V
    static constexpr uint32_t HT = VE + 8192;              // two bf16 state tiles: leave for the workspace by bulk stores; operand of Q h
    static constexpr uint32_t PT = HT + 16384;             // P (only when o is wanted)
    static constexpr uint32_t SMEM_BYTES = PT + (O ? 8192 : 0) + 1024;
    static_assert(2 * (SMEM_BYTES + 4096) <= 228 * 1024, "two CTAs per SM");
};
}  // namespace f64

template <bool O>
__global__ void __launch_bounds__(kThreads64, 2) tc64_fwd_kernel(const __grid_constant__ Tc64Params P) {
    wait_prerequisites();
    using C = f64::Cfg<O>;
    constexpr int STAGES = C::STAGES;
    constexpr uint32_t KT = C::KT, VT = C::VT, QT = C::QT, STAGE_BYTES = C::STAGE_BYTES, VE = C::VE, PT = C::PT;
    const Problem& p = P.p;
    const WsHeader* hdr = reinterpret_cast<const WsHeader*>(p.ws);
    if (hdr->status != GDN_OK) return;
    const int H = p.d.H;
    const int n = blockIdx.x / H, hd = blockIdx.x % H;
    const SeqGeom cg = seq_geom(p, n);
    const int c0 = cg.c0, nsteps = cg.n_chunks;

    extern __shared__ unsigned char smem_raw[];
    unsigned char* sm = align1024(smem_raw);
    __shared__ __align__(16) float gl2[2][kC], Gam2[2][kC], ee2[2][kC];   // two sets: a step's gate arrays are made during the step before
    __shared__ uint64_t bar_full[STAGES], bar_mma;
    __shared__ uint32_t tmem_slot;
    const int warp = warp_id(), lane = threadIdx.x & 31;
    const int q4 = warp & 3, half = warp >> 2;
    const int r = q4 * 16 + (lane & 15);      // row of the 64 x 64 accumulators / of the state held by this lane
    const bool act = lane < 16;               // (output path: its accumulators are on lanes 0..15)
    const int cb0 = half * 32;                // first of its 32 columns there
    const int sc0 = (act ? 0 : 32) + half * 16;   // first of its 16 state columns (lanes 16..31 hold columns 32..63)
    constexpr uint32_t LB = 16u << 16;
    const uint32_t lane_base = (uint32_t)(q4 * 32) << 16;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) mbar_init(&bar_full[s], 1);
        mbar_init(&bar_mma, 1);
        fence_mbar_init();
    }
    if (warp == 0) { tmem_alloc(&tmem_slot, 256); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;

    auto fill = [&](int s) {
        const int stage = s % STAGES, tok0 = cg.chunk_tok0(c0 + s);
        unsigned char* st = sm + stage * STAGE_BYTES;
        mbar_expect_tx(&bar_full[stage], STAGE_BYTES);
        tma_load_2d(st + KT, &P.tm_k, hd * D6, tok0, &bar_full[stage]);
        tma_load_2d(st + VT, &P.tm_v, hd * D6, tok0, &bar_full[stage]);
        if (O) tma_load_2d(st + QT, &P.tm_q, hd * D6, tok0, &bar_full[stage]);
    };
    if (threadIdx.x == 0)
        for (int s = 0; s < STAGES && s < nsteps; ++s) fill(s);

    float st[16];
    const size_t soff = ((size_t)n * H + hd) * D6 * D6 + (size_t)r * D6 + sc0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        float4 v = p.h0 ? *reinterpret_cast<const float4*>(p.h0 + soff + 4 * k) : make_float4(0.f, 0.f, 0.f, 0.f);
        st[4 * k] = v.x; st[4 * k + 1] = v.y; st[4 * k + 2] = v.z; st[4 * k + 3] = v.w;
    }
    const float* gamma = reinterpret_cast<const float*>(p.ws + p.L.gamma);
    auto gate_row = [&](int step) { return gamma + ((size_t)(c0 + step) * H + hd) * kC; };
    auto make_gates = [&](int set, float g, float gend) {
        gl2[set][threadIdx.x] = g * kLog2e;
        Gam2[set][threadIdx.x] = expf(g);
        ee2[set][threadIdx.x] = ex2((gend - g) * kLog2e);
    };
    float gnext = 0.f, gend_next = 0.f;   // of the step after next
    if (threadIdx.x < kC && nsteps > 0) {
        make_gates(0, gate_row(0)[threadIdx.x], gate_row(0)[kC - 1]);
        if (nsteps > 1) { gnext = gate_row(1)[threadIdx.x]; gend_next = gate_row(1)[kC - 1]; }
    }
    __syncthreads();
    bool ok = true;
    uint32_t mma_phase = 0;
    auto give_up = [&](int s) { if (threadIdx.x == 0) drain_ring<STAGES>(bar_full, s, nsteps); };
#pragma unroll 1
    for (int s = 0; s < nsteps; ++s) {
        const int c = c0 + s, stage = s % STAGES, len = cg.chunk_len(c);
        const size_t ch = (size_t)c * H + hd;
        unsigned char* tiles = sm + stage * STAGE_BYTES;
        unsigned char* HT = sm + C::HT + (s & 1) * 8192;
        const float *gl = gl2[s & 1], *Gam = Gam2[s & 1], *ee = ee2[s & 1];
        ok = mbar_wait(&bar_full[stage], (s / STAGES) & 1);
        if (!ok) { if (lane == 0) report_timeout(p.ws, 40); give_up(s); break; }
        if (len < kC) {
            zero_tail_rows64(tiles + KT, len);
            zero_tail_rows64(tiles + VT, len);
            if (O) zero_tail_rows64(tiles + QT, len);
            __syncthreads();
        }
        const float Ge = Gam[kC - 1];
#pragma unroll
        for (int t = 0; t < 2; ++t) {   // Diag(e) V
            const int i = (threadIdx.x >> 3) + 32 * t, cch = threadIdx.x & 7;
            float v[8];
            chunk_load(tiles + VT, 64, i, cch, v);
            const float e = ee[i];
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] *= e;
            chunk_store(sm + VE, 64, i, cch, v);
        }
        // state entering the chunk -> bf16 tile: the workspace copy (and, for o, the MMA operand)
#pragma unroll
        for (int k = 0; k < 2; ++k)
            *reinterpret_cast<uint4*>(HT + tile_chunk_off(64, r, (sc0 >> 3) + k)) = pack8(st + 8 * k);
        // the next step's gate arrays (read from the top of that step on: this step's barrier publishes them)
        if (threadIdx.x < kC && s + 1 < nsteps) {
            make_gates((s + 1) & 1, gnext, gend_next);
            if (s + 2 < nsteps) { gnext = gate_row(s + 2)[threadIdx.x]; gend_next = gate_row(s + 2)[kC - 1]; }
        }
        fence_async_smem();
        __syncthreads();
        if (warp == 0 && elect_one()) {
            tc_fence_after();
            mma_tile<64, 32, 64>(tmem + 0, op_mn_major(tiles + KT, 64), op_mn_major(sm + VE, 64), false);              // Kb^T V
            mma_tile<64, 32, 64>(tmem + 0 + LB, op_mn_major(tiles + KT, 64), op_mn_major(sm + VE + 64, 64), false);    // (columns 32..63)
            if (O) {
                mma_tile<64, 64, 64>(tmem + 64, op_k_major(tiles + QT, 64), op_k_major(tiles + KT, 64), false);         // Q K^T
                mma_tile<64, 64, 64>(tmem + 128, op_k_major(tiles + QT, 64), op_mn_major(HT, 64), false);               // Q h
            }
            // the tile leaves through the async proxy (generic global stores would stall the next proxy fence); waiting for the
            // store of the step before to have read its tile, ahead of the commit, orders that read before the overwrite in the next step
            bulk_store(p.ws + p.L.hc + ch * 8192, HT, 8192);
            bulk_commit();
            bulk_wait_read<1>();
            mma_commit(&bar_mma);
        }
        GDN_WAIT_MMA(41)
        if (!ok) { give_up(s); break; }
        // without o the slot's K and V have now been read for the last time: refill it while the state is updated
        if (!O && threadIdx.x == 96 && s + STAGES < nsteps) fill(s + STAGES);
        if (O) {   // o = scale (Gam_i (Q h)_i + (P V)_i)
#pragma unroll 1
            for (int part = 0; part < 4; ++part) {
                float v[8];
                const int jb = cb0 + part * 8;
                tmem_ld8(tmem + lane_base + 64 + jb, v);
                tmem_wait_ld();
                if (act) {
                    float g8[8];
                    ld8s(gl + jb, g8);
#pragma unroll
                    for (int j = 0; j < 8; ++j) v[j] = (jb + j <= r) ? v[j] * ex2(gl[r] - g8[j]) : 0.f;
                    chunk_store(sm + PT, 64, r, jb >> 3, v);
                }
            }
            tc_fence_before();
            fence_async_smem();
            __syncthreads();
            if (warp == 0 && elect_one()) {
                tc_fence_after();
                mma_tile<64, 64, 64>(tmem + 192, op_k_major(sm + PT, 64), op_mn_major(tiles + VT, 64), false);          // P V
                mma_commit(&bar_mma);
            }
            GDN_WAIT_MMA(42)
            if (!ok) { give_up(s); break; }
            __nv_bfloat16* go = reinterpret_cast<__nv_bfloat16*>(p.o) + ((size_t)(cg.chunk_tok0(c) + r) * H + hd) * D6;
#pragma unroll 1
            for (int part = 0; part < 4; ++part) {
                float a[8], b[8];
                const int jb = cb0 + part * 8;
                tmem_ld8(tmem + lane_base + 128 + jb, a);
                tmem_ld8(tmem + lane_base + 192 + jb, b);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 8; ++j) a[j] = p.d.scale * fmaf(Gam[r], a[j], b[j]);
                if (act && r < len) *reinterpret_cast<uint4*>(go + jb) = pack8(a);
            }
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {   // h' = Gam_e h + Kb^T V
            float bf[8];
            tmem_ld8(tmem + lane_base + 0 + half * 16 + 8 * k, bf);
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < 8; ++j) st[8 * k + j] = fmaf(Ge, st[8 * k + j], bf[j]);
        }
        tc_fence_before();
        if (O) {
            __syncthreads();   // every reader of this stage's tiles is done
            if (threadIdx.x == 0 && s + STAGES < nsteps) fill(s + STAGES);
        }
    }
    if (warp == 0) bulk_wait_read<0>();
    if (p.hT && ok) {
#pragma unroll
        for (int k = 0; k < 4; ++k) *reinterpret_cast<float4*>(p.hT + soff + 4 * k) = make_float4(st[4 * k], st[4 * k + 1], st[4 * k + 2], st[4 * k + 3]);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 256);
}

// ------------------------------------------------------------------------------------------------
// backward pass
// ------------------------------------------------------------------------------------------------
namespace b64 {
constexpr int STAGES = 2;
constexpr uint32_t QT = 0, KT = 8192, VT = 16384, OT = 24576, HT = 32768, STAGE_BYTES = 40960;   // Q, K, V, dO, h
constexpr uint32_t DH = STAGES * STAGE_BYTES;   // bf16 tile of the carried dh' during phase 1, then Diag(Gam) dO
constexpr uint32_t PX = DH + 8192;              // P
constexpr uint32_t DPD = PX + 8192;             // scale tril(dO V^T) . D
constexpr uint32_t SMEM_BYTES = DPD + 8192 + 1024;
static_assert(2 * (SMEM_BYTES + 4096) <= 227 * 1024, "two CTAs per SM");
// Tensor memory: 256 columns per CTA so that two CTAs share an SM.
//   columns       lanes 0..15 (A)                      lanes 16..31 (B)
//   C0  64        Q K^T;  (Diag(Gam) Q)^T dO, columns 0..31 (32 wide)      dO V^T;  ... columns 32..63
//   C1  64        K dh'                                V dh'^T
//   C2  64        P^T dO                               (dP.D)^T Q
//   C3  32        dO h^T, columns 0..31                dO h^T, columns 32..63
//   C4  32        (dP.D) K, columns 0..31              (dP.D) K, columns 32..63
constexpr uint32_t C0 = 0, C1 = 64, C2 = 128, C3 = 192, C4 = 224, LB = 16u << 16;
}  // namespace b64

__global__ void __launch_bounds__(kThreads64 + 32, 2) tc64_bwd_kernel(const __grid_constant__ Tc64Params P) {
    wait_prerequisites();
    using namespace b64;
    const Problem& p = P.p;
    const WsHeader* hdr = reinterpret_cast<const WsHeader*>(p.ws);
    if (hdr->status != GDN_OK) return;
    const int H = p.d.H;
    const int n = blockIdx.x / H, hd = blockIdx.x % H;
    const SeqGeom cg = seq_geom(p, n);
    const int c0 = cg.c0, nsteps = cg.n_chunks, c1 = c0 + nsteps;
    const float sc = p.d.scale;

    extern __shared__ unsigned char smem_raw[];
    unsigned char* sm = align1024(smem_raw);
    __shared__ __align__(16) float gl2[2][kC], Gam2[2][kC], ee2[2][kC], dgp[2][kC], scal[2][kThreads64 / 32];
    __shared__ uint64_t bar_full[STAGES], bar_st, bar_mma, bar_mma2;
    __shared__ uint32_t tmem_slot;
    const int warp = warp_id(), lane = threadIdx.x & 31;
    const int q4 = warp & 3, half = warp >> 2;
    const int r = q4 * 16 + (lane & 15);      // accumulator / state row of this lane
    const bool ga = lane < 16;                // group A: lanes 0..15, group B: lanes 16..31
    const int cb0 = half * 32;                // first of this thread's 32 columns of a whole accumulator
    const int sc0 = (ga ? 0 : 32) + half * 16;   // first of its 16 columns of one issued in halves, and of the state
    const uint32_t lane_base = (uint32_t)(q4 * 32) << 16;

    // Warp 8 only moves data: its first lane stores a step's staged gradients and then loads the tiles of the step
    // after next into the ring slot they came from.  It follows the other warps through an mbarrier and shares no
    // block-wide barrier with them inside the loop (they use a named barrier).
    const bool loader = warp == kThreads64 / 32;
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) mbar_init(&bar_full[s], 1);
        mbar_init(&bar_st, 1);
        mbar_init(&bar_mma, 1);
        mbar_init(&bar_mma2, 1);
        fence_mbar_init();
    }
    if (warp == 0) { tmem_alloc(&tmem_slot, 256); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;

    auto fill = [&](int s) {   // step s handles chunk c1 - 1 - s
        const int stage = s % STAGES, c = c1 - 1 - s, tok0 = cg.chunk_tok0(c);
        unsigned char* st = sm + stage * STAGE_BYTES;
        mbar_expect_tx(&bar_full[stage], 40960);
        tma_load_2d(st + QT, &P.tm_q, hd * D6, tok0, &bar_full[stage]);
        tma_load_2d(st + KT, &P.tm_k, hd * D6, tok0, &bar_full[stage]);
        tma_load_2d(st + VT, &P.tm_v, hd * D6, tok0, &bar_full[stage]);
        tma_load_2d(st + OT, &P.tm_do, hd * D6, tok0, &bar_full[stage]);
        bulk_load(st + HT, p.ws + p.L.hc + ((size_t)c * H + hd) * 8192, 8192, &bar_full[stage]);
    };
    if (loader) {
        if (lane == 0) {
            for (int s = 0; s < STAGES && s < nsteps; ++s) fill(s);
            int s = 0;
#pragma unroll 1
            for (; s < nsteps; ++s) {
                if (!mbar_wait(&bar_st, s & 1)) break;          // step s has staged its gradient rows (or flushed them)
                const int c = c1 - 1 - s;
                if (cg.chunk_len(c) == kC) {
                    const int tok0 = cg.chunk_tok0(c);
                    unsigned char* st = sm + (s % STAGES) * STAGE_BYTES;
                    tma_store_2d(&P.tm_dv, hd * D6, tok0, st + VT);
                    tma_store_2d(&P.tm_dk, hd * D6, tok0, st + KT);
                    tma_store_2d(&P.tm_dq, hd * D6, tok0, st + QT);
                    bulk_commit();
                    bulk_wait_read<0>();   // the ring slot is loaded over next
                }
                if (s + STAGES < nsteps) fill(s + STAGES);
            }
            bulk_wait_read<0>();
            drain_ring<STAGES>(bar_full, s, nsteps);
        }
        return;
    }
    auto cta_sync = [] { asm volatile("bar.sync 1, %0;" ::"n"(kThreads64) : "memory"); };   // all warps but the loader

    float st[16];   // dh' row r, columns sc0 .. sc0 + 15 (gradient w.r.t. the state leaving the current chunk)
    const size_t soff = ((size_t)n * H + hd) * D6 * D6 + (size_t)r * D6 + sc0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        float4 v = p.dhT ? *reinterpret_cast<const float4*>(p.dhT + soff + 4 * k) : make_float4(0.f, 0.f, 0.f, 0.f);
        st[4 * k] = v.x; st[4 * k + 1] = v.y; st[4 * k + 2] = v.z; st[4 * k + 3] = v.w;
    }
    // Gate arrays of a step (log2-scaled cumulative decay, Gam = exp(gam), e = exp(gam_end - gam)) are prepared one
    // step ahead, into the other of two sets, while the tensor pipe works; their inputs are fetched a step before that.
    const float* gamma = reinterpret_cast<const float*>(p.ws + p.L.gamma);
    auto gate_row = [&](int step) { return gamma + ((size_t)(c1 - 1 - step) * H + hd) * kC; };
    auto make_gates = [&](int set, float g, float gend) {
        gl2[set][threadIdx.x] = g * kLog2e;
        Gam2[set][threadIdx.x] = expf(g);
        ee2[set][threadIdx.x] = ex2((gend - g) * kLog2e);
    };
    float gnext = 0.f, gend_next = 0.f;
    if (threadIdx.x < kC && nsteps > 0) {
        make_gates(0, gate_row(0)[threadIdx.x], gate_row(0)[kC - 1]);
        if (nsteps > 1) { gnext = gate_row(1)[threadIdx.x]; gend_next = gate_row(1)[kC - 1]; }
    }
    bool ok = true;
    uint32_t mma_phase = 0;
    // a warp that gives up in step s behind `passed` of its barriers (three, and a fourth in the first step if that chunk is a ragged tail)
    auto leave = [&](int s, int passed) { stand_by((nsteps - s) * 3 - passed + (s == 0 && cg.chunk_len(c1 - 1) < kC ? 1 : 0), cta_sync); };
    int len_n = nsteps > 0 ? cg.chunk_len(c1 - 1) : 0, tok0_n = nsteps > 0 ? cg.chunk_tok0(c1 - 1) : 0;   // fetched a step ahead
#pragma unroll 1
    for (int s = 0; s < nsteps; ++s) {
        const int c = c1 - 1 - s, stage = s % STAGES, len = len_n, tok0 = tok0_n;
        if (s + 1 < nsteps) { len_n = cg.chunk_len(c - 1); tok0_n = cg.chunk_tok0(c - 1); }
        unsigned char* tiles = sm + stage * STAGE_BYTES;
        const float *gl = gl2[s & 1], *Gam = Gam2[s & 1], *ee = ee2[s & 1];
        ok = mbar_wait(&bar_full[stage], (s / STAGES) & 1);
        if (!ok) { if (lane == 0) report_timeout(p.ws, 50); leave(s, 0); break; }
        if (len < kC) {
            zero_tail_rows64(tiles + QT, len);
            zero_tail_rows64(tiles + KT, len);
            zero_tail_rows64(tiles + VT, len);
            zero_tail_rows64(tiles + OT, len);
        }
        float hh = 0.f;   // <dh', h> restricted to this thread's part of the state
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            float hv[8];
            chunk_load(tiles + HT, 64, r, (sc0 >> 3) + k, hv);
#pragma unroll
            for (int j = 0; j < 8; ++j) hh = fmaf(st[8 * k + j], hv[j], hh);
            chunk_store(sm + DH, 64, r, (sc0 >> 3) + k, st + 8 * k);
        }
        fence_async_smem();
        cta_sync();
        const float Ge = Gam[kC - 1];
        // ---- phase 1: Q K^T, dO V^T; under their readout K dh', V dh'^T, dO h^T
        if (warp == 0 && elect_one()) {
            tc_fence_after();
            mma_tile<64, 64, 64>(tmem + C0, op_k_major(tiles + QT, 64), op_k_major(tiles + KT, 64), false);
            mma_tile<64, 64, 64>(tmem + C0 + LB, op_k_major(tiles + OT, 64), op_k_major(tiles + VT, 64), false);
            mma_commit(&bar_mma);
            mma_tile<64, 64, 64>(tmem + C1, op_k_major(tiles + KT, 64), op_mn_major(sm + DH, 64), false);
            mma_tile<64, 64, 64>(tmem + C1 + LB, op_k_major(tiles + VT, 64), op_k_major(sm + DH, 64), false);
            mma_tile<64, 32, 64>(tmem + C3, op_k_major(tiles + OT, 64), op_k_major(tiles + HT, 64, 0), false);
            mma_tile<64, 32, 64>(tmem + C3 + LB, op_k_major(tiles + OT, 64), op_k_major(tiles + HT, 64, 32), false);
            mma_commit(&bar_mma2);
        }
        if (threadIdx.x < kC && s + 1 < nsteps) {
            make_gates((s + 1) & 1, gnext, gend_next);
            if (s + 2 < nsteps) { gnext = gate_row(s + 2)[threadIdx.x]; gend_next = gate_row(s + 2)[kC - 1]; }
        }
        GDN_WAIT_MMA(51)
        if (!ok) { leave(s, 1); break; }
        {   // A: P = tril(Q K^T . D)   B: dP . D = scale tril(dO V^T) . D
            const float glr = gl[r], f = ga ? 1.f : sc;
            unsigned char* dst = sm + (ga ? PX : DPD);
#pragma unroll 2
            for (int part = 0; part < 4; ++part) {
                float s8[8], g8[8];
                const int jb = cb0 + part * 8;
                tmem_ld8(tmem + lane_base + C0 + jb, s8);
                ld8s(gl + jb, g8);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 8; ++j) s8[j] *= (jb + j <= r) ? f * ex2(glr - g8[j]) : 0.f;   // masked first: the exponent is never positive
                chunk_store(dst, 64, r, jb >> 3, s8);
            }
        }
        ok = mbar_wait(&bar_mma2, 0);
        if (!ok) { if (lane == 0) report_timeout(p.ws, 53); leave(s, 1); break; }
        tc_fence_after();
#pragma unroll
        for (int t = 0; t < 2; ++t) {   // Diag(Gam) dO over the dh' tile, which no MMA reads any more
            const int i = (threadIdx.x >> 3) + 32 * t, cch = threadIdx.x & 7;
            float v[8];
            chunk_load(tiles + OT, 64, i, cch, v);
            const float G = Gam[i];
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] *= G;
            chunk_store(sm + DH, 64, i, cch, v);
        }
        tc_fence_before();
        fence_async_smem();
        cta_sync();
        // ---- phase 2: P^T dO, (dP.D)^T Q, (dP.D) K; under their readout (Diag(Gam) Q)^T dO
        if (warp == 0 && elect_one()) {
            tc_fence_after();
            mma_tile<64, 64, 64>(tmem + C2, op_mn_major(sm + PX, 64), op_mn_major(tiles + OT, 64), false);
            mma_tile<64, 64, 64>(tmem + C2 + LB, op_mn_major(sm + DPD, 64), op_mn_major(tiles + QT, 64), false);
            mma_tile<64, 32, 64>(tmem + C4, op_k_major(sm + DPD, 64), op_mn_major(tiles + KT, 64), false);
            mma_tile<64, 32, 64>(tmem + C4 + LB, op_k_major(sm + DPD, 64), op_mn_major(tiles + KT + 64, 64), false);
            mma_commit(&bar_mma);
            mma_tile<64, 32, 64>(tmem + C0, op_mn_major(tiles + QT, 64), op_mn_major(sm + DH, 64), false);
            mma_tile<64, 32, 64>(tmem + C0 + LB, op_mn_major(tiles + QT, 64), op_mn_major(sm + DH + 64, 64), false);
            mma_commit(&bar_mma2);
        }
        GDN_WAIT_MMA(52)
        if (!ok) { leave(s, 2); break; }
        // Gradient rows are staged token-major in place over this step's input tiles (dv over V, dk over K and dq over Q, where
        // a thread overwrites exactly the piece it has just read; every product that reads the tile is done) and leave by TMA
        // stores; generic global stores here would be one 16-byte piece per row.
        float rs = 0.f;    // A: sum_j r_j, r_j = e_j <(K dh')_j, V_j>
        float dot = 0.f;   // B: -<k_r, dk_r>;  both: <q_r, dq_r> over this thread's columns
        {   // A: dv = scale P^T dO + Diag(e) K dh'     B: dk = (dP.D)^T Q + Diag(e) V dh'^T
            const float e = ee[r], f = ga ? sc : 1.f;
            unsigned char* tile = tiles + (ga ? VT : KT);
#pragma unroll 2
            for (int part = 0; part < 4; ++part) {
                float a[8], b[8], x[8];
                const int jb = cb0 + part * 8;
                tmem_ld8(tmem + lane_base + C2 + jb, a);
                tmem_ld8(tmem + lane_base + C1 + jb, b);
                chunk_load(tile, 64, r, jb >> 3, x);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    rs = fmaf(b[j], x[j], rs);
                    a[j] = fmaf(f, a[j], e * b[j]);
                    dot = fmaf(-x[j], a[j], dot);
                }
                chunk_store(tile, 64, r, jb >> 3, a);
            }
            rs *= e;
            if (ga) dot = 0.f;
        }
        ok = mbar_wait(&bar_mma2, 1);
        if (!ok) { if (lane == 0) report_timeout(p.ws, 54); leave(s, 2); break; }
        tc_fence_after();
        {   // dq = scale Gam dO h^T + (dP.D) K ;  dh = Gam_e dh' + scale (Diag(Gam) Q)^T dO
            const float G = sc * Gam[r];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                float a[8], b[8], x[8], e8[8];
                tmem_ld8(tmem + lane_base + C3 + half * 16 + 8 * k, a);
                tmem_ld8(tmem + lane_base + C4 + half * 16 + 8 * k, b);
                tmem_ld8(tmem + lane_base + C0 + half * 16 + 8 * k, e8);
                chunk_load(tiles + QT, 64, r, (sc0 >> 3) + k, x);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    a[j] = fmaf(G, a[j], b[j]);
                    dot = fmaf(x[j], a[j], dot);
                    st[8 * k + j] = fmaf(Ge, st[8 * k + j], sc * e8[j]);
                }
                chunk_store(tiles + QT, 64, r, (sc0 >> 3) + k, a);
            }
        }
        dot += __shfl_xor_sync(0xffffffffu, dot, 16);
        if (ga) dgp[half][r] = dot;
        rs = warp_sum(ga ? rs : 0.f);
        hh = warp_sum(hh);
        if (lane == 0) { scal[0][warp] = rs; scal[1][warp] = hh; }
        tc_fence_before();
        fence_async_smem();
        cta_sync();   // every reader of this stage's tiles is done; partial sums and staged rows are visible
        if (len < kC) {   // ragged tail: rows beyond the sequence must not be written
            const size_t gbase = ((size_t)tok0 * H + hd) * D6;
            for (int t = threadIdx.x; t < kC * 8; t += kThreads64) {
                const int i = t >> 3, chk = t & 7;
                if (i < len) {
                    const size_t o = gbase + (size_t)i * H * D6 + chk * 8;
                    *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(p.dv) + o) = *reinterpret_cast<const uint4*>(tiles + VT + tile_chunk_off(64, i, chk));
                    *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(p.dk) + o) = *reinterpret_cast<const uint4*>(tiles + KT + tile_chunk_off(64, i, chk));
                    *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(p.dq) + o) = *reinterpret_cast<const uint4*>(tiles + QT + tile_chunk_off(64, i, chk));
                }
            }
            cta_sync();   // the ring slot is handed to the loader only after every row has been read
        }
        if (threadIdx.x == 32) mbar_arrive(&bar_st);
        if (warp == 0) {
            float rsum = 0.f, hsum = 0.f;
            for (int w = 0; w < kThreads64 / 32; ++w) { rsum += scal[0][w]; hsum += scal[1][w]; }
            write_dg_suffix(dgp[0], dgp[1], rsum + Ge * hsum, p.dg + (size_t)tok0 * H + hd, (size_t)H, len, lane);
        }
    }
    tc_fence_before();
    ok = named_barrier_and<kThreads64>(ok);
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, 256);
    }
    if (p.dh0 && ok) {
#pragma unroll
        for (int k = 0; k < 4; ++k) *reinterpret_cast<float4*>(p.dh0 + soff + 4 * k) = make_float4(st[4 * k], st[4 * k + 1], st[4 * k + 2], st[4 * k + 3]);
    }
}

}  // namespace

// ------------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------------
bool tc64_supported(const gdn_desc& d) {
    return d.dtype == GDN_BF16 && d.d_k == 64 && d.d_v == 64 && d.delta_rule == 0 && d.chunk == kC;
}

static bool fill_params64(Tc64Params& P, const Problem& p, bool with_bwd) {
    P.p = p;
    const uint64_t rows = (uint64_t)p.Ttot, cols = (uint64_t)p.d.H * D6, pitch = cols * 2;
    if (!tc::make_tmap_bf16_2d(&P.tm_q, p.q, rows, cols, pitch, 64)) return false;
    if (!tc::make_tmap_bf16_2d(&P.tm_k, p.k, rows, cols, pitch, 64)) return false;
    if (!tc::make_tmap_bf16_2d(&P.tm_v, p.v, rows, cols, pitch, 64)) return false;
    if (!tc::make_tmap_bf16_2d(&P.tm_do, with_bwd ? p.dO : p.v, rows, cols, pitch, 64)) return false;
    if (with_bwd) {
        if (!tc::make_tmap_bf16_2d(&P.tm_dq, p.dq, rows, cols, pitch, 64)) return false;
        if (!tc::make_tmap_bf16_2d(&P.tm_dk, p.dk, rows, cols, pitch, 64)) return false;
        if (!tc::make_tmap_bf16_2d(&P.tm_dv, p.dv, rows, cols, pitch, 64)) return false;
    }
    return true;
}

// fresh: gamma and the status word are those of the forward whose workspace the call consumes.
static cudaError_t tc64_prologue(const Problem& p, bool fresh, cudaStream_t st) {
    // the chunk table is needed for packed sequences only (and for an empty call, whose only kernel it is)
    if (p.cu || p.Ttot == 0) {
        const cudaError_t e = launch_table(p, st, fresh);
        if (e != cudaSuccess) return e;
    }
    if (!fresh && p.L.max_chunks > 0 && p.Ttot > 0) {
        StageScope t(ST_PREP, st);
        launch_kernel(tc64_gamma_kernel, dim3(p.L.max_chunks, (p.d.H + 31) / 32), 256, 0, st, p);
    }
    return cudaGetLastError();
}

static cudaError_t tc64_fwd_pass(const Tc64Params& P, cudaStream_t st) {
    static SmemLimitOnce once, once_o;
    const bool o = P.p.o != nullptr;
    const uint32_t smem = o ? f64::Cfg<true>::SMEM_BYTES : f64::Cfg<false>::SMEM_BYTES;
    const cudaError_t e0 = o ? once_o.ensure(tc64_fwd_kernel<true>, smem) : once.ensure(tc64_fwd_kernel<false>, smem);
    if (e0 != cudaSuccess) return e0;
    const int chains = P.p.d.N * P.p.d.H;
    if (chains > 0) {
        StageScope t(ST_FSCAN, st);
        launch_kernel(o ? tc64_fwd_kernel<true> : tc64_fwd_kernel<false>, chains, kThreads64, smem, st, P);
    }
    return cudaGetLastError();
}

cudaError_t tc64_launch_fwd(const Problem& p, cudaStream_t st) {
    Tc64Params P;
    cudaError_t e = tc64_prologue(p, false, st);
    if (e != cudaSuccess) return e;
    if (p.Ttot == 0) {
        const size_t bytes = (size_t)p.d.N * p.d.H * D6 * D6 * sizeof(float);
        if (!p.hT) return cudaSuccess;
        return p.h0 ? cudaMemcpyAsync(p.hT, p.h0, bytes, cudaMemcpyDeviceToDevice, st) : cudaMemsetAsync(p.hT, 0, bytes, st);
    }
    if (!fill_params64(P, p, false)) return cudaErrorUnknown;
    return tc64_fwd_pass(P, st);
}

cudaError_t tc64_launch_bwd(const Problem& p, bool skip_recompute, cudaStream_t st) {
    Tc64Params P;
    cudaError_t e = tc64_prologue(p, skip_recompute, st);
    if (e != cudaSuccess) return e;
    if (p.Ttot == 0) {
        const size_t bytes = (size_t)p.d.N * p.d.H * D6 * D6 * sizeof(float);
        if (!p.dh0) return cudaSuccess;
        return p.dhT ? cudaMemcpyAsync(p.dh0, p.dhT, bytes, cudaMemcpyDeviceToDevice, st) : cudaMemsetAsync(p.dh0, 0, bytes, st);
    }
    if (!fill_params64(P, p, true)) return cudaErrorUnknown;
    if (!skip_recompute) {
        Tc64Params F = P;
        F.p.o = nullptr;   // the backward never asks for the forward outputs
        F.p.hT = nullptr;
        if ((e = tc64_fwd_pass(F, st)) != cudaSuccess) return e;
    }
    static SmemLimitOnce once;
    if ((e = once.ensure(tc64_bwd_kernel, b64::SMEM_BYTES)) != cudaSuccess) return e;
    const int chains = p.d.N * p.d.H;
    if (chains > 0) {
        StageScope t(ST_RSCAN, st);
        launch_kernel(tc64_bwd_kernel, chains, kThreads64 + 32, b64::SMEM_BYTES, st, P);
    }
    return cudaGetLastError();
}

}  // namespace gdn

