// tcgen05 / TMEM / TMA kernels of the GDN backward for bf16 I/O, d_k = d_v = 128, chunk 64 (sm_100a).
//
// Kernels follow the stage map of the chunked method (Section 4.2 of the paper):
//   tc_prep  (one CTA per chunk-head)  gamma, A, T = (I + A)^-1, W, U~, Nm = Kb^T W, Bf = Kb^T U~ and, for the
//                                      backward, E = scale (Diag(Gam) Q - P W)^T dO
//   tc_scan  (one CTA per chain and direction)
//                                      forward carry  h'  = Gam_e h  - Nm   h  + Bf   (stores h per chunk)
//                                      reverse carry  dh  = Gam_e dh' - Nm^T dh' + E   (the paper's K#1; stores dh')
//   tc_prep_lr, tc_scan_lr             the same with the carries in low-rank form, which leave U and dU per chunk as well
//   tc_intra (one CTA per chunk-head)  every token gradient, including the VJP of the triangular solve (K#2)
//   tc_out   (optional)                forward output o
//
// All dense products run on tcgen05.mma with fp32 accumulators in tensor memory; operands are bf16 tiles in
// shared memory in the "blocked-64, 128-byte swizzle" format of tc_ptx.cuh, brought in by TMA (inputs) or by
// contiguous bulk copies of tile images (workspace).  Accumulators are produced with the feature dimension
// (128) on the TMEM lanes and the 64 tokens of the chunk on the columns, i.e. transposed, so that M = 128.
// The carried states stay fp32 in registers for the whole scan; tensor memory holds accumulators only and is
// allocated once per CTA and released once.  Every wait is bounded; a wait that gives up records
// GDN_ERR_DEVICE_TIMEOUT in the workspace header and the CTA leaves through its normal teardown.
// Loops over accumulator columns are kept rolled (8 columns per trip): the kernels run each piece of code once
// per chunk, so instruction-cache footprint matters more than loop overhead.
#include "tc_common.cuh"
#include "tc_inverse.cuh"

namespace gdn {


namespace {

constexpr int D = 128;          // d_k = d_v
constexpr int kThreads = 256;   // 8 warps: lane quadrant = warp % 4, column half = warp / 4 (scan, out)
// The chunk kernels run 16 readout warps: four warps share a TMEM lane quadrant and split the 64 token columns four
// ways, which shortens every thread's serial readout chain and gives the scheduler more warps to hide latencies with.
constexpr int kWideThreads = 512;
constexpr int kGroups = kWideThreads / 128;   // column groups
constexpr int kTG = kC / kGroups;             // token columns per group (16)
constexpr int kIntraThreads = kWideThreads + 32;   // ... plus one warp whose first lane only issues MMAs; the kernels are
                                                   // launched with one more warp on top (kIntraThreads + 32) that only
                                                   // issues bulk copies and takes no part in the named barrier
// values of TcParams::withhold and of gdn_debug_inject_timeout
enum { WITHHOLD_PREP = 1, WITHHOLD_CARRY = 2, WITHHOLD_GRADIENT = 3, DISAGREE_PREP = 4, DISAGREE_CARRY = 5, DISAGREE_GRADIENT = 6 };
struct TcParams {
    Problem p;
    CUtensorMap tm_q, tm_k, tm_v, tm_do;   // [T_total, H, d] bf16, boxes of 64 tokens x 64 features of a head
    CUtensorMap tm_dq, tm_dk, tm_dv;       // same geometry, for the gradient stores of full chunks
    CUtensorMap tm_o;                      // same geometry, for the forward output (forward calls that want it)
    int with_bwd;                          // prep: also produce E
    int scan_dirs;                         // scan: 0 = forward carry only, 1 = reverse only, 2 = both
    int lowrank;                           // carries in low-rank form (tc_scan_lr): prepared by tc_prep_lr without Nm, Bf
    int narrow_v;                          // d_v = 64: of the kernels whose CTAs carry 64 state columns only the first half is launched
    int withhold;                          // debugging hook: a kernel leaves out one of its first loads, so that the wait for
                                           // it runs out, or half of its warps take a first wait for one that did (exercises
                                           // the time-out path without any fault)
};

// ------------------------------------------------------------------------------------------------
// tc_prep
// ------------------------------------------------------------------------------------------------
namespace prep {
// The input tiles are never reused within a trip, so the next trip's inputs are loaded into them as soon as the last
// product that reads them is done; the three output images are staged over tiles that are dead by then.
constexpr uint32_t QK = 0;                    // [Q rows 0..63 ; K rows 64..127] x 128   32 KB
constexpr uint32_t VO = 32768;                // [V ; dO] x 128                           32 KB
constexpr uint32_t TT = 65536;                // T                      [64][64]           8 KB  (these four: finally
constexpr uint32_t TP = TT + 8192;            // T Diag(b Gam)                                    the Nm image)
constexpr uint32_t TPP = TP + 8192;           // T Diag(w)
constexpr uint32_t PT = TPP + 8192;           // P = tril(Q K^T . D)
constexpr uint32_t WT = PT + 8192;            // W^T   [128 dk][64 tokens]                16 KB
constexpr uint32_t UTT = WT + 16384;          // U~^T  [128 dv][64]
constexpr uint32_t WET = UTT + 16384;         // (Diag(e) W)^T                                    (these two: finally
constexpr uint32_t UET = WET + 16384;         // (Diag(e) U~)^T                                   the Bf image)
constexpr uint32_t X = UET + 16384;           // fp32 A and T during the inversion; then R = Diag(Gam) dO and
constexpr uint32_t XA = X, XT = X + 17408;    // (P^T dO)^T; finally the E image
constexpr uint32_t XR = X, XPDO = X + 16384;
constexpr uint32_t NMS = TT, BFS = WET, ES = X;   // staging of the three output images
constexpr uint32_t TILES_END = X + 34816;
constexpr uint32_t SMEM_BYTES = TILES_END + 1024 /* alignment slack */;
static_assert(SMEM_BYTES <= 227 * 1024, "shared memory budget");
// TMEM columns (512 allocated): accumulators at fixed offsets, allocated once, released once.
constexpr uint32_t C_S1 = 0, C_W = 64, C_U = 128, C_PDO = 192, C_NM = 256, C_BF = 384, C_E = 0;
}  // namespace prep

__global__ void __launch_bounds__(kIntraThreads + 32, 1) tc_prep_kernel(const __grid_constant__ TcParams P) {
    wait_prerequisites();
    using namespace prep;
    const Problem& p = P.p;
    // Persistent: a CTA walks over chunk-heads blockIdx.x, blockIdx.x + gridDim.x, ...; the inputs of its next one
    // are loaded while it works on the current one.
    const int H = p.d.H;
    init_header_if_untabled(p);
    const int n_items = n_chunks_of(p) * H;
    if ((int)blockIdx.x >= n_items) return;
    const bool bwd = P.with_bwd != 0;

    extern __shared__ unsigned char smem_raw[];
    unsigned char* sm = align1024(smem_raw);
    // gate arrays, two sets: a trip's set is written during the trip before it
    __shared__ __align__(16) float gate_sets[2][6][kC];
    __shared__ uint64_t bar_qk, bar_vo, bar_ld0, bar_t, bar_vofree, bar_ld1, bar_st, bar_tfree, bar_free1, bar_free2, bar_free, bar_mma;
    __shared__ uint32_t tmem_slot;
    const int warp = warp_id(), lane = threadIdx.x & 31;
    const int q4 = warp & 3, grp = warp >> 2;
    const uint32_t lane_base = (uint32_t)(q4 * 32) << 16;
    const bool worker = warp < 16;                       // warps 0..15 read accumulators and do the fp32 work
    const bool issuer = threadIdx.x == kWideThreads;     // first lane of warp 16 feeds the tensor pipe
    // Warp 17 only moves data: its first lane issues the bulk stores of a trip's results and the loads of the next
    // trip's inputs (each such instruction costs its issuer hundreds of cycles).  It follows the other warps through
    // mbarriers and shares no block-wide barrier with them inside the loop (they use a named barrier).
    const bool loader = warp == 17;

    if (threadIdx.x == 0) {
        mbar_init(&bar_qk, 1); mbar_init(&bar_vo, 1); mbar_init(&bar_ld0, 1); mbar_init(&bar_t, 1);
        mbar_init(&bar_vofree, 1); mbar_init(&bar_ld1, 1); mbar_init(&bar_st, 1); mbar_init(&bar_tfree, 1);
        mbar_init(&bar_free1, 1); mbar_init(&bar_free2, 1); mbar_init(&bar_free, 1); mbar_init(&bar_mma, 1);
        fence_mbar_init();
    }
    if (warp == 0) { tmem_alloc(&tmem_slot, 512); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    bool ok = true;
    const uint32_t VO_BYTES = bwd ? 32768 : 16384;
    auto load_piece = [&](int piece, const ChunkInfo& c) {   // 0,1: Q  2,3: K  4,5: V  6,7: dO   (column halves)
        const int cb = piece & 1;
        switch (piece >> 1) {
            case 0: tma_load_3d(sm + QK + cb * 16384, &P.tm_q, cb * 64, c.hd, c.tok0, &bar_qk); break;
            case 1: tma_load_3d(sm + QK + cb * 16384 + 8192, &P.tm_k, cb * 64, c.hd, c.tok0, &bar_qk); break;
            case 2: tma_load_3d(sm + VO + cb * 16384, &P.tm_v, cb * 64, c.hd, c.tok0, &bar_vo); break;
            case 3: if (bwd) tma_load_3d(sm + VO + cb * 16384 + 8192, &P.tm_do, cb * 64, c.hd, c.tok0, &bar_vo); break;
            default: break;
        }
    };

    if (loader) {
        if (lane == 0) {
            uint32_t ph = 0;
            bool lok = true, pend_qk = false, pend_vo = false;
#pragma unroll 1
            for (int item = blockIdx.x; item < n_items && lok; item += gridDim.x, ph ^= 1) {
                ChunkInfo x, nx;
                chunk_entry(p, x, item);
                const bool has_next = item + (int)gridDim.x < n_items;
                if (has_next) chunk_entry(p, nx, item + gridDim.x);
                pend_qk = pend_vo = false;
                // the trip is under way: the inputs of the next one (loaded late in this trip) -> L2
                if (!(lok = mbar_wait(&bar_ld0, ph))) break;
                if (has_next) {
                    for (int cb = 0; cb < 2; ++cb) {
                        prefetch_l2_tma_3d(&P.tm_v, cb * 64, nx.hd, nx.tok0);
                        if (bwd) prefetch_l2_tma_3d(&P.tm_do, cb * 64, nx.hd, nx.tok0);
                    }
                    for (int cb = 0; cb < 2; ++cb) {
                        prefetch_l2_tma_3d(&P.tm_q, cb * 64, nx.hd, nx.tok0);
                        prefetch_l2_tma_3d(&P.tm_k, cb * 64, nx.hd, nx.tok0);
                    }
                }
                // T is staged
                if (!(lok = mbar_wait(&bar_t, ph))) break;
                bulk_store(p.ws + p.L.Tm + (size_t)x.ch * 8192, sm + TT, 8192);
                bulk_store(p.ws + p.L.Pm + (size_t)x.ch * 8192, sm + PT, 8192);   // the forward output and the gradient stage read P from here
                bulk_commit();
                // W^T, U~^T are staged and V, dO have been read for the last time
                if (!(lok = mbar_wait(&bar_vofree, ph))) break;
                bulk_wait_read<0>();
                mbar_arrive(&bar_tfree);   // the T tile may be overwritten (by the staged Nm image)
                if (has_next) {            // (the loads first: the next trip starts with them, the stores have time)
                    mbar_expect_tx(&bar_vo, VO_BYTES);
                    pend_vo = true;
#pragma unroll 1
                    for (int piece = 4; piece < 8; ++piece) load_piece(piece, nx);
                }
                bulk_store(p.ws + p.L.W + (size_t)x.ch * 16384, sm + WT, 16384);
                bulk_store(p.ws + p.L.Ut + (size_t)x.ch * 16384, sm + UTT, 16384);
                bulk_commit();
                // phase 3 is done: Q, K have been read for the last time
                if (!(lok = mbar_wait(&bar_ld1, ph))) break;
                if (has_next) {
                    mbar_expect_tx(&bar_qk, 32768);
                    pend_qk = true;
#pragma unroll 1
                    for (int piece = 0; piece < 4; ++piece) {
                        load_piece(piece, nx);
                    }
                }
                // the three images are staged.  All CTAs store at about the same time, so the 96 KB drain at the rate of
                // HBM (some 22 bytes per cycle and SM); they leave in the order in which the next trip rewrites their
                // tiles: first the bytes under the fp32 A block (head of the E image) and under P (tail of the Nm image),
                // then those under the fp32 T block (rest of E), last what the T tiles and the second readout overwrite
                if (!(lok = mbar_wait(&bar_st, ph))) break;
                constexpr uint32_t A_BYTES = XT - XA;
                if (bwd) bulk_store(p.ws + p.L.E + (size_t)x.ch * 32768, sm + ES, A_BYTES);
                bulk_store(p.ws + p.L.Nm + (size_t)x.ch * 32768 + (PT - TT), sm + NMS + (PT - TT), 8192);
                bulk_commit();
                if (bwd) bulk_store(p.ws + p.L.E + (size_t)x.ch * 32768 + A_BYTES, sm + ES + A_BYTES, 32768 - A_BYTES);
                bulk_commit();
                bulk_wait_read<1>();       // (issuing a store takes hundreds of cycles: the first group has drained by now)
                mbar_arrive(&bar_free1);   // the fp32 A block and P may be written (and the scratch over W^T: its store is older)
                bulk_store(p.ws + p.L.Nm + (size_t)x.ch * 32768, sm + NMS, PT - TT);
                bulk_store(p.ws + p.L.Bf + (size_t)x.ch * 32768, sm + BFS, 32768);
                bulk_commit();
                bulk_wait_read<1>();
                mbar_arrive(&bar_free2);   // the fp32 T block may be written
                bulk_wait_read<0>();
                mbar_arrive(&bar_free);    // every staging tile may be rewritten
            }
            bulk_wait_read<0>();
            if (!lok) {   // after a timeout a copy may still be in flight, of this trip or of the next one: wait for it before the CTA may retire
                (void)mbar_wait(&bar_qk, pend_qk ? ph ^ 1 : ph);
                (void)mbar_wait(&bar_vo, pend_vo ? ph ^ 1 : ph);
            }
        }
        return;
    }

    auto cta_sync = [] { asm volatile("bar.sync 1, %0;" ::"n"(kIntraThreads) : "memory"); };   // all warps but the loader
    uint32_t mma_phase = 0, in_phase = 0;
    // The chunk table entry and the gate values of a trip are fetched one trip ahead into registers: they are tiny, but
    // read at the top of a trip their DRAM latency would be fully exposed.
    ChunkInfo xn;
    chunk_entry(p, xn, blockIdx.x);
    // Warp 0 owns the gates: lane l holds g (0 when padded) and the erase gate b of tokens l and l + 32.
    float ng[2] = {0.f, 0.f}, nb[2] = {0.f, 0.f};
    auto fetch_gates = [&](const ChunkInfo& c) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = lane + 32 * h;
            ng[h] = nb[h] = 0.f;
            if (i < c.len) {
                const size_t idx = (size_t)(c.tok0 + i) * H + c.hd;
                ng[h] = p.g[idx];
                if (p.d.delta_rule) nb[h] = p.beta[idx];   // delta rule off: erase gate 0 (T = I, W = 0 fall out of the same products)
            }
        }
    };
    // Warp 0 turns the fetched values into the gate arrays of chunk-head `ch` (set `set`): erase gate b, write gate w,
    // chunk-local cumulative decay gam (inclusive prefix sum of the 64 log decays), in registers.
    auto make_gates = [&](int set, int ch) {
        float a = ng[0], b = ng[1];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const float ua = __shfl_up_sync(0xffffffffu, a, o), ub = __shfl_up_sync(0xffffffffu, b, o);
            if (lane >= o) { a += ua; b += ub; }
        }
        b += __shfl_sync(0xffffffffu, a, 31);
        const float gend = __shfl_sync(0xffffffffu, b, 31);
        const float gc[2] = {a, b};
        float (*gs)[kC] = gate_sets[set];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = lane + 32 * h;
            const float G = expf(gc[h]);
            gs[0][i] = gc[h] * kLog2e;
            gs[1][i] = G;
            gs[2][i] = expf(gend - gc[h]);
            gs[3][i] = nb[h];
            gs[4][i] = p.d.delta_rule ? nb[h] : (i < xn.len ? 1.f : 0.f);   // write gate (delta rule off: 1)
            gs[5][i] = nb[h] * G;
            reinterpret_cast<float*>(p.ws + p.L.gamma)[(size_t)ch * kC + i] = gc[h];
        }
    };
    if (warp == 0) { fetch_gates(xn); make_gates(0, xn.ch); }
    // first trip: the inputs are loaded at once, one instruction per warp
    if (issuer) { mbar_expect_tx(&bar_qk, 32768); mbar_expect_tx(&bar_vo, VO_BYTES); }
    if (lane == 0 && warp < 8 && !(P.withhold == WITHHOLD_PREP && warp == 0)) load_piece(warp, xn);
#pragma unroll 1
    for (int item = blockIdx.x; item < n_items; item += gridDim.x, in_phase ^= 1) {
    const ChunkInfo x = xn;
    const bool has_next = item + (int)gridDim.x < n_items;
    const bool first = item == (int)blockIdx.x;
    if (has_next) chunk_entry(p, xn, item + gridDim.x);

    // this trip's gate arrays (written by warp 0 during the previous trip; the barrier before phase 1 publishes them)
    const float* gl = gate_sets[in_phase][0];
    const float* Gam = gate_sets[in_phase][1];
    const float* ee = gate_sets[in_phase][2];
    const float* bb = gate_sets[in_phase][3];
    const float* ww = gate_sets[in_phase][4];
    const float* bgam = gate_sets[in_phase][5];
    if (ok) {
        ok = mbar_wait(&bar_vo, in_phase);
        ok = ok && mbar_wait(&bar_qk, in_phase) && !(P.withhold == DISAGREE_PREP && (warp & 1));
        if (!ok && lane == 0) report_timeout(p.ws, 1);
    }
    if (ok && x.len < kC) {   // identity padding of a ragged tail: rows beyond the sequence read as zero
        zero_tail_rows(sm + QK, 128, 0, x.len, kIntraThreads);
        zero_tail_rows(sm + QK, 128, 64, x.len, kIntraThreads);
        zero_tail_rows(sm + VO, 128, 0, x.len, kIntraThreads);
        if (bwd) zero_tail_rows(sm + VO, 128, 64, x.len, kIntraThreads);
        fence_async_smem();
    }
    cta_sync();

    // ---- phase 1: S1 = [Q; K] K^T  (rows 0..63: Q K^T, rows 64..127: K K^T)
    if (warp == 16 && elect_one() && ok) {
        tc_fence_after();
        mma_tile<128, 64, 128>(tmem + C_S1, op_k_major(sm + QK, 128, 0), op_k_major(sm + QK, 128, 64), false);
        mma_commit(&bar_mma);
    }
    if (threadIdx.x == 32) mbar_arrive(&bar_ld0);   // this trip's inputs have arrived
    float* Af = reinterpret_cast<float*>(sm + XA);   // [64][kLdi]  strictly lower part of I + A
    float* Tf = reinterpret_cast<float*>(sm + XT);   // [64][kLdi]  T
    if (has_next && warp == 0) fetch_gates(xn);   // next trip's gates -> registers while the product runs
    // R = Diag(Gam) dO (token-major tile)
    auto form_R = [&](unsigned char* dst) {   // the 512 worker threads, two 16-byte pieces each (both loads in flight)
        if (worker) {
            float v[2][8];
#pragma unroll
            for (int it = 0; it < 2; ++it) chunk_load(sm + VO, 128, 64 + (threadIdx.x >> 4) + 32 * it, threadIdx.x & 15, v[it]);
#pragma unroll
            for (int it = 0; it < 2; ++it) {
                const int i = (threadIdx.x >> 4) + 32 * it;
                const float G = Gam[i];
#pragma unroll
                for (int k = 0; k < 8; ++k) v[it][k] *= G;
                chunk_store(dst, 64, i, threadIdx.x & 15, v[it]);
            }
        }
    };
    GDN_WAIT_MMA(2)
    if (ok && !first) {   // the previous trip's stores have read what lies under the fp32 A block and under P
        ok = mbar_wait(&bar_free1, in_phase ^ 1);
        if (!ok && lane == 0) report_timeout(p.ws, 6);
    }
    if (ok && worker) {
        const int i = (q4 & 1) * 32 + lane, j0 = grp * kTG;
#pragma unroll 1
        for (int part = 0; part < kTG / 8; ++part) {
            float v[8];
            tmem_ld8(tmem + lane_base + C_S1 + j0 + part * 8, v);
            tmem_wait_ld();
            const int jb = j0 + part * 8;
            if (q4 < 2) {   // P_ij = (q_i . k_j) exp(gam_i - gam_j), j <= i (mask before exponentiating)
                float g8[8];
                ld8s(gl + jb, g8);
#pragma unroll
                for (int j = 0; j < 8; ++j) v[j] = (jb + j <= i) ? v[j] * ex2(gl[i] - g8[j]) : 0.f;
                chunk_store(sm + PT, 64, i, jb >> 3, v);
            } else {        // A_ij = b_i (k_i . k_j) exp(gam_i - gam_j), j < i
                float g8[8];
                ld8s(gl + jb, g8);
#pragma unroll
                for (int j = 0; j < 8; ++j) v[j] = (jb + j < i) ? bb[i] * v[j] * ex2(gl[i] - g8[j]) : 0.f;
                *reinterpret_cast<float4*>(Af + i * kLdi + jb) = make_float4(v[0], v[1], v[2], v[3]);
                *reinterpret_cast<float4*>(Af + i * kLdi + jb + 4) = make_float4(v[4], v[5], v[6], v[7]);
            }
        }
    }
    tc_fence_before();
    fence_async_smem();
    cta_sync();
    // (P^T dO)^T = dO^T P needs nothing of the inversion: it runs under it and is covered by phase 2's commit
    if (warp == 16 && elect_one() && ok && bwd) {
        tc_fence_after();
        mma_tile<128, 64, 64>(tmem + C_PDO, op_mn_major(sm + VO, 128, 64), op_mn_major(sm + PT, 64), false);
    }
    // ---- T = (I + A)^-1, blocked, fp32 (invert64)
    if (ok && !first) {   // ... and what lies under the fp32 T block
        ok = mbar_wait(&bar_free2, in_phase ^ 1);
        if (!ok && lane == 0) report_timeout(p.ws, 8);
    }
    invert64(Af, Tf, cta_sync);
    if (ok && !first) {   // every store of the previous trip has read its tile (the T tiles and the second readout are next)
        ok = mbar_wait(&bar_free, in_phase ^ 1);
        if (!ok && lane == 0) report_timeout(p.ws, 5);
    }
    if (threadIdx.x < kC * 4) {   // T -> bf16 tiles T, T Diag(b Gam), T Diag(w): a thread scales two rows of one 8-column piece
        const int cch = threadIdx.x & 7;
        float gb[8], gw[8];
        *reinterpret_cast<float4*>(gb) = *reinterpret_cast<const float4*>(bgam + cch * 8);
        *reinterpret_cast<float4*>(gb + 4) = *reinterpret_cast<const float4*>(bgam + cch * 8 + 4);
        *reinterpret_cast<float4*>(gw) = *reinterpret_cast<const float4*>(ww + cch * 8);
        *reinterpret_cast<float4*>(gw + 4) = *reinterpret_cast<const float4*>(ww + cch * 8 + 4);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = (threadIdx.x >> 3) + 32 * h;
            float a[8], b[8], w8[8];
            if ((cch >> 1) <= (i >> 4)) {   // the blocks above the block diagonal are zero and were never written
                *reinterpret_cast<float4*>(a) = *reinterpret_cast<const float4*>(Tf + i * kLdi + cch * 8);
                *reinterpret_cast<float4*>(a + 4) = *reinterpret_cast<const float4*>(Tf + i * kLdi + cch * 8 + 4);
            } else {
#pragma unroll
                for (int k = 0; k < 8; ++k) a[k] = 0.f;
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) { b[k] = gb[k] * a[k]; w8[k] = gw[k] * a[k]; }
            chunk_store(sm + TT, 64, i, cch, a);
            chunk_store(sm + TP, 64, i, cch, b);
            chunk_store(sm + TPP, 64, i, cch, w8);
        }
    }
    fence_async_smem();
    cta_sync();

    // ---- phase 2: W^T = K^T (T Diag(b Gam))^T ; U~^T = V^T (T Diag(w))^T
    if (warp == 16 && elect_one() && ok) {
        tc_fence_after();
        mma_tile<128, 64, 64>(tmem + C_W, op_mn_major(sm + QK, 128, 64), op_k_major(sm + TP, 64), false);
        mma_tile<128, 64, 64>(tmem + C_U, op_mn_major(sm + VO, 128, 0), op_k_major(sm + TPP, 64), false);
        mma_commit(&bar_mma);
    }
    if (threadIdx.x == 32) mbar_arrive(&bar_t);   // the loader stores the T tile
    // R while the MMAs run, over the fp32 A / T scratch, which is dead by now
    if (bwd) form_R(sm + XR);
    GDN_WAIT_MMA(3)
    if (ok && worker) {
        const int f = q4 * 32 + lane, i0 = grp * kTG;
#pragma unroll 1
        for (int part = 0; part < kTG / 8; ++part) {
            const int ib = i0 + part * 8;
            float v[8], ve[8];
            tmem_ld8(tmem + lane_base + C_W + ib, v);
            tmem_wait_ld();
            float e8[8];
            ld8s(ee + ib, e8);
#pragma unroll
            for (int i = 0; i < 8; ++i) ve[i] = v[i] * e8[i];
            chunk_store(sm + WT, 128, f, ib >> 3, v);
            chunk_store(sm + WET, 128, f, ib >> 3, ve);
            tmem_ld8(tmem + lane_base + C_U + ib, v);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 8; ++i) ve[i] = v[i] * e8[i];
            chunk_store(sm + UTT, 128, f, ib >> 3, v);
            chunk_store(sm + UET, 128, f, ib >> 3, ve);
            if (bwd) {
                tmem_ld8(tmem + lane_base + C_PDO + ib, v);
                tmem_wait_ld();
                chunk_store(sm + XPDO, 128, f, ib >> 3, v);
            }
        }
    }
    tc_fence_before();
    fence_async_smem();
    cta_sync();

    // ---- phase 3: Nm = K^T (Diag(e) W) ; Bf = K^T (Diag(e) U~) ; E = Q^T R - W^T (P^T dO)
    if (warp == 16 && elect_one() && ok) {
        tc_fence_after();
        // Nm and Bf share the operand K^T; their other operands and their accumulators are neighbours: one N = 256 product
        static_assert(UET == WET + 16384 && C_BF == C_NM + 128, "Nm | Bf as one product");
        mma_tile<128, 256, 64>(tmem + C_NM, op_mn_major(sm + QK, 128, 64), op_k_major(sm + WET, 128), false);
        if (bwd) mma_tile<128, 128, 64>(tmem + C_E, op_mn_major(sm + QK, 128, 0), op_mn_major(sm + XR, 64), false);
        if (bwd) mma_tile<128, 128, 64>(tmem + C_E, op_k_major(sm + WT, 128), op_k_major(sm + XPDO, 128), true, /*neg_a=*/true);
        mma_commit(&bar_mma);
        mma_commit(&bar_ld1);   // Q, K have been read for the last time
    } else if (threadIdx.x == 32 && ok) {   // (a load is announced behind one that has arrived only)
        mbar_arrive(&bar_vofree);   // W^T, U~^T are staged; V, dO were last read by phase 2 and the pass that formed R
    }
    if (has_next && warp == 0) make_gates(in_phase ^ 1, xn.ch);   // the next trip's gate arrays, while the products run
    GDN_WAIT_MMA(4)
    if (ok) {   // the T tile, part of the Nm staging area, has left through its store
        ok = mbar_wait(&bar_tfree, in_phase);
        if (!ok && lane == 0) report_timeout(p.ws, 7);
    }
    if (ok && worker) {   // Nm, Bf, E -> bf16 tile images staged over tiles that no MMA reads any more
        const int r = q4 * 32 + lane, c0 = grp * (D / kGroups);
        const float sc = p.d.scale;
#pragma unroll 1
        for (int part = 0; part < D / kGroups / 8; ++part) {
            const int cb = c0 + part * 8;
            float v[8];
            tmem_ld8(tmem + lane_base + C_NM + cb, v);
            tmem_wait_ld();
            chunk_store(sm + NMS, 128, r, cb >> 3, v);
            tmem_ld8(tmem + lane_base + C_BF + cb, v);
            tmem_wait_ld();
            chunk_store(sm + BFS, 128, r, cb >> 3, v);
            if (bwd) {
                tmem_ld8(tmem + lane_base + C_E + cb, v);
                tmem_wait_ld();
#pragma unroll
                for (int k = 0; k < 8; ++k) v[k] *= sc;
                chunk_store(sm + ES, 128, r, cb >> 3, v);
            }
        }
    }
    tc_fence_before();
    fence_async_smem();
    cta_sync();
    if (threadIdx.x == 32) mbar_arrive(&bar_st);   // the three images are staged: the loader stores them
    if (!ok) {   // (the loader, which gives up in turn, waits for the loads that are in flight)
        stand_by_items<10>(item, n_items, cta_sync);
        break;
    }
    }
    if (warp == 0) tmem_dealloc(tmem, 512);
}

#include "tc_prep_split.cuh"

// ------------------------------------------------------------------------------------------------
// tc_scan: forward and reverse inter-chunk carries, one CTA per (chain, direction).
// Per chunk: the fp32 state (registers; thread = one row, 64 columns) is rounded to a bf16 tile, one tcgen05.mma
// forms Nm h (forward) or Nm^T dh (reverse), and the state is updated in fp32:  s <- Gam_e s - (Nm s) + add.
// The bf16 tile that fed the MMA is also what the chunk's gradient stage needs, so each thread writes its part
// of the tile image to the workspace as well.  Nm and the additive term (Bf or E) arrive through a two-stage
// ring of bulk copies; the chunk decays exp(gamma_e) are fetched once per chain.
// ------------------------------------------------------------------------------------------------
namespace scan {
constexpr int GE_CAP = 2048;                     // chunk decays cached per chain (longer chains read them from global)
constexpr uint32_t NM = 0, ADD = 32768;          // ring stage: Nm tile image (32 KB) + the CTA's columns of the additive image
// S = number of CTAs that share a chain, each carrying 128 / S state columns (the columns of the state evolve
// independently).  S = 2 is used when there are too few chains to fill the machine.
template <int S> struct Cfg {
    static constexpr int NS = D / S;                         // state columns of this CTA
    static constexpr int STAGES = S == 1 ? 2 : 3;
    static constexpr int PREFETCH_AHEAD = STAGES + 1;        // steps by which L2 prefetches run ahead of the ring loads
    static constexpr uint32_t ADD_BYTES = 32768 / S, STAGE_BYTES = 32768 + ADD_BYTES;
    static constexpr uint32_t HT = STAGES * STAGE_BYTES;     // two state tiles [128][NS] (one feeds the MMA and the bulk
    static constexpr uint32_t HT_BYTES = 32768 / S;          // store of this step while the next step's is being written)
    static constexpr uint32_t SMEM_BYTES = HT + 2 * HT_BYTES + 1024;
    static_assert(SMEM_BYTES + GE_CAP * 4 <= 227 * 1024, "shared memory budget");
};
}  // namespace scan

template <int S>
__global__ void __launch_bounds__(kThreads, 1) tc_scan_kernel(const __grid_constant__ TcParams P) {
    wait_prerequisites();
    using namespace scan;
    using C = Cfg<S>;
    constexpr int NS = C::NS, NSH = NS / 2, STAGES = C::STAGES, PREFETCH_AHEAD = C::PREFETCH_AHEAD;
    constexpr uint32_t STAGE_BYTES = C::STAGE_BYTES, ADD_BYTES = C::ADD_BYTES, HT = C::HT, HT_BYTES = C::HT_BYTES;
    const int blocks = S == 2 && P.narrow_v ? 1 : S;
    const int part = (int)blockIdx.x % blocks, bid = (int)blockIdx.x / blocks;   // column block of the state, (chain, direction)
    const Problem& p = P.p;
    const WsHeader* hdr = reinterpret_cast<const WsHeader*>(p.ws);
    if (hdr->status != GDN_OK) return;
    const int reverse = P.scan_dirs == 2 ? (bid & 1) : P.scan_dirs;
    const int chain = P.scan_dirs == 2 ? (bid >> 1) : bid;
    const int n = chain / p.d.H, hd = chain % p.d.H;
    const int c0 = seq_first_chunk(p, n), c1 = seq_first_chunk(p, n + 1), nsteps = c1 - c0;

    extern __shared__ unsigned char smem_raw[];
    unsigned char* sm = align1024(smem_raw);
    __shared__ float ge[GE_CAP];
    __shared__ uint64_t bar_full[STAGES], bar_mma;
    __shared__ uint32_t tmem_slot;
    const int warp = warp_id(), lane = threadIdx.x & 31;
    const int q4 = warp & 3, hf = warp >> 2;
    const int r = q4 * 32 + lane;              // state row owned by this thread
    const int lc0 = hf * NSH;                  // first of its NSH columns inside the CTA's block
    const int gc0 = part * NS + lc0;           // ... and inside the state
    const uint32_t lane_base = (uint32_t)(q4 * 32) << 16;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) mbar_init(&bar_full[s], 1);
        mbar_init(&bar_mma, 1);
        fence_mbar_init();
    }
    if (warp == 0) { tmem_alloc(&tmem_slot, NS); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;

    auto chunk_of = [&](int s) { return reverse ? (c1 - 1 - s) : (c0 + s); };
    const char* nm_base = p.ws + p.L.Nm;
    const char* add_base = p.ws + (reverse ? p.L.E : p.L.Bf) + part * ADD_BYTES;
    char* keep_base = p.ws + (reverse ? p.L.dhn : p.L.hc) + part * HT_BYTES;
    const float* gamma = reinterpret_cast<const float*>(p.ws + p.L.gamma);
    auto fill = [&](int s) {   // thread 0: bring chunk step s into ring slot s % STAGES
        const int stage = s % STAGES;
        const size_t ch = (size_t)chunk_of(s) * p.d.H + hd;
        mbar_expect_tx(&bar_full[stage], STAGE_BYTES);
        if (!(P.withhold == WITHHOLD_CARRY && s == 0)) bulk_load(sm + stage * STAGE_BYTES + NM, nm_base + ch * 32768, 32768, &bar_full[stage]);
        bulk_load(sm + stage * STAGE_BYTES + ADD, add_base + ch * 32768, ADD_BYTES, &bar_full[stage]);
        // The ring gives a load one step of lead, less than an HBM round trip; pull the step after next into L2 now.
        if (s + PREFETCH_AHEAD < nsteps) {
            const size_t chn = (size_t)chunk_of(s + PREFETCH_AHEAD) * p.d.H + hd;
            prefetch_l2_bulk(nm_base + chn * 32768, 32768);
            prefetch_l2_bulk(add_base + chn * 32768, ADD_BYTES);
        }
    };
    if (threadIdx.x == 32) {
        for (int s = STAGES; s < STAGES + PREFETCH_AHEAD && s < nsteps; ++s) {
            const size_t chn = (size_t)chunk_of(s) * p.d.H + hd;
            prefetch_l2_bulk(nm_base + chn * 32768, 32768);
            prefetch_l2_bulk(add_base + chn * 32768, ADD_BYTES);
        }
        for (int s = 0; s < STAGES && s < nsteps; ++s) fill(s);
    }
    for (int s = threadIdx.x; s < nsteps && s < GE_CAP; s += blockDim.x)
        ge[s] = expf(gamma[((size_t)chunk_of(s) * p.d.H + hd) * kC + kC - 1]);
    // initial state
    float st[NSH];
    {
        const float* init = reverse ? p.dhT : p.h0;
        const bool inside = r < p.d.d_k && gc0 < p.d.d_v;   // (a head dimension of 64: the rest of the state is zero)
        const size_t soff = (((size_t)n * p.d.H + hd) * p.d.d_k + r) * p.d.d_v + gc0;
#pragma unroll
        for (int k = 0; k < NSH / 4; ++k) {
            float4 v = init && inside ? *reinterpret_cast<const float4*>(init + soff + 4 * k) : make_float4(0.f, 0.f, 0.f, 0.f);
            st[4 * k] = v.x; st[4 * k + 1] = v.y; st[4 * k + 2] = v.z; st[4 * k + 3] = v.w;
        }
    }
    __syncthreads();
    const bool disagree = P.withhold == DISAGREE_CARRY && (warp & 1);
    bool ok = true;
    uint32_t mma_phase = 0;
    int s = 0;
#pragma unroll 1
    for (; s < nsteps; ++s) {
        unsigned char* Ht = sm + HT + (s & 1) * HT_BYTES;
        const size_t ch = (size_t)chunk_of(s) * p.d.H + hd;
        const int stage = s % STAGES;
        const unsigned char* ring = sm + stage * STAGE_BYTES;
        const float Ge = s < GE_CAP ? ge[s] : expf(gamma[ch * kC + kC - 1]);
        // state -> bf16: operand tile of the MMA; the same bytes are the per-chunk state the gradient stage reads
#pragma unroll
        for (int k = 0; k < NSH / 8; ++k) *reinterpret_cast<uint4*>(Ht + tile_chunk_off(128, r, (lc0 >> 3) + k)) = pack8(st + 8 * k);
        fence_async_smem();
        __syncthreads();
        if (warp == 0 && elect_one()) {
            ok = mbar_wait(&bar_full[stage], (s / STAGES) & 1);
            if (ok) {
                tc_fence_after();
                const Operand a = reverse ? op_mn_major(ring + NM, 128) : op_k_major(ring + NM, 128);
                mma_tile<128, NS, 128>(tmem, a, op_mn_major(Ht, 128), false);
            } else {
                report_timeout(p.ws, 10);
            }
            // The tile leaves through the async proxy: generic global stores here would stall the next step's proxy
            // fence until they drain.  Waiting for the previous step's store to have read its tile before committing the
            // MMA orders that read before the overwrite of the tile two steps later.
            bulk_store(keep_base + ch * 32768, Ht, HT_BYTES);
            bulk_commit();
            bulk_wait_read<1>();
            mma_commit(&bar_mma);
        } else if (threadIdx.x == 32) {
            // every thread has finished step s - 1, so its ring slot can take step s - 1 + STAGES.  Bulk copies are slow
            // to issue; a thread of another warp does it so that the MMA issue is not delayed.
            if (s >= 1 && s - 1 + STAGES < nsteps) fill(s - 1 + STAGES);
        }
        ok = mbar_wait(&bar_full[stage], (s / STAGES) & 1) && !disagree;   // the additive term of this step is in shared memory
        if (ok) ok = mbar_wait(&bar_mma, mma_phase);
        mma_phase ^= 1;
        if (!ok) {
            if (lane == 0) report_timeout(p.ws, 11);
            stand_by(nsteps - 1 - s, [] { __syncthreads(); });
            break;
        }
        tc_fence_after();
#pragma unroll
        for (int k = 0; k < NSH / 8; ++k) {
            float dl[8], ad[8];
            tmem_ld8(tmem + lane_base + lc0 + 8 * k, dl);
            chunk_load(ring + ADD, 128, r, (lc0 >> 3) + k, ad);
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < 8; ++j) st[8 * k + j] = fmaf(Ge, st[8 * k + j], ad[j] - dl[j]);
        }
        tc_fence_before();
    }
    if (threadIdx.x == 32) drain_ring<STAGES>(bar_full, s, nsteps);
    ok = __syncthreads_and(ok);
    float* fin = reverse ? p.dh0 : p.hT;
    if (fin && ok) {
        const bool inside = r < p.d.d_k && gc0 < p.d.d_v;   // (a head dimension of 64: the rest of the state is zero)
        const size_t soff = (((size_t)n * p.d.H + hd) * p.d.d_k + r) * p.d.d_v + gc0;
#pragma unroll
        for (int k = 0; k < NSH / 4; ++k) if (inside) *reinterpret_cast<float4*>(fin + soff + 4 * k) = make_float4(st[4 * k], st[4 * k + 1], st[4 * k + 2], st[4 * k + 3]);
    }
    if (warp == 0) {
        bulk_wait_read<0>();
        tc_fence_after();
        tmem_dealloc(tmem, NS);
    }
}

// ------------------------------------------------------------------------------------------------
// tc_scan_lr: the same carries without the d x d operator of a chunk, for shapes whose carries are bound by HBM
// bandwidth (one CTA per chain and direction fills the machine).  With e_j = exp(gam_e - gam_j):
//   forward   U  = U~ - W h (stored over U~),                 h' = Gam_e h   + K^T Diag(e) U
//   reverse   dU = scale P^T dO + Diag(e) K dh' (stored),     dh = Gam_e dh' + (scale Diag(Gam) Q)^T dO - W^T dU
// U and dU are what the forward output and the gradient stage need: both are operands of the second product here, so they cost a store of
// 16 KB each and save those kernels a phase, and with the whole of dU under W^T the additive term of the reverse carry needs neither P
// nor W: the preparation has no share in the backward, and a backward on a workspace fresh from the forward starts with the carry.
// Per step a ring slot receives W^T, the K tile of the chunk and U~^T (forward) or Q, dO and P (reverse); the first product leaves
// (W h)^T or (K dh')^T with features on TMEM lanes and tokens on columns, the readout forms the bf16 operand of the second product in the
// same orientation, the second product yields the d_k x d_v increment of the state, which lives in fp32 registers as in tc_scan.  P^T dO
// and Q^T dO do not depend on the state: they are issued behind the first product and run under its readout.
// 4 x 16 heads of 2048 tokens, both directions: 88 us, 216 KB per chunk-head at 4.8 TB/s, which bounds it (with the additive term E from the
// preparation, U and dU left to the consumers, 77; the preparation took 80 us for 64, the gradient stage 115 for 105, the output of 6 x 16
// heads of 1500 tokens 51 for 44, and a backward on the forward's workspace had a kernel more, of 38 us).  What it costs: a forward without output,
// which leaves U for a backward that may follow, 1 to 7 % (64 chains of 32 chunks 125 -> 134 us; with that backward 357 -> 333).
// ------------------------------------------------------------------------------------------------
namespace scanlr {
constexpr uint32_t WT = 0, KT = 16384, XT = 32768;   // ring slot: W^T | K | forward: this CTA's part of U~^T (16 KB / S), and room for U^T behind it
constexpr uint32_t UT = 49152;
constexpr uint32_t QT = 32768, PT = 49152, OT = 57344;   // reverse: Q | P | this CTA's columns of dO
constexpr uint32_t C_D1 = 0, C_D3 = 64, C_D2 = 128;      // TMEM columns: first product (64), (P^T dO)^T (64), second product (128 / S)
// S = number of CTAs that share a chain, each carrying 128 / S state columns (the columns of the state evolve
// independently; W and K are needed whole by every one of them).  S = 2 serves the reverse carry alone (the backward on a fresh workspace) with
// so few chains that half of the SMs would idle: a step of a half is shorter, and a step's latency is what bounds that launch; and every
// call with d_v = 64, where the first half is all there is.
template <int S> struct Cfg {
    static constexpr int NS = D / S;                          // state columns of this CTA = rows of the first product
    static constexpr int NSH = NS / 2;                        // ... of one thread
    static constexpr int STAGES = 2;
    static constexpr uint32_t STAGE_BYTES = OT + 16384 / S;
    static constexpr uint32_t HT = STAGES * STAGE_BYTES;      // two bf16 state tiles [128][NS]
    static constexpr uint32_t HT_BYTES = 32768 / S;
    static constexpr uint32_t GT = HT + 2 * HT_BYTES;         // operand of the second product, [NS features][64 tokens]
    static constexpr uint32_t SMEM_BYTES = GT + 16384 / S + 1024;
    static constexpr uint32_t TMEM_COLS = 256;
    static_assert(SMEM_BYTES + 1536 <= 227 * 1024, "shared memory budget");
    static_assert(UT + 16384 / S <= STAGE_BYTES && STAGE_BYTES % 1024 == 0, "U^T fits behind a forward slot's tiles");
};
struct Gates { float ee[2][kC], gq[2][kC], ge[2]; };   // e_j, scale Gam_j and Gam_e of a step, made during the step before it
// What the threads of a CTA share besides the tiles.
struct Shared {
    Gates gates;
    uint64_t full[2], mma;           // a ring slot has arrived; a product of the present step is done
    uint64_t free1[2], free2[2];     // by step parity: the tiles that the first product was the last to read, and all others, may be loaded over
    uint32_t tmem;
    uint32_t gave_up[2];             // a warp has given up (tc_common.cuh), by parity of the step that judges it: behind its first barrier
};
constexpr int kScanThreads = kThreads + 32;   // ... and a warp that only loads: a tile of the step after next goes over its predecessor as
                                              // soon as the product that read it last is done
}  // namespace scanlr

// One direction of one chain (the direction is a compile-time constant: the two differ in operands and readouts).
template <bool reverse, int S>
__device__ __forceinline__ void scan_lr_chain(const TcParams& P, int chain, int part, scanlr::Shared& sh) {
    using namespace scanlr;
    using C = Cfg<S>;
    constexpr int NS = C::NS, NSH = C::NSH, STAGES = C::STAGES;
    constexpr uint32_t STAGE_BYTES = C::STAGE_BYTES, HT = C::HT, HT_BYTES = C::HT_BYTES, GT = C::GT, VALUE_BYTES = 16384 / S;
    Gates& gates = sh.gates;
    uint64_t *bar_full = sh.full, &bar_mma = sh.mma;
    const Problem& p = P.p;
    const int H = p.d.H, n = chain / H, hd = chain % H;
    const SeqGeom sg = seq_geom(p, n);
    const int c0 = sg.c0, nsteps = sg.n_chunks, c1 = c0 + nsteps;
    auto chunk_of = [&](int s) { return reverse ? (c1 - 1 - s) : (c0 + s); };

    extern __shared__ unsigned char smem_raw[];
    unsigned char* sm = align1024(smem_raw);
    const int warp = warp_id(), lane = threadIdx.x & 31;
    const int q4 = warp & 3, hf = warp >> 2;
    const int r = q4 * 32 + lane;              // TMEM lane of this thread: state row (d_k) or feature of the first product (d_v)
    const int lc0 = hf * NSH;                  // first of its NSH state columns inside the CTA's block
    const int tk0 = hf * 32;                   // first of its 32 tokens in the first product
    // The first product has NS rows.  With 128 of them a thread's TMEM lane is its feature; with 64 (M = 64) the rows sit
    // on lanes 0..15 of each quadrant and the other lanes of a warp have nothing to read out.
    const int r1 = S == 1 ? r : q4 * 16 + (lane & 15);
    const bool act1 = S == 1 || lane < 16;
    const uint32_t lane_base = (uint32_t)(q4 * 32) << 16;
    const float sc = p.d.scale;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) { mbar_init(&bar_full[s], 1); mbar_init(&sh.free1[s], 1); mbar_init(&sh.free2[s], 1); }
        mbar_init(&bar_mma, 1);
        sh.gave_up[0] = sh.gave_up[1] = 0;
        fence_mbar_init();
    }
    if (warp == 0) { tmem_alloc(&sh.tmem, C::TMEM_COLS); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sh.tmem;

    // this CTA's rows of U~^T, then U^T, or of dU^T (both images [d_v][tokens])
    char* y_base = p.ws + (reverse ? p.L.E : p.L.Ut) + part * VALUE_BYTES;
    char* keep_base = p.ws + (reverse ? p.L.dhn : p.L.hc) + part * HT_BYTES;
    const float* gamma = reinterpret_cast<const float*>(p.ws + p.L.gamma);
    // (L2 prefetches running ahead of the ring, as in tc_scan, made this kernel slower: 79.7 -> 78.5 us without)
    // The tiles of step s into ring slot s % STAGES, in two parts: those whose predecessors are dead after the first product (W^T forward; K and P
    // in reverse), which announce the slot's bytes, and the rest.
    auto fill1 = [&](int s) {
        const int stage = s % STAGES, c = chunk_of(s), tok0 = sg.chunk_tok0(c);
        const size_t ch = (size_t)c * H + hd;
        unsigned char* slot = sm + stage * STAGE_BYTES;
        uint64_t* bar = &bar_full[stage];
        mbar_expect_tx(bar, 32768 + VALUE_BYTES + (reverse ? 24576 : 0));
        if (reverse) {
            for (int cb = 0; cb < 2; ++cb) tma_load_3d(slot + KT + cb * 8192, &P.tm_k, cb * 64, hd, tok0, bar);
            bulk_load(slot + PT, p.ws + p.L.Pm + ch * 8192, 8192, bar);
        } else if (!(P.withhold == WITHHOLD_CARRY && s == 0)) {
            bulk_load(slot + WT, p.ws + p.L.W + ch * 16384, 16384, bar);
        }
    };
    auto fill2 = [&](int s) {
        const int stage = s % STAGES, c = chunk_of(s), tok0 = sg.chunk_tok0(c);
        const size_t ch = (size_t)c * H + hd;
        unsigned char* slot = sm + stage * STAGE_BYTES;
        uint64_t* bar = &bar_full[stage];
        if (reverse) {
            for (int cb = 0; cb < 2 / S; ++cb) tma_load_3d(slot + OT + cb * 8192, &P.tm_do, part * NS + cb * 64, hd, tok0, bar);
            for (int cb = 0; cb < 2; ++cb) tma_load_3d(slot + QT + cb * 8192, &P.tm_q, cb * 64, hd, tok0, bar);
            if (!(P.withhold == WITHHOLD_CARRY && s == 0)) bulk_load(slot + WT, p.ws + p.L.W + ch * 16384, 16384, bar);
        } else {
            for (int cb = 0; cb < 2; ++cb) tma_load_3d(slot + KT + cb * 8192, &P.tm_k, cb * 64, hd, tok0, bar);
            bulk_load(slot + XT, y_base + ch * 16384, VALUE_BYTES, bar);
        }
    };
    if (warp == kThreads / 32) {
        if (lane == 0) {
            for (int s = 0; s < STAGES && s < nsteps; ++s) { fill1(s); fill2(s); }
            int s = 0;
            for (; s + STAGES < nsteps; ++s) {   // (a product two steps on needs the slot filled here: no phase of these barriers can be missed)
                if (!mbar_wait(&sh.free1[s & 1], (s >> 1) & 1)) break;
                fill1(s + STAGES);
                if (!mbar_wait(&sh.free2[s & 1], (s >> 1) & 1)) { ++s; break; }
                fill2(s + STAGES);
            }
            drain_ring<STAGES>(bar_full, s, nsteps);   // (what is still in flight after a time-out; otherwise the workers wait for the same loads)
        }
        return;
    }
    auto cta_sync = [] { asm volatile("bar.sync 1, %0;" ::"n"(kThreads) : "memory"); };   // all warps but the loader
    const bool disagree = P.withhold == DISAGREE_CARRY && (warp & 1);
    // the gate arrays of the first step; the cumulative decays of the second are fetched now
    auto gate_row = [&](int s) { return gamma + ((size_t)chunk_of(s) * H + hd) * kC; };
    auto make_gates = [&](int set, float g, float gend) {
        gates.ee[set][threadIdx.x] = expf(gend - g);
        if (reverse) gates.gq[set][threadIdx.x] = sc * expf(g);
        if (threadIdx.x == 0) gates.ge[set] = expf(gend);
    };
    float gnext = 0.f, gend_next = 0.f;
    if (threadIdx.x < kC && nsteps > 0) {
        make_gates(0, gate_row(0)[threadIdx.x], gate_row(0)[kC - 1]);
        if (nsteps > 1) { gnext = gate_row(1)[threadIdx.x]; gend_next = gate_row(1)[kC - 1]; }
    }
    float st[NSH];
    {
        const float* init = reverse ? p.dhT : p.h0;
        const bool inside = r < p.d.d_k && part * NS + lc0 < p.d.d_v;   // (a head dimension of 64: the rest of the state is zero)
        const size_t soff = (((size_t)n * H + hd) * p.d.d_k + r) * p.d.d_v + part * NS + lc0;
#pragma unroll
        for (int k = 0; k < NSH / 4; ++k) {
            float4 v = init && inside ? *reinterpret_cast<const float4*>(init + soff + 4 * k) : make_float4(0.f, 0.f, 0.f, 0.f);
            st[4 * k] = v.x; st[4 * k + 1] = v.y; st[4 * k + 2] = v.z; st[4 * k + 3] = v.w;
        }
    }
    cta_sync();
    bool ok = true;
    uint32_t mma_phase = 0;
    auto wait_for = [&](uint64_t* bar, uint32_t parity, int where, int judged) {
        if (!ok) return;
        ok = mbar_wait_inline(bar, parity);
        if (!ok) { report_timeout(p.ws, where); sh.gave_up[judged & 1] = 1; }
    };
    int s = 0;
#pragma unroll 1
    for (; s < nsteps; ++s) {
        unsigned char* Ht = sm + HT + (s & 1) * HT_BYTES;
        const int c = chunk_of(s), stage = s % STAGES, len = sg.chunk_len(c);
        const size_t ch = (size_t)c * H + hd;
        unsigned char* ring = sm + stage * STAGE_BYTES;
        const float* ee = gates.ee[s & 1];
        // state -> bf16: operand of the first product, and the per-chunk state the gradient stage reads
#pragma unroll
        for (int k = 0; k < NSH / 8; ++k) *reinterpret_cast<uint4*>(Ht + tile_chunk_off(128, r, (lc0 >> 3) + k)) = pack8(st + 8 * k);
        if (len < kC) {   // ragged tail: the rows beyond the sequence belong to somebody else
            wait_for(&bar_full[stage], (s / STAGES) & 1, 12, s);
            zero_tail_rows(ring + KT, 64, 0, len, kThreads);
            if (reverse) {
                zero_tail_rows(ring + QT, 64, 0, len, kThreads);
                for (int t = threadIdx.x; t < (kC - len) * (NS / 8); t += kThreads)
                    *reinterpret_cast<uint4*>(ring + OT + tile_chunk_off(64, len + t / (NS / 8), t % (NS / 8))) = make_uint4(0, 0, 0, 0);
            }
        }
        fence_async_smem();
        cta_sync();
        const uint32_t gone = sh.gave_up[s & 1];   // (of this step so far and of the step before)
        const float Ge = gates.ge[s & 1];   // decay of the state over the chunk
        wait_for(&bar_full[stage], (s / STAGES) & 1, 10, s + 1);
        if (warp == 0 && elect_one() && ok) {
            tc_fence_after();
            // forward (W h)^T = h^T W^T ; reverse (K dh')^T = dh'^T K^T : [d_v][tokens]
            const Operand b = reverse ? op_k_major(ring + KT, 64) : op_mn_major(ring + WT, 128);
            mma_tile<NS, 64, 128>(tmem + C_D1, op_mn_major(Ht, 128), b, false);
            if (reverse) mma_tile<NS, 64, 64>(tmem + C_D3, op_mn_major(ring + OT, 64), op_mn_major(ring + PT, 64), false);   // (P^T dO)^T
            bulk_store(keep_base + ch * 32768, Ht, HT_BYTES);
            bulk_commit();
            bulk_wait_read<1>();   // (the stores of the step before have read their tiles: they are rewritten from here on)
            mma_commit(&bar_mma);
            mma_commit(&sh.free1[s & 1]);
        }
        if (disagree) { ok = false; report_timeout(p.ws, 14); sh.gave_up[(s + 1) & 1] = 1; }
        if (reverse) {   // scale Diag(Gam) Q in place, under the first product; its product by dO runs under the readout
            if (ok) {
#pragma unroll
                for (int it = 0; it < 4; ++it) {
                    const int i = (threadIdx.x >> 4) + 16 * it;
                    float v[8];
                    chunk_load(ring + QT, 64, i, threadIdx.x & 15, v);
                    const float G = gates.gq[s & 1][i];
#pragma unroll
                    for (int k = 0; k < 8; ++k) v[k] *= G;
                    chunk_store(ring + QT, 64, i, threadIdx.x & 15, v);
                }
            }
            fence_async_smem();
            cta_sync();
            if (warp == 0 && elect_one() && ok && !gone) mma_tile<128, NS, 64>(tmem + C_D2, op_mn_major(ring + QT, 64), op_mn_major(ring + OT, 64), false);
        }
        wait_for(&bar_mma, mma_phase, 11, s + 1);
        mma_phase ^= 1;
        if (gone) break;   // (here, where no product is in flight any more and nobody waits for the word)
        tc_fence_after();
        // operand of the second product, transposed: forward Diag(e) U (and U, for the workspace), reverse dU
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            float d1[8], u[8], e8[8];
            tmem_ld8(tmem + lane_base + C_D1 + tk0 + 8 * k, d1);
            if (reverse) {
                tmem_ld8(tmem + lane_base + C_D3 + tk0 + 8 * k, u);
            } else if (act1) {
                chunk_load(ring + XT, NS, r1, (tk0 >> 3) + k, u);
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j) u[j] = 0.f;
            }
            ld8s(ee + tk0 + 8 * k, e8);
            tmem_wait_ld();
            if (reverse) {
#pragma unroll
                for (int j = 0; j < 8; ++j) d1[j] = fmaf(sc, u[j], e8[j] * d1[j]);
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j) u[j] -= d1[j];
                if (act1) chunk_store(ring + UT, NS, r1, (tk0 >> 3) + k, u);
#pragma unroll
                for (int j = 0; j < 8; ++j) d1[j] = e8[j] * u[j];
            }
            if (act1) chunk_store(sm + GT, NS, r1, (tk0 >> 3) + k, d1);
        }
        tc_fence_before();
        fence_async_smem();
        cta_sync();
        if (warp == 0 && elect_one() && ok) {
            tc_fence_after();
            if (reverse) mma_tile<128, NS, 64>(tmem + C_D2, op_k_major(ring + WT, 128), op_k_major(sm + GT, NS), true, /*neg_a=*/true);
            else mma_tile<128, NS, 64>(tmem + C_D2, op_mn_major(ring + KT, 64), op_k_major(sm + GT, NS), false);
            mma_commit(&bar_mma);
            mma_commit(&sh.free2[s & 1]);
            bulk_store(y_base + ch * 16384, reverse ? sm + GT : ring + UT, VALUE_BYTES);
            bulk_commit();
        }
        if (threadIdx.x < kC && s + 1 < nsteps) {   // the gate arrays of the next step, while the product runs
            make_gates((s + 1) & 1, gnext, gend_next);
            if (s + 2 < nsteps) { gnext = gate_row(s + 2)[threadIdx.x]; gend_next = gate_row(s + 2)[kC - 1]; }
        }
        wait_for(&bar_mma, mma_phase, 13, s + 1);
        mma_phase ^= 1;
        tc_fence_after();
#pragma unroll
        for (int k = 0; k < NSH / 8; ++k) {
            float d2[8];
            tmem_ld8(tmem + lane_base + C_D2 + lc0 + 8 * k, d2);
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < 8; ++j) st[8 * k + j] = fmaf(Ge, st[8 * k + j], d2[j]);
        }
        tc_fence_before();
    }
    cta_sync();   // every reader of the accumulators is done
    ok = !(sh.gave_up[0] | sh.gave_up[1]);
    float* fin = reverse ? p.dh0 : p.hT;
    if (fin && ok) {
        const bool inside = r < p.d.d_k && part * NS + lc0 < p.d.d_v;   // (a head dimension of 64: the rest of the state is zero)
        const size_t soff = (((size_t)n * H + hd) * p.d.d_k + r) * p.d.d_v + part * NS + lc0;
#pragma unroll
        for (int k = 0; k < NSH / 4; ++k) if (inside) *reinterpret_cast<float4*>(fin + soff + 4 * k) = make_float4(st[4 * k], st[4 * k + 1], st[4 * k + 2], st[4 * k + 3]);
    }
    if (warp == 0) {
        bulk_wait_read<0>();
        tc_fence_after();
        tmem_dealloc(tmem, C::TMEM_COLS);
    }
}

// Block index -> (chain, direction, column block): with both directions in one launch the direction is the low bit
// (S = 1, or narrow_v, where the second column block is not there); with S = 2 (one direction per launch) the low bit is the column block.
template <int S>
__global__ void __launch_bounds__(scanlr::kScanThreads, 1) tc_scan_lr_kernel(const __grid_constant__ TcParams P) {
    wait_prerequisites();
    using namespace scanlr;
    __shared__ __align__(16) scanlr::Shared sh;
    const int bid = (int)blockIdx.x;
    if (reinterpret_cast<const WsHeader*>(P.p.ws)->status != GDN_OK) return;
    const bool halves = S == 2 && !P.narrow_v;
    const int rev = (!halves && P.scan_dirs == 2) ? (bid & 1) : P.scan_dirs;
    const int chain = (halves || P.scan_dirs == 2) ? (bid >> 1) : bid;
    const int part = halves ? (bid & 1) : 0;
    if (rev) scan_lr_chain<true, S>(P, chain, part, sh);
    else scan_lr_chain<false, S>(P, chain, part, sh);
}

namespace scancw {
constexpr uint32_t WT = 0, KT = 16384, XT = 32768;   // ring slot: W^T | K | this CTA's part of U~^T (16 KB / S) or E (32 KB / S)
constexpr uint32_t C_D1 = 0, C_D2 = 64;              // TMEM columns: first product (64), second product (128 / S)
// S = number of CTAs that share a chain, each carrying 128 / S state columns (the columns of the state evolve
// independently; W and K are needed whole by every one of them).  S = 2 serves calls that run one direction only with so
// few chains that half of the SMs would idle (the forward, the backward on a fresh workspace): a step of a half is
// shorter, and a step's latency is what bounds those launches.
template <int S> struct Cfg {
    static constexpr int NS = D / S;                          // state columns of this CTA = rows of the first product
    static constexpr int NSH = NS / 2;                        // ... of one thread
    static constexpr int STAGES = S == 1 ? 2 : 3;
    static constexpr uint32_t STAGE_BYTES = 32768 + 32768 / S;
    static constexpr uint32_t HT = STAGES * STAGE_BYTES;      // two bf16 state tiles [128][NS]
    static constexpr uint32_t HT_BYTES = 32768 / S;
    static constexpr uint32_t GT = HT + 2 * HT_BYTES;         // operand of the second product, [NS features][64 tokens]
    static constexpr uint32_t SMEM_BYTES = GT + 16384 / S + 1024;
    static constexpr uint32_t TMEM_COLS = S == 1 ? 256 : 128;
    static_assert(SMEM_BYTES + 2048 <= 227 * 1024, "shared memory budget");
};
}  // namespace scancw

// The carries of the channel-wise path (per-channel gates, d_k = d_v = 128, bf16 I/O) on the same machinery, with the additive term E of
// the preparation in reverse: the decay of the state is a vector (one factor per state
// row, i.e. per thread), and the key tile arrives as K- = S k / Gam, a tile image from the
// workspace together with images of W^T, U~^T and E (written by the channel-wise preparation kernels), so the readout of the
// first product applies no per-token factor.  Those images are relative to a reference S = 2^ref of the chunk (gdn_tc_cw.cu), and
// so is the state that enters a chunk's products: S h forward, (Gam_e / S) dh' in reverse.  The registers carry it relative to a
// reference as well, so that a step has one factor per row and no operation more than without references:
//   forward   x = S h,             x'  = A (x + K-^T U)        with A = Gam_e S' / S     (S': of the next chunk, 1 after the last)
//   reverse   w = dh' / S'',       w'  = A w + E - W^T Y       with A = Gam_e S'' / S    (S'': of the chunk before in this order, 1 at first)
// (A scaled copy of an unscaled state, and a factor of its own for the increment, took 40 to 50 ns a step: 8 heads of 8192 tokens
// 383 -> 388 us.)
template <bool reverse, int S>
__device__ __forceinline__ void scan_cw_chain(const TcParams& P, int chain, int part, uint64_t* bar_full,
                                              uint64_t& bar_mma, uint32_t& tmem_slot) {
    using namespace scancw;
    using C = Cfg<S>;
    constexpr int NS = C::NS, NSH = C::NSH, STAGES = C::STAGES;
    constexpr uint32_t STAGE_BYTES = C::STAGE_BYTES, HT = C::HT, HT_BYTES = C::HT_BYTES, GT = C::GT;
    const Problem& p = P.p;
    const int H = p.d.H, n = chain / H, hd = chain % H;
    const SeqGeom sg = seq_geom(p, n);
    const int c0 = sg.c0, nsteps = sg.n_chunks, c1 = c0 + nsteps;
    auto chunk_of = [&](int s) { return reverse ? (c1 - 1 - s) : (c0 + s); };

    extern __shared__ unsigned char smem_raw[];
    unsigned char* sm = align1024(smem_raw);
    const int warp = warp_id(), lane = threadIdx.x & 31;
    const int q4 = warp & 3, hf = warp >> 2;
    const int r = q4 * 32 + lane;              // TMEM lane of this thread: state row (d_k) or feature of the first product (d_v)
    const int lc0 = hf * NSH;                  // first of its NSH state columns inside the CTA's block
    const int tk0 = hf * 32;                   // first of its 32 tokens in the first product
    // The first product has NS rows.  With 128 of them a thread's TMEM lane is its feature; with 64 (M = 64) the rows sit
    // on lanes 0..15 of each quadrant and the other lanes of a warp have nothing to read out.
    const int r1 = S == 1 ? r : q4 * 16 + (lane & 15);
    const bool act1 = S == 1 || lane < 16;
    const uint32_t lane_base = (uint32_t)(q4 * 32) << 16;
    // channel-wise: log decay over the chunk and reference of this thread's state row, fetched a step ahead
    struct { float gam; int ref; } cw_next{0.f, 0};
    auto cw_fetch = [&](int s) {
        if (s < nsteps) {
            const size_t ch = (size_t)chunk_of(s) * H + hd;
            cw_next.gam = reinterpret_cast<const float*>(p.ws + p.L.gamma)[(ch * kC + kC - 1) * D + r];
            cw_next.ref = reinterpret_cast<const int32_t*>(p.ws + p.L.ref)[ch * D + r];
        } else {
            cw_next.ref = 0;
        }
    };
    cw_fetch(0);

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) mbar_init(&bar_full[s], 1);
        mbar_init(&bar_mma, 1);
        fence_mbar_init();
    }
    if (warp == 0) { tmem_alloc(&tmem_slot, C::TMEM_COLS); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;

    const char* w_base = p.ws + p.L.img_W;
    // this CTA's part of the additive image: rows part * NS.. of U~^T [d_v][tokens], column block `part` of E [d_k][d_v]
    const uint32_t x_chunk = reverse ? 32768u : 16384u, x_bytes = x_chunk / S;
    const char* x_base = p.ws + (reverse ? p.L.img_E : p.L.img_U) + part * x_bytes;
    char* keep_base = p.ws + (reverse ? p.L.dhn : p.L.hc) + part * HT_BYTES;
    // (L2 prefetches running ahead of the ring, as in tc_scan, made this kernel slower: 79.7 -> 78.5 us without)
    auto fill = [&](int s) {   // thread 32: bring chunk step s into ring slot s % STAGES
        const int stage = s % STAGES, c = chunk_of(s);
        const size_t ch = (size_t)c * H + hd;
        unsigned char* slot = sm + stage * STAGE_BYTES;
        mbar_expect_tx(&bar_full[stage], 32768 + x_bytes);
        if (!(P.withhold == WITHHOLD_CARRY && s == 0)) bulk_load(slot + WT, w_base + ch * 16384, 16384, &bar_full[stage]);
        // k-, in both directions: what is left of the decay is applied to the state (row by row, below)
        bulk_load(slot + KT, p.ws + p.L.img_Km + ch * 16384, 16384, &bar_full[stage]);
        bulk_load(slot + XT, x_base + ch * x_chunk, x_bytes, &bar_full[stage]);
    };
    if (threadIdx.x == 32) {
        for (int s = 0; s < STAGES && s < nsteps; ++s) fill(s);
    }
    float st[NSH];
    {
        const float* init = reverse ? p.dhT : p.h0;
        const bool inside = r < p.d.d_k && part * NS + lc0 < p.d.d_v;   // (a head dimension of 64: the rest of the state is zero)
        const size_t soff = (((size_t)n * H + hd) * p.d.d_k + r) * p.d.d_v + part * NS + lc0;
#pragma unroll
        for (int k = 0; k < NSH / 4; ++k) {
            float4 v = init && inside ? *reinterpret_cast<const float4*>(init + soff + 4 * k) : make_float4(0.f, 0.f, 0.f, 0.f);
            st[4 * k] = v.x; st[4 * k + 1] = v.y; st[4 * k + 2] = v.z; st[4 * k + 3] = v.w;
        }
    }
    __syncthreads();
    bool ok = true;
    uint32_t mma_phase = 0;
    int cw_ref = 0;   // reverse: reference of the step before
    if (!reverse) {
        const float S_ref = pow2(cw_next.ref);
#pragma unroll
        for (int k = 0; k < NSH; ++k) st[k] *= S_ref;
    }
    int s = 0;
#pragma unroll 1
    for (; s < nsteps; ++s) {
        unsigned char* Ht = sm + HT + (s & 1) * HT_BYTES;
        const int c = chunk_of(s), stage = s % STAGES;
        const size_t ch = (size_t)c * H + hd;
        unsigned char* ring = sm + stage * STAGE_BYTES;
        float Ge = expf(cw_next.gam);   // decay of this thread's state row over the chunk
        const int ref = cw_next.ref;
        if (reverse) { Ge *= pow2(cw_ref - ref); cw_ref = ref; }   // A
        cw_fetch(s + 1);
        // state -> bf16: operand of the first product, and the per-chunk state the gradient stage reads
#pragma unroll
        for (int k = 0; k < NSH / 8; ++k) {
            if constexpr (reverse) {
                float sc8[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) sc8[j] = Ge * st[8 * k + j];
                *reinterpret_cast<uint4*>(Ht + tile_chunk_off(128, r, (lc0 >> 3) + k)) = pack8(sc8);
            } else {
                *reinterpret_cast<uint4*>(Ht + tile_chunk_off(128, r, (lc0 >> 3) + k)) = pack8(st + 8 * k);
            }
        }
        fence_async_smem();
        __syncthreads();
        if (warp == 0 && elect_one()) {
            ok = mbar_wait_inline(&bar_full[stage], (s / STAGES) & 1);
            if (ok) {
                tc_fence_after();
                // forward (W h)^T = h^T W^T ; reverse (K dh')^T = dh'^T K^T : [d_v][tokens]
                const Operand b = reverse ? op_k_major(ring + KT, 64) : op_mn_major(ring + WT, 128);
                mma_tile<NS, 64, 128>(tmem + C_D1, op_mn_major(Ht, 128), b, false);
            } else {
                report_timeout(p.ws, 10);
            }
            bulk_store(keep_base + ch * 32768, Ht, HT_BYTES);
            bulk_commit();
            bulk_wait_read<1>();   // (the store of the step before has read its tile: it is rewritten in the next step)
            mma_commit(&bar_mma);
        } else if (threadIdx.x == 32) {
            if (s >= 1 && s - 1 + STAGES < nsteps) fill(s - 1 + STAGES);
        }
        ok = mbar_wait_inline(&bar_full[stage], (s / STAGES) & 1);
        if (ok) ok = mbar_wait_inline(&bar_mma, mma_phase);
        mma_phase ^= 1;
        if (!ok) { if (lane == 0) report_timeout(p.ws, 11); break; }
        tc_fence_after();
        // operand of the second product: forward Diag(e)(U~ - W h), reverse Diag(e)(K dh'), transposed
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            float d1[8], u[8];
            if constexpr (S == 2) {
#pragma unroll
                for (int j = 0; j < 8; ++j) u[j] = 0.f;
            }
            tmem_ld8(tmem + lane_base + C_D1 + tk0 + 8 * k, d1);
            if (!reverse && act1) chunk_load(ring + XT, NS, r1, (tk0 >> 3) + k, u);
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < 8; ++j) d1[j] = reverse ? d1[j] : u[j] - d1[j];
            if (act1) chunk_store(sm + GT, NS, r1, (tk0 >> 3) + k, d1);
        }
        tc_fence_before();
        fence_async_smem();
        __syncthreads();
        if (warp == 0 && elect_one()) {
            tc_fence_after();
            if (reverse) mma_tile<128, NS, 64>(tmem + C_D2, op_k_major(ring + WT, 128), op_k_major(sm + GT, NS), false, /*neg_a=*/true);
            else mma_tile<128, NS, 64>(tmem + C_D2, op_mn_major(ring + KT, 64), op_k_major(sm + GT, NS), false);
            mma_commit(&bar_mma);
        }
        ok = mbar_wait_inline(&bar_mma, mma_phase);
        mma_phase ^= 1;
        if (!ok) { if (lane == 0) report_timeout(p.ws, 13); break; }
        tc_fence_after();
        if (!reverse) Ge *= pow2(cw_next.ref - ref);   // A
#pragma unroll
        for (int k = 0; k < NSH / 8; ++k) {
            float d2[8], ad[8];
            tmem_ld8(tmem + lane_base + C_D2 + lc0 + 8 * k, d2);
            if (reverse) chunk_load(ring + XT, 128, r, (lc0 >> 3) + k, ad);
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                if (!reverse) st[8 * k + j] = Ge * (st[8 * k + j] + d2[j]);
                else st[8 * k + j] = fmaf(Ge, st[8 * k + j], ad[j] + d2[j]);
            }
        }
        tc_fence_before();
    }
    float* fin = reverse ? p.dh0 : p.hT;
    if (reverse) {
        const float S_ref = pow2(cw_ref);
#pragma unroll
        for (int k = 0; k < NSH; ++k) st[k] *= S_ref;
    }
    if (fin && ok) {
        const bool inside = r < p.d.d_k && part * NS + lc0 < p.d.d_v;   // (a head dimension of 64: the rest of the state is zero)
        const size_t soff = (((size_t)n * H + hd) * p.d.d_k + r) * p.d.d_v + part * NS + lc0;
#pragma unroll
        for (int k = 0; k < NSH / 4; ++k) if (inside) *reinterpret_cast<float4*>(fin + soff + 4 * k) = make_float4(st[4 * k], st[4 * k + 1], st[4 * k + 2], st[4 * k + 3]);
    }
    if (warp == 0) bulk_wait_read<0>();
    if (threadIdx.x == 32) drain_ring<STAGES>(bar_full, s, nsteps);
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, C::TMEM_COLS);
}

template <int S>
__global__ void __launch_bounds__(kThreads, 1) tc_scan_cw_kernel(const __grid_constant__ TcParams P) {
    wait_prerequisites();
    using namespace scancw;
    __shared__ uint64_t bar_full[Cfg<S>::STAGES], bar_mma;
    __shared__ uint32_t tmem_slot;
    const int bid = (int)blockIdx.x;
    const WsHeader* hdr = reinterpret_cast<const WsHeader*>(P.p.ws);
    if (hdr->status != GDN_OK || hdr->cw_fallback) return;
    const int rev = (S == 1 && P.scan_dirs == 2) ? (bid & 1) : P.scan_dirs;
    const int chain = (S == 2 || P.scan_dirs == 2) ? (bid >> 1) : bid;
    const int part = S == 2 ? (bid & 1) : 0;
    if (rev) scan_cw_chain<true, S>(P, chain, part, bar_full, bar_mma, tmem_slot);
    else scan_cw_chain<false, S>(P, chain, part, bar_full, bar_mma, tmem_slot);
}

// ------------------------------------------------------------------------------------------------
// tc_intra: token gradients of one (chunk, head).
//
// Products (all on tcgen05), in four dependent phases:
//   phase 1  (W h)^T ; (K dh')^T ; (P^T dO)^T              -> U = U~ - W h ; dU = scale P^T dO + Diag(e) K dh'
//   phase 2  dO U^T ; T^T dU ; under the readout U dh'^T   -> dPD = scale tril(dO U^T) . D ; dXv ; dv ; dw
//   phase 3  dXv U^T ; under the readout [dO; dXv] h^T ; dPD^T Q   -> G = -stril(dXv U^T) . D ; Diag(b) G
//   phase 4  [dPD; G] K ; += (Diag(b) G)^T K               -> dq ; dk ; db ; dgamma -> dg
// (P = tril(Q K^T . D) comes from tc_prep, which forms it anyway.)  With carries in low-rank form phase 1 is not there: U and dU come from the
// carries (FACTORS), and sum_j r_j is made of U dh'^T in the last readout.
// The vector-Jacobian product of the triangular solve (K#2) is taken in a shorter form than its definition
// dW = -dU h^T, dXk = T^T dW, dXv = T^T dU, dA = -stril(dXk W^T + dXv U~^T):  T^T dW = -(T^T dU) h^T, so dXk = -dXv h^T,
// and with it dXk W^T + dXv U~^T = dXv (U~ - W h)^T = dXv U^T.  dW is never formed, dXv follows dU directly (beside dP,
// not after dW), and the sandwich is one product: a phase, a readout and twelve MMA instructions fewer per chunk-head.
// The decay gradient uses the identities  rowsum(dP.P) + scale Gam <q, dO h^T> = <q, dq>  and its analogues for
// k:  dgamma_i = <q_i, dq_i> + <k_i, dk_i^row> - <k_i, dk_i^col>, where dk^row = Diag(b)(G K + Diag(Gam) dXk)
// collects the terms in which k_i enters with exp(+gamma_i) and dk^col those with exp(-gamma_i); the last row
// of the chunk adds sum_j r_j + Gam_e <dh', h> (r_j = <(Kb dh')_j, U_j>).
//
// What bounds it: the chain of phases (issue and completion of the products, readout, barrier) and, within a readout, the
// instruction issue; HBM needs 10 k of the cycles.  The forms of the products follow from that:
// * Phase 1 is transposed (features on TMEM lanes) because its results feed later products.
// * The two pairs of products with a common second operand, dO h^T with dXv h^T and dPD K with G K, are stacked along M: one
//   instruction of M = 128 costs what one of M = 64 does (66 cycles at N = 128), and the last readout finds a
//   token of dq on each of lanes 0..63 and one of dk on each of lanes 64..127, where 64-row accumulators would leave half of
//   the lanes of every warp idle.  The two products of dk^col are issued with M = 128 as well, their A operand shifted by one
//   64-column block so that the 64 rows that count land on lanes 64..127, beside the other half of dk (the rows on lanes
//   0..63 are made from whatever lies there and are never read).
// * T^T dU is issued as two 64-column halves, one on lanes 0..15 and one on lanes 16..31 of each quadrant.
// Measured on 4 x 16 heads of 2048 tokens (2048 chunk-heads): 105 us with FACTORS, 116 us (14.7 k cycles per chunk-head) with phase 1; with separate M = 64
// products, gate gradients finished by two of the readout warps and dq assembled in a readout of its own it was 144 us.
// 8 packed sequences, 32768 tokens, 32 heads: 971 -> 763 us.
// ------------------------------------------------------------------------------------------------
namespace intra {
constexpr uint32_t OX = 0;                 // rows 0..63 dO, rows 64..127 dXv  x 128            32 KB
constexpr uint32_t QT = OX + 32768;        // Q  [64][128]                                      16 KB
constexpr uint32_t KT = QT + 16384;        // K  [64][128]                                      16 KB
constexpr uint32_t VT = KT + 16384;        // V  [64][128], later staged dv                     16 KB
constexpr uint32_t PG = VT + 16384;        // dPD [64][64]                                       8 KB  (these two: the stacked
constexpr uint32_t TT = PG + 8192;         // T [64][64], later G                                8 KB   operand [dPD; G])
constexpr uint32_t PT = TT + 8192;         // P [64][64], later Diag(b) G                        8 KB
constexpr uint32_t HH = PT + 8192;         // h [128][128]                                      32 KB
constexpr uint32_t DH = HH + 32768;        // dh' [128][128]                                    32 KB
constexpr uint32_t UTT = DH + 32768;       // U~^T [128][64]                                    16 KB
constexpr uint32_t UT = UTT + 16384;       // U^T [128][64], later staged dk                    16 KB
constexpr uint32_t DUT = UT + 16384;       // dU^T [128][64], later staged dq                   16 KB
constexpr uint32_t SMEM_BYTES = DUT + 16384 + 1024;
// W^T lies where dXv will be written (rows 64..127 of the two column blocks of OX: two pieces of 64 rows)
constexpr uint32_t W0 = OX + 8192, W1 = OX + 16384 + 8192;
constexpr uint32_t BGT = PT;
// Staging of dq, dv (in place: a thread overwrites exactly the piece it has just read) and dk: over tiles that no later
// product reads.
constexpr uint32_t STG_Q = DUT, STG_V = VT, STG_K = UT;
static_assert(SMEM_BYTES + 8192 <= 227 * 1024, "shared memory budget");
static_assert(TT == PG + 8192, "[dPD; G] is one operand tile");
// TMEM columns (512 allocated).  The four accumulators of the last readout fill all of them; what earlier phases read out
// lies where their products have not started yet.
constexpr uint32_t C_UH = 0, C_A1 = 128, C_A2 = 256, C_C2 = 384;    // U dh'^T | [dO; dXv] h^T | [dPD; G] K | rest of dk^col
constexpr uint32_t C_WH = 128, C_KD = 192, C_PD = 256;              // phase 1
constexpr uint32_t C_DP = 320, C_DX = 384;                          // phase 2
constexpr uint32_t C_DA = 256;                                      // phase 3
constexpr int kGateWarp = 18;                       // the warp of the gate arrays and gradients
constexpr int kThreadsAll = kIntraThreads + 64;     // 16 readout warps, issuer, loader, gates
constexpr int kBarThreads = kIntraThreads + 32;     // ... all but the loader meet at the named barrier
}  // namespace intra

template <int DV, bool FACTORS>   // FACTORS: the carries have left U and dU (low-rank form)
__global__ void __launch_bounds__(intra::kThreadsAll, 1) tc_intra_kernel(const __grid_constant__ TcParams P) {
    wait_prerequisites();
    using namespace intra;
    const Problem& p = P.p;
    // Persistent: a CTA walks over chunk-heads blockIdx.x, blockIdx.x + gridDim.x, ...  While it works on one, the
    // tiles of its next one are loaded into the regions the current one has finished with.
    const int H = p.d.H;
    if (reinterpret_cast<const WsHeader*>(p.ws)->status != GDN_OK) return;   // an earlier stage gave up: nothing is written
    const int n_items = n_chunks_of(p) * H;
    if ((int)blockIdx.x >= n_items) return;
    const float sc = p.d.scale;

    extern __shared__ unsigned char smem_raw[];
    unsigned char* sm = align1024(smem_raw);
    __shared__ __align__(16) float gate_sets[2][5][kC];   // two sets: a trip's gate arrays are written during the trip before
    __shared__ float red[4][kGroups][kC];       // four token-wise partial sums: [which][column group][token]
    __shared__ float scal[2][kWideThreads / 32];
    __shared__ uint64_t bar_a, bar_u, bar_b, bar_ld0, bar_e0, bar_e1, bar_e2, bar_e3, bar_st1, bar_st2, bar_v, bar_kq, bar_free, bar_mma;
    __shared__ uint32_t tmem_slot;
    // where dq and dk are staged: over dU^T and U^T, or, when the next trip's are loaded over these as early as they can be, over the place of U~^T
    // (not used then) and dXv (rows 64..127 of its tile)
    constexpr uint32_t SQ = FACTORS ? UTT : STG_Q, SK = FACTORS ? OX : STG_K;
    constexpr int SK_ROWS = FACTORS ? 128 : 64, SK_ROW0 = FACTORS ? 64 : 0;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int q4 = warp & 3, grp = warp >> 2;
    const uint32_t lane_base = (uint32_t)(q4 * 32) << 16;
    // Warps 0..15 read accumulators; the first lane of warp 16 only feeds the tensor pipe.  Because the issuer has no
    // readout duties, a phase can commit the products the next readout needs first and keep issuing the ones that
    // are only needed later while the readout already runs.
    const bool worker = warp < 16;
    const bool issuer = threadIdx.x == kWideThreads;
    // Warp 17 only moves data.  Its first lane issues every bulk / TMA instruction of the steady state (each costs its
    // issuer hundreds of cycles): the stores of the staged gradients, and the loads of the NEXT trip's tiles, each as
    // soon as the region it goes to has been read for the last time in this trip.  It shares no block-wide barrier
    // with the other warps inside the loop (they use a named barrier); it follows them through mbarriers.
    const bool loader = warp == 17;
    // Warp 18 makes the next trip's gate arrays and finishes the previous trip's gate gradients beside the readouts.
    const bool gates = warp == kGateWarp;

    if (threadIdx.x == 0) {
        mbar_init(&bar_a, 1); mbar_init(&bar_u, 1); mbar_init(&bar_b, 1);
        mbar_init(&bar_ld0, 1); mbar_init(&bar_e0, 1); mbar_init(&bar_e1, 1); mbar_init(&bar_e2, 1); mbar_init(&bar_e3, 1);
        mbar_init(&bar_st1, 1); mbar_init(&bar_st2, 1); mbar_init(&bar_v, 1); mbar_init(&bar_kq, 16); mbar_init(&bar_free, 1);
        mbar_init(&bar_mma, 1);
        fence_mbar_init();
    }
    if (warp == 0) { tmem_alloc(&tmem_slot, 512); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    bool ok = true;

    // The tiles of a trip arrive in three groups, one mbarrier each, loaded during the previous trip as their regions fall free:
    // (with FACTORS: u is dU^T (once T^T dU is done, e1), U^T (with h and dO, e2) and T; K comes with b; no U~^T, W^T, P)
    //   u  U~^T             once the first readout is done (e0)
    //   a  dh'              once U dh'^T is done (e1)
    //      h, dO, W^T       once [dO; dXv] h^T is done (e2)
    //      P, K             once the products of phase 4 are done (e3); K also read by the last readout
    //   b  V                once the staged dv has left (needed by the second readout)
    //      T, Q             once the products of phase 4 are done; Q also read by the last readout
    constexpr uint32_t STATE_BYTES = 256 * DV, VALUE_BYTES = 128 * DV;   // h or dh'; dO, V or U~ (d_v = 64: the first half of the tiles, the rest is never looked at)
    constexpr uint32_t A_BYTES = 2 * STATE_BYTES + VALUE_BYTES + (FACTORS ? 0 : 16384 + 16384 + 8192), B_BYTES = 16384 + VALUE_BYTES + (FACTORS ? 16384 : 8192),
                       U_BYTES = FACTORS ? 2 * VALUE_BYTES + 8192 : VALUE_BYTES;
    auto load_piece = [&](int piece, const ChunkInfo& c) {
        const int cb = piece & 1;
        switch (piece) {
            case 0: case 1: tma_load_3d(sm + KT + cb * 8192, &P.tm_k, cb * 64, c.hd, c.tok0, FACTORS ? &bar_b : &bar_a); break;
            case 2: case 3: if (cb * 64 < DV) tma_load_3d(sm + OX + cb * 16384, &P.tm_do, cb * 64, c.hd, c.tok0, &bar_a); break;
            case 4: bulk_load(sm + DH, p.ws + p.L.dhn + (size_t)c.ch * 32768, STATE_BYTES, &bar_a); break;
            case 5: bulk_load(sm + HH, p.ws + p.L.hc + (size_t)c.ch * 32768, STATE_BYTES, &bar_a); break;
            case 6: if (!FACTORS) bulk_load(sm + W0, p.ws + p.L.W + (size_t)c.ch * 16384, 8192, &bar_a); break;
            case 7: if (!FACTORS) bulk_load(sm + W1, p.ws + p.L.W + (size_t)c.ch * 16384 + 8192, 8192, &bar_a); break;
            case 8: if (!FACTORS) bulk_load(sm + PT, p.ws + p.L.Pm + (size_t)c.ch * 8192, 8192, &bar_a); break;
            case 9: bulk_load(sm + (FACTORS ? UT : UTT), p.ws + p.L.Ut + (size_t)c.ch * 16384, VALUE_BYTES, &bar_u); break;
            case 10: case 11: tma_load_3d(sm + QT + cb * 8192, &P.tm_q, cb * 64, c.hd, c.tok0, &bar_b); break;
            case 12: case 13: if (cb * 64 < DV) tma_load_3d(sm + VT + cb * 8192, &P.tm_v, cb * 64, c.hd, c.tok0, &bar_b); break;
            case 15: if (FACTORS) bulk_load(sm + DUT, p.ws + p.L.E + (size_t)c.ch * 16384, VALUE_BYTES, &bar_u); break;
            case 14: bulk_load(sm + TT, p.ws + p.L.Tm + (size_t)c.ch * 8192, 8192, FACTORS ? &bar_u : &bar_b); break;
            default: break;
        }
    };

    if (loader) {
        if (lane == 0) {
            uint32_t ph = 0;
            bool lok = true, pend_a = false, pend_b = false, pend_u = false;
#pragma unroll 1
            for (int item = blockIdx.x; item < n_items && lok; item += gridDim.x, ph ^= 1) {
                ChunkInfo x, nx;
                chunk_entry(p, x, item);
                const bool has_next = item + (int)gridDim.x < n_items;
                if (has_next) chunk_entry(p, nx, item + gridDim.x);
                const bool full = x.len == kC;
                pend_a = pend_b = pend_u = false;
                // (Early loads not in a CTA's first trip: there every CTA of the grid reaches these points at the same moment,
                // the loads come as one burst of 25 MB, and the instruction fetches of the last phases, which run for the
                // first time, queue behind it for microseconds.  The first trip loads at its end instead.)
                const bool early = has_next && item != (int)blockIdx.x;
                if (!(lok = mbar_wait(&bar_ld0, ph))) break;   // the trip is under way: the late loads of the next one -> L2
                if (early) {
                    for (int cb = 0; cb < 2; ++cb) prefetch_l2_tma_3d(&P.tm_k, cb * 64, nx.hd, nx.tok0);
                    if (!FACTORS) prefetch_l2_bulk(p.ws + p.L.Pm + (size_t)nx.ch * 8192, 8192);
                    prefetch_l2_bulk(p.ws + p.L.Tm + (size_t)nx.ch * 8192, 8192);
                    for (int cb = 0; cb * 64 < DV; ++cb) prefetch_l2_tma_3d(&P.tm_do, cb * 64, nx.hd, nx.tok0);
                }
                if (!FACTORS && !(lok = mbar_wait(&bar_e0, ph))) break;    // U~^T has been read by the first readout
                if (early && !FACTORS) { mbar_expect_tx(&bar_u, U_BYTES); pend_u = true; load_piece(9, nx); }
                if (!(lok = mbar_wait(&bar_e1, ph))) break;    // dh'
                if (early) { mbar_expect_tx(&bar_a, A_BYTES); pend_a = true; load_piece(4, nx); }   // (the first piece announces the group)
                if (early && FACTORS) { mbar_expect_tx(&bar_u, U_BYTES); pend_u = true; load_piece(15, nx); }   // dU
                if (!(lok = mbar_wait(&bar_st1, ph))) break;   // dv is staged
                if (full) {
                    for (int cb = 0; cb * 64 < DV; ++cb) tma_store_3d(&P.tm_dv, cb * 64, x.hd, x.tok0, sm + STG_V + cb * 8192);
                    bulk_commit();
                }
                if (!(lok = mbar_wait(&bar_e2, ph))) break;    // dO, h and dXv (over W^T)
                if (early) {
                    if (FACTORS) load_piece(9, nx);
                    load_piece(5, nx);
                    load_piece(6, nx);
                    load_piece(7, nx);
                    load_piece(2, nx);
                    load_piece(3, nx);
                }
                if (!(lok = mbar_wait(&bar_v, ph))) break;     // (a ragged tail's dv has been flushed)
                bulk_wait_read<0>();
                if (early) {
                    mbar_expect_tx(&bar_b, B_BYTES);
                    pend_b = true;
                    load_piece(12, nx);
                    load_piece(13, nx);
                }
                if (!(lok = mbar_wait(&bar_e3, ph))) break;    // the products of phase 4 are done: Diag(b) G (over P), G (over T)
                if (early) { load_piece(FACTORS ? 14 : 8, nx); }
                if (!(lok = mbar_wait(&bar_kq, ph))) break;    // ... and the readout holds its rows of K and Q
                if (early) {
                    load_piece(0, nx);
                    load_piece(1, nx);
                    if (!FACTORS) load_piece(14, nx);
                    load_piece(10, nx);
                    load_piece(11, nx);
                }
                if (!(lok = mbar_wait(&bar_st2, ph))) break;   // dq, dk are staged
                if (full) {
                    for (int cb = 0; cb * 64 < p.d.d_k; ++cb) {
                        tma_store_3d(&P.tm_dq, cb * 64, x.hd, x.tok0, sm + SQ + cb * 8192);
                        tma_store_3d(&P.tm_dk, cb * 64, x.hd, x.tok0, sm + SK + SK_ROW0 * 128 + cb * SK_ROWS * 128);
                    }
                    bulk_commit();
                }
                if (has_next && !early) {
                    mbar_expect_tx(&bar_a, A_BYTES);
                    mbar_expect_tx(&bar_b, B_BYTES);
                    mbar_expect_tx(&bar_u, U_BYTES);
                    pend_a = pend_b = pend_u = true;
#pragma unroll 1
                    for (int piece = 0; piece <= 15; ++piece) load_piece(piece, nx);
                }
                bulk_wait_read<0>();
                mbar_arrive(&bar_free);   // the staging regions may be rewritten
            }
            bulk_wait_read<0>();
            if (!lok) {   // after a timeout a copy may still be in flight, of this trip or of the next one: wait for it before the CTA may retire
                (void)mbar_wait(&bar_a, pend_a ? ph ^ 1 : ph);
                (void)mbar_wait(&bar_b, pend_b ? ph ^ 1 : ph);
                (void)mbar_wait(&bar_u, pend_u ? ph ^ 1 : ph);
            }
        }
        return;
    }

    auto cta_sync = [] { asm volatile("bar.sync 1, %0;" ::"n"(kBarThreads) : "memory"); };   // all warps but the loader
    uint32_t mma_phase = 0, in_phase = 0;
    ChunkInfo xn;
    chunk_entry(p, xn, blockIdx.x);
    // The gate warp: lane l owns tokens l and l + 32.  Values are fetched one phase before they are turned into arrays.
    float ng[2] = {0.f, 0.f}, nb[2] = {0.f, 0.f}, ngend = 0.f, bb_prev[2] = {0.f, 0.f}, Gam_last_prev = 0.f;
    auto fetch_gates = [&](const ChunkInfo& c) {   // cumulative log decays and the one of the chunk end, erase gates
        const float* gsrc = reinterpret_cast<const float*>(p.ws + p.L.gamma) + (size_t)c.ch * kC;
        ngend = gsrc[kC - 1];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = lane + 32 * h;
            ng[h] = gsrc[i];
            nb[h] = (i < c.len && p.d.delta_rule) ? p.beta[(size_t)(c.tok0 + i) * H + c.hd] : 0.f;
        }
    };
    auto make_gates = [&](int set) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = lane + 32 * h;
            gate_sets[set][0][i] = ng[h] * kLog2e;
            gate_sets[set][1][i] = expf(ng[h]);
            gate_sets[set][2][i] = expf(ngend - ng[h]);
            gate_sets[set][3][i] = nb[h];                                                 // erase gate
            gate_sets[set][4][i] = p.d.delta_rule ? nb[h] : (i < xn.len ? 1.f : 0.f);     // write gate (delta rule off: 0 and 1)
        }
    };
    // dbeta and dg of the previous trip's chunk, from its token-wise partial sums
    ChunkInfo xp = xn;
    bool have_prev = false;
    auto finish_gates = [&]() {
        float v[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = lane + 32 * h;
            auto tot = [&](int w) { return (red[w][0][i] + red[w][1][i]) + (red[w][2][i] + red[w][3][i]); };
            const float qdq = tot(0), dw = tot(1), db = tot(2), kcol = tot(3);
            if (i < xp.len && p.dbeta) p.dbeta[(size_t)(xp.tok0 + i) * H + xp.hd] = db + dw;
            v[h] = fmaf(bb_prev[h], db, qdq - kcol);
        }
        constexpr int nw = kWideThreads / 32;   // per-warp partial sums, one per lane
        const float rsum = warp_sum(lane < nw ? scal[0][lane] : 0.f), hsum = warp_sum(lane < nw ? scal[1][lane] : 0.f);
        // dg_j = sum_{i >= j} dgam_i inside the chunk
        float a = v[0], b = v[1] + (lane == 31 ? rsum + Gam_last_prev * hsum : 0.f);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const float ta = __shfl_down_sync(0xffffffffu, a, o), tb = __shfl_down_sync(0xffffffffu, b, o);
            if (lane + o < 32) { a += ta; b += tb; }
        }
        a += __shfl_sync(0xffffffffu, b, 0);
        float* dg = p.dg + (size_t)xp.tok0 * H + xp.hd;
        if (lane < xp.len) dg[(size_t)lane * H] = a;
        if (lane + 32 < xp.len) dg[(size_t)(lane + 32) * H] = b;
    };
    // first trip: every group is loaded at once, one instruction per warp
    if (issuer) { mbar_expect_tx(&bar_a, A_BYTES); mbar_expect_tx(&bar_b, B_BYTES); mbar_expect_tx(&bar_u, U_BYTES); }
    if (lane == 0 && warp < 16 && !(P.withhold == WITHHOLD_GRADIENT && warp == 9)) load_piece(warp, xn);
    if (gates) { fetch_gates(xn); make_gates(0); }
    unsigned char* const sm_base = sm;
#pragma unroll 1
    for (int item = blockIdx.x; item < n_items; item += gridDim.x, in_phase ^= 1) {
    unsigned char* sm = sm_base;
    if (FACTORS) asm volatile("" : "+l"(sm));   // (addresses of tiles are made where they are used: kept over the trip they cost spills)
    const ChunkInfo x = xn;
    // this trip's gate arrays (the barrier before phase 1 publishes them)
    const float* gl = gate_sets[in_phase][0];
    const float* Gam = gate_sets[in_phase][1];
    const float* ee = gate_sets[in_phase][2];
    const float* bb = gate_sets[in_phase][3];
    const bool has_next = item + (int)gridDim.x < n_items;
    const bool first = item == (int)blockIdx.x, full = x.len == kC;
    if (has_next) chunk_entry(p, xn, item + gridDim.x);

    const int i0 = grp * kTG;          // first of this thread's 16 tokens (or columns of a 64-column accumulator)
    float rs = 0.f;
    if (FACTORS && gates && have_prev && ok) finish_gates();   // the previous chunk's gate gradients (what they are made of is rewritten below)
    if (ok) {
        ok = mbar_wait(&bar_a, in_phase) && !(FACTORS && P.withhold == DISAGREE_GRADIENT && (warp & 1));
        if (!FACTORS && P.withhold == DISAGREE_GRADIENT && (warp & 1)) ok = false;
        if (!ok && lane == 0) report_timeout(p.ws, 20);
    }
    if (FACTORS && ok) {
        ok = mbar_wait(&bar_u, in_phase);
        if (!ok && lane == 0) report_timeout(p.ws, 27);
    }
    if (FACTORS && ok && !first) {   // dXv goes where the previous trip's dk is staged, dq over its dq: the stores must have read them
        ok = mbar_wait(&bar_free, in_phase ^ 1);
        if (!ok && lane == 0) report_timeout(p.ws, 28);
    }
    if (ok && !full) {
        if (!FACTORS) zero_tail_rows(sm + KT, 64, 0, x.len, kWideThreads);
        zero_tail_rows(sm + OX, 128, 0, x.len, kWideThreads);
        fence_async_smem();
    }
    if constexpr (!FACTORS) {
    cta_sync();

    // ---- phase 1: (W h)^T, (K dh')^T, (P^T dO)^T
    if (ok && issuer) {
        tc_fence_after();
        Operand w = op_mn_major(sm + W0, 64);   // W^T in two pieces of 64 rows
        w.jump = (W1 - W0 - 8192) / 16;
        mma_tile<128, 64, 128>(tmem + C_WH, op_mn_major(sm + HH, 128), w, false);
        mma_tile<128, 64, 128>(tmem + C_KD, op_mn_major(sm + DH, 128), op_k_major(sm + KT, 64), false);
        mma_tile<128, 64, 64>(tmem + C_PD, op_mn_major(sm + OX, 128), op_mn_major(sm + PT, 64), false);
        mma_commit(&bar_mma);
    }
    if (threadIdx.x == 32) mbar_arrive(&bar_ld0);
    if (gates && have_prev && ok) finish_gates();   // the previous chunk's gate gradients
    if (ok) {
        ok = mbar_wait(&bar_u, in_phase);
        if (!ok && lane == 0) report_timeout(p.ws, 27);
    }
    GDN_WAIT_MMA(22)
    if (ok && !first) {   // U^T and dU^T held the previous trip's staged dk and dq: their stores must have read them
        ok = mbar_wait(&bar_free, in_phase ^ 1);
        if (!ok && lane == 0) report_timeout(p.ws, 28);
    }
    if (ok && worker && (DV == 128 || q4 < 2)) {
        const int f = q4 * 32 + lane;      // feature (lane of the transposed accumulators)
        float t2[2][8], kb2[2][8], pd2[2][8];
#pragma unroll
        for (int part = 0; part < 2; ++part) {
            tmem_ld8(tmem + lane_base + C_WH + i0 + part * 8, t2[part]);
            tmem_ld8(tmem + lane_base + C_KD + i0 + part * 8, kb2[part]);
            tmem_ld8(tmem + lane_base + C_PD + i0 + part * 8, pd2[part]);
        }
        tmem_wait_ld();
#pragma unroll
        for (int part = 0; part < 2; ++part) {
            const int ib = i0 + part * 8;
            float u[8], e8[8];
            float (&t)[8] = t2[part], (&kb)[8] = kb2[part], (&pd)[8] = pd2[part];
            chunk_load(sm + UTT, 128, f, ib >> 3, u);
            ld8s(ee + ib, e8);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                u[i] -= t[i];                                       // U = U~ - W h
                const float kbe = e8[i] * kb[i];
                rs = fmaf(kbe, u[i], rs);                           // sum_j r_j
                pd[i] = fmaf(sc, pd[i], kbe);                       // dU = scale P^T dO + Diag(e) K dh'
            }
            chunk_store(sm + UT, 128, f, ib >> 3, u);
            chunk_store(sm + DUT, 128, f, ib >> 3, pd);
        }
    }
    if (ok) {   // T and V are needed from phase 2 on, Q from phase 3 on
        ok = mbar_wait(&bar_b, in_phase);
        if (!ok && lane == 0) report_timeout(p.ws, 31);
    }
    if (ok && !full) zero_tail_rows(sm + QT, 64, 0, x.len, kWideThreads);
    tc_fence_before();
    fence_async_smem();
    cta_sync();
    if (threadIdx.x == 32 && ok) mbar_arrive(&bar_e0);   // U~^T has been read (a load is announced behind one that has arrived only)
    }
    else { cta_sync(); }

    // Token-major accumulators with 64 rows (M = 64) occupy lanes 0..15 of each quadrant, or lanes 16..31 (address + 16 lanes).
    constexpr uint32_t LB = 16u << 16;
    const bool ga = lane < 16;
    const int tr = q4 * 16 + (lane & 15);   // token row of this lane there

    // ---- phase 2: dO U^T and dXv = T^T dU (features 0..63 on lanes 0..15, 64..127 on lanes 16..31)
    if (ok && issuer) {
        tc_fence_after();
        mma_tile<64, 64, DV>(tmem + C_DP, op_k_major(sm + OX, 128), op_mn_major(sm + UT, 128), false);
        mma_tile<64, 64, 64>(tmem + C_DX, op_mn_major(sm + TT, 64), op_k_major(sm + DUT, 128, 0), false);
        if (DV == 128) mma_tile<64, 64, 64>(tmem + C_DX + LB, op_mn_major(sm + TT, 64), op_k_major(sm + DUT, 128, 64), false);
        mma_commit(&bar_mma);
        // U dh'^T, rows on lanes 64..127, is first read after phase 4: it runs under the readout
        mma_tile<128, 128, DV>(tmem + C_UH, op_mn_major(sm + UT - 16384, 128), op_k_major(sm + DH, 128), false);
    }
    // <dh', h> over the whole state, while the products run (both tiles share one format, so offsets pair up)
    float hh = 0.f;
    if (worker) {
#pragma unroll
        for (int t = 0; t < DV / 32; ++t) {
            float a[8], b[8];
            unpack8(*reinterpret_cast<const uint4*>(sm + HH + (threadIdx.x + t * kWideThreads) * 16), a);
            unpack8(*reinterpret_cast<const uint4*>(sm + DH + (threadIdx.x + t * kWideThreads) * 16), b);
#pragma unroll
            for (int k = 0; k < 8; ++k) hh = fmaf(a[k], b[k], hh);
        }
        if (FACTORS) {   // (the gate warp has read the previous trip's)
            hh = warp_sum(hh);
            if (lane == 0) scal[1][warp] = hh;
        }
    }
    if (FACTORS && threadIdx.x == 32) mbar_arrive(&bar_ld0);
    if (gates && has_next) fetch_gates(xn);
    if (FACTORS && ok) {   // V is needed now, Q from phase 3 on, K from phase 4 on
        ok = mbar_wait(&bar_b, in_phase);
        if (!ok && lane == 0) report_timeout(p.ws, 31);
        if (ok && !full) {
            zero_tail_rows(sm + QT, 64, 0, x.len, kWideThreads);
            zero_tail_rows(sm + KT, 64, 0, x.len, kWideThreads);
        }
    }
    GDN_WAIT_MMA(23)
    if (ok && worker) {
        float v2[2][8];
        tmem_ld8(tmem + lane_base + C_DP + i0, v2[0]);
        tmem_ld8(tmem + lane_base + C_DP + i0 + 8, v2[1]);
        tmem_wait_ld();
        if (ga) {   // dPD = scale tril(dO U^T) . D
#pragma unroll
            for (int part = 0; part < 2; ++part) {
                const int jb = i0 + part * 8;
                float (&v)[8] = v2[part];
                float g8[8];
                ld8s(gl + jb, g8);
#pragma unroll
                for (int j = 0; j < 8; ++j) v[j] = (jb + j <= tr) ? sc * v[j] * ex2(gl[tr] - g8[j]) : 0.f;
                chunk_store(sm + PG, 128, tr, jb >> 3, v);
            }
        }
        // dXv -> operand tile beside dO (over W^T) ; <v, dXv> (dw partial) ; dv = w dXv, staged over V
        tmem_ld8(tmem + lane_base + C_DX + i0, v2[0]);
        tmem_ld8(tmem + lane_base + C_DX + i0 + 8, v2[1]);
        tmem_wait_ld();
        float acc = 0.f;
        const float wg = gate_sets[in_phase][4][tr];
#pragma unroll
        for (int part = 0; part < 2; ++part) {
            if (DV == 64 && !ga) break;
            const int chk = (ga ? 0 : 8) + (i0 >> 3) + part;   // 8-feature piece
            float (&b)[8] = v2[part];
            float t8[8];
            chunk_load(sm + VT, 64, tr, chk, t8);
            chunk_store(sm + OX, 128, 64 + tr, chk, b);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                acc = fmaf(t8[j], b[j], acc);
                b[j] *= wg;
            }
            chunk_store(sm + STG_V, 64, tr, chk, b);
        }
        if (DV == 128) acc += __shfl_xor_sync(0xffffffffu, acc, 16);
        if (ga) red[1][grp][tr] = acc;
    }
    tc_fence_before();
    fence_async_smem();
    cta_sync();
    if (threadIdx.x == 32) mbar_arrive(&bar_st1);   // dv is staged: the loader stores it (async proxy)
    if (ok && !full) flush_rows(sm + STG_V, p.dv, x, H, p.d.d_v, kWideThreads);   // rows beyond the sequence must not be written

    // ---- phase 3: dA = -stril(dXv U^T) ; under its readout [dO; dXv] h^T and dPD^T Q (rows on lanes 64..127)
    if (ok && issuer) {
        tc_fence_after();
        mma_commit(&bar_e1);   // U dh'^T is done: dh' has been read for the last time
        mma_tile<64, 64, DV>(tmem + C_DA, op_k_major(sm + OX, 128, 64), op_mn_major(sm + UT, 128), false);
        mma_commit(&bar_mma);
        mma_tile<128, 128, DV>(tmem + C_A1, op_k_major(sm + OX, 128), op_k_major(sm + HH, 128), false);
        mma_commit(&bar_e2);   // dO, dXv and h have been read for the last time
        mma_tile<128, 128, 64>(tmem + C_C2, op_mn_major(sm + PG - 8192, 64), op_mn_major(sm + QT, 64), false);
    }
    if (gates && has_next) make_gates(in_phase ^ 1);   // the next trip's gate arrays
    GDN_WAIT_MMA(24)
    if (ok && worker) {   // G = dA . D and Diag(b) G (over T and P, which no product reads any more)
        float v2[2][8];
        tmem_ld8(tmem + lane_base + C_DA + i0, v2[0]);
        tmem_ld8(tmem + lane_base + C_DA + i0 + 8, v2[1]);
        tmem_wait_ld();
        if (ga) {
#pragma unroll
            for (int part = 0; part < 2; ++part) {
                float (&v)[8] = v2[part];
                float w[8], g8[8];
                const int jb = i0 + part * 8;
                ld8s(gl + jb, g8);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    v[j] = (jb + j < tr) ? -v[j] * ex2(gl[tr] - g8[j]) : 0.f;
                    w[j] = bb[tr] * v[j];
                }
                chunk_store(sm + PG, 128, 64 + tr, jb >> 3, v);
                chunk_store(sm + BGT, 64, tr, jb >> 3, w);
            }
        }
    }
    tc_fence_before();
    fence_async_smem();
    cta_sync();
    if (threadIdx.x == 32) mbar_arrive(&bar_v);     // the flush of a ragged dv is done

    // ---- phase 4: [dPD; G] K ; += (Diag(b) G)^T K
    if (ok && issuer) {
        tc_fence_after();
        mma_tile<128, 128, 64>(tmem + C_A2, op_k_major(sm + PG, 128), op_mn_major(sm + KT, 64), false);
        mma_tile<128, 128, 64>(tmem + C_C2, op_mn_major(sm + BGT - 8192, 64), op_mn_major(sm + KT, 64), true);
        mma_commit(&bar_mma);
        mma_commit(&bar_e3);   // every product of this trip is done
    }
    GDN_WAIT_MMA(26)
    if (worker) {
        // Warps of quadrants 0, 1 (lanes 0..63) assemble dq = scale Gam (dO h^T) + dPD K, those of quadrants 2, 3
        // dk = Diag(b)(G K - Gam dXv h^T) + e U dh'^T + dPD^T Q + (Diag(b) G)^T K, and the row dots.
        const bool is_k = q4 >= 2;
        const int i = (q4 & 1) * 32 + lane, c0 = grp * 32;
        uint4 raw[4];   // this thread's part of its row of K or Q leaves shared memory now: the next trip's is loaded over it
#pragma unroll
        for (int part = 0; part < 4; ++part)
            raw[part] = *reinterpret_cast<const uint4*>(sm + (is_k ? KT : QT) + tile_chunk_off(64, i, (c0 >> 3) + part));
        __syncwarp();
        if (lane == 0) mbar_arrive(&bar_kq);
        const float G = Gam[i];
        if (ok && !is_k) {
            float acc = 0.f;
            const float coef = sc * G;
#pragma unroll
            for (int part = 0; part < 4; ++part) {
                const int cb = c0 + part * 8;
                float a[8], b[8], t8[8];
                tmem_ld8(tmem + lane_base + C_A1 + cb, a);     // dO h^T
                tmem_ld8(tmem + lane_base + C_A2 + cb, b);     // dPD K
                tmem_wait_ld();
                unpack8(raw[part], t8);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    b[j] = fmaf(coef, a[j], b[j]);
                    acc = fmaf(t8[j], b[j], acc);
                }
                chunk_store(sm + SQ, 64, i, cb >> 3, b);
            }
            red[0][grp][i] = acc;     // <q, dq>
        } else if (ok) {
            float acc_c = 0.f, acc_r = 0.f, acc_db = 0.f;   // <k, dk^col> in its two parts ; db = <k, G K + Gam dXk>
            const float e6 = ee[i], b6 = bb[i];
#pragma unroll
            for (int part = 0; part < 4; ++part) {
                const int cb = c0 + part * 8;
                float a[8], b[8], c8[8], d8[8], kk[8];
                tmem_ld8(tmem + lane_base + C_A2 + cb, a);     // G K
                tmem_ld8(tmem + lane_base + C_A1 + cb, b);     // dXv h^T = -dXk
                tmem_ld8(tmem + lane_base + C_C2 + cb, c8);    // dPD^T Q + (bG)^T K
                tmem_ld8(tmem + lane_base + C_UH + cb, d8);    // U dh'^T
                tmem_wait_ld();
                unpack8(raw[part], kk);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float kcol = fmaf(e6, d8[j], c8[j]);       // dk^col
                    const float t = fmaf(-G, b[j], a[j]);            // G K + Gam dXk
                    acc_c = fmaf(kk[j], kcol, acc_c);
                    if (FACTORS) acc_r = fmaf(kk[j], d8[j], acc_r);
                    acc_db = fmaf(kk[j], t, acc_db);
                    a[j] = fmaf(b6, t, kcol);
                }
                chunk_store(sm + SK, SK_ROWS, SK_ROW0 + i, cb >> 3, a);
            }
            red[2][grp][i] = acc_db;
            if (FACTORS) rs = e6 * acc_r;   // (its share of sum_j r_j; in the other form the first readout has made it)
            red[3][grp][i] = acc_c;
        }
        // block totals of sum_j r_j and <dh', h>
        rs = warp_sum(rs);
        if (!FACTORS) hh = warp_sum(hh);
        if (lane == 0) {
            scal[0][warp] = rs;
            if (!FACTORS) scal[1][warp] = hh;
        }
    }
    // The token-wise sums are turned into dbeta and dg by the gate warp during the next trip's first products.  It keeps what
    // the next trip overwrites: this chunk's gates and place.
    if (gates) {
        bb_prev[0] = bb[lane]; bb_prev[1] = bb[lane + 32];
        Gam_last_prev = Gam[kC - 1];
    }
    xp = x;
    have_prev = true;
    tc_fence_before();
    fence_async_smem();
    // every reader of this trip's tiles and scratch is done.  (Without FACTORS the warps leave together on the outcome of the barrier: to stand by
    // takes registers there, and spills: 16 heads of 16384 tokens 635 -> 646 us.  With FACTORS the outcome costs 0.2 %.)
    if (FACTORS) {
        cta_sync();
    } else if (!named_barrier_and<kBarThreads>(ok)) {
        if (warp == 0) tmem_dealloc(tmem, 512);
        return;   // (the loader, which gives up in turn, waits for the loads that are in flight)
    }
    if (threadIdx.x == 32) mbar_arrive(&bar_st2);   // dq, dk are staged: the loader stores them
    if (ok && !full) {
        flush_rows(sm + SQ, p.dq, x, H, p.d.d_k, kWideThreads);
        flush_rows(sm + SK, p.dk, x, H, p.d.d_k, kWideThreads, SK_ROWS, SK_ROW0);
    }
    if (FACTORS && !ok) {
        stand_by_items<4>(item, n_items, cta_sync);
        break;
    }
    }
    if (ok && have_prev && gates) finish_gates();
    if (warp == 0) tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------------------------------------------------
// tc_out (optional forward output): o = scale (Diag(Gam) Q h + P U),  P = tril(Q K^T . D),  U = U~ - W h made here or, with carries in
// low-rank form, left by the forward carry (FACTORS: one step instead of two; 6 x 16 heads of 1500 tokens 51 -> 44 us)
//
// Persistent, two CTAs per SM (89 KB of shared memory, 256 TMEM columns each): a CTA walks through the dependent
// steps of one chunk-head while its neighbour is in another step of another one.  The tiles of the next trip are
// loaded as soon as the last product (or store) that reads their region is done.  Q h and P U are formed token-major
// (M = 64: a thread owns a token row), so the output tile is staged with 16-byte stores and leaves by TMA.
// CW: the channel-wise path.  Its preparation kernels leave Q~, P = tril(Q~ K-^T), W^T, U~^T and the per-chunk
// states h~ in the workspace as tile images, the decay is inside them, so o = scale (Q~ h~ + P (U~ - W h~)): no
// gates here, and P U accumulates onto Q~ h~.
// ------------------------------------------------------------------------------------------------
namespace outk {
constexpr uint32_t QT = 0;                  // Q or Q~ [64][128]                                     16 KB
constexpr uint32_t PT = 16384;              // P [64][64]                                             8 KB
constexpr uint32_t WT = PT + 8192;          // W^T [128][64]                                         16 KB
constexpr uint32_t UTT = WT + 16384;        // U~^T [128][64]; U^T in place                         16 KB
constexpr uint32_t HH = UTT + 16384;        // h [128][128]; after the first products: staged o     32 KB
constexpr uint32_t STG = HH;
constexpr uint32_t SMEM_BYTES = HH + 32768 + 1024 /* alignment slack */;
constexpr uint32_t C_WH = 0, C_QH = 128, C_PU = 0;   // TMEM columns (256 allocated; P U over (W h)^T, which is read by then)
constexpr uint32_t IN_BYTES = 16384 + 8192 + 16384 + 16384 + 32768;
static_assert(2 * (SMEM_BYTES + 4096) <= 228 * 1024, "two CTAs per SM");
}  // namespace outk

template <bool CW, int DV, bool FACTORS>   // FACTORS: the forward carry has left U where U~ was (low-rank form)
__global__ void __launch_bounds__(kThreads, 2) tc_out_kernel(const __grid_constant__ TcParams P) {
    wait_prerequisites();
    using namespace outk;
    const Problem& p = P.p;
    const int H = p.d.H;
    const WsHeader* hdr = reinterpret_cast<const WsHeader*>(p.ws);
    if (hdr->status != GDN_OK || (CW && hdr->cw_fallback)) return;
    const int n_items = n_chunks_of(p) * H;
    if ((int)blockIdx.x >= n_items) return;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* sm = align1024(smem_raw);
    __shared__ float Gam[kC];
    __shared__ uint64_t bar_in, bar_mma;
    __shared__ uint32_t tmem_slot;
    const int warp = warp_id(), lane = threadIdx.x & 31;
    const int q4 = warp & 3, half = warp >> 2;
    const uint32_t lane_base = (uint32_t)(q4 * 32) << 16;
    if (threadIdx.x == 0) { mbar_init(&bar_in, 1); mbar_init(&bar_mma, 1); fence_mbar_init(); }
    if (warp == 0) { tmem_alloc(&tmem_slot, 256); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    bool ok = true, pending = false;
    uint32_t mma_phase = 0, in_phase = 0, pending_phase = 0;   // (pending_phase: the phase of bar_in the loads in flight belong to)
    // One mbarrier phase per trip collects all five tiles; they are issued in three pieces, each when its region is free.
    auto load_q = [&](const ChunkInfo& c, uint32_t phase) {   // thread 0; first piece of a trip: announces the whole trip's bytes
        pending_phase = phase;
        mbar_expect_tx(&bar_in, IN_BYTES - (128 - DV) * 384 - (FACTORS ? 16384 : 0));
        for (int cb = 0; cb < 2; ++cb) {
            if (CW) bulk_load(sm + QT + cb * 8192, p.ws + p.L.img_QKp + (size_t)c.ch * 32768 + cb * 16384, 8192, &bar_in);
            else tma_load_3d(sm + QT + cb * 8192, &P.tm_q, cb * 64, c.hd, c.tok0, &bar_in);
        }
        if (!FACTORS) bulk_load(sm + WT, p.ws + (CW ? p.L.img_W : p.L.W) + (size_t)c.ch * 16384, 16384, &bar_in);
        pending = true;
    };
    auto load_up = [&](const ChunkInfo& c) {
        bulk_load(sm + UTT, p.ws + (CW ? p.L.img_U : p.L.Ut) + (size_t)c.ch * 16384, 128 * DV, &bar_in);
        bulk_load(sm + PT, p.ws + p.L.Pm + (size_t)c.ch * 8192, 8192, &bar_in);
    };
    auto load_h = [&](const ChunkInfo& c) { bulk_load(sm + HH, p.ws + p.L.hc + (size_t)c.ch * 32768, 256 * DV, &bar_in); };
    auto fetch_gamma = [&](const ChunkInfo& c) {   // threads 0..63: cumulative log decay of their token
        return reinterpret_cast<const float*>(p.ws + p.L.gamma)[(size_t)c.ch * kC + threadIdx.x];
    };
    ChunkInfo x;
    chunk_entry(p, x, blockIdx.x);
    if (threadIdx.x == 0) { load_q(x, 0); load_up(x); load_h(x); }
    float gnext = (!CW && threadIdx.x < kC) ? fetch_gamma(x) : 0.f;
    const int f = q4 * 32 + lane;            // feature row of the transposed accumulator (W h)^T
    const int tr = q4 * 16 + (lane & 15);    // token row of the M = 64 accumulators (lanes 0..15 of a quadrant hold them)
    const bool ga = lane < 16;
    const float sc = p.d.scale;
#pragma unroll 1
    for (int item = blockIdx.x; item < n_items; item += gridDim.x, in_phase ^= 1) {
        const bool has_next = item + (int)gridDim.x < n_items;
        ChunkInfo xn = x;
        if (has_next) chunk_entry(p, xn, item + gridDim.x);
        if (!CW && threadIdx.x < kC) {
            Gam[threadIdx.x] = expf(gnext);
        }
        if (ok) {
            ok = mbar_wait(&bar_in, in_phase);
            if (!ok && lane == 0) report_timeout(p.ws, 30);
            if (ok && threadIdx.x == 0) pending = false;
        }
        if (!CW && ok && x.len < kC) {   // ragged tail: rows beyond the sequence belong to somebody else (the images are padded)
            zero_tail_rows(sm + QT, 64, 0, x.len);
            fence_async_smem();
        }
        __syncthreads();
        if constexpr (!FACTORS) {
        // ---- step 1: (W h)^T ; under its readout Q h
        if (warp == 0 && elect_one() && ok) {
            tc_fence_after();
            mma_tile<128, 64, 128>(tmem + C_WH, op_mn_major(sm + HH, 128), op_mn_major(sm + WT, 128), false);
            mma_commit(&bar_mma);
            mma_tile<64, DV, 128>(tmem + C_QH, op_k_major(sm + QT, 64), op_mn_major(sm + HH, 128), false);
        }
        GDN_WAIT_MMA(31)
        if (ok && (DV == 128 || q4 < 2)) {   // U = U~ - W h in place
            const int i0 = half * 32;
#pragma unroll 2
            for (int part = 0; part < 4; ++part) {
                float u[8], t[8];
                const int ib = i0 + part * 8;
                tmem_ld8(tmem + lane_base + C_WH + ib, t);
                chunk_load(sm + UTT, 128, f, ib >> 3, u);
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 8; ++i) u[i] -= t[i];
                chunk_store(sm + UTT, 128, f, ib >> 3, u);
            }
        }
        tc_fence_before();
        fence_async_smem();
        __syncthreads();
        }
        if (!CW && ok && has_next && threadIdx.x < kC) gnext = fetch_gamma(xn);
        // ---- step 2: P U (token-major)
        if (warp == 0 && elect_one() && ok) {
            tc_fence_after();
            if (FACTORS) mma_tile<64, DV, 128>(tmem + C_QH, op_k_major(sm + QT, 64), op_mn_major(sm + HH, 128), false);   // Q h
            if (CW) mma_tile<64, DV, 64>(tmem + C_QH, op_k_major(sm + PT, 64), op_k_major(sm + UTT, 128), true);
            else mma_tile<64, DV, 64>(tmem + C_PU, op_k_major(sm + PT, 64), op_k_major(sm + UTT, 128), false);
            mma_commit(&bar_mma);
        }
        GDN_WAIT_MMA(32)
        if (ok && has_next && threadIdx.x == 0) { load_q(xn, in_phase ^ 1); load_up(xn); }   // every tile has been read for the last time
        if (ok) {   // o = scale (Gam . (Q h) + P U): the sixteen low lanes of a warp own a token row and half of the columns each
            const float coef = CW ? sc : sc * Gam[tr];
#pragma unroll 1
            for (int part = 0; part < DV / 16; ++part) {
                const int cb = half * (DV / 2) + part * 8;
                float a[8], b[8];
                tmem_ld8(tmem + lane_base + C_QH + cb, a);
                if (!CW) tmem_ld8(tmem + lane_base + C_PU + cb, b);
                tmem_wait_ld();
                if (ga) {
#pragma unroll
                    for (int j = 0; j < 8; ++j) b[j] = CW ? coef * a[j] : fmaf(coef, a[j], sc * b[j]);
                    chunk_store(sm + STG, 64, tr, cb >> 3, b);
                }
            }
        }
        tc_fence_before();
        fence_async_smem();
        __syncthreads();
        if (ok) {
            if (x.len == kC) {
                if (threadIdx.x == 0) {
                    for (int cb = 0; cb * 64 < DV; ++cb) tma_store_3d(&P.tm_o, cb * 64, x.hd, x.tok0, sm + STG + cb * 8192);
                    bulk_commit();
                }
            } else {
                flush_rows(sm + STG, p.o, x, H, p.d.d_v, kThreads);
                __syncthreads();
            }
            if (threadIdx.x == 0) {
                bulk_wait_read<0>();            // the store has read the staged tile: h of the next trip may land on it
                if (has_next) load_h(xn);
            }
        }
        if (!ok) break;
        x = xn;
    }
    if (threadIdx.x == 0) {
        bulk_wait_read<0>();
        if (pending) (void)mbar_wait(&bar_in, pending_phase);   // after a timeout a load may still be in flight
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 256);
}

#undef GDN_WAIT_MMA

}  // namespace

// ------------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------------
bool tc_supported(const gdn_desc& d) {
    return d.dtype == GDN_BF16 && (d.d_k == 64 || d.d_k == 128) && (d.d_v == 64 || d.d_v == 128) && d.chunk == kC;
}

thread_local int g_inject_timeout = 0;   // set by gdn_debug_inject_timeout, consumed by the next gdn_bwd of this family

static int sm_count();
// Up to 37 chains (on 148 SMs) the operator form gives each direction of a chain two CTAs, and its one product per step wins; from
// 38 on it would have one, and the low-rank form moves less.  Backward, us, operator / low-rank: 16 chains of 8 chunks 35.6 / 42.4, 16 of
// 128 317 / 413, 32 of 32 155.4 / 158.9, 37 of 32 172.4 / 170.2; 38 of 32 197 / 177, 64 of 32 290 / 243.  One line for all numbers of chunks and
// both calls has its price: 24 to 37 chains of 8 chunks (a step 79.0 / 74.4 at 32), steps of one chunk at any number of chains (42.5 / 39.0), and
// steps of 38 to 48 chains of 128 chunks (823 / 914).  With d_v = 64 the operator form has one CTA of 64 columns per direction up to 74
// chains; there too the low-rank form is faster from 38 on (38 of 32 172.6 / 159.6, 64 of 32 255 / 217; 38 of 128 570 / 574), in short calls from 24 on.
// The rule looks at the chains only, so the forward, the backward and a backward on a workspace fresh from the forward agree on the form (and
// on the workspace layout that follows from it).  All of it: profiles/carry_forms.md
bool tc_carries_lowrank(const gdn_desc& d) {
    if (g_force_carries) return g_force_carries == 2;
    return 4 * (long long)d.N * d.H > sm_count();
}
static bool fill_params(TcParams& P, const Problem& p, bool with_bwd, int scan_dirs) {
    P.p = p;
    P.with_bwd = with_bwd ? 1 : 0;
    P.scan_dirs = scan_dirs;
    P.lowrank = tc_carries_lowrank(p.d) ? 1 : 0;
    P.narrow_v = p.d.d_v == 64 ? 1 : 0;
    P.withhold = 0;
    auto map = [&](CUtensorMap* m, const void* base, int d) { return tc::make_tmap_bf16_heads(m, base, p.Ttot, p.d.H, d); };
    if (!map(&P.tm_q, p.q, p.d.d_k) || !map(&P.tm_k, p.k, p.d.d_k) || !map(&P.tm_v, p.v, p.d.d_v)) return false;
    if (!map(&P.tm_do, with_bwd ? p.dO : p.v, p.d.d_v)) return false;
    if (!with_bwd && p.o && !map(&P.tm_o, p.o, p.d.d_v)) return false;
    if (with_bwd && (!map(&P.tm_dq, p.dq, p.d.d_k) || !map(&P.tm_dk, p.dk, p.d.d_k) || !map(&P.tm_dv, p.dv, p.d.d_v))) return false;
    return true;
}

template <class Kernel>
static cudaError_t launch_chunk_kernel(Kernel kernel, SmemLimitOnce& once, uint32_t smem, Stage stage, int grid, int threads,
                                       const TcParams& P, cudaStream_t st) {
    const cudaError_t e = once.ensure(kernel, smem);
    if (e != cudaSuccess) return e;
    if (grid > 0) {
        StageScope t(stage, st);
        launch_kernel(kernel, grid, threads, smem, st, P);
    }
    return cudaGetLastError();
}

static int sm_count();
static cudaError_t launch_prep(const TcParams& P, cudaStream_t st) {
    static SmemLimitOnce done;
    const int items = P.p.L.max_chunks * P.p.d.H, sms = sm_count();
    return launch_chunk_kernel(tc_prep_kernel, done, prep::SMEM_BYTES, ST_PREP, items < sms ? items : sms, kIntraThreads + 32, P, st);
}
// Number of SMs of the current device (persistent kernels launch one CTA per SM).
static int sm_count() {
    static int cached[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 148;
    if (!cached[dev]) {
        int n = 0;
        cached[dev] = (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && n > 0) ? n : 148;
    }
    return cached[dev];
}

// The small preparation kernels, two CTAs per SM.
static cudaError_t launch_eprep(const TcParams& P, cudaStream_t st) {
    static SmemLimitOnce done, done64;
    const int items = P.p.L.max_chunks * P.p.d.H, ctas = 2 * sm_count();
    if (P.narrow_v) return launch_chunk_kernel(tc_eprep_kernel<64>, done64, eprep::SMEM_BYTES, ST_EPREP, items < ctas ? items : ctas, split::kT, P, st);
    return launch_chunk_kernel(tc_eprep_kernel<128>, done, eprep::SMEM_BYTES, ST_EPREP, items < ctas ? items : ctas, split::kT, P, st);
}

template <int DV>
static cudaError_t launch_prep_lr_t(const TcParams& P, cudaStream_t st) {
    static SmemLimitOnce done;
    const int items = P.p.L.max_chunks * P.p.d.H, ctas = 2 * sm_count();
    return launch_chunk_kernel(tc_prep_lr_kernel<DV>, done, preplr::SMEM_BYTES, ST_PREP, items < ctas ? items : ctas, split::kT, P, st);
}
static cudaError_t launch_prep_lr(const TcParams& P, cudaStream_t st) { return P.narrow_v ? launch_prep_lr_t<64>(P, st) : launch_prep_lr_t<128>(P, st); }

static cudaError_t launch_scan(const TcParams& P, cudaStream_t st) {
    static SmemLimitOnce done;
    static SmemLimitOnce done2;
    const int ctas = P.p.d.N * P.p.d.H * (P.scan_dirs == 2 ? 2 : 1);
    const int half_ctas = P.narrow_v ? ctas : 2 * ctas;   // ... of the kernels whose CTAs carry 64 state columns each
    if (P.lowrank) {
        static SmemLimitOnce done_lr, done_lr2;
        // the reverse carry alone (backward on a fresh workspace) with few chains: two CTAs per chain, each carrying half of
        // the state columns (measured on 64 chains of 32 chunks: reverse 64 -> 58 us; the forward carry alone became
        // slower that way, 62 -> 66 us, and keeps one CTA per chain).  d_v = 64: half of the columns are all there are.
        if (P.narrow_v || (P.scan_dirs == 1 && half_ctas <= sm_count()))
            return launch_chunk_kernel(tc_scan_lr_kernel<2>, done_lr2, scanlr::Cfg<2>::SMEM_BYTES, ST_SCANS, half_ctas, scanlr::kScanThreads, P, st);
        return launch_chunk_kernel(tc_scan_lr_kernel<1>, done_lr, scanlr::Cfg<1>::SMEM_BYTES, ST_SCANS, ctas, scanlr::kScanThreads, P, st);
    }
    // few chains: two CTAs per (chain, direction), each carrying half of the state columns
    if (half_ctas <= sm_count())
        return launch_chunk_kernel(tc_scan_kernel<2>, done2, scan::Cfg<2>::SMEM_BYTES, ST_SCANS, half_ctas, kThreads, P, st);
    return launch_chunk_kernel(tc_scan_kernel<1>, done, scan::Cfg<1>::SMEM_BYTES, ST_SCANS, ctas, kThreads, P, st);
}
template <int DV, bool FACTORS>
static cudaError_t launch_intra_t(const TcParams& P, cudaStream_t st) {
    static SmemLimitOnce done;
    const int items = P.p.L.max_chunks * P.p.d.H, sms = sm_count();
    return launch_chunk_kernel(tc_intra_kernel<DV, FACTORS>, done, intra::SMEM_BYTES, ST_INTRA, items < sms ? items : sms, intra::kThreadsAll, P, st);
}
static cudaError_t launch_intra(const TcParams& P, cudaStream_t st) {
    if (P.lowrank) return P.narrow_v ? launch_intra_t<64, true>(P, st) : launch_intra_t<128, true>(P, st);
    return P.narrow_v ? launch_intra_t<64, false>(P, st) : launch_intra_t<128, false>(P, st);
}
template <int DV, bool FACTORS>
static cudaError_t launch_out_t(const TcParams& P, cudaStream_t st) {
    static SmemLimitOnce done;
    const int items = P.p.L.max_chunks * P.p.d.H, ctas = 2 * sm_count();
    return launch_chunk_kernel(tc_out_kernel<false, DV, FACTORS>, done, outk::SMEM_BYTES, ST_OUT, items < ctas ? items : ctas, kThreads, P, st);
}
static cudaError_t launch_out(const TcParams& P, cudaStream_t st) {
    if (P.lowrank) return P.narrow_v ? launch_out_t<64, true>(P, st) : launch_out_t<128, true>(P, st);
    return P.narrow_v ? launch_out_t<64, false>(P, st) : launch_out_t<128, false>(P, st);
}

int tc_sm_count() { return sm_count(); }

// Forward output of the channel-wise path from the tile images its preparation kernels and carries left in the workspace.
cudaError_t tc_launch_out_channelwise(const Problem& p, cudaStream_t st) {
    static SmemLimitOnce done;
    TcParams P{};
    P.p = p;
    if (!tc::make_tmap_bf16_heads(&P.tm_o, p.o, p.Ttot, p.d.H, p.d.d_v)) return cudaErrorUnknown;
    const int items = p.L.max_chunks * p.d.H, ctas = 2 * sm_count();
    return launch_chunk_kernel(tc_out_kernel<true, 128, false>, done, outk::SMEM_BYTES, ST_OUT, items < ctas ? items : ctas, kThreads, P, st);
}

// Carries of the channel-wise path: dirs = 0 forward, 1 reverse, 2 both in one launch.  Needs the tile images the
// channel-wise preparation kernels leave in the workspace; no tensor map is used.
cudaError_t tc_launch_scan_channelwise(const Problem& p, int dirs, cudaStream_t st) {
    static SmemLimitOnce done;
    TcParams P{};
    P.p = p;
    P.scan_dirs = dirs;
    P.lowrank = 1;
    const int ctas = p.d.N * p.d.H * (dirs == 2 ? 2 : 1);
    static SmemLimitOnce done2;
    if (dirs != 2 && 2 * ctas <= sm_count())
        return launch_chunk_kernel(tc_scan_cw_kernel<2>, done2, scancw::Cfg<2>::SMEM_BYTES, ST_SCANS, 2 * ctas, kThreads, P, st);
    return launch_chunk_kernel(tc_scan_cw_kernel<1>, done, scancw::Cfg<1>::SMEM_BYTES, ST_SCANS, ctas, kThreads, P, st);
}

// A call with no tokens still owes the pass-through of the states.
static cudaError_t empty_call(const Problem& p, bool bwd, cudaStream_t st) {
    const size_t bytes = (size_t)p.d.N * p.d.H * p.d.d_k * p.d.d_v * sizeof(float);
    float* dst = bwd ? p.dh0 : p.hT;
    const float* src = bwd ? p.dhT : p.h0;
    if (!dst) return cudaSuccess;
    return src ? cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToDevice, st) : cudaMemsetAsync(dst, 0, bytes, st);
}

// The chunk table is needed for packed sequences only (and for an empty call, whose only kernel it is).
static cudaError_t launch_table_if_needed(const Problem& p, bool fresh, cudaStream_t st) {
    return (p.cu || p.Ttot == 0) ? launch_table(p, st, fresh) : cudaSuccess;
}

// Carries in low-rank form take the chunk factors from tc_prep_lr; in operator form they also need Nm and Bf, which only
// tc_prep makes.
cudaError_t tc_launch_fwd(const Problem& p, cudaStream_t st) {
    TcParams P;
    cudaError_t e = launch_table_if_needed(p, false, st);
    if (e != cudaSuccess) return e;
    if (p.Ttot == 0) return empty_call(p, false, st);
    if (!fill_params(P, p, false, 0)) return cudaErrorUnknown;
    if ((e = P.lowrank ? launch_prep_lr(P, st) : launch_prep(P, st)) != cudaSuccess) return e;
    if ((e = launch_scan(P, st)) != cudaSuccess) return e;
    return p.o ? launch_out(P, st) : cudaSuccess;
}

// With a workspace fresh from gdn_fwd_recompute nothing of the forward is repeated: P, T, W, U~ and the per-chunk states
// are taken from it; the reverse carry and the gradient stage follow, in operator form behind E (tc_eprep).  A status that the forward left stands.
cudaError_t tc_launch_bwd(const Problem& p, bool skip_recompute, cudaStream_t st) {
    TcParams P;
    cudaError_t e = launch_table_if_needed(p, skip_recompute, st);
    if (e != cudaSuccess) return e;
    if (p.Ttot == 0) return empty_call(p, true, st);
    if (!fill_params(P, p, true, skip_recompute ? 1 : 2)) return cudaErrorUnknown;
    const bool inject = g_inject_timeout && !skip_recompute;
    if (inject) {   // debugging hook, this call only: a millisecond of patience, and one kernel withholds a load
        const unsigned long long ns = 1000000ull;
        P.withhold = g_inject_timeout;
        g_inject_timeout = 0;
        if ((e = cudaMemcpyToSymbolAsync(g_wait_limit_ns, &ns, sizeof(ns), 0, cudaMemcpyHostToDevice, st)) != cudaSuccess) return e;
    }
    if (!(skip_recompute && P.lowrank)) {
        if ((e = skip_recompute ? launch_eprep(P, st) : P.lowrank ? launch_prep_lr(P, st) : launch_prep(P, st)) != cudaSuccess) return e;
    }
    if ((e = launch_scan(P, st)) != cudaSuccess) return e;
    e = launch_intra(P, st);
    if (inject) {
        const unsigned long long ns = 2000000000ull;
        const cudaError_t e2 = cudaMemcpyToSymbolAsync(g_wait_limit_ns, &ns, sizeof(ns), 0, cudaMemcpyHostToDevice, st);
        if (e == cudaSuccess) e = e2;
    }
    return e;
}

}  // namespace gdn

