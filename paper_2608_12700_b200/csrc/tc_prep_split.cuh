// The chunk-local preparation of the tcgen05 d = 128 family with the carries in low-rank form (included by gdn_tc.cu), as
// small kernels: about 90 KB of shared memory and 256 columns of tensor memory each, so that two CTAs share an SM.  A CTA
// works through the dependent phases of one chunk-head (product -> readout -> product ...) while its neighbour is in another
// phase of another chunk-head, which is what keeps the tensor pipe and the load/store path busy.  A trip's inputs are
// dead once its last product is done, so the next trip's are loaded right then, under the last readout and the stores
// (look-ahead without a second buffer).
//
//   tc_prep_lr  gamma, P, T = (I + A)^-1, W^T, U~^T (Section 4.2): all that carries in low-rank form need
//   tc_eprep    carries in operator form: E alone, for a backward that consumes a workspace fresh from the forward (no product,
//               inversion or store of the forward is repeated)
// The tc_prep kernel remains for carries in operator form, which also need Nm, Bf and E.
#pragma once

namespace split {
constexpr int kT = 256;   // 8 warps: TMEM lane quadrant = warp % 4, column half = warp / 4
}

// ------------------------------------------------------------------------------------------------
// tc_eprep: E alone, for a backward on a workspace fresh from the forward, from the stored P and W^T.
// ------------------------------------------------------------------------------------------------
namespace eprep {
constexpr uint32_t QT = 0;                  // Q [64][128]                                     16 KB
constexpr uint32_t DOT = 16384;             // dO [64][128]                                    16 KB
constexpr uint32_t WT = DOT + 16384;        // W^T [128][64] (image from the workspace)         16 KB
constexpr uint32_t PT = WT + 16384;         // P [64][64] (image from the workspace)             8 KB
constexpr uint32_t RT = PT + 8192;          // R = Diag(Gam) dO [64][128]                       16 KB  (these two: finally
constexpr uint32_t PDOT = RT + 16384;       // (P^T dO)^T [128][64]                             16 KB   the staged E image)
static_assert(RT % 1024 == 0 && PDOT == RT + 16384, "the E image [128][128] is two column blocks of 16 KB");
constexpr uint32_t SMEM_BYTES = PDOT + 16384 + 1024 /* alignment slack */;
constexpr uint32_t C_PDO = 0, C_E = 128;    // TMEM columns (256 allocated)
static_assert(2 * (SMEM_BYTES + 4096) <= 228 * 1024, "two CTAs per SM");
}  // namespace eprep

template <int DV>
__global__ void __launch_bounds__(split::kT, 2) tc_eprep_kernel(const __grid_constant__ TcParams P) {
    wait_prerequisites();
    using namespace eprep;
    const Problem& p = P.p;
    const int H = p.d.H;
    if (reinterpret_cast<const WsHeader*>(p.ws)->status != GDN_OK) return;
    const int n_items = n_chunks_of(p) * H;
    if ((int)blockIdx.x >= n_items) return;

    extern __shared__ unsigned char smem_raw[];
    unsigned char* sm = align1024(smem_raw);
    __shared__ float Gam[kC];
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
    // Q, dO, P and W of a trip are dead once its last product is done: the next trip's are loaded right then, under the
    // readout of E and its store (E is staged over R and (P^T dO)^T, which are dead by then too, not over an input).
    auto issue_loads = [&](const ChunkInfo& c) {   // thread 0
        mbar_expect_tx(&bar_in, 40960 + 128 * DV);
        for (int cb = 0; cb < 2; ++cb) {
            tma_load_3d(sm + QT + cb * 8192, &P.tm_q, cb * 64, c.hd, c.tok0, &bar_in);
            if (cb * 64 < DV) tma_load_3d(sm + DOT + cb * 8192, &P.tm_do, cb * 64, c.hd, c.tok0, &bar_in);
        }
        bulk_load(sm + PT, p.ws + p.L.Pm + (size_t)c.ch * 8192, 8192, &bar_in);
        bulk_load(sm + WT, p.ws + p.L.W + (size_t)c.ch * 16384, 16384, &bar_in);
        pending = true;
    };
    float gnext = 0.f;   // threads 0..63: cumulative decay of the next trip's chunk, fetched a trip ahead
    auto fetch_gamma = [&](const ChunkInfo& c) {
        if (threadIdx.x < kC) gnext = reinterpret_cast<const float*>(p.ws + p.L.gamma)[(size_t)c.ch * kC + threadIdx.x];
    };
    ChunkInfo x;
    chunk_entry(p, x, blockIdx.x);
    if (threadIdx.x == 0) issue_loads(x);
    fetch_gamma(x);
#pragma unroll 1
    for (int item = blockIdx.x; item < n_items; item += gridDim.x, in_phase ^= 1) {
        const bool has_next = item + (int)gridDim.x < n_items;
        ChunkInfo xn = x;
        if (has_next) chunk_entry(p, xn, item + gridDim.x);
        if (threadIdx.x < kC) {   // chunk-local cumulative decay, left in the workspace by the factor stage
            Gam[threadIdx.x] = expf(gnext);
        }
        if (ok) {
            ok = mbar_wait(&bar_in, in_phase);
            if (!ok && lane == 0) report_timeout(p.ws, 24);
            if (ok && threadIdx.x == 0) pending = false;
        }
        if (ok && x.len < kC) {   // identity padding of a ragged tail
            zero_tail_rows(sm + QT, 64, 0, x.len, split::kT);
            zero_tail_rows(sm + DOT, 64, 0, x.len, split::kT);
            fence_async_smem();
        }
        __syncthreads();
        // ---- phase 1: (P^T dO)^T = dO^T P, and meanwhile R = Diag(Gam) dO (four 16-byte pieces per thread)
        if (warp == 0 && elect_one() && ok) {
            tc_fence_after();
            mma_tile<128, 64, 64>(tmem + C_PDO, op_mn_major(sm + DOT, 64), op_mn_major(sm + PT, 64), false);
            mma_commit(&bar_mma);
        }
        if (warp == 0) bulk_wait_read<0>();   // the previous trip's store has read the staged E image
        GDN_WAIT_MMA(25)
        __syncthreads();
#pragma unroll
        for (int it = 0; it < 4; ++it) {
            const int i = (threadIdx.x >> 4) + 16 * it;
            float v[8];
            chunk_load(sm + DOT, 64, i, threadIdx.x & 15, v);
            const float G = Gam[i];
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] *= G;
            chunk_store(sm + RT, 64, i, threadIdx.x & 15, v);
        }
        if (ok) {
            const int f = q4 * 32 + lane, i0 = grp * 32;
#pragma unroll 1
            for (int part = 0; part < 4; ++part) {
                const int ib = i0 + part * 8;
                float v[8];
                tmem_ld8(tmem + lane_base + C_PDO + ib, v);
                tmem_wait_ld();
                chunk_store(sm + PDOT, 128, f, ib >> 3, v);
            }
        }
        tc_fence_before();
        fence_async_smem();
        __syncthreads();
        // ---- phase 2: E = Q^T R - W^T (P^T dO)
        if (warp == 0 && elect_one() && ok) {
            tc_fence_after();
            mma_tile<128, DV, 64>(tmem + C_E, op_mn_major(sm + QT, 64), op_mn_major(sm + RT, 64), false);
            mma_tile<128, DV, 64>(tmem + C_E, op_k_major(sm + WT, 128), op_k_major(sm + PDOT, 128), true, /*neg_a=*/true);
            mma_commit(&bar_mma);
        }
        GDN_WAIT_MMA(27)
        if (ok && has_next) {   // every input tile has been read for the last time
            if (threadIdx.x == 0) issue_loads(xn);
            fetch_gamma(xn);
        }
        if (ok) {   // E -> bf16 tile image over R and (P^T dO)^T, which no product reads any more
            const int r = q4 * 32 + lane, c0 = grp * (DV / 2);
#pragma unroll 1
            for (int part = 0; part < DV / 16; ++part) {
                const int cb = c0 + part * 8;
                float v[8];
                tmem_ld8(tmem + lane_base + C_E + cb, v);
                tmem_wait_ld();
#pragma unroll
                for (int k = 0; k < 8; ++k) v[k] *= sc;
                chunk_store(sm + RT, 128, r, cb >> 3, v);
            }
        }
        tc_fence_before();
        fence_async_smem();
        __syncthreads();
        if (warp == 0 && elect_one() && ok) {
            bulk_store(p.ws + p.L.E + (size_t)x.ch * 32768, sm + RT, 256 * DV);
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
// tc_prep_lr: gamma, P = tril(Q K^T . D), T = (I + A)^-1, W^T, U~^T.  The forward's and the backward's preparation are the same: the
// reverse carry takes Q, dO and P itself (tc_scan_lr).
// Against one CTA per SM with sixteen readout warps, a loader and an issuer warp (the form tc_prep still has), two CTAs fill each
// other's waits (both are bound by the chain of dependent phases of a chunk-head).  4 x 16 heads of 2048 tokens 64.5 us, 8 packed
// sequences, 32768 tokens, 32 heads 447 us (98 KB of traffic per chunk-head); with E for a backward 80 and 562 us.
// P is made here, although the forward output and the reverse carry use it: Q K^T rides along with K K^T in one M = 128
// product, and neither of those has to load K and wait for a product of its own.
// ------------------------------------------------------------------------------------------------
namespace preplr {
constexpr uint32_t QK = 0;                  // [Q rows 0..63 ; K rows 64..127] x 128                            32 KB
constexpr uint32_t VT = 32768;              // V [64][128], later U~^T [128][64]                                16 KB
constexpr uint32_t XA = VT + 16384;         // fp32 A [64][kLdi], then the bf16 tiles T, T Diag(b Gam), T Diag(w) over A and T,
constexpr uint32_t XT = XA + 17408;         // fp32 T [64][kLdi]        then W^T over the last two
constexpr uint32_t PT = XT + 17408;         // P = tril(Q K^T . D)                                               8 KB
constexpr uint32_t TT = XA, TP = XA + 8192, TPP = XA + 16384, WT = TP, UTT = VT;
constexpr uint32_t SMEM_BYTES = PT + 8192 + 1024 /* alignment slack */;
constexpr uint32_t C_S1 = 0, C_W = 128, C_U = 192;   // TMEM columns (256 allocated)
static_assert(TPP + 8192 <= PT && PT % 1024 == 0, "T tiles fit over the fp32 blocks");
static_assert(2 * (SMEM_BYTES + 4096) <= 228 * 1024, "two CTAs per SM");
}  // namespace preplr

template <int DV>
__global__ void __launch_bounds__(split::kT, 2) tc_prep_lr_kernel(const __grid_constant__ TcParams P) {
    wait_prerequisites();
    using namespace preplr;
    const Problem& p = P.p;
    const int H = p.d.H;
    init_header_if_untabled(p);
    const int n_items = n_chunks_of(p) * H;
    if ((int)blockIdx.x >= n_items) return;

    extern __shared__ unsigned char smem_raw[];
    unsigned char* sm = align1024(smem_raw);
    __shared__ __align__(16) float gates[4][kC];   // gam log2e, b, w, b Gam
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
    const float *gl = gates[0], *bb = gates[1], *ww = gates[2], *bgam = gates[3];
    float* Af = reinterpret_cast<float*>(sm + XA);
    float* Tf = reinterpret_cast<float*>(sm + XT);
    bool ok = true, pending = false;
    uint32_t mma_phase = 0, in_phase = 0;
    // Q and K of a trip are dead once its last product is done, V when U~^T, staged over it, has left: the next trip's are loaded right then, the
    // gate values of the next trip fetched into registers at the same moment.
    auto load_qk = [&](const ChunkInfo& c, bool withhold) {   // thread 0; announces the trip's bytes
        mbar_expect_tx(&bar_in, 49152);
        for (int cb = 0; cb < 2; ++cb) {
            if (!(withhold && cb == 0)) tma_load_3d(sm + QK + cb * 16384, &P.tm_q, cb * 64, c.hd, c.tok0, &bar_in);
            tma_load_3d(sm + QK + cb * 16384 + 8192, &P.tm_k, cb * 64, c.hd, c.tok0, &bar_in);
        }
        pending = true;
    };
    auto load_v = [&](const ChunkInfo& c) {
        for (int cb = 0; cb < 2; ++cb) tma_load_3d(sm + VT + cb * 8192, &P.tm_v, cb * 64, c.hd, c.tok0, &bar_in);
    };
    float gg[2] = {0.f, 0.f}, gb[2] = {0.f, 0.f}, gw[2] = {0.f, 0.f};   // warp 0: log decay, erase gate, write gate of tokens lane, lane + 32
    auto fetch_gates = [&](const ChunkInfo& c) {   // warp 0
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = lane + 32 * h;
            gg[h] = gb[h] = gw[h] = 0.f;
            if (i < c.len) {
                const size_t idx = (size_t)(c.tok0 + i) * H + c.hd;
                gg[h] = p.g[idx];
                gb[h] = p.d.delta_rule ? p.beta[idx] : 0.f;   // delta rule off: erase 0, write 1
                gw[h] = p.d.delta_rule ? gb[h] : 1.f;
            }
        }
    };
    ChunkInfo x;
    chunk_entry(p, x, blockIdx.x);
    if (threadIdx.x == 0) { load_qk(x, P.withhold == WITHHOLD_PREP); load_v(x); }
    if (warp == 0) fetch_gates(x);
#pragma unroll 1
    for (int item = blockIdx.x; item < n_items; item += gridDim.x, in_phase ^= 1) {
        const bool has_next = item + (int)gridDim.x < n_items;
        ChunkInfo xn = x;
        if (has_next) chunk_entry(p, xn, item + gridDim.x);
        if (warp == 0) {   // gate arrays of the chunk from the values fetched a trip ahead
            float a = gg[0], b = gg[1];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const float ua = __shfl_up_sync(0xffffffffu, a, o), ub = __shfl_up_sync(0xffffffffu, b, o);
                if (lane >= o) { a += ua; b += ub; }
            }
            b += __shfl_sync(0xffffffffu, a, 31);
            const float gc[2] = {a, b};
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int i = lane + 32 * h;
                const float G = expf(gc[h]);
                gates[0][i] = gc[h] * kLog2e;
                gates[1][i] = gb[h];
                gates[2][i] = gw[h];
                gates[3][i] = gb[h] * G;
                reinterpret_cast<float*>(p.ws + p.L.gamma)[(size_t)x.ch * kC + i] = gc[h];
            }
        }
        if (ok) {
            ok = mbar_wait(&bar_in, in_phase);
            if (P.withhold == DISAGREE_PREP && (warp & 1)) ok = false;
            if (!ok && lane == 0) report_timeout(p.ws, 1);
            if (ok && threadIdx.x == 0) pending = false;
        }
        if (ok && x.len < kC) {   // identity padding of a ragged tail
            zero_tail_rows(sm + QK, 128, 0, x.len, split::kT);
            zero_tail_rows(sm + QK, 128, 64, x.len, split::kT);
            zero_tail_rows(sm + VT, 64, 0, x.len, split::kT);
            fence_async_smem();
        }
        __syncthreads();
        // ---- phase 1: S1 = [Q; K] K^T  (rows 0..63: Q K^T, rows 64..127: K K^T)
        if (warp == 0 && elect_one() && ok) {
            tc_fence_after();
            mma_tile<128, 64, 128>(tmem + C_S1, op_k_major(sm + QK, 128, 0), op_k_major(sm + QK, 128, 64), false);
            bulk_wait_read<0>();   // (the previous trip's stores have read P and T: rewritten from here on)
            mma_commit(&bar_mma);
        }
        GDN_WAIT_MMA(2)
        if (ok) {
            const int i = (q4 & 1) * 32 + lane, j0 = grp * 32;
#pragma unroll 2
            for (int part = 0; part < 4; ++part) {
                float v[8], g8[8];
                const int jb = j0 + part * 8;
                tmem_ld8(tmem + lane_base + C_S1 + jb, v);
                ld8s(gl + jb, g8);
                tmem_wait_ld();
                if (q4 < 2) {   // P_ij = (q_i . k_j) exp(gam_i - gam_j), j <= i (mask before exponentiating)
#pragma unroll
                    for (int j = 0; j < 8; ++j) v[j] = (jb + j <= i) ? v[j] * ex2(gl[i] - g8[j]) : 0.f;
                    chunk_store(sm + PT, 64, i, jb >> 3, v);
                } else {        // A_ij = b_i (k_i . k_j) exp(gam_i - gam_j), j < i
#pragma unroll
                    for (int j = 0; j < 8; ++j) v[j] = (jb + j < i) ? bb[i] * v[j] * ex2(gl[i] - g8[j]) : 0.f;
                    *reinterpret_cast<float4*>(Af + i * kLdi + jb) = make_float4(v[0], v[1], v[2], v[3]);
                    *reinterpret_cast<float4*>(Af + i * kLdi + jb + 4) = make_float4(v[4], v[5], v[6], v[7]);
                }
            }
        }
        tc_fence_before();
        fence_async_smem();
        __syncthreads();
        if (warp == 0 && elect_one() && ok) {
            bulk_store(p.ws + p.L.Pm + (size_t)x.ch * 8192, sm + PT, 8192);   // the forward output and the reverse carry read P from here
            bulk_commit();
        }
        invert64(Af, Tf, [] { __syncthreads(); });
        {   // T -> bf16 tiles T, T Diag(b Gam), T Diag(w): a thread scales two rows of one 8-column piece.  The tiles lie over A
            // and T, so every row is in registers before the first one is written.
            const int cch = threadIdx.x & 7;
            float a[2][8], gb8[8], gw8[8];
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
            ld8s(bgam + cch * 8, gb8);
            ld8s(ww + cch * 8, gw8);
            __syncthreads();
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int i = (threadIdx.x >> 3) + 32 * h;
                float b[8], w8[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) { b[k] = gb8[k] * a[h][k]; w8[k] = gw8[k] * a[h][k]; }
                chunk_store(sm + TT, 64, i, cch, a[h]);
                chunk_store(sm + TP, 64, i, cch, b);
                chunk_store(sm + TPP, 64, i, cch, w8);
            }
        }
        fence_async_smem();
        __syncthreads();
        // ---- phase 2: W^T = K^T (T Diag(b Gam))^T ; U~^T = V^T (T Diag(w))^T
        if (warp == 0 && elect_one() && ok) {
            tc_fence_after();
            mma_tile<128, 64, 64>(tmem + C_W, op_mn_major(sm + QK, 128, 64), op_k_major(sm + TP, 64), false);
            mma_tile<128, 64, 64>(tmem + C_U, op_mn_major(sm + VT, 64), op_k_major(sm + TPP, 64), false);
            mma_commit(&bar_mma);
            bulk_store(p.ws + p.L.Tm + (size_t)x.ch * 8192, sm + TT, 8192);
            bulk_commit();
        }
        GDN_WAIT_MMA(3)
        if (ok && has_next && threadIdx.x == 0) load_qk(xn, false);
        if (ok) {
            const int f = q4 * 32 + lane, i0 = grp * 32;
#pragma unroll 1
            for (int part = 0; part < 4; ++part) {
                const int ib = i0 + part * 8;
                float a[8], b[8];
                tmem_ld8(tmem + lane_base + C_W + ib, a);
                tmem_ld8(tmem + lane_base + C_U + ib, b);
                tmem_wait_ld();
                chunk_store(sm + WT, 128, f, ib >> 3, a);
                chunk_store(sm + UTT, 128, f, ib >> 3, b);
            }
        }
        tc_fence_before();
        fence_async_smem();
        __syncthreads();
        if (threadIdx.x == 0 && ok) {
            bulk_store(p.ws + p.L.W + (size_t)x.ch * 16384, sm + WT, 16384);
            bulk_store(p.ws + p.L.Ut + (size_t)x.ch * 16384, sm + UTT, 128 * DV);
            bulk_commit();
            bulk_wait_read<0>();   // W^T and U~^T have left: the fp32 blocks and V of the next trip (it waits for V) go over them
            if (has_next) load_v(xn);
        }
        if (ok && has_next && warp == 0) fetch_gates(xn);
        if (!ok) {
            stand_by_items<10>(item, n_items, [] { __syncthreads(); });
            break;
        }
        x = xn;
    }
    if (warp == 0) bulk_wait_read<0>();
    if (threadIdx.x == 0 && pending) (void)mbar_wait(&bar_in, in_phase);   // after a timeout a load may still be in flight
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 256);
}
