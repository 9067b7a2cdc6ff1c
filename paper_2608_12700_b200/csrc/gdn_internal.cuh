// Internal declarations shared by the host API and the kernel translation units.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <utility>

#include "gdn.h"

namespace gdn {

constexpr int kC = 64;  // chunk length (Section 4.2: chunks of 64 steps)

// Workspace header, first 256 bytes of the workspace.
struct WsHeader {
    int32_t status;    // device-side gdn_status (0 = ok)
    int32_t n_chunks;  // chunks actually present (<= max_chunks)
    int32_t detail;    // where a bounded wait gave up / offending sequence index
    int32_t cw_fallback;   // channel-wise calls on the tensor-core route: 1 if the gates of the call leave its range (set by its first
                           // stage, cleared by the table kernel of a call that does not consume a forward's workspace).  The
                           // tensor-core kernels then stand down and the FFMA kernels enqueued behind them compute the call, and
                           // the backward on the workspace of such a forward.
    int32_t seqlens_ok;    // 1 if the sequences that the workspace was filled for were valid: a status of GDN_ERR_BAD_SEQLENS then comes from a
                           // backward on the forward's workspace, whose data is whole, and the next such backward may have better ones
    int32_t pad[59];
};
static_assert(sizeof(WsHeader) == 256, "header size");

// Byte offsets of every workspace region.  Chunk-head index = chunk * H + head.
struct WsLayout {
    int max_chunks;        // bound on the number of chunks: sum over sequences of ceil(len/64) <= ceil(T_total/64) + N
    size_t seq_first;      // int32 [N + 1]   first chunk index of each sequence
    size_t seq_tok0;       // int32 [N + 1]   first token of each sequence: cu_seqlens as validated (no tokens: not written; the region has
                           //                 room for max_chunks entries, which is N then)
    size_t chunk_tok0;     // int32 [max_chunks]   global token index of the chunk's first row
    size_t chunk_len;      // int32 [max_chunks]   valid rows (1..64)
    size_t gamma;          // f32 [CH, 64]         chunk-local cumulative log decay (channel-wise calls: [CH, 64, d_k])
    size_t ref;            // int32 [CH, d_k]      channel-wise path on the tensor cores: the reference of a chunk's decays is 2^ref
    size_t Tm;             // f32|bf16 [CH, 64, 64]    T = (I + A)^-1
    size_t W;              // [CH, 64, d_k]
    size_t Ut;             // [CH, 64, d_v]            U~ = T Diag(w) V (tcgen05 d = 128 family, low-rank carries: U = U~ - W h after the forward carry)
    size_t Nm;             // [CH, d_k, d_k]           Kb^T W        (these two only when the carries run in operator
    size_t Bf;             // [CH, d_k, d_v]           Kb^T U~        form: has_operator; otherwise they take no space)
    int has_operator;
    size_t hc;             // [CH, d_k, d_v]           state entering the chunk
    size_t fwd_end;        // bytes needed by the forward recompute
    size_t E;              // [CH, d_k, d_v]           scale (Gam Q - P W)^T dO (FFMA families: scale (Gam Q)^T dO; tcgen05 d = 128 family, low-rank carries: dU [CH, 64, d_v])
    size_t dhn;            // [CH, d_k, d_v]           gradient w.r.t. the state leaving the chunk
    size_t Pm;             // [CH, 64, 64]             P = tril(Q K^T . D) (tcgen05 d = 128 family: made once, by tc_prep)
    size_t img_W, img_U, img_E;    // channel-wise path on the tensor cores (bf16, d = 128): bf16 tile images of W^T, U~^T (16 KB
                                   // per chunk-head each) and E (32 KB); else unused
    size_t img_QKp, img_Km, img_Vt;   // ... of [Q~; K+] (32 KB), K- and V~ (16 KB each)
    int tc_scans;                        // ... and T, P, hc, dhn are bf16 tile images as well (8, 8, 32, 32 KB)
    size_t Kb, U, dU;      // FFMA families (fp32): keys scaled to the chunk end [CH, 64, d_k]; U = U~ - W h and dU [CH, 64, d_v]
    size_t total;
};

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Layout of the scalar-gate tcgen05 families: every factor, state and additive term of the carries is a bf16 tile image.
inline WsLayout make_layout_tc(const gdn_desc& d, bool with_operator) {
    WsLayout L{};
    const size_t Ttot = (size_t)d.B * (size_t)d.T;
    L.max_chunks = (int)((Ttot + kC - 1) / kC + (size_t)d.N);
    const size_t CH = (size_t)L.max_chunks * d.H;
    size_t o = sizeof(WsHeader);
    auto take = [&](size_t bytes) { size_t r = o; o = align_up(o + bytes, 256); return r; };
    L.seq_first = take(4 * ((size_t)d.N + 1));
    L.seq_tok0 = take(4 * (size_t)L.max_chunks);
    L.chunk_tok0 = take(4 * (size_t)L.max_chunks);
    L.chunk_len = take(4 * (size_t)L.max_chunks);
    L.gamma = take(4 * CH * kC);
    L.Tm = take(2 * CH * kC * kC);
    L.W = take(2 * CH * kC * d.d_k);
    L.Ut = take(2 * CH * kC * d.d_v);
    L.Pm = take(2 * CH * kC * kC);
    L.has_operator = with_operator ? 1 : 0;
    L.Nm = take(with_operator ? 2 * CH * d.d_k * d.d_k : 0);
    L.Bf = take(with_operator ? 2 * CH * d.d_k * d.d_v : 0);
    L.hc = take(2 * CH * d.d_k * d.d_v);
    L.fwd_end = o;
    L.E = take(2 * CH * d.d_k * d.d_v);
    L.dhn = take(2 * CH * d.d_k * d.d_v);
    L.total = o;
    return L;
}

// Layout of the scalar-gate FFMA family: everything fp32, carries in low-rank form.
inline WsLayout make_layout_ffma(const gdn_desc& d) {
    WsLayout L{};
    const size_t Ttot = (size_t)d.B * (size_t)d.T;
    L.max_chunks = (int)((Ttot + kC - 1) / kC + (size_t)d.N);
    const size_t CH = (size_t)L.max_chunks * d.H;
    size_t o = sizeof(WsHeader);
    auto take = [&](size_t bytes) { size_t r = o; o = align_up(o + bytes, 256); return r; };
    L.seq_first = take(4 * ((size_t)d.N + 1));
    L.seq_tok0 = take(4 * (size_t)L.max_chunks);
    L.chunk_tok0 = take(4 * (size_t)L.max_chunks);
    L.chunk_len = take(4 * (size_t)L.max_chunks);
    L.gamma = take(4 * CH * kC);
    L.Tm = take(4 * CH * kC * kC);
    L.W = take(4 * CH * kC * d.d_k);
    L.Ut = take(4 * CH * kC * d.d_v);
    L.Pm = take(4 * CH * kC * kC);
    L.Kb = take(4 * CH * kC * d.d_k);
    L.U = take(4 * CH * kC * d.d_v);
    L.hc = take(4 * CH * d.d_k * d.d_v);
    L.Nm = L.Bf = L.fwd_end = o;
    L.E = take(4 * CH * d.d_k * d.d_v);
    L.dhn = take(4 * CH * d.d_k * d.d_v);
    L.dU = take(4 * CH * kC * d.d_v);
    L.total = o;
    return L;
}

// Layout of the channel-wise FFMA family: everything fp32; gamma is per channel ([CH, 64, d_k]), no chunk operator.
inline bool vec_tc_scans(const gdn_desc& d) { return d.dtype == GDN_BF16 && d.d_k == 128 && d.d_v == 128; }
inline WsLayout make_layout_vec(const gdn_desc& d) {
    WsLayout L{};
    const size_t Ttot = (size_t)d.B * (size_t)d.T;
    L.max_chunks = (int)((Ttot + kC - 1) / kC + (size_t)d.N);
    const size_t CH = (size_t)L.max_chunks * d.H;
    size_t o = sizeof(WsHeader);
    auto take = [&](size_t bytes) { size_t r = o; o = align_up(o + bytes, 256); return r; };
    L.tc_scans = vec_tc_scans(d) ? 1 : 0;
    L.seq_first = take(4 * ((size_t)d.N + 1));
    L.seq_tok0 = take(4 * (size_t)L.max_chunks);
    L.chunk_tok0 = take(4 * (size_t)L.max_chunks);
    L.chunk_len = take(4 * (size_t)L.max_chunks);
    L.gamma = take(4 * CH * kC * d.d_k);
    L.Tm = take(4 * CH * kC * kC);
    L.W = take(4 * CH * kC * d.d_k);
    L.Ut = take(4 * CH * kC * d.d_v);
    L.Pm = take(4 * CH * kC * kC);
    L.Nm = L.Bf = o;
    L.ref = take(L.tc_scans ? 4 * CH * d.d_k : 0);
    L.img_W = take(L.tc_scans ? CH * 16384 : 0);
    L.img_U = take(L.tc_scans ? CH * 16384 : 0);
    L.img_QKp = take(L.tc_scans ? CH * 32768 : 0);
    L.img_Km = take(L.tc_scans ? CH * 16384 : 0);
    L.img_Vt = take(L.tc_scans ? CH * 16384 : 0);
    L.Kb = take(4 * CH * kC * d.d_k);
    L.U = take(4 * CH * kC * d.d_v);
    L.hc = take(4 * CH * d.d_k * d.d_v);   // (fp32, or a bf16 tile image in the first half of each slot)
    L.fwd_end = o;
    L.E = take(4 * CH * d.d_k * d.d_v);
    L.img_E = take(L.tc_scans ? CH * 32768 : 0);
    L.dhn = take(4 * CH * d.d_k * d.d_v);
    L.dU = take(4 * CH * kC * d.d_v);
    L.total = o;
    return L;
}

// Everything a kernel needs to know about one call.
struct Problem {
    gdn_desc d;
    int Ttot;  // B * T
    const void *q, *k, *v, *dO;
    const float *g, *beta, *h0, *dhT;
    const int32_t* cu;
    void *o, *dq, *dk, *dv;
    float *hT, *dg, *dbeta, *dh0;
    // channel-wise entry points only: gate vectors g, b [.., d_k], w [.., d_v] and their gradients (g, dg above unused)
    const float *gv, *bv, *wv;
    float *dgv, *dbv, *dwv;
    int fallback;   // channel-wise FFMA kernels only: 1 = run only if the tensor-core route has refused the gates (status word)
    char* ws;
    WsLayout L;
};

// Launch bookkeeping: every kernel launch goes through stage_begin / stage_end so that launches can be
// counted and, when enabled, timed per stage with CUDA events on the launching stream.
enum Stage { ST_TABLE = 0, ST_PREP, ST_FSCAN, ST_OUT, ST_EPREP, ST_RSCAN, ST_INTRA, ST_SCANS, ST_SCALE, ST_FALLBACK, ST_COUNT };
void stage_begin(Stage s, cudaStream_t st);
void stage_end(Stage s, cudaStream_t st);
struct StageScope {
    Stage s; cudaStream_t st;
    StageScope(Stage s_, cudaStream_t st_) : s(s_), st(st_) { stage_begin(s, st); }
    ~StageScope() { stage_end(s, st); }
};

// Raising a kernel's dynamic shared-memory limit is a per-device function attribute: remember, per kernel, on which
// devices it has been done (a process may drive several GPUs).
struct SmemLimitOnce {
    bool done[64] = {};
    template <class Kernel>
    cudaError_t ensure(Kernel kernel, uint32_t bytes) {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64 && done[dev]) return cudaSuccess;
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (e == cudaSuccess && dev >= 0 && dev < 64) done[dev] = true;
        return e;
    }
};

// Programmatic dependent launch.  Every launch allows its kernel to be set up while the one before it in the stream runs, and
// every kernel of the library begins with wait_prerequisites(), which returns when that one is complete and its writes are
// visible: what a launch costs between two dependent kernels shrinks by about two microseconds.  (A training step of 4 heads
// of 333 tokens, six launches: 63.5 -> 51.8 us; a backward of 4 x 16 heads of 2048 tokens, three: 307 -> 301 us.)  All threads
// of all blocks wait, those without work too: a grid that ended without waiting would let the kernel after it run beside the
// one before it.  No kernel triggers its dependents early (griddepcontrol.launch_dependents): their blocks then take up
// room while others still work; the same two calls took 54.4 and 326 us that way.  In the last trip or step of every kernel it is no
// better: the instruction itself costs some 2.7 us a launch (a six-launch call 89 -> 105 us).
__device__ __forceinline__ void wait_prerequisites() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <class... Params, class... Args>
cudaError_t launch_kernel_cluster(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, unsigned cluster, Args&&... args) {
    cudaLaunchAttribute attr[2]{};
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}
template <class... Params, class... Args>
cudaError_t launch_kernel(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
    return launch_kernel_cluster(kernel, grid, block, smem, st, 1, std::forward<Args>(args)...);
}

gdn_status check_desc(const gdn_desc* d);                       // shape / dtype envelope
gdn_status check_seq(const gdn_desc& d, const int32_t* cu);     // B, N against cu_seqlens
void call_begin();                                              // stage-timing bookkeeping at the top of an entry point

// Host-side argument checks of gdn_bwd (everything that can be refused before a launch), shared with the entry point
// that brings its own workspace.
gdn_status check_bwd_args(const gdn_desc* desc, const void* q, const void* k, const void* v, const float* g, const float* beta,
                          const float* h0, const void* dO, const float* dhT, const int32_t* cu, void* dq, void* dk, void* dv,
                          float* dg, float* dbeta, float* dh0, const void* workspace, size_t workspace_bytes);

// Kernel families (each defined in its own translation unit).  They enqueue on `st` and return the
// first CUDA error seen.
// Chunk table of a call with packed sequences (or without tokens).  It validates cu_seqlens; nothing else reads them but
// check_fresh_seqlens.  `fresh`: the workspace is the forward's, whose status and fall-back words stay as they are.
cudaError_t launch_table(const Problem& p, cudaStream_t st, bool fresh = false);
cudaError_t simt_launch_fwd(const Problem& p, cudaStream_t st);
cudaError_t simt_launch_bwd(const Problem& p, bool skip_recompute, cudaStream_t st);

// FFMA family for per-channel gates (Eq. 1 with gate vectors).
cudaError_t vec_launch_fwd(const Problem& p, cudaStream_t st);
cudaError_t vec_launch_bwd(const Problem& p, bool skip_recompute, cudaStream_t st);
// ... and its tensor-core route (bf16 I/O, d_k = d_v = 128; gdn_tc_cw.cu): forward (bwd = false) or backward.
cudaError_t cw_tc_launch(const Problem& p, bool bwd, bool skip_recompute, cudaStream_t st);

// tcgen05 family (bf16 I/O; tiles of 128 features, a head dimension of 64 fills half of them).
extern thread_local int g_force_carries;   // form of the inter-chunk carries: 0 = chosen by shape, 1 = operator form, 2 = low-rank
extern thread_local int g_inject_timeout;   // debugging hook: the next gdn_bwd of this family provokes a device-side time-out (which
                                            // kernel's: see TcParams::withhold)
bool tc_supported(const gdn_desc& d);
// Form of the carries for a descriptor: one rule for the forward, the backward and a backward that consumes a workspace
// fresh from the forward, so that the layout of a workspace does not depend on which call sized it.
bool tc_carries_lowrank(const gdn_desc& d);
cudaError_t tc_launch_scan_channelwise(const Problem& p, int dirs, cudaStream_t st);   // carries of the channel-wise path
cudaError_t tc_launch_out_channelwise(const Problem& p, cudaStream_t st);              // its forward output (p.o non-null)
int tc_sm_count();                                                                     // SMs of the current device
cudaError_t tc_launch_fwd(const Problem& p, cudaStream_t st);
cudaError_t tc_launch_bwd(const Problem& p, bool skip_recompute, cudaStream_t st);


// Channel-wise calls with bf16 I/O and a head dimension of 64, zero-padded onto the d = 128 kernels (gdn_pad.cu).
bool tc_padded_supported(const gdn_desc& d);
gdn_desc tc_padded_desc(const gdn_desc& d);          // the widened descriptor (d_k = d_v = 128)
size_t tc_padded_extra_bytes(const gdn_desc& d);     // bytes of padded copies behind the widened problem's own workspace
cudaError_t tc_padded_launch(const Problem& p, const WsLayout& inner, bool bwd, bool skip_recompute, cudaStream_t st);

// tcgen05 family for the scalar-gate recurrence (bf16 I/O, d_k = d_v = 64, delta rule off).
bool tc64_supported(const gdn_desc& d);
cudaError_t tc64_launch_fwd(const Problem& p, cudaStream_t st);
cudaError_t tc64_launch_bwd(const Problem& p, bool skip_recompute, cudaStream_t st);

}  // namespace gdn
