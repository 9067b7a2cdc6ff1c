// Chunk geometry on the device and the reset of the workspace header, shared by every kernel family.
#pragma once
#include "gdn_internal.cuh"

namespace gdn {
namespace {

// Chunk geometry.  With packed sequences (cu_seqlens given) it is read from the table the table kernel wrote into the
// workspace; with equal-length sequences it is plain arithmetic and that kernel is not launched at all (the first
// kernel of the call initialises the header instead, see init_header_if_untabled).
struct ChunkInfo { int c, hd, ch, tok0, len; };
__device__ __forceinline__ int chunks_per_sequence(const Problem& p) { return (p.d.T + kC - 1) / kC; }
__device__ __forceinline__ int n_chunks_of(const Problem& p) {
    return p.cu ? reinterpret_cast<const WsHeader*>(p.ws)->n_chunks : p.d.N * chunks_per_sequence(p);
}
__device__ __forceinline__ int seq_first_chunk(const Problem& p, int n) {
    return p.cu ? reinterpret_cast<const int32_t*>(p.ws + p.L.seq_first)[n] : n * chunks_per_sequence(p);
}
// Entry of an item known to exist: no header read and no branch on loaded data, so the two table loads can stay in
// flight until their values are used (the persistent kernels fetch the entry one trip ahead).
__device__ __forceinline__ void chunk_entry(const Problem& p, ChunkInfo& x, int item) {
    x.c = item / p.d.H;
    x.hd = item % p.d.H;
    x.ch = item;
    if (p.cu) {
        x.tok0 = reinterpret_cast<const int32_t*>(p.ws + p.L.chunk_tok0)[x.c];
        x.len = reinterpret_cast<const int32_t*>(p.ws + p.L.chunk_len)[x.c];
    } else {
        const int cps = chunks_per_sequence(p), n = x.c / cps, pos = x.c - n * cps;
        x.tok0 = n * p.d.T + pos * kC;
        x.len = min(kC, p.d.T - pos * kC);
    }
}
// ... and from the table, for calls that build it whatever the sequences (the channel-wise ones).
__device__ __forceinline__ void chunk_entry_tab(const Problem& p, ChunkInfo& x, int item) {
    x.c = item / p.d.H;
    x.hd = item % p.d.H;
    x.ch = item;
    x.tok0 = reinterpret_cast<const int32_t*>(p.ws + p.L.chunk_tok0)[x.c];
    x.len = reinterpret_cast<const int32_t*>(p.ws + p.L.chunk_len)[x.c];
}
// The same geometry for kernels that walk along whole sequences.
struct ChunkGeom {
    const int32_t *first, *tok0, *len;   // tables (packed sequences), else null
    int cps, T;                          // equal lengths: chunks per sequence, tokens per sequence
    __device__ __forceinline__ int seq_first(int n) const { return first ? first[n] : n * cps; }
    __device__ __forceinline__ int chunk_tok0(int c) const {
        if (tok0) return tok0[c];
        const int n = c / cps;
        return n * T + (c - n * cps) * kC;
    }
    __device__ __forceinline__ int chunk_len(int c) const { return len ? len[c] : min(kC, T - (c % cps) * kC); }
};
__device__ __forceinline__ ChunkGeom chunk_geom(const Problem& p) {
    ChunkGeom g;
    g.first = p.cu ? reinterpret_cast<const int32_t*>(p.ws + p.L.seq_first) : nullptr;
    g.tok0 = p.cu ? reinterpret_cast<const int32_t*>(p.ws + p.L.chunk_tok0) : nullptr;
    g.len = p.cu ? reinterpret_cast<const int32_t*>(p.ws + p.L.chunk_len) : nullptr;
    g.cps = max(1, chunks_per_sequence(p));
    g.T = p.d.T;
    return g;
}
// One sequence, for the kernels that walk along it: its chunks are consecutive, each starts 64 tokens after the one
// before, only the last can be short.  (Packed sequences: from the table, never from the caller's cu_seqlens, which in a backward on
// the forward's workspace may no longer be what they were.)
struct SeqGeom {
    int c0, n_chunks, tok0, len;   // first chunk, number of chunks, first token, tokens
    __device__ __forceinline__ int chunk_tok0(int c) const { return tok0 + (c - c0) * kC; }
    __device__ __forceinline__ int chunk_len(int c) const { return min(kC, len - (c - c0) * kC); }
};
__device__ __forceinline__ SeqGeom seq_geom(const Problem& p, int n) {
    SeqGeom g;
    if (p.cu && p.Ttot > 0) {
        const int32_t* tok0 = reinterpret_cast<const int32_t*>(p.ws + p.L.seq_tok0);
        g.tok0 = tok0[n];
        g.len = tok0[n + 1] - g.tok0;
        g.c0 = reinterpret_cast<const int32_t*>(p.ws + p.L.seq_first)[n];
    } else {
        g.tok0 = n * p.d.T;
        g.len = p.d.T;
        g.c0 = n * chunks_per_sequence(p);
    }
    g.n_chunks = (g.len + kC - 1) / kC;
    return g;
}
__device__ __forceinline__ bool chunk_info(const Problem& p, ChunkInfo& x, int item) {
    if (item / p.d.H >= n_chunks_of(p)) return false;
    chunk_entry(p, x, item);
    return true;
}
__device__ __forceinline__ bool chunk_info(const Problem& p, ChunkInfo& x) { return chunk_info(p, x, (int)blockIdx.x); }
// Called at the top of the first kernel of a call: without the table kernel somebody has to reset the status word.
__device__ __forceinline__ void init_header_if_untabled(const Problem& p) {
    if (!p.cu && blockIdx.x == 0 && threadIdx.x == 0) {
        WsHeader* hdr = reinterpret_cast<WsHeader*>(p.ws);
        hdr->status = GDN_OK;
        hdr->n_chunks = n_chunks_of(p);
        hdr->detail = 0;
        hdr->seqlens_ok = 1;
    }
}
// Called by all threads at the top of the first kernel of a backward on the forward's workspace, in the families that do not build
// the table again: the cu_seqlens have to be the forward's.  One block looks, the last one, which has no chunk to work on in a grid
// of max_chunks x heads (the bound allows one chunk more than there can be); the others work from the table meanwhile, and the kernels
// behind, which write the outputs, see the status.  (As a launch of the table kernel ahead of it the check took 2.5 us.)
__device__ __forceinline__ bool status_from_fresh(const WsHeader* hdr) { return hdr->status == GDN_ERR_BAD_SEQLENS && hdr->seqlens_ok; }
__device__ __forceinline__ void check_fresh_seqlens(const Problem& p) {
    if (!p.cu || blockIdx.x != gridDim.x - 1) return;
    const int32_t* tok0 = reinterpret_cast<const int32_t*>(p.ws + p.L.seq_tok0);
    int same = 1, at = p.d.N;
    for (int n = threadIdx.x; n <= p.d.N; n += blockDim.x)
        if (p.cu[n] != (p.Ttot > 0 ? tok0[n] : 0)) { same = 0; at = n; }
    const int all = __syncthreads_and(same);
    WsHeader* hdr = reinterpret_cast<WsHeader*>(p.ws);
    if (all ? threadIdx.x == 0 : !same) {   // (several threads may find a difference: any of them will do)
        if (hdr->status == GDN_OK || status_from_fresh(hdr)) {
            hdr->status = all ? GDN_OK : GDN_ERR_BAD_SEQLENS;
            hdr->detail = all ? 0 : at;
        }
    }
}

}  // namespace
}  // namespace gdn
