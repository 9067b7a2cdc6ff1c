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
// before, only the last can be short.  (cu_seqlens has been validated by the table kernel by the time it is read here.)
struct SeqGeom {
    int c0, n_chunks, tok0, len;   // first chunk, number of chunks, first token, tokens
    __device__ __forceinline__ int chunk_tok0(int c) const { return tok0 + (c - c0) * kC; }
    __device__ __forceinline__ int chunk_len(int c) const { return min(kC, len - (c - c0) * kC); }
};
__device__ __forceinline__ SeqGeom seq_geom(const Problem& p, int n) {
    SeqGeom g;
    if (p.cu) {
        g.tok0 = p.cu[n];
        g.len = p.cu[n + 1] - g.tok0;
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
    }
}

}  // namespace
}  // namespace gdn
