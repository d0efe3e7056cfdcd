// Chunked prefill: shared layout of the workspace and of the per-(chunk, v-head) record.
//
// Inside a chunk of C = 64 tokens entering with state S0 (dv x dk), with
// b_r = sum_{i<=r} g_i (inclusive, chunk-local) the gated delta rule unrolls to
//
//   A_ri = beta_r e^{b_r-b_i} (k_r.k_i)  (i <  r),   T = (I + A)^{-1}
//   P_ri =        e^{b_r-b_i} (q_r.k_i)  (i <= r)
//   W  = T diag(beta e^b) K   (C x dk),   U~ = T diag(beta) V   (C x dv)
//   U  = U~ - W S0^T
//   O  = scale ( diag(e^b) Q S0^T + P U )
//   S' = e^{b_C} S0 + U^T diag(e^{b_C-b}) K
//
// Three launches: a prep kernel builds the chunk table from cu_seqlens; the
// intra-chunk kernel (all chunks and v-heads in parallel, a pipeline per SM)
// computes W, U~, P and b with tcgen05 GEMMs and an fp32 triangular solve and
// writes them as a record; the state pass (one persistent CTA per SM that takes
// sequence after sequence of a v-head from a list) walks the chunks in order
// carrying S in fp32 registers.  A fused variant runs the last two as one
// cooperative launch, another produces part of the records beside the state pass.
#pragma once
#include "gdn_common.cuh"
#include <cuda.h>

namespace gdn {

// One record per (chunk, v-head), written by the intra-chunk kernel in exactly the
// byte image the state-pass kernel wants in shared memory (linear bulk copies):
//   [0, 16384)      W   as one MN-major 128B-swizzled tile [128 dk][64 tokens] bf16 (a row per dk)
//   [16384, 32768)  Qg  = diag(scale e^b) Q as two K-major 128B-swizzled halves [64 tokens][64 dk] bf16:
//                   in the cooperative launch only
//   [32768, 40960)  P   as one K-major 128B-swizzled tile   [64 r][64 i]      bf16, scale folded in
//   [40960, 73728)  U~  as [2 halves of dv][16 token-groups][64 dv][4 tokens] fp32, dv swizzled (rec_u_index)
//   [73728, 73984)  e^{b_C - b_c} for c = 0..63, fp32 (rows past the chunk's length hold 1)
//   [73984, 74240)  scale e^{b_r} for r = 0..63, fp32
//   [74240, 74496)  e^{b_C}, then (int32) the number of 16-token blocks that hold tokens, rest unused
// Of a chunk with fewer than 64 tokens only the 16-token blocks that hold tokens (rows of P, token groups of U~) are
// written, copied and read; W is zero in the others, the state pass puts zeros in U~'s place, and so U is zero there.
// The output's first term is diag(scale e^b) Q S0^T.  Cooperative launch (kScaledQ): the record carries Qg and
// both terms meet in one accumulator, since whatever the output warps do there comes out of the chain's issue
// slots (32768 tokens 792 us, with raw Q 854).  Elsewhere the state pass loads the raw Q tile and scales the
// rows of the product: the intra-chunk kernel saves a pass over Q and a fifth of its writes and can load V
// early, the state pass pays with a second accumulator to read (4 x 2048 tokens at 32 heads 163 us, with the
// scaled Q 172; 512 + 1024 + 2048 + 4096 200.7 and 203.3, 57 sequences 223 and 240).
constexpr uint32_t kRecW = 0;
constexpr uint32_t kRecQg = 16384;
constexpr uint32_t kRecP = 32768;
constexpr uint32_t kRecU = 40960;
constexpr uint32_t kRecDecay = 73728;
constexpr uint32_t kRecEb = 73984;
constexpr uint32_t kRecGammaC = 74240;
constexpr uint32_t kRecBytes = 74496;
constexpr uint32_t kRecUHalf = (kRecDecay - kRecU) / 2;
constexpr uint32_t kRecUBlock = kRecUHalf / 4, kRecPBlock = (kRecU - kRecP) / 4;      // bytes of a 16-token block
__device__ __forceinline__ int token_blocks(int seq_len, int chunk) { return (min(kChunk, seq_len - chunk * kChunk) + 15) >> 4; }
// The same by the record's own word.  Where a producer has left after a wait that ran out, that is whatever the workspace
// held, and what is addressed by it has four blocks.
__device__ __forceinline__ int record_blocks(const void* word) {
    const uint32_t n = *reinterpret_cast<const uint32_t*>(word);
    return static_cast<int>(n < 4u ? n : 4u);
}
// Place (in 16-byte units) of a token group and dv within one half of U~.  Odd groups have their dv swapped in fours,
// so that a fragment read (four dv of two neighbouring groups per half warp) touches every bank once.
__device__ __forceinline__ int rec_u_index(int group, int dv) { return group * 64 + (dv ^ ((group & 1) << 2)); }

// Batches of at most this many sequences need no table-building launch in front of the intra-chunk kernel and the state
// pass: a warp reads all bounds at once.
constexpr int kSmallSeqs = 32;

struct ChunkInfo {      // 16 bytes
    int32_t seq;        // sequence the chunk belongs to
    int32_t t0;         // first packed token of the chunk
    int32_t len;        // valid tokens (1..64)
    int32_t pad;
};

// Which sequences count.  One does if its own bounds are in order (0 <= t0 <= t1 <= T) and no earlier sequence whose
// bounds are in order ends behind its start; the others have no chunks and are flagged.  Those that count do not
// overlap, so they have at most T / 64 + N chunks, which is what the workspace is laid out for.  Where every
// sequence's own bounds are in order each starts where the one before ends: only where a vote finds one that is not
// are starts and ends compared.
__device__ __forceinline__ bool bounds_in_order(int32_t t0, int32_t t1, int32_t T) {
    return t0 >= 0 && t1 >= t0 && t1 <= T;
}
// By one converged warp, a sequence a lane; lanes past the last one hold t0 = t1 = 0.
__device__ __forceinline__ bool warp_bounds_ok(int32_t t0, int32_t t1, int32_t T, int lane) {
    bool ok = bounds_in_order(t0, t1, T);
    if (!__all_sync(0xffffffffu, ok)) {
        const int32_t end = ok ? t1 : 0;
#pragma unroll 1
        for (int m = 0; m < 32; ++m) {
            const int32_t e = __shfl_sync(0xffffffffu, end, m);
            if (m < lane && t0 < e) ok = false;
        }
    }
    return ok;
}
// By a block, a sequence a thread (`here`: the thread has one).  `ends`: shared, one per thread, holds the ends of the
// thread's sequences whose own bounds are in order afterwards; `before`: the largest such end of the sequences in
// front.
__device__ __forceinline__ bool block_bounds_ok(bool here, int32_t t0, int32_t t1, int32_t T, int32_t before,
                                                int32_t* ends, int tid) {
    const bool in_order = here && bounds_in_order(t0, t1, T);
    bool ok = in_order && t0 >= before;
    ends[tid] = in_order ? t1 : 0;
    if (!__syncthreads_and(ok || !here))
#pragma unroll 1
        for (int m = 0; m < tid; ++m) ok = ok && t0 >= ends[m];
    return ok;
}

// Workspace layout (all offsets multiples of 256 bytes):
//   [0,256)                      int32 header: [0] total_chunks, [1] total_items
//                                (= total_chunks * Hv), [2] item queue head,
//                                [4] items produced before the state pass starts, [5] 1 once the
//                                producers of the others run, [6] the chunk that the first
//                                chain has come to (two-part route)
//   seq_first[N+1]               int32: first chunk of each sequence (prefix sum); an invalid
//                                sequence has zero chunks and seq_bad[n] = 1
//   seq_bad[N]                   int32
//   chunks[max_chunks]           ChunkInfo
//   seq_by_rank[N]               int32: sequences sorted by chunk count, longest first
//   -- used by the cooperative launch and the two-part route only --
//   rank_of[N]                   int32: the inverse (rank of each sequence)
//   order[max_chunks]            int32: chunk ids in processing order: by position inside the
//                                sequence first, by sequence rank second (so that the records
//                                every state-pass unit needs next are produced first)
//   hist, fill, cnt, pos[max_nc+2]  int32 scratch of the counting sort (max_nc = T/64 + 1); in the two-part route hist
//                                then holds how far in the processing order the second part's producers may go when
//                                the first chain is at a chunk
//   flags[max_chunks][Hv]        uint32: 1 once the record is complete and visible
//   done[N][Hv][2]               uint16: 1 once the two-part route's state pass has finished the half unit
//                                (rank-major, like the unit list); the rest is left to a last launch
//   -- every route --
//   records[max_chunks][Hv]      kRecBytes each
struct WorkspaceLayout {
    size_t seq_first, seq_bad, chunks, seq_by_rank, rank_of, order, hist, fill, cnt, pos, flags,
        done, records, total;
    int32_t max_chunks, max_nc;
};

constexpr int kHdrTotalChunks = 0, kHdrTotalItems = 1, kHdrItemHead = 2, kHdrSplit = 4, kHdrStarted = 5, kHdrProgress = 6;

inline size_t round256(size_t x) { return (x + 255) & ~static_cast<size_t>(255); }

inline WorkspaceLayout workspace_layout(int32_t T, int32_t N, int32_t Hv) {
    WorkspaceLayout w;
    w.max_chunks = T / kChunk + N;
    w.max_nc = T / kChunk + 1;
    const size_t nchunks = static_cast<size_t>(w.max_chunks ? w.max_chunks : 1);
    const size_t nbins = round256(sizeof(int32_t) * (static_cast<size_t>(w.max_nc) + 2));
    w.seq_first = 256;
    w.seq_bad = w.seq_first + round256(sizeof(int32_t) * (static_cast<size_t>(N) + 1));
    w.chunks = w.seq_bad + round256(sizeof(int32_t) * static_cast<size_t>(N ? N : 1));
    w.seq_by_rank = w.chunks + round256(sizeof(ChunkInfo) * nchunks);
    w.rank_of = w.seq_by_rank + round256(sizeof(int32_t) * static_cast<size_t>(N ? N : 1));
    w.order = w.rank_of + round256(sizeof(int32_t) * static_cast<size_t>(N ? N : 1));
    w.hist = w.order + round256(sizeof(int32_t) * nchunks);
    w.fill = w.hist + nbins;
    w.cnt = w.fill + nbins;
    w.pos = w.cnt + nbins;
    w.flags = w.pos + nbins;
    w.done = w.flags + round256(sizeof(uint32_t) * nchunks * Hv);
    w.records = w.done + round256(sizeof(int32_t) * static_cast<size_t>(N ? N : 1) * Hv);
    w.total = w.records + static_cast<size_t>(w.max_chunks) * Hv * kRecBytes;
    return w;
}

struct ChunkedParams {
    PrefillParams p;
    uint8_t* ws;
    WorkspaceLayout lay;
    int32_t longest = 0;      // known_longest(): picks kernels only
};

// Tokens of the longest sequence as far as the host can know them, 0: not at all.  The caller's bound counts only if T
// tokens in N sequences can reach it (empty ones aside): one beyond, a model's context length for example, tells
// nothing.
inline int32_t known_longest(int32_t T, int32_t N, int32_t max_seqlen_hint) {
    if (N == 1) return T;
    return max_seqlen_hint > 0 && max_seqlen_hint <= T - (N - 1) ? max_seqlen_hint : 0;
}

cudaError_t launch_prefill_chunked(const ChunkedParams& cp, cudaStream_t stream);
// One cooperative launch: some CTAs produce the records, the others run the state pass behind them.
cudaError_t launch_prefill_fused(const ChunkedParams& cp, cudaStream_t stream);
// Three launches (for small batches two: no table-building one): CTAs of the state pass walk lists of
// (sequence, v-head) units and stream their records without draining between units.
cudaError_t launch_prefill_stream(const ChunkedParams& cp, cudaStream_t stream);
// Pieces shared by the launchers: the prep kernel that also ranks the sequences by chunk count
// (longest first) and, for the fused launch, orders the chunks and clears the queues and flags;
// the intra-chunk kernel over all items.
// mode 0: chunk table and ranking; 1: + processing order, cleared queue heads and flags (fused
// launch); 2: + the cut of the two-part production (split_permille < 0: the kernel's own model).
cudaError_t launch_prefill_ranked_prep(const ChunkedParams& cp, cudaStream_t stream, int mode,
                                       int split_permille = -1, int sms = 0);
// SMs that a batch in two parts must leave to the producers of the second part, one half unit an SM.
constexpr int kOverlapSpareSms = 8;
// The intra-chunk kernel in two parts around a flag-gated state pass of two CTAs per unit: the second part
// of the records is produced beside the chains, on the SMs the state pass leaves free.  (The three launches where it
// leaves too few.)
cudaError_t launch_prefill_overlap(const ChunkedParams& cp, cudaStream_t stream, int split_permille);

}  // namespace gdn
