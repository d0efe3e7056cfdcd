// Inter-chunk state pass as a PERSISTENT role: a CTA of 512 threads walks a fixed list of
// (sequence, v-head) units and streams their chunk records through one two-stage pipeline that
// does not drain between units.  Two kernels run it: the persistent state pass after the
// intra-chunk kernel (one CTA per SM), and the state CTAs of the fused cooperative launch, whose
// records are produced by other CTAs while the pass runs.
//
// One CTA per unit would pay, for every unit, a launch slot, barrier and TMEM set-up, the first
// record's memory latency and the tail of its last chunk; with thousands of short units (many
// short sequences) that overhead is longer than the chunk steps themselves.  Here
//   * warps 13-15 (loaders) copy records and K tiles in unit order, running up to two chunks ahead
//     of the consumers and straight across unit boundaries (in the fused launch they first wait for
//     each record's flag); a stage is released in three parts and each warp refills one, so that no
//     part waits behind another's release or flag;
//   * warp 12 (issuer) issues every tcgen05.mma;
//   * warps 0-7 (chain) carry the dependent chain  U = U~ - S W^T  ->  D4 = (U decayed)^T K  ->
//     S = e^{b_C} S + D4  and nothing else; U~ is already in the accumulator of S W^T when the
//     product runs (negated B operand), so the chain warps read U itself;
//   * warps 8-11 (output) put U~ of the next chunk into that accumulator and turn
//     Y = diag(scale e^b) (Q S^T) + P U into o rows one chunk behind.  Whatever these warps issue comes out of
//     the chain warps' issue slots, so the rows are made with few instructions (fragment loads,
//     paired conversions, transposing matrix stores).
// The CTA is compiled for 512 threads (128 registers); the chain warps take 144 registers each
// from what the other groups hand back (setmaxnreg).
// The roles never meet at a CTA barrier inside the loop: each derives the same unit list
// (unit = cta + i * n_ctas over the rank-sorted units, longest sequences first) and the same
// running chunk count, from which every mbarrier parity follows.  Every barrier phase is consumed
// by its waiters before the next one can complete (a parity wait cannot tell a barrier that is two
// phases ahead), which is why the state hand-over after a unit's last chunk is omitted rather than
// left unconsumed.
//
// The fp32 master state lives in the chain threads' registers (64 per thread; TMEM lane = state
// row, two column halves).
#pragma once
#include "gdn_prefill_device.cuh"

namespace gdn {

constexpr int kSEpiWarps = 8;                 // warps 0-7: the dependent chain
constexpr int kSEpiThreads = kSEpiWarps * 32;
constexpr int kSOutWarp0 = 8;                 // warps 8-11: output rows (one per TMEM lane quadrant)
constexpr int kSOutThreads = 128;
constexpr int kSIssueWarp = 12;               // warp 12: tcgen05.mma issue
constexpr int kSLoadWarp = 13;                // warps 13-15: record and K-tile copies, one part of a stage each
constexpr int kStreamThreads = 512;
constexpr uint32_t kStreamSmem = 2 * kStageBytes + 16384 + 1024;


// What every role needs to know about one unit; derived identically by each of them.
struct UnitInfo {
    int n, hv, hqk, c_first, nc, seq_t0, seq_len, slot;
    bool skip;          // invalid sequence, padding / out-of-range slot, or no chunks
    bool bad_seq, bad_slot;
};

// After the intra-chunk kernel alone (no order of production to agree on), batches of at most kSmallSeqs sequences: a
// warp of the state pass works the per-sequence table out from cu_seqlens itself, into shared memory.  Behind the
// launch before it a CTA then waits for one round trip to global memory, not for the three of rank -> sequence ->
// first chunk and bounds (1.3 -> 0.6 us; a call of 100 tokens takes 13.5).
struct SeqEntry {       // by rank
    int32_t n, c_first, nc, t0, len, slot, bad, pad;
};

// Which of the rank-sorted units a CTA takes: its first one by its number, then more in passes that turn round, so
// that a CTA that took a long one of a pass takes a short one of the next.  The CTAs whose first unit is longer than
// half the longest are left out of the later passes where the others can do the rest in the longest one's time.
struct UnitWalk {
    int cta, n_ctas, first_later;       // CTAs first_later .. n_ctas - 1 walk the later passes
    __device__ __forceinline__ int at(int i) const {       // i-th unit, or one past the end
        if (i == 0) return cta;
        if (cta < first_later) return 0x7fffffff;
        const int n = n_ctas - first_later, c = cta - first_later;
        return n_ctas + (i - 1) * n + ((i & 1) ? n - 1 - c : c);
    }
};

// By one converged warp, N <= kSmallSeqs; returns UnitWalk::first_later for `per_seq` units a sequence.  The rules are
// the table-building kernels': see warp_bounds_ok; more chunks first, ties by index.
__device__ __forceinline__ int build_seq_table(SeqEntry* tab, const PrefillParams& p, const int lane, const int per_seq,
                                               const int n_ctas) {
    SeqEntry e = {lane, 0, 0, 0, 0, lane, 0, 0};
    int32_t t1 = 0;
    if (lane < p.N) {
        e.t0 = p.cu_seqlens[lane];
        t1 = p.cu_seqlens[lane + 1];
        if (p.slot_idx) e.slot = p.slot_idx[lane];
    }
    e.bad = warp_bounds_ok(e.t0, t1, p.T, lane) ? 0 : 1;
    e.len = t1 - e.t0;
    e.nc = e.bad ? 0 : (e.len + kChunk - 1) / kChunk;
    int32_t incl = e.nc;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += y;
    }
    e.c_first = incl - e.nc;
    int rank = 0;
#pragma unroll 1
    for (int m = 0; m < p.N; ++m) {
        const int32_t nm = __shfl_sync(0xffffffffu, e.nc, m);
        rank += (nm > e.nc || (nm == e.nc && m < lane)) ? 1 : 0;
    }
    if (lane < p.N) tab[rank] = e;
    if (p.N * per_seq <= n_ctas) return 0;          // one pass
    const int longest = __reduce_max_sync(0xffffffffu, e.nc);
    const bool is_long = 2 * e.nc > longest;
    const int n_long = __popc(__ballot_sync(0xffffffffu, is_long)) * per_seq;
    const long long rest = static_cast<long long>(__reduce_add_sync(0xffffffffu, is_long ? 0 : e.nc)) * per_seq;
    return n_long < n_ctas && rest <= static_cast<long long>(longest) * (n_ctas - n_long) ? n_long : 0;
}

// `tab`: that table, or null for the one in the workspace.
__device__ __forceinline__ UnitInfo unit_info(const PrefillParams& p, const uint8_t* ws, const WorkspaceLayout& lay,
                                              const SeqEntry* tab, int unit) {
    UnitInfo u;
    const int rank = unit / p.by_hv;
    u.hv = unit - rank * p.Hv;
    u.hqk = u.hv / p.by_group;
    if (tab) {
        const SeqEntry e = tab[rank];
        u.n = e.n;
        u.c_first = e.c_first;
        u.nc = e.nc;
        u.seq_t0 = e.t0;
        u.seq_len = e.len;
        u.slot = e.slot;
        u.bad_seq = e.bad != 0;
    } else {
        const int32_t* seq_first = reinterpret_cast<const int32_t*>(ws + lay.seq_first);
        const int32_t* seq_bad = reinterpret_cast<const int32_t*>(ws + lay.seq_bad);
        const int32_t* seq_by_rank = reinterpret_cast<const int32_t*>(ws + lay.seq_by_rank);
        u.n = seq_by_rank[rank];
        u.c_first = seq_first[u.n];
        u.nc = seq_first[u.n + 1] - u.c_first;
        u.seq_t0 = p.cu_seqlens[u.n];
        u.seq_len = p.cu_seqlens[u.n + 1] - u.seq_t0;
        u.slot = p.slot_idx ? p.slot_idx[u.n] : u.n;
        u.bad_seq = seq_bad[u.n] != 0;
    }
    u.bad_slot = u.slot < 0 || u.slot >= p.num_slots;
    u.skip = u.bad_seq || u.bad_slot || u.nc == 0;
    return u;
}

constexpr uint32_t kSpinFlagLimit = 1u << 22;

// The state pass of one CTA of 512 threads over its share of the rank-sorted units.  kGated = false: every record
// exists (the intra-chunk kernel ran before).  true: records are being produced by other CTAs of the same cooperative
// launch and the loading warps wait for each record's flag first.  `tmem` = 512 allocated columns; ends with a CTA
// barrier.
template <bool kGated>
__device__ __forceinline__ void state_stream_role(const TensorMaps& maps, const PrefillParams& p,
                                                  uint8_t* ws, const WorkspaceLayout& lay,
                                                  uint8_t* smem, const uint32_t tmem, const int cta,
                                                  const int n_ctas) {
    __shared__ uint64_t bar_full[2], bar_free_a[2], bar_free_b[2], bar_free_c[2], bar_y[2],
        bar_y_read, bar_d1, bar_d4, bar_s, bar_u;
    __shared__ int abort_flag;
    __shared__ uint32_t armed_chunks;     // chunks of the CTA's stream whose copies a loader has started
    // Only the cooperative launch's records carry the scaled Q (gdn_prefill_chunk.cuh).
    constexpr bool kScaledQ = kGated;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int half = (warp >> 2) & 1;                 // which half of the columns this thread owns
    const int dv = (warp & 3) * 32 + lane;            // TMEM lane = state row
    const uint32_t lane_base = static_cast<uint32_t>((warp & 3) * 32) << 16;
    const int total_units = p.N * p.Hv;

    if (tid == 0) {
        mbar_init(&bar_full[0], 3);      // one arrival (and its bytes) per loading warp
        mbar_init(&bar_full[1], 3);
        // A stage is released in three parts as its readers finish with them, so that the next
        // record's copies start up to half a chunk step earlier (one chunk step of look-ahead is
        // shorter than a cold copy): W and Q once S W^T and S Q^T have retired, U~ and the
        // decay vector once every chain warp has read them, P and the K tile once U P^T and the
        // state product have retired.
        for (int st = 0; st < 2; ++st) {
            mbar_init(&bar_free_a[st], 1);
            mbar_init(&bar_free_b[st], kSEpiWarps);
            mbar_init(&bar_free_c[st], 1);
        }
        mbar_init(&bar_d1, 1);
        mbar_init(&bar_d4, 1);
        mbar_init(&bar_y_read, kSOutThreads / 32);      // (raw Q) the output warps have read S Q^T and U P^T
        mbar_init(&bar_y[0], 1);      // one per Y tile: with a single barrier the output warps could
        mbar_init(&bar_y[1], 1);      // find it two phases ahead, which a parity wait cannot tell
        // bar_s: everything the chunk's first product needs is in TMEM: the bf16 state (one arrival
        // per chain warp) and U~ in the accumulator (one per output warp).  The output warps copy
        // U~ only after they have seen the record land and have read Y of two chunks ago, so this one
        // wait also tells the issuing warp that the record is in shared memory (and, with scaled Q, that
        // the Y tile may be overwritten).
        mbar_init(&bar_s, kSEpiWarps + kSOutThreads / 32);
        mbar_init(&bar_u, kSEpiWarps);
        abort_flag = 0;
        armed_chunks = 0;
        fence_barrier_init();
    }
    __shared__ __align__(16) SeqEntry seq_entries[kGated ? 1 : kSmallSeqs];
    const SeqEntry* const seq_tab = !kGated && p.N <= kSmallSeqs ? seq_entries : nullptr;
    if constexpr (!kGated) pdl_wait();     // tables and records are the previous kernels'
    __shared__ int first_later;
    if (warp == kStreamThreads / 32 - 1) {
        const int v = seq_tab ? build_seq_table(seq_entries, p, lane, p.Hv, n_ctas) : 0;
        if (lane == 0) first_later = v;
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    volatile int* abortp = &abort_flag;
    const UnitWalk walk = {cta, n_ctas, first_later};
    auto at = [&](int i) { return walk.at(i); };

    // gc = chunks of earlier units of this CTA; chunk j of the current unit is chunk g = gc + j of
    // the CTA's stream: stage g & 1, phase g >> 1 of bar_full / bar_free_* of that stage, phase g of
    // bar_d1 / bar_d4 / bar_y / bar_u and of bar_s (one state hand-over per chunk: the initial one
    // and one after every chunk but the unit's last).
    uint32_t gc = 0;

    // Register budget: setmaxnreg waits, unbounded, until the registers it asks for have been given
    // back by other warps of the same CTA, so keep room to spare and use multiples of 16.  The CTA
    // starts with 512 x 128; the issuing group gives back 128 x 64, the output warps 128 x 16, the
    // chain warps take 256 x 16.
    if (warp >= kSIssueWarp) {
    reg_dealloc<64>();
    if (warp >= kSLoadWarp) {
        // ===================== loaders: records and K tiles, in stream order
        const int part = warp - kSLoadWarp;
        uint64_t* const bar_free = part == 0 ? bar_free_a : part == 1 ? bar_free_b : bar_free_c;
        if (lane == 0) {
            const size_t rec_stride = static_cast<size_t>(p.Hv) * kRecBytes;
            const uint32_t* flags = reinterpret_cast<const uint32_t*>(ws + lay.flags);
            (void)flags;
            bool live = true;
            // the next unit's table entries are fetched while the current unit is processed
            UnitInfo nxt = unit_info(p, ws, lay, seq_tab, min(cta, total_units - 1));
#pragma unroll 1
            for (int i = 0, unit = cta; unit < total_units && live; unit = at(++i)) {
                const UnitInfo u = nxt;
                nxt = unit_info(p, ws, lay, seq_tab, min(at(i + 1), total_units - 1));
                if (u.skip) continue;
                const uint8_t* records =
                    ws + lay.records + (static_cast<size_t>(u.c_first) * p.Hv + u.hv) * kRecBytes;
#pragma unroll 1
                for (int j = 0; j < u.nc; ++j) {
                    const uint32_t g = gc + j;
                    const int st = g & 1;
                    // the stage held chunk g - 2; each part is refilled as soon as it is free
                    const uint32_t par_free = ((g - 2) >> 1) & 1u;
                    uint8_t* base = smem + st * kStageBytes;
                    const uint8_t* rec = records + j * rec_stride;
                    if constexpr (kGated) {
                        // the record must have been published by its producer CTA
                        const uint32_t* f = flags + (static_cast<size_t>(u.c_first + j) * p.Hv + u.hv);
                        uint32_t v = 0;
                        for (uint32_t k = 0; k < kSpinFlagLimit; ++k) {
                            v = ld_acquire_u32(f);
                            if (v != 0 || *abortp) break;
                            __nanosleep(64);
                        }
                        if (v != 1) {
                            if (*abortp == 0) *abortp = 1;
                            live = false;
                            break;
                        }
                        // No proxy fence here: the producer put one between its generic stores and
                        // the flag's release, which is on the path from those stores to the copies
                        // below; one here would also wait for this thread's copies in flight (3 %
                        // of a long sequence's run time).
                    }
                    if (g >= 2 && !wait_or_abort<40>(&bar_free[st], par_free, abortp)) { live = false; break; }
                    atomicMax(&armed_chunks, g + 1);
                    const int tok = u.seq_t0 + j * kChunk, nb = token_blocks(u.seq_len, j);
                    if (part == 0) {
                        mbar_expect_tx(&bar_full[st], kRecP - kRecW);
                        if constexpr (kScaledQ) {
                            bulk_load(base + kS_Rec + kRecW, rec + kRecW, kRecP - kRecW, &bar_full[st]);
                        } else {
                            bulk_load(base + kS_Rec + kRecW, rec + kRecW, kRecQg - kRecW, &bar_full[st]);
                            tma_load_2d(base + kS_Q, &maps.q, u.hqk * kD, tok, &bar_full[st]);
                            tma_load_2d(base + kS_Q + 8192, &maps.q, u.hqk * kD + 64, tok, &bar_full[st]);
                        }
                    } else if (part == 1) {
                        mbar_expect_tx(&bar_full[st], 2 * nb * kRecUBlock + (kRecBytes - kRecDecay));
                        bulk_load(base + kS_Rec + kRecU, rec + kRecU, nb * kRecUBlock, &bar_full[st]);
                        bulk_load(base + kS_Rec + kRecU + kRecUHalf, rec + kRecU + kRecUHalf, nb * kRecUBlock, &bar_full[st]);
                        bulk_load(base + kS_Rec + kRecDecay, rec + kRecDecay, kRecBytes - kRecDecay, &bar_full[st]);
                    } else {
                        mbar_expect_tx(&bar_full[st], nb * kRecPBlock + 16384);
                        bulk_load(base + kS_Rec + kRecP, rec + kRecP, nb * kRecPBlock, &bar_full[st]);
                        tma_load_2d(base + kS_K, &maps.k, u.hqk * kD, tok, &bar_full[st]);
                        tma_load_2d(base + kS_K + 8192, &maps.k, u.hqk * kD + 64, tok, &bar_full[st]);
                    }
                }
                gc += u.nc;
            }
        }
        __syncwarp();
    } else {
        // ===================== issuer: tensor-core instructions
        {   // the whole warp waits, one elected lane issues a product and its commit
            const uint32_t id64 = make_idesc_bf16(128, 64, false, false);
            const uint32_t id128mn = make_idesc_bf16(128, 128, false, true);
            const uint32_t id64mn = make_idesc_bf16(128, 64, false, true) | kIdescNegateB;
            const uint32_t sRec0 = smem_u32(smem + kS_Rec), sRec1 = sRec0 + kStageBytes;
            const uint64_t dW0 = make_sdesc_sw128(sRec0 + kRecW, 8192, 1024);
            const uint64_t dQ0 = make_sdesc_sw128(sRec0 + kRecQg, 16, 1024);
            const uint64_t dP0 = make_sdesc_sw128(sRec0 + kRecP, 16, 1024);
            const uint64_t dK0 = make_sdesc_sw128(sRec0 + kS_K, 8192, 1024);
            const uint64_t dW1 = make_sdesc_sw128(sRec1 + kRecW, 8192, 1024);
            const uint64_t dQ1 = make_sdesc_sw128(sRec1 + kRecQg, 16, 1024);
            const uint64_t dP1 = make_sdesc_sw128(sRec1 + kRecP, 16, 1024);
            const uint64_t dK1 = make_sdesc_sw128(sRec1 + kS_K, 8192, 1024);
            const uint32_t tS = tmem + kT_S, tD1 = tmem + kT_D1, tD4 = tmem + kT_D4;
            bool live = true;
            // the next unit's table entries are fetched while the current unit is processed
            UnitInfo nxt = unit_info(p, ws, lay, seq_tab, min(cta, total_units - 1));
#pragma unroll 1
            for (int i = 0, unit = cta; unit < total_units && live; unit = at(++i)) {
                const UnitInfo u = nxt;
                nxt = unit_info(p, ws, lay, seq_tab, min(at(i + 1), total_units - 1));
                if (u.skip) continue;
#pragma unroll 1
                for (int j = 0; j < u.nc; ++j) {
                    const uint32_t g = gc + j;
                    const int st = g & 1;
                    const uint64_t w = st ? dW1 : dW0, qg = st ? dQ1 : dQ0, pp = st ? dP1 : dP0,
                                   kk = st ? dK1 : dK0;
                    // Y.  Scaled Q: both terms in one of two tiles.  Raw Q: a tile for each term.
                    const uint32_t tY1 = tmem + kT_Y + (kScaledQ ? 64 * st : 0);
                    const uint32_t tY2 = tmem + kT_Y + (kScaledQ ? 64 * st : 64);
                    if (!warp_wait_or_abort(&bar_s, g & 1u, abortp)) {      // record landed, bf16 S and U~ in TMEM
                        live = false;
                        break;
                    }
                    tc_fence_after_sync();
                    // U = U~ - S W^T  (on the chain): the accumulator holds U~, the B operand is negated;
                    // W is MN-major: k-step ks reads 16 dk rows = 2048 bytes
                    if (elect_one()) {
                        mma_ts_c<true>(tD1, tS, w, id64mn);
                        mma_ts_c<true>(tD1, tS + 8, sdesc_advance(w, 2048), id64mn);
                        mma_ts_c<true>(tD1, tS + 16, sdesc_advance(w, 4096), id64mn);
                        mma_ts_c<true>(tD1, tS + 24, sdesc_advance(w, 6144), id64mn);
                        mma_ts_c<true>(tD1, tS + 32, sdesc_advance(w, 8192), id64mn);
                        mma_ts_c<true>(tD1, tS + 40, sdesc_advance(w, 10240), id64mn);
                        mma_ts_c<true>(tD1, tS + 48, sdesc_advance(w, 12288), id64mn);
                        mma_ts_c<true>(tD1, tS + 56, sdesc_advance(w, 14336), id64mn);
                        mma_commit(&bar_d1);
                    }
                    // S Q^T  (off the chain) overwrites the tile the output warps read two chunks ago (raw Q: one
                    // chunk ago)
                    if (!kScaledQ && g > 0 && !warp_wait_or_abort(&bar_y_read, (g - 1) & 1u, abortp)) {
                        live = false;
                        break;
                    }
                    if (!kScaledQ) tc_fence_after_sync();
                    if (elect_one()) {
                        mma_ts_c<false>(tY1, tS, qg, id64);
                        mma_ts_c<true>(tY1, tS + 8, sdesc_advance(qg, 32), id64);
                        mma_ts_c<true>(tY1, tS + 16, sdesc_advance(qg, 64), id64);
                        mma_ts_c<true>(tY1, tS + 24, sdesc_advance(qg, 96), id64);
                        mma_ts_c<true>(tY1, tS + 32, sdesc_advance(qg, 8192), id64);
                        mma_ts_c<true>(tY1, tS + 40, sdesc_advance(qg, 8192 + 32), id64);
                        mma_ts_c<true>(tY1, tS + 48, sdesc_advance(qg, 8192 + 64), id64);
                        mma_ts_c<true>(tY1, tS + 56, sdesc_advance(qg, 8192 + 96), id64);
                        mma_commit(&bar_free_a[st]);                          // W and Q have been read
                    }
                    if (!warp_wait_or_abort(&bar_u, g & 1u, abortp)) {         // U operands in TMEM
                        live = false;
                        break;
                    }
                    tc_fence_after_sync();
                    // D4 = (U decayed, hi + lo) K   (K tile MN-major: 16 tokens = 2048 bytes)
                    if (elect_one()) {
                        mma_ts_c<false>(tD4, tmem + kT_Us, kk, id128mn);
                        mma_ts_c<true>(tD4, tmem + kT_Us + 8, sdesc_advance(kk, 2048), id128mn);
                        mma_ts_c<true>(tD4, tmem + kT_Us + 16, sdesc_advance(kk, 4096), id128mn);
                        mma_ts_c<true>(tD4, tmem + kT_Us + 24, sdesc_advance(kk, 6144), id128mn);
                        mma_ts_c<true>(tD4, tmem + kT_UsLo, kk, id128mn);
                        mma_ts_c<true>(tD4, tmem + kT_UsLo + 8, sdesc_advance(kk, 2048), id128mn);
                        mma_ts_c<true>(tD4, tmem + kT_UsLo + 16, sdesc_advance(kk, 4096), id128mn);
                        mma_ts_c<true>(tD4, tmem + kT_UsLo + 24, sdesc_advance(kk, 6144), id128mn);
                        mma_commit(&bar_d4);
                    }
                    // U P^T
                    if (elect_one()) {
                        mma_ts_c<kScaledQ>(tY2, tmem + kT_U, pp, id64);
                        mma_ts_c<true>(tY2, tmem + kT_U + 8, sdesc_advance(pp, 32), id64);
                        mma_ts_c<true>(tY2, tmem + kT_U + 16, sdesc_advance(pp, 64), id64);
                        mma_ts_c<true>(tY2, tmem + kT_U + 24, sdesc_advance(pp, 96), id64);
                        mma_commit(&bar_y[st]);
                        mma_commit(&bar_free_c[st]);                          // P and the K tile have been read
                    }
                }
                gc += u.nc;
            }
        }
        __syncwarp();
    }
    } else if (warp < kSEpiWarps) {
        reg_alloc<144>();
        // ===================== chain warps: U and the state refresh (the dependent chain)
        auto hand_over = [&](uint64_t* bar) {     // after tcgen05.st: publish to the issuing lane
            tmem_wait_st();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar);
        };
        float S[64];      // the thread's 64 state columns [64*half, 64*half+64) of row dv, fp32 master
        auto store_state_bf16 = [&]() {           // S (fp32 regs) -> bf16 A operand in TMEM
#pragma unroll
            for (int c0 = 0; c0 < 64; c0 += 32) {
                uint32_t pk[16];
#pragma unroll
                for (int j = 0; j < 16; ++j) pk[j] = pack_bf16(S[c0 + 2 * j], S[c0 + 2 * j + 1]);
                tmem_st16(tmem + kT_S + lane_base + half * 32 + (c0 >> 1), pk);
            }
        };
        bool ok = true;
        // Whole states move between global memory and the chain threads through TMEM, whose fragment
        // shape gives a warp access 8 rows of 32 bytes.  Straight from the threads' own rows it touched
        // 32 rows of 16 bytes, 4100 load/store cycles per state, in front of the next unit (8192 tokens
        // in 57 sequences 246 -> 225 us, with initial states 306 -> 250 us; 100 tokens 18.5 -> 16.9 us).
        // Fragment piece i (0..3): rows 16 (i & 1) .., columns 64 half + 32 (i >> 1) ..
        auto frag_off = [&] { return ((warp & 3) * 32 + (lane >> 2)) * kD + half * 64 + 2 * (lane & 3); };
        auto piece_off = [&](int i, int b, int r) { return ((i & 1) * 16 + 8 * r) * kD + 32 * (i >> 1) + 8 * b; };
        // The final state of the unit before, still in the D4 tile: written once the next unit's first
        // product is on its way (which does not touch that tile; the next state product waits for
        // these warps).
        int pending = -1;
        auto flush = [&] {
            if (pending < 0) return;
            float* out = p.final_state + static_cast<size_t>(pending) * (kD * kD) + frag_off();
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                uint32_t y[16];
                tmem_ld_16x256b_x4(tmem + kT_D4 + lane_base + half * 64 + (static_cast<uint32_t>(i & 1) << 20) +
                                       32 * (i >> 1),
                                   y);
                tmem_wait_ld();
#pragma unroll
                for (int b = 0; b < 4; ++b)
#pragma unroll
                    for (int r = 0; r < 2; ++r)
                        *reinterpret_cast<uint2*>(out + piece_off(i, b, r)) =
                            make_uint2(y[4 * b + 2 * r], y[4 * b + 2 * r + 1]);
            }
            pending = -1;
        };
        // Bounded wait + tcgen05 fence.  `ok` is each warp's own until the unit's last chunk, where the group
        // agrees on it.
        auto await = [&](uint64_t* bar, uint32_t parity) {
            if (!warp_wait_or_abort(bar, parity, abortp)) ok = false;
            tc_fence_after_sync();
        };
        // Every warp runs every group barrier and hand-over below, also after a wait has failed
        // (ok == false), so that no warp is ever left alone at a barrier.  It then works on with whatever
        // is there; nothing of it is written out.  (A branch around each phase costs 60 cycles a
        // chunk step: 32768 tokens at 8 v-heads 793 -> 769 us without them.)
        // A unit's chunks (0: nothing for the chain) and state tile; the rest of its entry is read again
        // where a unit is left out (registers).
        auto brief = [&](int unit) {
            const UnitInfo u = unit_info(p, ws, lay, seq_tab, min(unit, total_units - 1));
            return make_int2(u.skip ? 0 : u.nc, u.slot * p.Hv + u.hv);
        };
        int2 nxt = brief(cta);
#pragma unroll 1
        for (int i = 0, unit = cta; unit < total_units; unit = at(++i)) {
            const int nc = nxt.x, tile = nxt.y;
            nxt = brief(at(i + 1));
            if (nc == 0) {
                const UnitInfo u = unit_info(p, ws, lay, seq_tab, unit);
                const size_t tile_off = (static_cast<size_t>(u.bad_slot ? 0 : u.slot) * p.Hv + u.hv) * (kD * kD) +
                                        static_cast<size_t>(dv) * kD + half * 64;
                if (u.bad_seq) continue;
                if (u.bad_slot) {          // padding / out-of-range slot: zero rows, no state
                    if (u.slot >= p.num_slots && tid == 0) report(p.dev_status, kDevBadSlot);
                    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
                    for (int idx = tid; idx < u.seq_len * 16; idx += kSEpiThreads)
                        *reinterpret_cast<uint4*>(p.o + (static_cast<size_t>(u.seq_t0 + (idx >> 4)) * p.Hv + u.hv) * kD +
                                                  (idx & 15) * 8) = zero;
                } else {                   // empty sequence: the state passes through untouched
#pragma unroll 4
                    for (int j = 0; j < 64; j += 4) {
                        const float4 x = p.init_state
                                             ? *reinterpret_cast<const float4*>(p.init_state + tile_off + j)
                                             : make_float4(0.f, 0.f, 0.f, 0.f);
                        *reinterpret_cast<float4*>(p.final_state + tile_off + j) = x;
                    }
                }
                continue;
            }
            // the unit's initial state
            if (p.init_state) {
                const float* in = p.init_state + static_cast<size_t>(tile) * (kD * kD) + frag_off();
                uint32_t x[4][16];
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int b = 0; b < 4; ++b)
#pragma unroll
                        for (int r = 0; r < 2; ++r) {
                            const uint2 v = *reinterpret_cast<const uint2*>(in + piece_off(i, b, r));
                            x[i][4 * b + 2 * r] = v.x;
                            x[i][4 * b + 2 * r + 1] = v.y;
                        }
                // (through the columns of the decayed U, which the last state product has read)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const uint32_t t = tmem + kT_Us + lane_base + half * 32;
                    tmem_st_16x256b_x4(t, x[2 * h]);
                    tmem_st_16x256b_x4(t + (16u << 16), x[2 * h + 1]);
                    tmem_wait_st();
                    __syncwarp();
                    uint32_t y0[16], y1[16];
                    tmem_ld16(t, y0);
                    tmem_ld16(t + 16, y1);
                    tmem_wait_ld();
                    __syncwarp();
#pragma unroll
                    for (int q = 0; q < 16; ++q) {
                        S[32 * h + q] = __uint_as_float(y0[q]);
                        S[32 * h + 16 + q] = __uint_as_float(y1[q]);
                    }
                }
            } else {
#pragma unroll
                for (int j = 0; j < 64; ++j) S[j] = 0.f;
            }
            store_state_bf16();
            hand_over(&bar_s);
            // the next unit's initial state, towards L2
            if (p.init_state && tid == 0 && nxt.x > 0 && at(i + 1) < total_units)
                bulk_prefetch_l2(p.init_state + static_cast<size_t>(nxt.y) * (kD * kD), kD * kD * 4);
            flush();
#pragma unroll 1
            for (int j = 0; j < nc; ++j) {
                const uint32_t g = gc + j;
                const int st = g & 1;
                const uint8_t* base = smem + st * kStageBytes;
                await(&bar_full[st], (g >> 1) & 1u);
                await(&bar_d1, g & 1u);
                {   // U^T[dv][c] (the accumulator holds U~ - S W^T) for the thread's 32 tokens [32*half, 32*half+32)
                    const float* sdec = reinterpret_cast<const float*>(base + kS_Rec + kRecDecay);
#pragma unroll
                    for (int c0 = 0; c0 < 32; c0 += 16) {
                        const int cb = half * 32 + c0;
                        uint32_t x[16];
                        tmem_ld16(tmem + kT_D1 + lane_base + cb, x);
                        tmem_wait_ld();
                        uint32_t pu[8], ph[8], pl[8];
#pragma unroll
                        for (int q4 = 0; q4 < 4; ++q4) {
                            const float4 dd = *reinterpret_cast<const float4*>(sdec + cb + 4 * q4);
                            const float u0 = __uint_as_float(x[4 * q4 + 0]);
                            const float u1 = __uint_as_float(x[4 * q4 + 1]);
                            const float u2 = __uint_as_float(x[4 * q4 + 2]);
                            const float u3 = __uint_as_float(x[4 * q4 + 3]);
                            const float s0 = u0 * dd.x, s1 = u1 * dd.y, s2 = u2 * dd.z, s3 = u3 * dd.w;
                            pu[2 * q4] = pack_bf16(u0, u1);
                            pu[2 * q4 + 1] = pack_bf16(u2, u3);
                            ph[2 * q4] = pack_bf16(s0, s1);
                            ph[2 * q4 + 1] = pack_bf16(s2, s3);
                            pl[2 * q4] = pack_bf16(s0 - __uint_as_float(ph[2 * q4] << 16),
                                                   s1 - __uint_as_float(ph[2 * q4] & 0xffff0000u));
                            pl[2 * q4 + 1] = pack_bf16(s2 - __uint_as_float(ph[2 * q4 + 1] << 16),
                                                       s3 - __uint_as_float(ph[2 * q4 + 1] & 0xffff0000u));
                        }
                        tmem_st8(tmem + kT_Us + lane_base + (cb >> 1), ph);
                        tmem_st8(tmem + kT_UsLo + lane_base + (cb >> 1), pl);
                        tmem_st8(tmem + kT_U + lane_base + (cb >> 1), pu);
                    }
                }
                const float gC = reinterpret_cast<const float*>(base + kS_Rec + kRecGammaC)[0];
                hand_over(&bar_u);
                if (lane == 0) mbar_arrive(&bar_free_b[st]);    // this warp has read U~, decay, e^{b_C}
                const bool last = j + 1 == nc;
                await(&bar_d4, g & 1u);
                {   // S <- e^{b_C} S + D4 on the thread's 64 dk columns
#pragma unroll
                    for (int c0 = 0; c0 < 64; c0 += 32) {
                        uint32_t xa[16], xb[16];
                        tmem_ld16(tmem + kT_D4 + lane_base + half * 64 + c0, xa);
                        tmem_ld16(tmem + kT_D4 + lane_base + half * 64 + c0 + 16, xb);
                        tmem_wait_ld();
#pragma unroll
                        for (int jj = 0; jj < 16; ++jj) {
                            S[c0 + jj] = fmaf(gC, S[c0 + jj], __uint_as_float(xa[jj]));
                            S[c0 + 16 + jj] = fmaf(gC, S[c0 + 16 + jj], __uint_as_float(xb[jj]));
                        }
                    }
                }
                if (last) {
                    // nothing of a unit is written after a failed wait
                    ok = group_all<2, kSEpiThreads>(ok);
                    if (ok) {
#pragma unroll
                        for (int c0 = 0; c0 < 64; c0 += 8) {
                            uint32_t y[8];
#pragma unroll
                            for (int q = 0; q < 8; ++q) y[q] = __float_as_uint(S[c0 + q]);
                            tmem_st8(tmem + kT_D4 + lane_base + half * 64 + c0, y);
                        }
                        tmem_wait_st();
                        __syncwarp();
                        pending = tile;
                    }
                } else {
                    store_state_bf16();          // the next chunk's A operand
                    hand_over(&bar_s);
                }
            }
            gc += nc;
        }
        flush();
    } else {
        reg_dealloc<112>();
        // ===================== output warps: Y = scale e^b (S Q^T) + U P^T (fp32, TMEM) -> o rows.  Warp 8 + q
        // reads TMEM lanes 32 q .. 32 q + 31 (dv indices), scales and rounds, transposes through
        // shared memory, and the four warps write whole rows in 16-byte pieces.
        const int q4 = warp & 3;
        const uint32_t olane = static_cast<uint32_t>(q4 * 32) << 16;
        const int ot = tid - kSOutWarp0 * 32;
        const size_t tok_stride = static_cast<size_t>(p.Hv) * kD;
        auto out_sync = [] { asm volatile("bar.sync 1, %0;" ::"n"(kSOutThreads) : "memory"); };
        // As in the chain warps: each warp's own, and after a failed wait the work goes on with whatever is there; only
        // the stores of rows depend on it.
        bool ok = true;
        auto await = [&](uint64_t* bar, uint32_t parity) {
            if (ok) ok = wait_or_abort<40>(bar, parity, abortp);
            __syncwarp();
        };
        // U~ (fp32, 32 KB per chunk) reaches the chain through the accumulator of S W^T: this group
        // copies it from the record into TMEM one chunk ahead, the product then subtracts S W^T
        // from it (negated B operand), and the chain warps read U itself.  (Read by the chain warps
        // from shared memory, the 32 KB took 300 of the 3700 cycles of a chunk step.)
        const int odv = q4 * 32 + lane;
        // (raw Q) the chunk's scale e^{b_r} outlives its stage: a copy per warp, two chunks deep
        __shared__ __align__(8) float s_eb[kScaledQ ? 1 : kSOutThreads / 32][2][kChunk];
        auto preload = [&](uint32_t gq) {       // chunk gq of the CTA's stream -> accumulator
            const int sq = gq & 1;
            await(&bar_full[sq], (gq >> 1) & 1u);
            if constexpr (!kScaledQ)
                *reinterpret_cast<float2*>(&s_eb[q4][sq][2 * lane]) = *reinterpret_cast<const float2*>(
                    smem + sq * kStageBytes + kS_Rec + kRecEb + 8 * lane);
            const float4* sU = reinterpret_cast<const float4*>(smem + sq * kStageBytes + kS_Rec + kRecU +
                                                                   (odv >> 6) * kRecUHalf);
            const int nb = record_blocks(smem + sq * kStageBytes + kS_Rec + kRecGammaC + 4);
#pragma unroll
            for (int c0 = 0; c0 < 64; c0 += 32) {       // eight reads in flight
                uint32_t r[2][16];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const float4 v = sU[rec_u_index((c0 >> 2) + q, odv & 63)];
                    uint32_t(&x)[16] = r[q >> 2];
                    x[4 * (q & 3)] = __float_as_uint(v.x); x[4 * (q & 3) + 1] = __float_as_uint(v.y);
                    x[4 * (q & 3) + 2] = __float_as_uint(v.z); x[4 * (q & 3) + 3] = __float_as_uint(v.w);
                }
                tmem_st16(tmem + kT_D1 + olane + c0, r[0]);
                tmem_st16(tmem + kT_D1 + olane + c0 + 16, r[1]);
            }
            // blocks without tokens were not copied: whatever was there is replaced
#pragma unroll 1
            for (int b = nb; b < 4; ++b) {
                const uint32_t zero[16] = {};
                tmem_st16(tmem + kT_D1 + olane + 16 * b, zero);
            }
            tmem_wait_st();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_s);
        };
        bool preloaded = false;     // U~ of the chunk about to be processed is already in place
        UnitInfo nxt = unit_info(p, ws, lay, seq_tab, min(cta, total_units - 1));
#pragma unroll 1
        for (int i = 0, unit = cta; unit < total_units; unit = at(++i)) {
            const UnitInfo u = nxt;
            nxt = unit_info(p, ws, lay, seq_tab, min(at(i + 1), total_units - 1));
            if (u.skip) continue;
#pragma unroll 1
            for (int j = 0; j < u.nc; ++j) {
                const uint32_t g = gc + j;
                const int buf = g & 1;
                // k = 0: this chunk's U~ (first chunk of the stream, or after a skipped unit).
                // k = 1: once the chain warps have read U of this chunk the accumulator is free for
                // the next chunk's U~ (when the next chunk is known without looking past a skipped
                // unit), which is then in place long before the chain warps hand the state over.
                const bool ahead = j + 1 < u.nc || (at(i + 1) < total_units && !nxt.skip);
#pragma unroll 1
                for (int k = preloaded ? 1 : 0; k < 2; ++k) {
                    if (k == 1) {
                        await(&bar_u, g & 1u);
                        tc_fence_after_sync();
                        if (!ahead) break;
                    }
                    preload(g + k);
                }
                preloaded = ahead;
                // every warp runs both group barriers of every chunk, also after a failed wait
                if (ot == 0) bulk_wait_read_all();       // the last chunk's rows have left the staging tile
                out_sync();
                await(&bar_y[buf], (g >> 1) & 1u);
                tc_fence_after_sync();
                // The tile (lanes = dv, columns = tokens) is read as accumulator fragments (lane 4 x + t holds columns
                // 8 i + 2 t, + 1; raw Q: both tiles, and added), rounded in pairs and stored transposed, 8 dv of one
                // token per 16 bytes, into a [token][dv] tile of two 128B-swizzled halves of 64 dv (what these warps
                // issue comes out of the chain warps' issue slots).
                {
                    const int dv0 = q4 * 32 + 8 * (lane >> 3);         // the 8 dv this lane's address covers
                    const uint32_t dst = smem_u32(smem + kS_Out) + (dv0 >> 6) * 8192;
#pragma unroll
                    for (int c = 0; c < 2; ++c) {        // 32 columns at a time
                        float2 eb[4];
                        if constexpr (!kScaledQ) {
#pragma unroll
                            for (int i = 0; i < 4; ++i)
                                eb[i] = *reinterpret_cast<const float2*>(&s_eb[q4][buf][2 * (lane & 3) + 8 * (4 * c + i)]);
                        }
                        uint32_t pk[2][8];               // packed pairs: lanes 0-15 / 16-31 of the quadrant
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            uint32_t y1[16], y2[16];
                            const uint32_t at = tmem + kT_Y + olane + (static_cast<uint32_t>(h) << 20) + 32 * c;
                            tmem_ld_16x256b_x4(at + (kScaledQ ? 64 * buf : 0), y1);
                            if constexpr (!kScaledQ) tmem_ld_16x256b_x4(at + 64, y2);
                            tmem_wait_ld();
#pragma unroll
                            for (int i = 0; i < 8; ++i) {
                                float2 y = make_float2(__uint_as_float(y1[2 * i]), __uint_as_float(y1[2 * i + 1]));
                                if constexpr (!kScaledQ)
                                    y = fma2(eb[i >> 1], y, make_float2(__uint_as_float(y2[2 * i]), __uint_as_float(y2[2 * i + 1])));
                                pk[h][i] = pack_bf16(y.x, y.y);
                            }
                        }
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            stmatrix_x4_trans(dst + sw128_offset(8 * (4 * c + i) + (lane & 7), (dv0 & 63) >> 3),
                                              pk[0][2 * i], pk[0][2 * i + 1], pk[1][2 * i], pk[1][2 * i + 1]);
                    }
                }
                tc_fence_before_sync();
                fence_proxy_async_smem();
                __syncwarp();
                if (!kScaledQ && lane == 0) mbar_arrive(&bar_y_read);
                out_sync();
                const int len = min(kChunk, u.seq_len - j * kChunk), tok = u.seq_t0 + j * kChunk;
                if (len == kChunk) {
                    if (ot == 0 && ok) {     // two tiled copies (16-byte loops of the group's threads took 960 cycles)
                        tma_store_2d(&maps.o, u.hv * kD, tok, smem + kS_Out);
                        tma_store_2d(&maps.o, u.hv * kD + 64, tok, smem + kS_Out + 8192);
                        bulk_commit();
                    }
                } else if (ok) {             // a ragged tail: the rows behind it are another sequence's
                    const int piece = ot & 15;
                    const uint8_t* src = smem + kS_Out + (piece >> 3) * 8192;
                    __nv_bfloat16* og = p.o + (static_cast<size_t>(tok) * p.Hv + u.hv) * kD + piece * 8;
                    for (int row = ot >> 4; row < len; row += 8)
                        *reinterpret_cast<uint4*>(og + row * tok_stride) =
                            *reinterpret_cast<const uint4*>(src + sw128_offset(row, piece & 7));
                }
            }
            gc += u.nc;
        }
        if (ot == 0) bulk_wait_all();        // before the CTA's shared memory goes away
    }

    tc_fence_before_sync();
    __syncthreads();
    if (abort_flag != 0 && warp == kSIssueWarp && lane == 0) {
        report(p.dev_status, kDevTimeout);
        // let copies already in flight land before the CTA's shared memory goes away: the last two
        // chunks a loader started, each on its stage's barrier at that chunk's own parity
        const uint32_t armed = *reinterpret_cast<volatile uint32_t*>(&armed_chunks);
        for (uint32_t back = 1; back <= 2 && back <= armed; ++back) {
            const uint32_t gq = armed - back;
            mbar_wait(&bar_full[gq & 1], (gq >> 1) & 1u, 1u << 12);
        }
    }
}

}  // namespace gdn
