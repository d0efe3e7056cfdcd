// Inter-chunk state pass with TWO CTAs per (sequence, v-head) unit, each carrying 64 of the 128 state rows.
//
// The rows of the state evolve independently (U = U~ - S W^T and S' = e^{b_C} S + (U decayed)^T K act on each dv
// row alone), so a unit can be cut along dv.  The chain of a chunk step is two tensor-core products and two passes
// over their results; the passes are bound by what the CTA's four schedulers can issue and by the tiles' way
// through TMEM, so half the rows take about half the time there, and so does the state product (below).  The CTA
// copies the same W, Q, K and P as a whole unit's would and half of U~.
//
// Everything 64 rows wide lies in TMEM as M = 64 tiles do: 16 rows in the lower 16 lanes of each of the four lane
// quadrants.  The fragment shapes (16x256b for fp32, 16x128b for packed bf16 pairs) spread such a quadrant over all 32
// lanes of a warp, so no lane idles, and they agree: what one loads as fp32 pairs the other stores as bf16 pairs.  The
// decayed U enters the state product as bf16 hi + lo: hi goes to the lower, lo to the upper 16 lanes, so that one
// M = 128 product of four instructions forms both terms (an M = 64 instruction takes as long as an M = 128 one: eight
// of them for hi and lo apart would take twice as long); the chain warps add the two halves of the result.
//
// The roles, their barriers and the unit order are those of gdn_prefill_stream.cuh, with these differences: the fp32
// master state is held as fragments (32 registers a thread), so whole states cross to and from global memory directly,
// 8 rows of 32 bytes an access; the bf16 state is double-buffered, so the outputs' products may read the last
// one while the next is stored; and a CTA's list of half units turns round at each pass over the CTAs (a CTA that took a long one of a pass
// takes a short one of the next).
#pragma once
#include "gdn_prefill_stream.cuh"

namespace gdn {

constexpr int kHalfRows = kD / 2;
// warps 0-7 chain, 8-11 outputs, 12 and 13 issuers, 14 loader
constexpr int kHLoadWarp = 14;
// Three rings, each filled and released by itself: W with the Q tile, the K tile with P, half of U~ with the vectors
// (two places: U~ goes on to TMEM a chunk ahead).
constexpr int kHStages = 3;
constexpr uint32_t kHA_W = 0, kHA_Q = 16384, kHABytes = 32768;
constexpr uint32_t kHC_K = 0, kHC_P = 16384, kHCBytes = 24576;
constexpr uint32_t kHB_U = 0, kHB_Vec = kRecUHalf, kHBBytes = kRecUHalf + 1024;
static_assert(kHB_Vec + (kRecBytes - kRecDecay) <= kHBBytes, "the vectors fit");
constexpr uint32_t kHS_A = 0, kHS_C = kHS_A + kHStages * kHABytes, kHS_B = kHS_C + kHStages * kHCBytes;
constexpr uint32_t kHS_Out = kHS_B + 2 * kHBBytes;              // o staging, two tiles [64 tokens][64 dv] bf16
constexpr uint32_t kHalfSmem = kHS_Out + 2 * 8192 + 1024;
// TMEM columns: S W^T, S Q^T, U P^T, the state product, bf16 S (of odd chunks, of even ones: the next is stored while S Q^T
// still reads the last), decayed U (hi / lo lanes), U
constexpr uint32_t kH_D1 = 0, kH_Y1 = 128, kH_Y2 = 192, kH_D4 = 256, kH_SOdd = 64, kH_SEven = 384, kH_Us = 448, kH_U = 480;
__device__ __forceinline__ uint32_t half_s_col(uint32_t g) { return g & 1 ? kH_SOdd : kH_SEven; }

// Polls of a record's flag, about 0.4 us each.  A few milliseconds: far longer than the producers ever lag
// when they do run beside the state pass, far shorter than the other roles' mbarrier waits (which would report an
// error).  And how long to wait if they have not even started: two launches in a row start within some ten
// microseconds of each other unless another stream's kernel holds the SMs between them (32768 tokens beside 57
// sequences on a second stream: at half this limit the chains give up for that).  What is lost by giving up too early
// is no more than the chain has done so far.
constexpr uint32_t kSpinFlagLimitSoft = 1u << 13, kSpinStartLimit = 1u << 9;

// Which records exist when the state pass starts.
enum HalfMode {
    kHalfAll,       // every one (the intra-chunk kernel ran before)
    kHalfGated,     // those of the first hdr[kHdrSplit] items of the processing order; the others are being produced by a
                    // concurrent kernel and are waited for.  A wait that runs out ends the CTA's work without an error
                    // (the half units it has finished are marked in the done table, the others are left to a later
                    // launch).
    kHalfRest       // every one, by that later launch: the half units marked done are left out
};

// The state pass of one CTA of 512 threads over its share of the rank-sorted half units.  `tmem` = 512 allocated
// columns; ends with a CTA barrier.
template <HalfMode kMode>
__device__ __forceinline__ void state_half_role(const TensorMaps& maps, const PrefillParams& p, uint8_t* ws,
                                                const WorkspaceLayout& lay, uint8_t* smem, const uint32_t tmem,
                                                const int cta, const int n_ctas) {
    __shared__ uint64_t bar_full_a[kHStages], bar_full_b[2], bar_full_c[kHStages], bar_free_a[kHStages], bar_free_b[2],
        bar_free_c[kHStages], bar_y[2], bar_p[2], bar_y_read, bar_d1, bar_d4[2], bar_s[2][2], bar_u,
        bar_drain[2];
    __shared__ int abort_flag;
    __shared__ uint32_t armed[3];         // chunks of the CTA's stream whose copies the loader has started, per ring
    // kHalfGated waits for records of a launch that may not be running beside this one: there no
    // wait that runs out is an error, whichever role it happens in (the loader's own wait for a
    // flag is the shortest, but the limits are counted in polls, not in time): the half units this CTA
    // has not finished are left to the last launch, which reports real failures.
    constexpr int kWaitReason = kMode == kHalfGated ? 2 : 1;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g8 = lane >> 2, t4 = lane & 3;          // fragment coordinates: row g8 (and + 8), column pair t4
    const uint32_t lane_base = static_cast<uint32_t>((warp & 3) * 32) << 16;
    const int total = 2 * p.N * p.Hv;                 // half units, rank-sorted: 2 unit + half
    uint16_t* done = reinterpret_cast<uint16_t*>(ws + lay.done);     // a mark per half unit
    auto is_done = [&](int hu) { return kMode == kHalfRest && done[hu] != 0; };

    if (tid == 0) {
        for (int st = 0; st < 2; ++st) {
            mbar_init(&bar_full_b[st], 1);
            mbar_init(&bar_free_b[st], kSEpiWarps);
            mbar_init(&bar_y[st], 1);
            mbar_init(&bar_p[st], kSOutThreads / 32); // U~ in the accumulator
            mbar_init(&bar_drain[st], 1);             // an issuer that gave up: its products
            mbar_init(&bar_d4[st], 1);                // by halves of dk
            for (int h = 0; h < 2; ++h)               // the bf16 state in TMEM, by odd and even chunks and halves of dk
                mbar_init(&bar_s[st][h], kSEpiWarps / 2);
        }
        for (int st = 0; st < kHStages; ++st) {
            mbar_init(&bar_full_a[st], 1);
            mbar_init(&bar_full_c[st], 1);
            mbar_init(&bar_free_a[st], 2);            // a product of either issuer
            mbar_init(&bar_free_c[st], 1);
        }
        mbar_init(&bar_d1, 1);
        mbar_init(&bar_y_read, kSOutThreads / 32);
        mbar_init(&bar_u, kSEpiWarps);
        abort_flag = 0;
        armed[0] = armed[1] = armed[2] = 0;
        fence_barrier_init();
    }
    // (the two parts go by the order of production in the workspace)
    __shared__ __align__(16) SeqEntry seq_entries[kMode == kHalfAll ? kSmallSeqs : 1];
    const SeqEntry* const seq_tab = kMode == kHalfAll && p.N <= kSmallSeqs ? seq_entries : nullptr;
    if constexpr (kMode == kHalfAll) pdl_wait();     // tables and records are the previous kernels'
    __shared__ int first_later;
    if (warp > kHLoadWarp) {
        const int v = seq_tab ? build_seq_table(seq_entries, p, lane, 2 * p.Hv, n_ctas) : 0;
        if (lane == 0) first_later = v;
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    volatile int* abortp = &abort_flag;

    // Every role walks the CTA's list of half units.
    const UnitWalk walk = {cta, n_ctas, first_later};
    auto at = [&](int i) { return walk.at(i); };
    auto info = [&](int hu) { return unit_info(p, ws, lay, seq_tab, min(hu, total - 1) >> 1); };
    // chunks of earlier units of this CTA; chunk j of the current one is chunk g = gc + j of the CTA's stream: stage
    // g & 1, phase g >> 1 of the barriers that come in pairs, phase g of the others and of bar_d4's two, which are halves
    // of one chunk's product
    uint32_t gc = 0;

    // place and parity of a chunk's use in the three-place rings
    struct Ring {
        int st = 0;
        uint32_t par = 0;
        __device__ __forceinline__ void next() {
            if (++st == kHStages) {
                st = 0;
                par ^= 1u;
            }
        }
    } ring;

    if (warp == kHLoadWarp) {
        // ===================== loader: records and Q, K tiles, in stream order; a stage's parts in the order in which
        // the chunk before last releases them
        const size_t rec_stride = static_cast<size_t>(p.Hv) * kRecBytes;
        const uint32_t* flags = reinterpret_cast<const uint32_t*>(ws + lay.flags);
        const int32_t* pos = reinterpret_cast<const int32_t*>(ws + lay.pos);
        const int32_t cut = kMode == kHalfGated ? reinterpret_cast<const int32_t*>(ws)[kHdrSplit] : 0;
        (void)flags;
        (void)pos;
        (void)cut;
        volatile int32_t* progress = reinterpret_cast<int32_t*>(ws) + kHdrProgress;
        (void)progress;
        uint32_t started = 0;           // (kHalfGated) the producers have been seen to run
        (void)started;
        bool live = true;
        UnitInfo nxt = info(at(0));
#pragma unroll 1
        for (int i = 0, hu = at(0); hu < total && live; hu = at(++i)) {
            const UnitInfo u = nxt;
            nxt = info(at(i + 1));
            if (u.skip || is_done(hu)) continue;
            const uint8_t* rec = ws + lay.records + (static_cast<size_t>(u.c_first) * p.Hv + u.hv) * kRecBytes;
            const uint32_t u_off = kRecU + (hu & 1) * kRecUHalf;
            const int32_t rank = (hu >> 1) / p.by_hv;
            int32_t pos_j = kMode == kHalfGated ? pos[0] : 0;       // fetched one chunk ahead
#pragma unroll 1
            for (int j = 0; j < u.nc; ++j, rec += rec_stride) {
                const uint32_t g = gc + j;
                if constexpr (kMode == kHalfGated) {
                    const bool gated = (pos_j + rank) * p.Hv + u.hv >= cut;
                    pos_j = pos[j + 1];                     // pos has an entry past the longest chain
                    if (gated) {
                        // (no proxy fence behind the acquire: see state_stream_role)
                        const uint32_t* f = flags + (static_cast<size_t>(u.c_first + j) * p.Hv + u.hv);
                        uint32_t v = 0;
#pragma unroll 1
                        for (uint32_t k = 0; k < kSpinFlagLimitSoft; ++k) {
                            v = __shfl_sync(0xffffffffu, ld_acquire_u32(f), 0);
                            if (v != 0 || __any_sync(0xffffffffu, *abortp)) break;
                            if (k >= kSpinStartLimit && !started) {
                                const uint32_t* word = reinterpret_cast<const uint32_t*>(ws) + kHdrStarted;
                                started = __shfl_sync(0xffffffffu, ld_acquire_u32(word), 0);
                                if (!started) break;
                            }
                            __nanosleep(64);
                        }
                        if (v != 1) {
                            if (*abortp == 0) *abortp = v == 0 ? 2 : 1;
                            live = false;
                            break;
                        }
                    }
                }
                const int tok = u.seq_t0 + j * kChunk, nb = token_blocks(u.seq_len, j);
                const int sb = g & 1;
                uint8_t* const b_at = smem + kHS_B + sb * kHBBytes;
                uint8_t* const a_at = smem + kHS_A + ring.st * kHABytes;
                uint8_t* const c_at = smem + kHS_C + ring.st * kHCBytes;
                // (parity of the use before: a ring's first uses find the barrier's "previous" phase complete)
                if (!(live = warp_wait(&bar_free_b[sb], ~(g >> 1) & 1u, abortp, kWaitReason))) break;
                if (elect_one()) {
                    armed[1] = g + 1;
                    mbar_expect_tx(&bar_full_b[sb], nb * kRecUBlock + (kRecBytes - kRecDecay));
                    bulk_load(b_at + kHB_U, rec + u_off, nb * kRecUBlock, &bar_full_b[sb]);
                    bulk_load(b_at + kHB_Vec, rec + kRecDecay, kRecBytes - kRecDecay, &bar_full_b[sb]);
                }
                if (!(live = warp_wait(&bar_free_a[ring.st], ring.par ^ 1u, abortp, kWaitReason))) break;
                if (elect_one()) {
                    armed[0] = g + 1;
                    mbar_expect_tx(&bar_full_a[ring.st], kHABytes);
                    bulk_load(a_at + kHA_W, rec + kRecW, 16384, &bar_full_a[ring.st]);
                    tma_load_2d(a_at + kHA_Q, &maps.q, u.hqk * kD, tok, &bar_full_a[ring.st]);
                    tma_load_2d(a_at + kHA_Q + 8192, &maps.q, u.hqk * kD + 64, tok, &bar_full_a[ring.st]);
                }
                if (!(live = warp_wait(&bar_free_c[ring.st], ring.par ^ 1u, abortp, kWaitReason))) break;
                if (elect_one()) {
                    armed[2] = g + 1;
                    mbar_expect_tx(&bar_full_c[ring.st], 16384 + nb * kRecPBlock);
                    bulk_load(c_at + kHC_P, rec + kRecP, nb * kRecPBlock, &bar_full_c[ring.st]);
                    tma_load_2d(c_at + kHC_K, &maps.k, u.hqk * kD, tok, &bar_full_c[ring.st]);
                    tma_load_2d(c_at + kHC_K + 8192, &maps.k, u.hqk * kD + 64, tok, &bar_full_c[ring.st]);
                }
                ring.next();
                if (kMode == kHalfGated && cta == 0 && lane == 0) *progress = j;     // (paces the producers)
            }
            gc += u.nc;
        }
        if (kMode == kHalfGated && cta == 0 && lane == 0) *progress = 0x7fffffff;
        __syncwarp();
    } else if (warp > kHLoadWarp) {
        // one warp to spare
    } else if (warp >= kSIssueWarp) {
        // ===================== issuers: the whole warp waits, one elected lane issues.  Two warps: S W^T; and, in this order,
        // the state product, S Q^T and U P^T.  The products run in the order of issue, so the outputs' two run while the
        // chain warps are at the state, and neither in front of a product of the chain's nor beside it: with S Q^T right
        // behind S W^T (beside the U phase, which is shorter) the state product came 130 cycles later.
        const bool outputs = warp > kSIssueWarp;
        const uint32_t id_w = make_idesc_bf16(64, 64, false, true) | kIdescNegateB;
        const uint32_t id_qp = make_idesc_bf16(64, 64, false, false);
        const uint32_t id_k = make_idesc_bf16(128, 64, false, true);
        const uint32_t s0 = smem_u32(smem);
        bool live = true;
        UnitInfo nxt = info(at(0));
        for (int i = 0, hu = at(0); hu < total && live; hu = at(++i)) {
            const UnitInfo u = nxt;
            nxt = info(at(i + 1));
            if (u.skip || is_done(hu)) continue;
            if (!outputs) {
                const uint64_t dW0 = make_sdesc_sw128(s0 + kHS_A + kHA_W, 8192, 1024);
#pragma unroll 1
                for (int j = 0; j < u.nc; ++j, ring.next()) {
                    const uint32_t g = gc + j;
                    const uint64_t w = sdesc_advance(dW0, ring.st * kHABytes);
                    const uint32_t tD1 = tmem + kH_D1, tS = tmem + half_s_col(g);
                    if (!warp_wait(&bar_full_a[ring.st], ring.par, abortp, kWaitReason) ||
                        !warp_wait(&bar_p[g & 1], (g >> 1) & 1u, abortp, kWaitReason) ||      // U~ in place
                        !warp_wait(&bar_s[g & 1][0], (g >> 1) & 1u, abortp, kWaitReason)) {                 // bf16 S in TMEM, dk 0-63
                        live = false;
                        break;
                    }
                    tc_fence_after_sync();
                    // U = U~ - S W^T; W is MN-major: k-step ks reads 16 dk rows = 2048 bytes
                    if (elect_one()) {
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks)
                            mma_ts_c<true>(tD1, tS + 8 * ks, sdesc_advance(w, 2048 * ks), id_w);
                    }
                    if (!warp_wait(&bar_s[g & 1][1], (g >> 1) & 1u, abortp, kWaitReason)) {                 // dk 64-127
                        live = false;
                        break;
                    }
                    tc_fence_after_sync();
                    if (elect_one()) {
#pragma unroll
                        for (int ks = 4; ks < 8; ++ks)
                            mma_ts_c<true>(tD1, tS + 8 * ks, sdesc_advance(w, 2048 * ks), id_w);
                        mma_commit(&bar_d1);
                        mma_commit(&bar_free_a[ring.st]);                     // W has been read
                    }
                }
            } else {
                const uint64_t dQ0 = make_sdesc_sw128(s0 + kHS_A + kHA_Q, 16, 1024), dP0 = make_sdesc_sw128(s0 + kHS_C + kHC_P, 16, 1024),
                               dK0 = make_sdesc_sw128(s0 + kHS_C + kHC_K, 8192, 1024);
                const uint32_t tY1 = tmem + kH_Y1, tY2 = tmem + kH_Y2, tU = tmem + kH_U, tD4 = tmem + kH_D4, tUs = tmem + kH_Us;
#pragma unroll 1
                for (int j = 0; j < u.nc; ++j, ring.next()) {
                    const uint32_t g = gc + j, tS = tmem + half_s_col(g);
                    const uint64_t q = sdesc_advance(dQ0, ring.st * kHABytes), pp = sdesc_advance(dP0, ring.st * kHCBytes),
                                   kk = sdesc_advance(dK0, ring.st * kHCBytes);
                    if (!warp_wait(&bar_full_c[ring.st], ring.par, abortp, kWaitReason) ||
                        !warp_wait(&bar_u, g & 1u, abortp, kWaitReason)) {        // U operands in TMEM
                        live = false;
                        break;
                    }
                    tc_fence_after_sync();
                    if (elect_one()) {
                        // (U decayed) K, hi and lo terms in the lower and upper lanes (K tile MN-major: 16 tokens = 2048
                        // bytes)
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            mma_ts_c<false>(tD4 + 64 * h, tUs, sdesc_advance(kk, 8192 * h), id_k);
#pragma unroll
                            for (int ks = 1; ks < 4; ++ks)
                                mma_ts_c<true>(tD4 + 64 * h, tUs + 8 * ks, sdesc_advance(kk, 8192 * h + 2048 * ks), id_k);
                            mma_commit(&bar_d4[h]);
                        }
                    }
                    // S Q^T (its tile has landed with W's), into the tile that the output warps read a chunk ago
                    if (g > 0 && !warp_wait(&bar_y_read, (g - 1) & 1u, abortp, kWaitReason)) {
                        live = false;
                        break;
                    }
                    tc_fence_after_sync();
                    if (elect_one()) {
                        mma_ts_c<false>(tY1, tS, q, id_qp);
#pragma unroll
                        for (int ks = 1; ks < 8; ++ks)
                            mma_ts_c<true>(tY1, tS + 8 * ks, sdesc_advance(q, (ks >> 2) * 8192 + (ks & 3) * 32), id_qp);
                        mma_commit(&bar_free_a[ring.st]);                     // Q has been read
                        // U P^T
                        mma_ts_c<false>(tY2, tU, pp, id_qp);
#pragma unroll
                        for (int ks = 1; ks < 4; ++ks)
                            mma_ts_c<true>(tY2, tU + 8 * ks, sdesc_advance(pp, 32 * ks), id_qp);
                        mma_commit(&bar_y[g & 1]);
                        mma_commit(&bar_free_c[ring.st]);                     // K and P have been read
                    }
                }
            }
            gc += u.nc;
        }
        __syncwarp();
        if (!live) {        // products still running read shared memory and TMEM that the CTA is about to give back
            if (elect_one()) mma_commit(&bar_drain[outputs]);
            mbar_wait(&bar_drain[outputs], 0u, 1u << 12);
            __syncwarp();
        }
    } else if (warp < kSEpiWarps) {
        // ===================== chain warps: U and the state refresh (the dependent chain)
        // Warp (q, h): rows 16 q .. + 15 of the half (TMEM lanes 32 q .. + 15), tokens 32 h .. of U, dk 64 h .. of S.
        const int ch = warp >> 2, q16 = (warp & 3) * 16;
        auto hand_over = [&](uint64_t* bar) {     // after tcgen05.st: publish to the issuing warp
            tmem_wait_st();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar);
        };
        // fp32 master state as fragments: S[4 b + 2 r + e] = row q16 + g8 + 8 r, dk 64 ch + 8 b + 2 t4 + e
        float S[32];
        auto store_state_bf16 = [&](uint32_t g) {       // -> chunk g's bf16 A operand in TMEM
            uint32_t pk[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) pk[k] = pack_bf16(S[2 * k], S[2 * k + 1]);
            tmem_st_16x128b_x8(tmem + half_s_col(g) + lane_base + 32 * ch, pk);
        };
        // element offset of a thread's first pair inside a half tile, and of pair (b, r) from there
        const int frag = (q16 + g8) * kD + 64 * ch + 2 * t4;
        auto pair_off = [](int b, int r) { return 8 * r * kD + 8 * b; };
        bool ok = true;
        // As in state_stream_role: each lane's own verdict until the unit's last chunk; after a failed wait the work
        // goes on with whatever is there and nothing of it is written out.
        auto await = [&](uint64_t* bar, uint32_t parity) {
            if (!warp_wait(bar, parity, abortp, kWaitReason)) ok = false;
            tc_fence_after_sync();
        };
        // a half unit's chunks (0: nothing for the chain) and its half tile
        auto brief = [&](int hu) {
            const UnitInfo u = info(hu);
            return make_int2(u.skip || is_done(min(hu, total - 1)) ? 0 : u.nc, (u.slot * p.Hv + u.hv) * 2 + (hu & 1));
        };
        int2 nxt = brief(at(0));
        for (int i = 0, hu = at(0); hu < total; hu = at(++i)) {
            const int nc = nxt.x, tile = nxt.y;
            const int hu_next = at(i + 1);
            nxt = brief(hu_next);
            if (nc == 0) {
                const UnitInfo u = info(hu);
                if (is_done(hu)) continue;
                if constexpr (kMode == kHalfGated) {
                    if (tid == 0) done[hu] = 1;
                }
                if (u.bad_seq) continue;
                const int half = hu & 1;
                if (u.bad_slot) {          // padding / out-of-range slot: zero rows, no state
                    if (u.slot >= p.num_slots && tid == 0) report(p.dev_status, kDevBadSlot);
                    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
                    for (int k = tid; k < u.seq_len * 8; k += kSEpiThreads)
                        *reinterpret_cast<uint4*>(p.o + (static_cast<size_t>(u.seq_t0 + (k >> 3)) * p.Hv + u.hv) * kD +
                                                  half * kHalfRows + (k & 7) * 8) = zero;
                } else {                   // empty sequence: the state passes through untouched
                    const size_t off = static_cast<size_t>(tile) * (kHalfRows * kD);
                    for (int k = 4 * tid; k < kHalfRows * kD; k += 4 * kSEpiThreads)
                        *reinterpret_cast<float4*>(p.final_state + off + k) =
                            p.init_state ? *reinterpret_cast<const float4*>(p.init_state + off + k)
                                         : make_float4(0.f, 0.f, 0.f, 0.f);
                }
                continue;
            }
            if (p.init_state) {
                const float* in = p.init_state + static_cast<size_t>(tile) * (kHalfRows * kD) + frag;
#pragma unroll
                for (int b = 0; b < 8; ++b)
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        const float2 v = *reinterpret_cast<const float2*>(in + pair_off(b, r));
                        S[4 * b + 2 * r] = v.x;
                        S[4 * b + 2 * r + 1] = v.y;
                    }
            } else {
#pragma unroll
                for (int k = 0; k < 32; ++k) S[k] = 0.f;
            }
            store_state_bf16(gc);
            hand_over(&bar_s[gc & 1][ch]);
            // the next initial state, towards L2
            if (p.init_state && tid == 0 && nxt.x > 0 && hu_next < total)
                bulk_prefetch_l2(p.init_state + static_cast<size_t>(nxt.y) * (kHalfRows * kD), kHalfRows * kD * 4);
#pragma unroll 1
            for (int j = 0; j < nc; ++j) {
                // (left to the last launch: the rest of the half unit would be a failing wait after another)
                if (kMode == kHalfGated && !ok) break;
                const uint32_t g = gc + j;
                const int st = g & 1;
                const uint8_t* vec = smem + kHS_B + st * kHBBytes + kHB_Vec;
                await(&bar_full_b[st], (g >> 1) & 1u);
                float2 dec[4];                    // e^{b_C - b} of tokens 32 ch + 8 b + 2 t4, + 1
#pragma unroll
                for (int b = 0; b < 4; ++b)
                    dec[b] = *reinterpret_cast<const float2*>(vec + 4 * (32 * ch + 8 * b + 2 * t4));
                const float gC = *reinterpret_cast<const float*>(vec + (kRecGammaC - kRecDecay));
                // U P^T of the chunk before has read the last U, and S Q^T before it the bf16 state in whose place the next
                // will be.  (A wait that finds its phase completed takes more than 100 cycles all the same: this one stands
                // where a product is in flight anyway.)
                if (g > 0) await(&bar_y[st ^ 1], ((g - 1) >> 1) & 1u);
                await(&bar_d1, g & 1u);
                {   // U (the accumulator holds U~ - S W^T): rounded, and decayed as hi + lo
                    uint32_t x[16], pu[8], ph[8], pl[8];
                    tmem_ld_16x256b_x4(tmem + kH_D1 + lane_base + 32 * ch, x);
                    tmem_wait_ld();
#pragma unroll
                    for (int b = 0; b < 4; ++b)
#pragma unroll
                        for (int r = 0; r < 2; ++r) {
                            const float u0 = __uint_as_float(x[4 * b + 2 * r]), u1 = __uint_as_float(x[4 * b + 2 * r + 1]);
                            const float s0 = u0 * dec[b].x, s1 = u1 * dec[b].y;
                            const uint32_t h = pack_bf16(s0, s1);
                            ph[2 * b + r] = h;
                            pl[2 * b + r] = pack_bf16(s0 - __uint_as_float(h << 16), s1 - __uint_as_float(h & 0xffff0000u));
                            pu[2 * b + r] = pack_bf16(u0, u1);
                        }
                    const uint32_t at_us = tmem + kH_Us + lane_base + 16 * ch;
                    tmem_st_16x128b_x4(at_us, ph);
                    tmem_st_16x128b_x4(at_us + (16u << 16), pl);
                    tmem_st_16x128b_x4(tmem + kH_U + lane_base + 16 * ch, pu);
                }
                hand_over(&bar_u);
                if (lane == 0) mbar_arrive(&bar_free_b[st]);    // this warp has read the vectors
                await(&bar_d4[ch], g & 1u);
                // S <- e^{b_C} S + (hi + lo terms)
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    uint32_t xh[16], xl[16];
                    const uint32_t at_d4 = tmem + kH_D4 + lane_base + 64 * ch + 32 * c;
                    tmem_ld_16x256b_x4(at_d4, xh);
                    tmem_ld_16x256b_x4(at_d4 + (16u << 16), xl);
                    tmem_wait_ld();
#pragma unroll
                    for (int k = 0; k < 16; ++k)
                        S[16 * c + k] = fmaf(gC, S[16 * c + k], __uint_as_float(xh[k]) + __uint_as_float(xl[k]));
                }
                if (j + 1 < nc) {
                    store_state_bf16(g + 1);     // the next chunk's A operand
                    hand_over(&bar_s[(g + 1) & 1][ch]);
                }
            }
            // nothing of a unit is written after a failed wait (every record of the unit has been loaded by now: no
            // flag wait of it can fail any more)
            ok = group_all<2, kSEpiThreads>(ok);
            if (ok) {
                float* out = p.final_state + static_cast<size_t>(tile) * (kHalfRows * kD) + frag;
#pragma unroll
                for (int b = 0; b < 8; ++b)
#pragma unroll
                    for (int r = 0; r < 2; ++r)
                        *reinterpret_cast<float2*>(out + pair_off(b, r)) = make_float2(S[4 * b + 2 * r], S[4 * b + 2 * r + 1]);
                if constexpr (kMode == kHalfGated) {
                    if (tid == 0) done[hu] = 1;
                }
            }
            gc += nc;
        }
    } else {
        // ===================== output warps: U~ into the accumulator of S W^T a chunk ahead, and
        // scale e^b (S Q^T) + U P^T -> o rows.  Warp 8 + q has rows 16 q .. + 15 of the half.
        const int q4 = warp & 3;
        const int ot = tid - kSOutWarp0 * 32;
        const size_t tok_stride = static_cast<size_t>(p.Hv) * kD;
        bool ok = true;
        auto await = [&](uint64_t* bar, uint32_t parity) {
            if (!warp_wait(bar, parity, abortp, kWaitReason)) ok = false;
        };
        // the chunk's scale e^{b_r} outlives its stage: a copy per warp, two chunks deep
        __shared__ __align__(8) float s_eb[kSOutThreads / 32][2][kChunk];
        auto preload = [&](uint32_t gq) {       // chunk gq of the CTA's stream -> accumulator
            const int sq = gq & 1;
            const uint8_t* base = smem + kHS_B + sq * kHBBytes;
            await(&bar_full_b[sq], (gq >> 1) & 1u);
            // tokens 8 b + 2 t4, + 1 of row 16 q + g8 + 8 r: token group 2 b + (t4 >> 1), see rec_u_index
            const float* sU = reinterpret_cast<const float*>(base + kHB_U) + 2 * (t4 & 1);
            uint32_t x[2][16];
#pragma unroll
            for (int c = 0; c < 2; ++c)
#pragma unroll
                for (int b = 0; b < 4; ++b)
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        const float2 v = *reinterpret_cast<const float2*>(
                            sU + 4 * rec_u_index(8 * c + 2 * b + (t4 >> 1), 16 * q4 + g8 + 8 * r));
                        x[c][4 * b + 2 * r] = __float_as_uint(v.x);
                        x[c][4 * b + 2 * r + 1] = __float_as_uint(v.y);
                    }
            const float2 eb = *reinterpret_cast<const float2*>(base + kHB_Vec + (kRecEb - kRecDecay) + 8 * lane);
            const int nb = record_blocks(base + kHB_Vec + (kRecGammaC + 4 - kRecDecay));
#pragma unroll
            for (int c = 0; c < 2; ++c) tmem_st_16x256b_x4(tmem + kH_D1 + lane_base + 32 * c, x[c]);
            // blocks without tokens were not copied: whatever was there is replaced
#pragma unroll 1
            for (int b = nb; b < 4; ++b) tmem_zero_16x256b_x2(tmem + kH_D1 + lane_base + 16 * b);
            *reinterpret_cast<float2*>(&s_eb[q4][sq][2 * lane]) = eb;
            tmem_wait_st();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_p[sq]);
        };
        // The rows of a chunk leave their staging tile once the next U~ is in place, for which the next S W^T waits (right
        // behind the rows they put it off by 200 cycles).  One group barrier a chunk, which every warp runs also after a
        // failed wait: the tile's rows are complete, and the rows in the other one, sent a chunk ago, have left.
        struct {
            bool any = false;
            int tok, len, hv, half;
            uint32_t tile;
        } rows;
        auto rows_out = [&] {
            if (ot == 0) bulk_wait_read_all();
            if constexpr (kMode == kHalfGated) ok = group_all<1, kSOutThreads>(ok);
            else asm volatile("bar.sync 1, %0;" ::"n"(kSOutThreads) : "memory");
            if (rows.any && ok) {
                const uint8_t* tile = smem + rows.tile;
                if (rows.len == kChunk) {
                    if (ot == 0) {
                        tma_store_2d(&maps.o, rows.hv * kD + rows.half * kHalfRows, rows.tok, tile);
                        bulk_commit();
                    }
                } else {                     // a ragged tail: the rows behind it are another sequence's
                    const int piece = ot & 7;
                    __nv_bfloat16* og = p.o + (static_cast<size_t>(rows.tok) * p.Hv + rows.hv) * kD + rows.half * kHalfRows + piece * 8;
                    for (int row = ot >> 3; row < rows.len; row += 16)
                        *reinterpret_cast<uint4*>(og + row * tok_stride) =
                            *reinterpret_cast<const uint4*>(tile + sw128_offset(row, piece));
                }
            }
            rows.any = false;
        };
        bool preloaded = false;     // U~ of the chunk about to be processed is already in place
        UnitInfo nxt = info(at(0));
        bool nxt_done = is_done(min(at(0), total - 1));
        for (int i = 0, hu = at(0); hu < total; hu = at(++i)) {
            const UnitInfo u = nxt;
            const bool skip = u.skip || nxt_done;
            const int hu_next = at(i + 1);
            nxt = info(hu_next);
            nxt_done = is_done(min(hu_next, total - 1));
            if (skip) continue;
#pragma unroll 1
            for (int j = 0; j < u.nc; ++j) {
                const uint32_t g = gc + j;
                const int buf = g & 1;
                // The next U~ goes into the accumulator as soon as the chain warps have read this chunk's U out of it (where
                // it was not put in ahead, this group has waited for the products that follow).
                const bool ahead = j + 1 < u.nc || (hu_next < total && !nxt.skip && !nxt_done);
#pragma unroll 1
                for (int k = preloaded ? 1 : 0; k < (ahead ? 2 : 1); ++k) {
                    if (k == 1) await(&bar_u, g & 1u);
                    tc_fence_after_sync();
                    preload(g + k);
                }
                preloaded = ahead;
                rows_out();
                if (kMode == kHalfGated && !ok) break;   // (the verdict is the group's)
                await(&bar_y[buf], (g >> 1) & 1u);
                // The rows are made once the chain warps have handed the next state over and wait behind the next
                // product: beside the refresh they take its issue slots (4096 tokens at 8 v-heads 91.5 us, 88.3 this
                // way).  The chain warps may by now have handed over the state after that one, but no more: it goes on from
                // the U~ that these warps put in place after these rows.  So the hand-overs have two barriers, in turn (a
                // parity cannot tell a phase from the one after the next).
                if (j + 1 < u.nc) await(&bar_s[(g + 1) & 1][1], ((g + 1) >> 1) & 1u);
                tc_fence_after_sync();
                {
                    // Fragments (rows = dv, columns = tokens), rounded in pairs and stored transposed into a
                    // [token][dv] tile: lane l gives the address of matrix l / 8: tokens 8 (b + (l >> 4)) .., dv 8 (l
                    // >> 3 & 1) ..
                    const uint32_t dst = smem_u32(smem + kHS_Out + 8192 * buf);
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        uint32_t y1[16], y2[16], pk[8];
                        tmem_ld_16x256b_x4(tmem + kH_Y1 + lane_base + 32 * c, y1);
                        tmem_ld_16x256b_x4(tmem + kH_Y2 + lane_base + 32 * c, y2);
                        tmem_wait_ld();
#pragma unroll
                        for (int b = 0; b < 4; ++b) {
                            const float2 eb = *reinterpret_cast<const float2*>(&s_eb[q4][buf][2 * t4 + 8 * (4 * c + b)]);
#pragma unroll
                            for (int r = 0; r < 2; ++r) {
                                const int k = 4 * b + 2 * r;
                                const float2 y = fma2(eb, make_float2(__uint_as_float(y1[k]), __uint_as_float(y1[k + 1])),
                                                      make_float2(__uint_as_float(y2[k]), __uint_as_float(y2[k + 1])));
                                pk[2 * b + r] = pack_bf16(y.x, y.y);
                            }
                        }
#pragma unroll
                        for (int b = 0; b < 4; b += 2)
                            stmatrix_x4_trans(dst + sw128_offset(8 * (4 * c + b + (lane >> 4)) + (lane & 7), 2 * q4 + ((lane >> 3) & 1)),
                                              pk[2 * b], pk[2 * b + 1], pk[2 * b + 2], pk[2 * b + 3]);
                    }
                }
                tc_fence_before_sync();
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bar_y_read);
                rows = {true, u.seq_t0 + j * kChunk, min(kChunk, u.seq_len - j * kChunk), u.hv, hu & 1, kHS_Out + 8192 * buf};
            }
            gc += u.nc;
        }
        rows_out();
        if (ot == 0) bulk_wait_all();        // before the CTA's shared memory goes away
    }

    tc_fence_before_sync();
    __syncthreads();
    if (abort_flag != 0 && warp == kSIssueWarp && lane == 0) {
        if (abort_flag == 1) report(p.dev_status, kDevTimeout);     // 2: a record not produced yet, no error
        // let copies already in flight land before the CTA's shared memory goes away: the last chunks of each ring
        // that the loader started, each on its place's barrier at that chunk's own parity
        for (uint32_t back = 1; back <= kHStages; ++back) {
            for (int r = 0; r < 3; ++r) {
                const uint32_t n = *reinterpret_cast<volatile uint32_t*>(&armed[r]), places = r == 1 ? 2 : kHStages;
                if (back > n || back > places) continue;
                uint64_t* full = r == 0 ? bar_full_a : r == 1 ? bar_full_b : bar_full_c;
                mbar_wait(&full[(n - back) % places], ((n - back) / places) & 1u, 1u << 12);
            }
        }
    }
}

}  // namespace gdn
