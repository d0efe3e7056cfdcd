// Device-side building blocks shared by the chunked prefill kernels (the three-launch path and
// the fused single-launch path): shared-memory maps, the fp32 triangular solve, the intra-chunk
// item routine, and the bounded-wait helpers.  See gdn_prefill_chunk.cuh for the algebra.
#pragma once
#include "gdn_prefill_chunk.cuh"
#include "gdn_sm100.cuh"

namespace gdn {
using namespace sm100;

constexpr int kIntraThreads = 256;
constexpr uint32_t kIntraTmemCols = 128;    // the Gram accumulator, then W^T in the same columns; U~^T
constexpr int kLdA = 68;               // row stride (floats) of the fp32 A / T matrix
// Shared memory map (bytes from a 1024-aligned base).  Regions are reused as their contents die
// so that four CTAs fit on an SM:
//   R1  Q/K tiles.  Q halves (-> Qg image, stored early) -> V tile, loaded once the Gram product (or
//       the store) has read Q;  K halves -> W image.
//   R2  A, then T, in fp32 -> T_w -> T_u(lo);  T_u(hi).
// The P image goes straight from registers to the record; T_u(lo) waits in registers until the
// product that reads T_w has retired.
constexpr uint32_t kI_QK = 0;          // 2 halves x [128 rows x 128 B]: rows 0-63 Q, 64-127 K
constexpr uint32_t kI_V = 0;           // over Q: 2 halves x [64 x 128 B], 16384 apart
constexpr uint32_t kI_A = 32768;       // A, then T in place: fp32 [64][kLdA]
constexpr uint32_t kI_Tw = kI_A;       // over A: T diag(beta e^b) [64 r x 64 i] bf16, K-major
constexpr uint32_t kI_TuLo = kI_A;     // ... and later the bf16 remainder of T diag(beta)
constexpr uint32_t kI_Tu = kI_A + 8192;                // T diag(beta) rounded to bf16
constexpr uint32_t kI_End = kI_A + 64 * kLdA * 4;      // 50176
constexpr uint32_t kIntraSmem = kI_End + 1024;         // + alignment slack
static_assert(kI_End % 1024 == 0 && 64 * kLdA * 4 >= 16384, "the T images must fit over A");

struct TensorMaps {
    CUtensorMap q, k, v, o;
};
// Host side: 2-D maps over the packed q, k, v, o (64 x 64 boxes, 128B swizzle); false on failure.
bool make_prefill_tensor_maps(TensorMaps* maps, const PrefillParams& p);
// Launch of the intra-chunk kernel over every (chunk, v-head) item of the batch.
// inline_tables: no table-building launch went before; every CTA finds its chunk from cu_seqlens.  For batches of few
// sequences: see prefill_tables_inline().
cudaError_t launch_prefill_intra(const TensorMaps& maps, const ChunkedParams& cp, cudaStream_t stream,
                                 bool inline_tables);
bool prefill_tables_inline(const ChunkedParams& cp);

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// One 16x8 output tile  C += A[16 x 8*ksteps] * B[8*ksteps x 8]  on mma.sync m16n8k8 with tf32
// operands (rounded to nearest, one product per k-step) and fp32 accumulation.  A, B: fp32
// row-major in shared memory; g = lane / 4, t = lane % 4.
// Accuracy: these products only form the OFF-diagonal blocks of T = (I + A)^-1 from blocks that
// are exact to fp32; an operand error of 2^-11 there moves the final state by about 1e-5 of its
// norm on random keys and 3e-4 when all keys coincide (the worst case for the solve), against
// 1.6e-4 and 1.4e-3 from the bf16 operands of the other products.  Split operands (three
// products per k-step) bought nothing measurable and cost 2.3x the instructions.
__device__ __forceinline__ uint32_t to_tf32(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ void mma_m16n8k8_tf32(float (&c)[4], const uint32_t (&a)[4],
                                                 const uint32_t (&b)[2]) {
    asm volatile(
        "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
// kN tiles side by side: columns 8 nb .. of B and of the output.
template <int kSteps, int kN>
__device__ __forceinline__ void mma_tile_tf32(const float* A, int lda, const float* B, int ldb,
                                              float (&c)[kN][4], int g, int t) {
    uint32_t a[kSteps][4], b[kSteps][kN][2];
#pragma unroll
    for (int ks = 0; ks < kSteps; ++ks) {          // every load first, then the products
        const float* a_ = A + 8 * ks;
        const float* b_ = B + (8 * ks) * ldb;
        a[ks][0] = to_tf32(a_[g * lda + t]);
        a[ks][1] = to_tf32(a_[(g + 8) * lda + t]);
        a[ks][2] = to_tf32(a_[g * lda + t + 4]);
        a[ks][3] = to_tf32(a_[(g + 8) * lda + t + 4]);
#pragma unroll
        for (int nb = 0; nb < kN; ++nb) {
            b[ks][nb][0] = to_tf32(b_[t * ldb + 8 * nb + g]);
            b[ks][nb][1] = to_tf32(b_[(t + 4) * ldb + 8 * nb + g]);
        }
    }
#pragma unroll
    for (int ks = 0; ks < kSteps; ++ks)
#pragma unroll
        for (int nb = 0; nb < kN; ++nb) mma_m16n8k8_tf32(c[nb], a[ks], b[ks][nb]);
}

__device__ __forceinline__ uint32_t scale_bf16x2(uint32_t packed, float f) {
    return pack_bf16(__uint_as_float(packed << 16) * f, __uint_as_float(packed & 0xffff0000u) * f);
}

// Per-group statics of the intra-chunk work (one instance per concurrently processed item).
struct IntraStatics {
    uint64_t bar_tma, bar_v, bar_mma;
    int abort_flag;
    int item;                          // work-queue slot (persistent variant)
    alignas(16) float s_b2[kChunk];    // b_r log2(e): inclusive log-decay prefix
    alignas(16) float s_beta[kChunk];  // beta_r (0 past the chunk's length)
    alignas(16) float s_bg[kChunk];    // beta_r e^{b_r}
};

// T = (I + A)^{-1} for the strictly lower-triangular 64x64 A in sA (fp32, row-major, stride kLdA),
// in place, in two stages:
//   solve_blocks_16_32: a warp inverts two neighbouring diagonal 16x16 blocks by forward
//     substitution (thread (I, j) computes column j of (I + A_II)^{-1}, right-looking, four columns of A
//     at a time so that a row's are one 16-byte read) and joins them into the inverse of their 32x32 block,
//   solve_merge_64: four warps compute the last off-diagonal 32x32 block, a 16x16 quarter each,
// both by block elimination  [[Ta, 0], [X, Tb]],  X = -Tb (A_ba Ta),  whose small products run on
// the legacy mma.sync path (tcgen05 needs M >= 64).  The intermediate product A_ba Ta changes
// from accumulator to operand layout through the block of sA that mirrors X above the diagonal.
// What is left there is not cleared: readers of T take every 16x16 block above the diagonal as zero.
// Warp `pr` (0 or 1) of the group: diagonal blocks 2 pr, 2 pr + 1 and block (2 pr + 1, 2 pr).
__device__ __forceinline__ void solve_blocks_16_32(float* sA, const int pr, const int lane,
                                                   const int len) {
    {
        const int I = 2 * pr + (lane >> 4), j = lane & 15;
        float* blk = sA + (16 * I) * kLdA + 16 * I;
        float t[16];
#pragma unroll
        for (int r = 0; r < 16; ++r) t[r] = (r == j) ? 1.f : 0.f;
#pragma unroll
        for (int c = 0; c < 16; c += 4) {
#pragma unroll
            for (int r = c + 1; r < 16; ++r) {
                const float4 a = *reinterpret_cast<const float4*>(blk + r * kLdA + c);
                t[r] = fmaf(-a.x, t[c], t[r]);
                if (r > c + 1) t[r] = fmaf(-a.y, t[c + 1], t[r]);
                if (r > c + 2) t[r] = fmaf(-a.z, t[c + 2], t[r]);
                if (r > c + 3) t[r] = fmaf(-a.w, t[c + 3], t[r]);
            }
        }
        __syncwarp();                      // every column of the block has read A_II
#pragma unroll
        for (int r = 0; r < 16; ++r) blk[r * kLdA + j] = t[r];
    }
    if (len <= 32 * pr + 16) return;       // block (2 pr + 1, 2 pr) lies in rows past the chunk's length: zero
    __syncwarp();
    const int g = lane >> 2, t = lane & 3;
    const int I = 2 * pr + 1, J = 2 * pr;
    float* A_IJ = sA + (16 * I) * kLdA + 16 * J;
    float* X = sA + (16 * J) * kLdA + 16 * I;          // the mirror block
    float c[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
    mma_tile_tf32<2, 2>(A_IJ, kLdA, sA + (16 * J) * kLdA + 16 * J, kLdA, c, g, t);      // X = A_IJ T_JJ
#pragma unroll
    for (int nb = 0; nb < 2; ++nb) {
        *reinterpret_cast<float2*>(X + g * kLdA + 8 * nb + 2 * t) = make_float2(c[nb][0], c[nb][1]);
        *reinterpret_cast<float2*>(X + (g + 8) * kLdA + 8 * nb + 2 * t) = make_float2(c[nb][2], c[nb][3]);
        c[nb][0] = c[nb][1] = c[nb][2] = c[nb][3] = 0.f;
    }
    __syncwarp();
    mma_tile_tf32<2, 2>(sA + (16 * I) * kLdA + 16 * I, kLdA, X, kLdA, c, g, t);         // T_IJ = -T_II X
    __syncwarp();                                      // every lane has read A_IJ (above)
#pragma unroll
    for (int nb = 0; nb < 2; ++nb) {
        float* dst = A_IJ + 8 * nb;
        *reinterpret_cast<float2*>(dst + g * kLdA + 2 * t) = make_float2(-c[nb][0], -c[nb][1]);
        *reinterpret_cast<float2*>(dst + (g + 8) * kLdA + 2 * t) = make_float2(-c[nb][2], -c[nb][3]);
    }
}

// Quarter w (0..3: rows 16 (w & 1), columns 16 (w >> 1)) of the 32x32 block (1, 0), given the inverses of
// the two diagonal 32x32 blocks.  Called by four consecutive warps together, which meet at a
// barrier of their own (`bar_id`, 128 threads) between the products: the second reads what two warps
// wrote and overwrites what all four have read.
__device__ __forceinline__ void solve_merge_64(float* sA, const int w, const int lane,
                                               const int bar_id) {
    const int g = lane >> 2, t = lane & 3;
    const int r0 = 16 * (w & 1), c0 = 16 * (w >> 1);
    float* Y = sA + 32 + c0;                           // rows 0-31 of the mirror block
    float c[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
    // Y = A_ba Ta; Ta is lower triangular: its columns 16-31 have rows 16-31 only
    if (c0 == 0)
        mma_tile_tf32<4, 2>(sA + (32 + r0) * kLdA, kLdA, sA, kLdA, c, g, t);
    else
        mma_tile_tf32<2, 2>(sA + (32 + r0) * kLdA + 16, kLdA, sA + 16 * kLdA + 16, kLdA, c, g, t);
#pragma unroll
    for (int nb = 0; nb < 2; ++nb) {
        *reinterpret_cast<float2*>(Y + (r0 + g) * kLdA + 8 * nb + 2 * t) = make_float2(c[nb][0], c[nb][1]);
        *reinterpret_cast<float2*>(Y + (r0 + g + 8) * kLdA + 8 * nb + 2 * t) = make_float2(c[nb][2], c[nb][3]);
        c[nb][0] = c[nb][1] = c[nb][2] = c[nb][3] = 0.f;
    }
    asm volatile("bar.sync %0, 128;" ::"r"(bar_id) : "memory");
    // X = -Tb Y; the rows 0-15 of Tb have columns 0-15 only
    if (r0 == 0)
        mma_tile_tf32<2, 2>(sA + 32 * kLdA + 32, kLdA, Y, kLdA, c, g, t);
    else
        mma_tile_tf32<4, 2>(sA + 48 * kLdA + 32, kLdA, Y, kLdA, c, g, t);
#pragma unroll
    for (int nb = 0; nb < 2; ++nb) {
        float* dst = sA + (32 + r0) * kLdA + c0 + 8 * nb;
        *reinterpret_cast<float2*>(dst + g * kLdA + 2 * t) = make_float2(-c[nb][0], -c[nb][1]);
        *reinterpret_cast<float2*>(dst + (g + 8) * kLdA + 2 * t) = make_float2(-c[nb][2], -c[nb][3]);
    }
}

// bounded wait that also gives up as soon as another role has flagged an abort.  `reason` is what a
// wait that runs out writes into the flag: 1 = an error (reported as a timeout), 2 = give up
// without an error (the caller's work is finished by a later launch).
// kSleepNs: pause between polls.  Polls take issue slots and shared-memory cycles from whatever is being
// waited for, so every wait but the shortest pauses.
template <int kSleepNs = 0>
__device__ __forceinline__ bool wait_or_abort(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                              const int reason = 1) {
#pragma unroll 1
    for (uint32_t i = 0; i < kSpinLimit; ++i) {
        if (mbar_try_wait(bar, parity)) return true;
        if (kSleepNs) __nanosleep(kSleepNs);
        if ((i & 255u) == 255u && *abort_flag) return false;
    }
    if (*abort_flag == 0) *abort_flag = reason;      // keep an earlier, different reason
    return false;
}

// Barrier `kId` over kThreads threads; the AND of their arguments.
template <int kId, int kThreads> __device__ __forceinline__ bool group_all(const bool mine) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %1, 0;\n\t"
        "bar.red.and.pred p, %2, %3, q;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(r)
        : "r"(static_cast<uint32_t>(mine)), "n"(kId), "n"(kThreads)
        : "memory");
    return r != 0;
}

// Same, for a whole converged warp: every lane polls, so the instruction stays warp-wide, and what ends the loop is a
// vote, so the verdict is the same on every lane whatever each lane's poll answers: callers issue warp-wide
// instructions on the strength of it.  (Polling by one lane and broadcasting the verdict costs a divergent branch and
// a shuffle, and that lane alone wakes later: a waiting warp saw an arrival after 200 cycles instead of 89.)
__device__ __forceinline__ bool warp_wait_or_abort(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                                   const int reason = 1) {
#pragma unroll 1
    for (uint32_t i = 0; i < kSpinLimit; ++i) {
        if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
        // (a poll that fails has blocked for some microseconds)
        if ((i & 7u) == 0u && __any_sync(0xffffffffu, *abort_flag)) return false;
    }
    if (*abort_flag == 0) *abort_flag = reason;      // keep an earlier, different reason
    return false;
}

// The same with the first poll in one piece with its vote (it blocks for a while by itself and so is nearly always the
// last) and the rest out of line.  The roles of a warp-specialised kernel share 32 KB of instruction cache, and past
// it each runs at the pace of its instruction misses: eight roles of 3 KB a round take 573 cycles, of 4 KB 929; the
// half-unit state pass had 128 misses a chunk step with its waits in line and unrolled, and has 2.
static __device__ __noinline__ bool warp_wait_more(uint64_t* bar, uint32_t parity, volatile int* abort_flag, const int reason) {
    return warp_wait_or_abort(bar, parity, abort_flag, reason);
}
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag, const int reason = 1) {
    return mbar_try_wait_all(bar, parity) || warp_wait_more(bar, parity, abort_flag, reason);
}

// kScaledQ: whether the record carries the scaled Q (gdn_prefill_chunk.cuh).
// The intra-chunk quantities of one (chunk, v-head) item, computed by a group of 256 threads (tid = 0..255 within the
// group; its warps must be CTA warps 0-3 mod 4 aligned, because a warp reaches TMEM lanes 32 (warp % 4) ...).  `smem`
// is the group's 1024-aligned slice of kI_End bytes, `tmem_base` + `tmem_off` its 128 TMEM columns (read behind the
// group's first barrier, which so also covers their allocation), `sync` a barrier over exactly the group.  Writes the
// item's record; returns false after a bounded wait gave up (status word set, nothing left in flight).
template <bool kScaledQ, class Sync>
__device__ __forceinline__ bool intra_item(const TensorMaps& maps, const PrefillParams& p,
                                           uint8_t* rec, const ChunkInfo ci, const int hqk,
                                           const int hv, uint8_t* smem, IntraStatics& st,
                                           const uint32_t* tmem_base, const uint32_t tmem_off, const int tid, Sync sync,
                                           const uint32_t n_done = 0) {
    // `n_done` = items this group has processed before (persistent callers): the mbarriers are
    // initialised once and keep flipping phase, one completion of bar_tma and bar_v and three
    // of bar_mma per item.
    const uint32_t par1 = n_done & 1u;           // parity of this item's bar_tma / bar_v phase
    const uint32_t par3 = (3u * n_done) & 1u;    // parity of this item's first bar_mma phase
    const int warp = tid >> 5;
    const int colhalf = warp >> 2;                   // which 32 of the 64 accumulator columns
    const int nb = (ci.len + 15) >> 4;               // 16-token blocks that hold tokens
    if (tid == 0) {
        if (n_done == 0) {
            mbar_init(&st.bar_tma, 1);
            mbar_init(&st.bar_v, 1);
            mbar_init(&st.bar_mma, 1);
            fence_barrier_init();
        }
        st.abort_flag = 0;
        // Q and K first: everything below overlaps their flight (V comes later, over Q)
        mbar_expect_tx(&st.bar_tma, 32768);
        tma_load_2d(smem + kI_QK, &maps.q, hqk * kD, ci.t0, &st.bar_tma);
        tma_load_2d(smem + kI_QK + 8192, &maps.k, hqk * kD, ci.t0, &st.bar_tma);
        tma_load_2d(smem + kI_QK + 16384, &maps.q, hqk * kD + 64, ci.t0, &st.bar_tma);
        tma_load_2d(smem + kI_QK + 24576, &maps.k, hqk * kD + 64, ci.t0, &st.bar_tma);
    }
    if (warp == 1) {
        // inclusive prefix sum of the log gates over the chunk (two tokens per lane); rows past
        // the chunk's length get g = 0, beta = 0 and so change nothing downstream
        const int lane = tid & 31;
        float g0 = 0.f, g1 = 0.f, be0 = 0.f, be1 = 0.f;
        if (2 * lane < ci.len) {
            const size_t th = static_cast<size_t>(ci.t0 + 2 * lane) * p.Hv + hv;
            g0 = p.g[th]; be0 = p.beta[th];
        }
        if (2 * lane + 1 < ci.len) {
            const size_t th = static_cast<size_t>(ci.t0 + 2 * lane + 1) * p.Hv + hv;
            g1 = p.g[th]; be1 = p.beta[th];
        }
        float incl = g0 + g1;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const float y = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += y;
        }
        const float kLog2e = 1.4426950408889634f;
        const float b1 = incl, b0 = incl - g1;
        const float bC = __shfl_sync(0xffffffffu, incl, 31);
        st.s_b2[2 * lane] = b0 * kLog2e; st.s_b2[2 * lane + 1] = b1 * kLog2e;
        st.s_beta[2 * lane] = be0; st.s_beta[2 * lane + 1] = be1;
        const float e0 = ex2_approx(b0 * kLog2e), e1 = ex2_approx(b1 * kLog2e);
        st.s_bg[2 * lane] = be0 * e0; st.s_bg[2 * lane + 1] = be1 * e1;
        // the record's vectors: e^{b_C - b_c}, scale e^{b_r}, and e^{b_C}
        *reinterpret_cast<float2*>(rec + kRecDecay + 8 * lane) =
            make_float2(ex2_approx((bC - b0) * kLog2e), ex2_approx((bC - b1) * kLog2e));
        *reinterpret_cast<float2*>(rec + kRecEb + 8 * lane) = make_float2(p.scale * e0, p.scale * e1);
        if (lane == 0)
            *reinterpret_cast<float2*>(rec + kRecGammaC) = make_float2(ex2_approx(bC * kLog2e), __int_as_float(nb));
    }
    sync();
    tc_fence_after_sync();
    const uint32_t tmem = *tmem_base + tmem_off;
    // Every warp polls the barriers it needs itself.  A wait that runs out flags the item and the group
    // goes on to its next barrier, behind which everyone leaves together; thread 0 drains what it has
    // in flight and the caller unwinds.
    volatile int* abortp = &st.abort_flag;
    // (the cooperative launch re-allocates registers, which functions out of line do not go with)
    auto wait_bar = [](uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
        if constexpr (kScaledQ) return warp_wait_or_abort(bar, parity, abort_flag);
        else return warp_wait(bar, parity, abort_flag);
    };
    bool v_started = false;         // (thread 0's)
    auto bail = [&](bool stores_pending) {
        if (tid == 0) {
            report(p.dev_status, kDevTimeout);
            mbar_wait(&st.bar_tma, par1, 1u << 12);
            if (v_started) mbar_wait(&st.bar_v, par1, 1u << 12);
            if (stores_pending) bulk_wait_read_all();
        }
    };

    const uint32_t tG = tmem, tW = tmem, tU = tmem + 64;     // W reuses the Gram columns
    const uint32_t sQK = smem_u32(smem + kI_QK);
    // Tensor-core instructions are issued by warp 0, converged, a product by one elected lane (elect_one).
    if (warp == 0 && wait_bar(&st.bar_tma, par1, abortp)) {
        tc_fence_after_sync();
        // [Q;K] (128 x 128, K-major) times K^T: lanes 0-63 = q.k, lanes 64-127 = k.k
        const uint32_t idesc = make_idesc_bf16(128, 64, false, false);
        const uint64_t dA = make_sdesc_sw128(sQK, 16, 1024), dB = make_sdesc_sw128(sQK + 8192, 16, 1024);
        if (elect_one()) {
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) {
                const uint32_t off = (ks >> 2) * 16384 + (ks & 3) * 32;
                mma_ss(tG, sdesc_advance(dA, off), sdesc_advance(dB, off), idesc, ks > 0);
            }
            mma_commit(&st.bar_mma);
        }
    }
    const bool gram_ok = wait_bar(&st.bar_mma, par3, abortp);
    tc_fence_after_sync();
    auto load_v = [&] {             // thread 0, once Q is dead
        v_started = true;
        mbar_expect_tx(&st.bar_v, 16384);
        tma_load_2d(smem + kI_V, &maps.v, hv * kD, ci.t0, &st.bar_v);
        tma_load_2d(smem + kI_V + 16384, &maps.v, hv * kD + 64, ci.t0, &st.bar_v);
    };
    if (!kScaledQ && tid == 0 && gram_ok) load_v();
    __syncwarp();

    const uint32_t lane_base = static_cast<uint32_t>((warp & 3) * 32) << 16;
    float* sA = reinterpret_cast<float*>(smem + kI_A);
    {
        // Accumulator row of this thread: TMEM lane 32 (warp % 4) + lane; lanes 0-63 hold q.k
        // rows (-> P), lanes 64-127 hold k.k rows (-> A).  The thread covers 32 of the 64 columns,
        // 16 at a time.
        const int row = (warp & 3) * 32 + (tid & 31);
        const int r = row & 63;
        const bool is_p = row < 64;
        const float br2 = st.s_b2[r];
        const float rowscale = is_p ? p.scale : st.s_beta[r];      // the output scale rides on P
        const int limit = is_p ? r : r - 1;              // keep columns i <= limit
        // (rows of a half without tokens are not read)
        if ((row & 32) < ci.len)
#pragma unroll
        for (int step = 0; step < 2; ++step) {
            const int cbase = colhalf * 32 + step * 16;
            float val[16];
            // a 16-column block that lies wholly above the diagonal for every row of the warp is
            // zero (warp-uniform test: no accumulator read, no exponentials), one that lies wholly
            // below it needs no mask
            if (cbase > (row & 32) + 31) {
#pragma unroll
                for (int jj = 0; jj < 16; ++jj) val[jj] = 0.f;
            } else {
                uint32_t x[16];
                tmem_ld16(tG + lane_base + cbase, x);
                tmem_wait_ld();
#pragma unroll
                for (int q4 = 0; q4 < 4; ++q4) {
                    const float4 bb = *reinterpret_cast<const float4*>(st.s_b2 + cbase + 4 * q4);
                    const float bv[4] = {bb.x, bb.y, bb.z, bb.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e)          // times e^{b_r - b_i} (above the diagonal: discarded)
                        val[4 * q4 + e] = rowscale * __uint_as_float(x[4 * q4 + e]) * ex2_approx(br2 - bv[e]);
                }
                if (cbase + 15 >= (row & 32)) {
#pragma unroll
                    for (int jj = 0; jj < 16; ++jj) val[jj] = cbase + jj <= limit ? val[jj] : 0.f;
                }
            }
            if (is_p) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint4 w;
                    w.x = pack_bf16(val[8 * h + 0], val[8 * h + 1]);
                    w.y = pack_bf16(val[8 * h + 2], val[8 * h + 3]);
                    w.z = pack_bf16(val[8 * h + 4], val[8 * h + 5]);
                    w.w = pack_bf16(val[8 * h + 6], val[8 * h + 7]);
                    *reinterpret_cast<uint4*>(rec + kRecP + sw128_offset(r, (cbase >> 3) + h)) = w;
                }
            } else {
#pragma unroll
                for (int q4 = 0; q4 < 4; ++q4)
                    *reinterpret_cast<float4*>(sA + r * kLdA + cbase + 4 * q4) =
                        make_float4(val[4 * q4], val[4 * q4 + 1], val[4 * q4 + 2], val[4 * q4 + 3]);
            }
        }
    }
    tc_fence_before_sync();
    sync();
    if (st.abort_flag) { bail(false); return false; }
    // Warps 0-1 invert the two diagonal 32x32 blocks of I + A (serial forward substitutions and two
    // small products each, all inside the warp), then warps 4-7 the block below them.
    if (warp < 2) {
        if (32 * warp < ci.len) solve_blocks_16_32(sA, warp, tid & 31, ci.len);
    } else if constexpr (kScaledQ) {
        // beside them the others scale the Q rows by scale * e^{b_r} in place: the Qg image
#pragma unroll 2
        for (int idx = tid - 64; idx < 1024; idx += kIntraThreads - 64) {      // 1024 16-byte pieces
            const int rem = idx & 511;
            uint4* ptr = reinterpret_cast<uint4*>(smem + kI_QK + (idx >> 9) * 16384 + rem * 16);
            const float f = ex2_approx(st.s_b2[rem >> 3]) * p.scale;
            uint4 w = *ptr;
            w.x = scale_bf16x2(w.x, f); w.y = scale_bf16x2(w.y, f);
            w.z = scale_bf16x2(w.z, f); w.w = scale_bf16x2(w.w, f);
            *ptr = w;
        }
        fence_proxy_async_smem();
    }
    sync();
    if (kScaledQ && tid == 0) {     // Qg is final: store it, and fetch V over it once the store has read it
        bulk_store(rec + kRecQg, smem + kI_QK, 8192);
        bulk_store(rec + kRecQg + 8192, smem + kI_QK + 16384, 8192);
        bulk_commit();
        bulk_wait_read_all();
        load_v();
    }
    // (rows past the length are zero: nothing to do then).  Barrier ids 4.. are this routine's: one per
    // group of 256 threads of the CTA.
    if (warp >= 4 && ci.len > 32)
        solve_merge_64(sA, warp - 4, tid & 31, 4 + (static_cast<int>(threadIdx.x) >> 8));
    sync();

    // T (fp32, row-major) -> bf16 B operands T diag(beta e^b), T diag(beta) (hi, lo).  A thread takes four
    // columns of every 16th row: its column factors stay in registers and both the reads of T and
    // the writes of the images cover whole 128-byte rows (eight columns a thread conflicted twice
    // over on every access: a quarter of this kernel's shared-memory cycles).
    uint32_t tu_lo[4][2];    // T diag(beta) - bf16(T diag(beta)), parked until T_w is dead
    const int icol = tid & 15, irow = tid >> 4;
    auto image_offset = [&](int it) { return sw128_offset(irow + 16 * it, icol >> 1) + 8u * (icol & 1); };
    {
        const float4 fg = *reinterpret_cast<const float4*>(st.s_bg + 4 * icol);
        const float4 fb = *reinterpret_cast<const float4*>(st.s_beta + 4 * icol);
        uint32_t tw[4][2], tu[4][2];
#pragma unroll
        for (int it = 0; it < 4; ++it) {
            // (a 16x16 block above the diagonal is zero whatever the solve has left there)
            float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
            if (icol >> 2 <= it) t = *reinterpret_cast<const float4*>(sA + (irow + 16 * it) * kLdA + 4 * icol);
            const float u0 = t.x * fb.x, u1 = t.y * fb.y, u2 = t.z * fb.z, u3 = t.w * fb.w;
            const uint32_t h0 = pack_bf16(u0, u1), h1 = pack_bf16(u2, u3);
            tu_lo[it][0] = pack_bf16(u0 - __uint_as_float(h0 << 16), u1 - __uint_as_float(h0 & 0xffff0000u));
            tu_lo[it][1] = pack_bf16(u2 - __uint_as_float(h1 << 16), u3 - __uint_as_float(h1 & 0xffff0000u));
            tu[it][0] = h0; tu[it][1] = h1;
            tw[it][0] = pack_bf16(t.x * fg.x, t.y * fg.y);
            tw[it][1] = pack_bf16(t.z * fg.z, t.w * fg.w);
        }
        sync();              // T has been read: the images take its place
#pragma unroll
        for (int it = 0; it < 4; ++it) {
            const uint32_t off = image_offset(it);
            *reinterpret_cast<uint2*>(smem + kI_Tw + off) = make_uint2(tw[it][0], tw[it][1]);
            *reinterpret_cast<uint2*>(smem + kI_Tu + off) = make_uint2(tu[it][0], tu[it][1]);
        }
    }
    fence_proxy_async_smem();
    sync();

    const uint32_t sV = smem_u32(smem + kI_V);
    // the blocks that hold tokens, as columns (N) and as k-steps
    const uint32_t idesc_t = make_idesc_bf16(128, 16 * nb, true, false);
    if (warp == 0) {     // W^T (dk x r) = K^T T_w^T with the raw K tile read MN-major
        const uint64_t dK = make_sdesc_sw128(sQK + 8192, 16384, 1024), dT = make_sdesc_sw128(smem_u32(smem + kI_Tw), 16, 1024);
        if (elect_one()) {
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
                if (ks < nb)
                    mma_ss(tW, sdesc_advance(dK, ks * 2048), sdesc_advance(dT, ks * 32), idesc_t, ks > 0);
            mma_commit(&st.bar_mma);
        }
    }
    wait_bar(&st.bar_mma, par3 ^ 1u, abortp);
    tc_fence_after_sync();

    const int d = (warp & 3) * 32 + (tid & 31);   // TMEM lane of this thread: a dk / dv index
    {   // W^T[d][32 tokens] -> bf16 -> W image staged over the (now dead) K halves.  The image
        // is MN-major for the state pass's product S W^T (one 128-byte row of 64 tokens per dk
        // index), so a thread writes its own row in 16-byte pieces.
        uint8_t* sW = smem + kI_QK + 8192 + (d >> 6) * 16384;
#pragma unroll
        for (int step = 0; step < 2; ++step) {
            const int cbase = colhalf * 32 + step * 16;
            uint32_t x[16] = {};            // (no tokens: W is zero there, and so U)
            if (cbase < ci.len) {
                tmem_ld16(tW + lane_base + cbase, x);
                tmem_wait_ld();
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint4 w;
                w.x = pack_bf16(__uint_as_float(x[8 * h + 0]), __uint_as_float(x[8 * h + 1]));
                w.y = pack_bf16(__uint_as_float(x[8 * h + 2]), __uint_as_float(x[8 * h + 3]));
                w.z = pack_bf16(__uint_as_float(x[8 * h + 4]), __uint_as_float(x[8 * h + 5]));
                w.w = pack_bf16(__uint_as_float(x[8 * h + 6]), __uint_as_float(x[8 * h + 7]));
                *reinterpret_cast<uint4*>(sW + sw128_offset(d & 63, (cbase >> 3) + h)) = w;
            }
        }
    }
    // the product that read T_w has retired: its place takes the remainder of T diag(beta)
#pragma unroll
    for (int it = 0; it < 4; ++it)
        *reinterpret_cast<uint2*>(smem + kI_TuLo + image_offset(it)) = make_uint2(tu_lo[it][0], tu_lo[it][1]);
    fence_proxy_async_smem();
    tc_fence_before_sync();
    sync();
    if (st.abort_flag) { bail(false); return false; }      // nothing of thread 0's stores is pending here
    if (tid == 0) {
        bulk_store(rec + kRecW, smem + kI_QK + 8192, 8192);
        bulk_store(rec + kRecW + 8192, smem + kI_QK + 24576, 8192);
        bulk_commit();
    }
    __syncwarp();
    if (warp == 0 && wait_bar(&st.bar_v, par1, abortp)) {        // V has landed
        tc_fence_after_sync();
        // U~^T (dv x r) = V^T T_u^T with T_u = hi + lo
        const uint64_t dV = make_sdesc_sw128(sV, 16384, 1024);
        const uint64_t dH = make_sdesc_sw128(smem_u32(smem + kI_Tu), 16, 1024), dL = make_sdesc_sw128(smem_u32(smem + kI_TuLo), 16, 1024);
        if (elect_one()) {
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
                if (ks < nb)
                    mma_ss(tU, sdesc_advance(dV, ks * 2048), sdesc_advance(dH, ks * 32), idesc_t, ks > 0);
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
                if (ks < nb)
                    mma_ss(tU, sdesc_advance(dV, ks * 2048), sdesc_advance(dL, ks * 32), idesc_t, true);
            mma_commit(&st.bar_mma);
        }
    }
    wait_bar(&st.bar_mma, par3, abortp);
    tc_fence_after_sync();

    {   // U~^T[d][32 tokens] -> record, [half of dv][token group][dv][4 tokens] fp32
        float4* urec = reinterpret_cast<float4*>(rec + kRecU + (d >> 6) * kRecUHalf);
#pragma unroll
        for (int step = 0; step < 2; ++step) {
            const int cbase = colhalf * 32 + step * 16;
            if (cbase >= ci.len) break;     // (neither written nor read)
            uint32_t y[16];
            tmem_ld16(tU + lane_base + cbase, y);
            tmem_wait_ld();
#pragma unroll
            for (int q4 = 0; q4 < 4; ++q4)
                urec[rec_u_index((cbase >> 2) + q4, d & 63)] =
                    make_float4(__uint_as_float(y[4 * q4]), __uint_as_float(y[4 * q4 + 1]),
                                __uint_as_float(y[4 * q4 + 2]), __uint_as_float(y[4 * q4 + 3]));
        }
    }
    tc_fence_before_sync();
    sync();
    if (st.abort_flag) { bail(true); return false; }
    if (tid == 0) bulk_wait_read_all();
    return true;
}

constexpr uint32_t kStateTmemCols = 512;
constexpr uint32_t kS_Rec = 0;                 // record image (74496 B, padded to 74752)
constexpr uint32_t kS_Q = kRecQg;              // Q tile in Qg's place, 2 halves [64 x 128 B]
constexpr uint32_t kS_K = 74752;               // K tile, 2 halves [64 x 128 B]
constexpr uint32_t kStageBytes = kS_K + 16384;                  // 91136
static_assert(kRecBytes <= kS_K && kS_K % 1024 == 0, "tiles are 1024-byte aligned");
constexpr uint32_t kS_Out = 2 * kStageBytes;   // o staging [64 tokens][128 dv] bf16
// TMEM columns
constexpr uint32_t kT_D1 = 0, kT_Y = 64 /* two tiles of 64 */, kT_D4 = 192, kT_S = 320, kT_U = 384,
                   kT_Us = 416, kT_UsLo = 448;


}  // namespace gdn
