// The intra-chunk quantities as a PERSISTENT pipeline: one CTA of 25 warps per SM streams (chunk, v-head) items through
// roles that hand over by mbarriers, so that the loads, the two groups of tensor-core products, the masks, the
// triangular solves and the write-out of different items run side by side.
//
//   warps 0-3, 17, 19  masks     the accumulator of [Q;K] K^T -> P (bf16, staged over Q) and A (fp32)
//   warps 4-7          write-out U~ and W from TMEM, staged over what the products have read
//   warps 8-15         solves    two groups of four warps, every other item each: T = (I + A)^{-1} straight into the
//                                bf16 images of T diag(beta) (hi, lo) and T diag(beta e^b) that the products read
//   warp 16            Q and K tiles in
//   warp 18            P images out, V tiles in, in Q's place
//   warp 20            items     which chunk and head comes next, gate prefix sums, the record's vectors
//   warp 21            [Q;K] K^T
//   warp 22            V^T T_u^T and K^T T_w^T
//   warps 23, 24       U~ and W images out, every other item each; where a concurrent state pass waits for the records
//                      they publish them
//
// What bounds it: 7680 tokens at 32 heads move 128 MB in and 164 of 222 MB out to DRAM, 45 us at the copy rate, in 64 us;
// the rest is the first item's way through (6 us) and the last's.  One CTA of 256 threads per item, four to an SM
// (intra_item, which few items still run as), takes 88 us there: its warps meet at barriers between phases in which two
// or four of eight have work, and four items' 46 KB of code run at the pace of instruction fetches.  What was found on
// the way, 7680 tokens:
//   * the code that the roles repeat must fit the SM's instruction cache: loops unrolled and waits in line (64 KB) 155 us,
//     rolled 93, waits out of line (46 KB) 72;
//   * records leave by bulk copies from staged images: written by the warps' own stores 66 us, of which 10 went to U~'s 32
//     KB and 6 to P's 8 KB at whatever address, because stores held up in the load/store unit hold up every shared-memory
//     access behind them (the same values to shared memory only: 58);
//   * a load into a register is waited for at the next call of a function: the gates come by asynchronous copies (72 -> 67).
//
// Shared memory: four slots of Q/K tiles, three buffers of A, the three images of T once per solve group, and a ring of
// eight items' vectors.  A slot in turn holds Q and K, P over half of Q, V over Q, then half of U~ over V and W over K; the
// other half of U~ is staged over the images of T_u.
#pragma once
#include "gdn_prefill_device.cuh"

namespace gdn {

constexpr int kProdWarps = 25, kProdThreads = kProdWarps * 32;
constexpr int kPWriteWarp0 = 4, kPSolveWarp0 = 8, kPLoadWarp = 16, kPMaskWarpP = 17, kPLoadVWarp = 18, kPMaskWarpA = 19, kPItemWarp = 20,
              kPGramWarp = 21, kPMmaWarp = 22, kPStoreWarp0 = 23;
static_assert(kPMaskWarpP % 4 == 1 && kPMaskWarpA % 4 == 3, "they read the accumulator's rows 32-63 and 96-127");
constexpr int kProdSlots = 4;            // Q/K tiles in flight
constexpr int kProdInfos = 8;            // items announced and not written out
// A slot: 2 halves x [128 rows x 128 B], rows 0-63 Q (then V), rows 64-127 K (then the W image)
constexpr uint32_t kPSlotBytes = 32768;
// images of T, MN-major: a 128-byte row per column i of T, 64 rows r of T in it, 128B-swizzled
constexpr uint32_t kPImgW = 0, kPImgHi = 8192, kPImgLo = 16384, kPImgBytes = 24576;
// A and T^T, fp32: rows 0-31 have 32 columns, rows 32-63 all 64 (pitches of 4 mod 32 words: no bank conflicts)
constexpr int kPAs = 3, kPLdTop = 36, kPLdLow = 68, kPLow = 32 * kPLdTop;
constexpr uint32_t kPABytes = (kPLow + 32 * kPLdLow) * 4;
struct ItemInfo {
    alignas(16) float nb2[kChunk];       // -b_r log2(e), b the inclusive log-decay prefix
    float beta[kChunk];                  // beta_r (0 past the chunk's length)
    float bg[kChunk];                    // beta_r e^{b_r}
    int32_t t0, len, hv, hqk;
    int32_t rec;                         // record number, chunk * Hv + hv; < 0: no more items
    int32_t pad[3];
};
constexpr uint32_t kPS_Slot = 0, kPS_Img = kPS_Slot + kProdSlots * kPSlotBytes, kPS_A = kPS_Img + 2 * kPImgBytes,
                   kPS_Info = kPS_A + kPAs * kPABytes, kPS_End = kPS_Info + kProdInfos * sizeof(ItemInfo);
constexpr uint32_t kProdSmem = kPS_End + 1024;
static_assert(kPS_A % 1024 == 0 && kPS_Info % 16 == 0 && sizeof(ItemInfo) % 16 == 0, "alignment");
constexpr uint32_t kProdTmemCols = 512;
// TMEM columns, two tiles of 64 each
constexpr uint32_t kPT_Gram = 0, kPT_U = 128, kPT_W = 256;

// How often a producer of the second part that is as far ahead of the first chain as the tables allow asks again before
// it goes on regardless.
constexpr int kPacePolls = 1 << 11;

// Where a CTA's items come from.
enum ItemSource {
    kItemsInline,       // every chunk of a batch of at most kSmallSeqs sequences, found from cu_seqlens
    kItemsTable,        // every chunk, from the chunk table
    kItemsFirst,        // the items before the cut, in processing order
    kItemsQueue         // those behind it, from a queue; each record is published through its flag
};

// Four 8x8 matrices of 16-bit pairs, i.e. 8 rows x 4 fp32 each: lane l supplies the address of row l % 8 of matrix l / 8
// and gets word l % 4 of row l / 4 of each.
__device__ __forceinline__ void ldmatrix_x4(const void* row, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(smem_u32(row))
                 : "memory");
}
__device__ __forceinline__ void mma_m16n8k8_tf32(float (&c)[4], const uint32_t (&a)[4], const uint32_t b0, const uint32_t b1) {
    const uint32_t b[2] = {b0, b1};
    mma_m16n8k8_tf32(c, a, b);
}
__device__ __forceinline__ float round_tf32(float x) { return __uint_as_float(to_tf32(x)); }

// ------------------------------------------------------------------ the solve
// T = (I + A)^{-1} of the strictly lower-triangular 64x64 A (fp32, row-major), by two warps p = 0, 1 and two helpers:
//   1. warp p inverts the diagonal 16x16 blocks 2p and 2p + 1 by forward substitution (thread = column),
//   2. joins them into the inverse of their 32x32 block: T_IJ = -T_II (A_IJ T_JJ),
//   3. and takes, with a helper for half of the columns, the rows 16 p .. of the transpose of the last block:
//      X = -T_b (A_ba T_a).
// Everything is formed TRANSPOSED.  A thread of step 1 holds a column of T, which is a row of the images that the
// products read; a product of steps 2 and 3 has T's own transpose as its left operand, its result is the left
// operand of the next one as it lies in registers (accumulator columns 2t, 2t + 1 taken as k = t and t + 4, the right
// operand's rows to match), and the last result goes to the images in pairs.  T^T is kept, rounded to tf32, where A's
// transposed blocks would be: on and above the diagonal, which only these products read.
struct SolveImages {
    uint8_t* img;
    // an adjacent pair of rows r, r + 1 of T in the column whose factors these are
    __device__ __forceinline__ static void pair(const float2 t, const float fb, const float fg, uint32_t& w, uint32_t& hi, uint32_t& lo) {
        const float2 u = mul2(t, make_float2(fb, fb)), v = mul2(t, make_float2(fg, fg));
        hi = pack_bf16(u.x, u.y);
        const float2 rest = fma2(make_float2(__uint_as_float(hi << 16), __uint_as_float(hi & 0xffff0000u)), make_float2(-1.f, -1.f), u);
        lo = pack_bf16(rest.x, rest.y);
        w = pack_bf16(v.x, v.y);
    }
    // an accumulator fragment of -T^T: rows i0 + g (+ 8), columns r0 + 2t, + 1; the rows' factors negated
    __device__ __forceinline__ void fragment(const float (&c)[4], const int i, const int r0, const int t, const float (&fb)[2],
                                             const float (&fg)[2]) const {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            uint32_t w, hi, lo;
            pair(make_float2(c[2 * h], c[2 * h + 1]), fb[h], fg[h], w, hi, lo);
            uint8_t* at = img + sw128_offset(i + 8 * h, r0 >> 3) + 4 * t;
            *reinterpret_cast<uint32_t*>(at + kPImgW) = w;
            *reinterpret_cast<uint32_t*>(at + kPImgHi) = hi;
            *reinterpret_cast<uint32_t*>(at + kPImgLo) = lo;
        }
    }
};

// Step 1's substitution: column j of (I + A_II)^{-1}, right-looking, four columns of A at a time.
__device__ __forceinline__ void invert_column(const float* blk, const int ld, const int j, float (&t)[16]) {
#pragma unroll
    for (int r = 0; r < 16; ++r) t[r] = (r == j) ? 1.f : 0.f;
#pragma unroll
    for (int c = 0; c < 16; c += 4) {
#pragma unroll
        for (int r = c + 1; r < 16; ++r) {
            const float4 a = *reinterpret_cast<const float4*>(blk + r * ld + c);
            t[r] = fmaf(-a.x, t[c], t[r]);
            if (r > c + 1) t[r] = fmaf(-a.y, t[c + 1], t[r]);
            if (r > c + 2) t[r] = fmaf(-a.z, t[c + 2], t[r]);
            if (r > c + 3) t[r] = fmaf(-a.w, t[c + 3], t[r]);
        }
    }
}

// An accumulator fragment (rounded) as the left operand of eight k, columns 2t and 2t + 1 as k = t and t + 4.
__device__ __forceinline__ void as_left_operand(const float (&c)[4], uint32_t (&a)[4]) {
    a[0] = to_tf32(c[0]);
    a[1] = to_tf32(c[2]);
    a[2] = to_tf32(c[1]);
    a[3] = to_tf32(c[3]);
}

// Step 2 for the 32x32 diagonal block L whose columns begin at i0.
__device__ __forceinline__ void join_blocks(float* L, const int ld, const int i0, const int lane, const SolveImages im,
                                            const ItemInfo& info) {
    const int g = lane >> 2, t = lane & 3;
    float x[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
    {   // X^T = T_JJ^T A_IJ^T
        uint32_t a[2][4], b[2][4];
#pragma unroll
        for (int ks = 0; ks < 2; ++ks) ldmatrix_x4(L + (lane & 15) * ld + 8 * ks + 4 * (lane >> 4), a[ks]);
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) {         // both k-steps of eight rows of A_IJ
            ldmatrix_x4(L + (16 + 8 * nt + (lane & 7)) * ld + 4 * (lane >> 3), b[nt]);
#pragma unroll
            for (int k = 0; k < 4; ++k) b[nt][k] = to_tf32(__uint_as_float(b[nt][k]));
        }
#pragma unroll
        for (int ks = 0; ks < 2; ++ks)
#pragma unroll
            for (int nt = 0; nt < 2; ++nt) mma_m16n8k8_tf32(x[nt], a[ks], b[nt][2 * ks], b[nt][2 * ks + 1]);
    }
    const int i = i0 + g;
    const float fb[2] = {-info.beta[i], -info.beta[i + 8]}, fg[2] = {-info.bg[i], -info.bg[i + 8]};
    uint32_t xa[2][4];
#pragma unroll
    for (int kk = 0; kk < 2; ++kk) as_left_operand(x[kk], xa[kk]);
#pragma unroll 1
    for (int nt = 0; nt < 2; ++nt) {             // -T_IJ^T = X^T T_II^T, T_II^T upper triangular
        float d[4] = {0.f, 0.f, 0.f, 0.f};
        const float* b = L + (16 + 2 * t) * ld + 16 + 8 * nt + g;
        mma_m16n8k8_tf32(d, xa[0], __float_as_uint(b[0]), __float_as_uint(b[ld]));
        if (nt > 0) mma_m16n8k8_tf32(d, xa[1], __float_as_uint(b[8 * ld]), __float_as_uint(b[9 * ld]));
        float* dst = L + g * ld + 16 + 8 * nt + 2 * t;
        *reinterpret_cast<float2*>(dst) = make_float2(round_tf32(-d[0]), round_tf32(-d[1]));
        *reinterpret_cast<float2*>(dst + 8 * ld) = make_float2(round_tf32(-d[2]), round_tf32(-d[3]));
        im.fragment(d, i, i0 + 16 + 8 * nt, t, fb, fg);
    }
}

// Step 3, rows 16 J .. (J = 0, 1) and columns 32 + 8 n0 .. 32 + 8 n1 - 1 of X^T.
__device__ __forceinline__ void merge_blocks(const float* sA, const int J, const int n0, const int n1, const int lane, const SolveImages im,
                                             const ItemInfo& info) {
    const int g = lane >> 2, t = lane & 3;
    float y[4][4] = {};
#pragma unroll 1
    for (int K = J; K < 2; ++K) {                // Y^T = T_a^T A_ba^T, T_a^T upper triangular
        uint32_t a[2][4];
#pragma unroll
        for (int ks = 0; ks < 2; ++ks)
            ldmatrix_x4(sA + (16 * J + (lane & 15)) * kPLdTop + 16 * K + 8 * ks + 4 * (lane >> 4), a[ks]);
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            if (nt >= 2 && n1 == 2) break;
            uint32_t b[4];                       // (rounded by the mask warps)
            ldmatrix_x4(sA + kPLow + (8 * nt + (lane & 7)) * kPLdLow + 16 * K + 4 * (lane >> 3), b);
            mma_m16n8k8_tf32(y[nt], a[0], b[0], b[1]);
            mma_m16n8k8_tf32(y[nt], a[1], b[2], b[3]);
        }
    }
    const int i = 16 * J + g;
    const float fb[2] = {-info.beta[i], -info.beta[i + 8]}, fg[2] = {-info.bg[i], -info.bg[i + 8]};
    uint32_t ya[4][4];
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) as_left_operand(y[kk], ya[kk]);
#pragma unroll 1
    for (int nt = n0; nt < n1; ++nt) {           // -X^T = Y^T T_b^T
        float d[4] = {0.f, 0.f, 0.f, 0.f};
        const float* b = sA + kPLow + 2 * t * kPLdLow + 32 + 8 * nt + g;
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
            if (kk <= nt)
                mma_m16n8k8_tf32(d, ya[kk], __float_as_uint(b[8 * kk * kPLdLow]), __float_as_uint(b[(8 * kk + 1) * kPLdLow]));
        im.fragment(d, i, 32 + 8 * nt, t, fb, fg);
    }
}

// ------------------------------------------------------------------ the role of a CTA
// Item k of the CTA's stream uses place k mod depth of each ring, in its use k / depth.
template <int kDepth> struct Place {
    int at;
    uint32_t par;            // parity of the k-th item's phase
    __device__ __forceinline__ explicit Place(uint32_t k) : at(k % kDepth), par((k / kDepth) & 1u) {}
};

// The mbarriers: a place per slot, announced item or tile.
enum ProdBars {
    kBQk = 0,                                // Q and K tiles have landed
    kBP = kBQk + kProdSlots,                 // the P image is staged
    kBV = kBP + kProdSlots,                  // the V tile has landed
    kBStaged = kBV + kProdSlots,             // the W image is staged
    kBSlot = kBStaged + kProdSlots,          // both have left: the slot is free
    kBItem = kBSlot + kProdSlots,            // an item's place is known
    kBGates = kBItem + kProdInfos,           // its vectors too
    kBInfoFree = kBGates + kProdInfos,       // all that read them have
    kBPub = kBInfoFree + kProdInfos,         // (published records) the vectors and P are complete
    kBGram = kBPub + kProdInfos,             // [Q;K] K^T
    kBGramFree = kBGram + 2,                 // it has been read
    kBA = kBGramFree + 2,                    // A in shared memory
    kBAFree = kBA + kPAs,
    kBHalf = kBAFree + kPAs,                 // the two warps of a solve between its second and third step
    kBImg = kBHalf + 2,                      // images of T
    kBImgFree = kBImg + 2,
    kBU = kBImgFree + 2,                     // U~^T
    kBW = kBU + 2,                           // W^T
    kBUwFree = kBW + 2,
    kBUStaged = kBUwFree + 2,                // the U~ image is staged
    kBDrain = kBUStaged + 2,                 // an issuer that gave up: its products
    kBCount = kBDrain + 2
};
__device__ __forceinline__ uint32_t prod_bar_count(int i) {
    return i >= kBDrain      ? 1
           : i >= kBUwFree   ? 4             // write-out warps
           : i >= kBImgFree  ? 1
           : i >= kBImg      ? 4             // solving warps
           : i >= kBHalf     ? 2             // the two of the diagonal blocks
           : i >= kBAFree    ? 4             // solving warps
           : i >= kBA        ? 3             // mask warps of A
           : i >= kBGramFree ? 6             // mask warps
           : i >= kBGram     ? 1
           : i >= kBPub      ? 2             // vectors, P
           : i >= kBInfoFree ? 2             // the warps that store
           : i >= kBSlot     ? 1
           : i >= kBStaged   ? 4             // write-out warps
           : i >= kBV        ? 1
           : i >= kBP        ? 3             // mask warps of P
                             : 1;
}

// Bounded wait of a converged warp, the verdict by vote.  A wait that runs out, or finds that another has, sets the
// flag: the role goes on with whatever is there to the end of its item (every access stays inside its buffers) and
// leaves.  Nothing is returned, and nothing branches on it, and the function is out of line, for the sake of the code's
// size: in line each of the kernel's waits is 640 bytes.
static __device__ __noinline__ void prod_wait(const uint32_t bar, const uint32_t parity, const uint32_t abort_flag) {
#pragma unroll 1
    for (uint32_t n = kSpinLimit;;) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "vote.sync.all.pred p, p, 0xffffffff;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return;
        uint32_t f;
        asm volatile("ld.volatile.shared.u32 %0, [%1];" : "=r"(f) : "r"(abort_flag) : "memory");
        if (__any_sync(0xffffffffu, f != 0u)) return;
        if (--n == 0) break;
    }
    asm volatile("st.volatile.shared.u32 [%0], 1;" ::"r"(abort_flag) : "memory");
}

// The role of one CTA of kProdThreads threads; ends with a CTA barrier.
template <ItemSource kSource>
__device__ __forceinline__ void produce_role(const TensorMaps& maps, const PrefillParams& p, uint8_t* ws,
                                             const WorkspaceLayout& lay, uint8_t* smem, const uint32_t* tmem_base) {
    constexpr bool kPublish = kSource == kItemsQueue;
    __shared__ uint64_t bars[kBCount];
    __shared__ int abort_flag;
    __shared__ uint32_t armed[2];            // items whose Q/K and V copies have been started
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    ItemInfo* const infos = reinterpret_cast<ItemInfo*>(smem + kPS_Info);

    if (tid < kBCount) mbar_init(&bars[tid], prod_bar_count(tid));
    if (tid == 0) {
        abort_flag = 0;
        armed[0] = armed[1] = 0;
        prefetch_tensormap(&maps.q);
        prefetch_tensormap(&maps.k);
        prefetch_tensormap(&maps.v);
    }
    fence_barrier_init();
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    // the tables are the previous kernel's, and the workspace its to read (the queue's launch feeds its predecessor)
    if constexpr (kSource != kItemsQueue) pdl_wait();
    const uint32_t tmem = *tmem_base;
    auto wait = [&](const int first, const int at, const uint32_t parity) { prod_wait(smem_u32(&bars[first + at]), parity, smem_u32(&abort_flag)); };
    auto arrive = [&](const int first, const int at) {       // by a warp that has finished something
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars[first + at]);
    };
    // a warp's item: false where there is none, or where a wait has run out
    auto item_at = [&](const int first, const uint32_t k) {
        const Place<kProdInfos> f(k);
        wait(first, f.at, f.par);
        return (infos[f.at].rec | -*reinterpret_cast<volatile int*>(&abort_flag)) >= 0;
    };

    if (warp == kPItemWarp) {
        // ===================== items: the next one's place and gates are fetched while this one's are worked on
        int32_t* hdr = reinterpret_cast<int32_t*>(ws);
        int n_items = 0;
        int32_t s_t0 = 0, s_t1 = 0, s_first = 0, s_nc = 0;       // kItemsInline: a sequence a lane
        if constexpr (kSource == kItemsInline) {
            if (lane < p.N) {
                s_t0 = p.cu_seqlens[lane];
                s_t1 = p.cu_seqlens[lane + 1];
            }
            const bool ok = warp_bounds_ok(s_t0, s_t1, p.T, lane);
            s_nc = ok ? (s_t1 - s_t0 + kChunk - 1) / kChunk : 0;
            int32_t incl = s_nc;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, d);
                if (lane >= d) incl += y;
            }
            s_first = incl - s_nc;
            n_items = __shfl_sync(0xffffffffu, incl, 31) * p.Hv;
            if (blockIdx.x == 0 && (!ok || (lane == 0 && s_t0 != 0) || (lane == p.N - 1 && s_t1 != p.T)))
                report(p.dev_status, kDevBadCuSeqlens);
        } else if constexpr (kSource == kItemsTable) {
            n_items = hdr[kHdrTotalChunks] * p.Hv;
        } else if constexpr (kSource == kItemsFirst) {
            n_items = hdr[kHdrSplit];
        } else {
            n_items = hdr[kHdrTotalItems];
        }
        int ticket = 0;                          // (kItemsQueue) the next item of the queue, asked for one item ahead
        auto pull = [&] {
            if constexpr (kSource == kItemsQueue) {
                if (lane == 0) ticket = hdr[kHdrSplit] + atomicAdd(&hdr[kHdrItemHead], 1);
            }
        };
        pull();
        // (kItemsQueue) No further ahead of the chains than that what they read next is still in L2, or than it takes to be
        // done in time, as far as the first of them tells; where none seems to come on, no bound.
        int allowed = 0;
        auto pace = [&](const int item) {
            if constexpr (kSource == kItemsQueue) {
#pragma unroll 1
                for (int n = 0; item >= allowed; ++n) {
                    const int at = *reinterpret_cast<volatile int32_t*>(hdr + kHdrProgress);
                    allowed = n == kPacePolls || at >= lay.max_nc ? 0x7fffffff : reinterpret_cast<const int32_t*>(ws + lay.hist)[at];
                    allowed = __shfl_sync(0xffffffffu, allowed, 0);
                }
            }
        };
        // Round k finds item k, works on item k - kAhead's gates, then announces item k and starts the copies of its
        // gates: to shared memory, asynchronously, since a load into a register is waited for at the next call.  (From
        // the queue only one item is announced ahead, and none is left lying while the next has to wait.)
        constexpr int kAhead = kSource == kItemsQueue ? 1 : 3;
        bool more = true;
        int ends = 0, ends_done = 0;            // the end is announced twice, once to either solve group
#pragma unroll 1
        for (uint32_t k = 0;; ++k) {
            int item = static_cast<int>(blockIdx.x + k * gridDim.x);
            if constexpr (kSource == kItemsQueue) item = __shfl_sync(0xffffffffu, ticket, 0);
            more = more && item < n_items;
            int32_t t0 = 0, len = 0, hv = 0, rec_no = -1;
            if (more) {
                pull();
                // the last chunks first, so that what the state pass opens with was written last
                const int place = kSource == kItemsInline || kSource == kItemsTable ? n_items - 1 - item : item;
                int c = place / p.by_hv;
                hv = place - c * p.Hv;
                if constexpr (kSource == kItemsInline) {
                    const unsigned here = __ballot_sync(0xffffffffu, c >= s_first && c < s_first + s_nc);
                    const int seq = (__ffs(here) - 1) & 31;
                    t0 = __shfl_sync(0xffffffffu, s_t0 + (c - s_first) * kChunk, seq);
                    len = min(kChunk, __shfl_sync(0xffffffffu, s_t1, seq) - t0);
                } else {
                    if constexpr (kSource != kItemsTable) c = reinterpret_cast<const int32_t*>(ws + lay.order)[c];
                    const ChunkInfo ci = reinterpret_cast<const ChunkInfo*>(ws + lay.chunks)[c];
                    t0 = ci.t0;
                    len = ci.len;
                }
                rec_no = c * p.Hv + hv;
            }
            if (k >= kAhead) {
                cp_async_wait<kAhead - 1>();
                __syncwarp();
                const Place<kProdInfos> f(k - kAhead);
                ItemInfo& info = infos[f.at];
                const int rec_done = info.rec;
                if (rec_done >= 0) {
                    // inclusive prefix sum of the log gates over the chunk, two tokens per lane
                    const float2 g = *reinterpret_cast<const float2*>(&info.nb2[2 * lane]), beta = *reinterpret_cast<const float2*>(&info.beta[2 * lane]);
                    float incl = g.x + g.y;
#pragma unroll 1
                    for (int d = 1; d < 32; d <<= 1) {
                        const float y = __shfl_up_sync(0xffffffffu, incl, d);
                        if (lane >= d) incl += y;
                    }
                    const float kLog2e = 1.4426950408889634f;
                    const float b1 = incl, b0 = incl - g.y;
                    const float bC = __shfl_sync(0xffffffffu, incl, 31);
                    const float e0 = ex2_approx(b0 * kLog2e), e1 = ex2_approx(b1 * kLog2e);
                    *reinterpret_cast<float2*>(&info.nb2[2 * lane]) = make_float2(-b0 * kLog2e, -b1 * kLog2e);
                    *reinterpret_cast<float2*>(&info.bg[2 * lane]) = make_float2(beta.x * e0, beta.y * e1);
                    arrive(kBGates, f.at);
                    // the record's vectors: e^{b_C - b_c}, scale e^{b_r}, and e^{b_C}
                    uint8_t* rec = ws + lay.records + static_cast<size_t>(rec_done) * kRecBytes;
                    *reinterpret_cast<float2*>(rec + kRecDecay + 8 * lane) =
                        make_float2(ex2_approx((bC - b0) * kLog2e), ex2_approx((bC - b1) * kLog2e));
                    *reinterpret_cast<float2*>(rec + kRecEb + 8 * lane) = make_float2(p.scale * e0, p.scale * e1);
                    if (lane == 0)
                        *reinterpret_cast<float2*>(rec + kRecGammaC) =
                            make_float2(ex2_approx(bC * kLog2e), __int_as_float((info.len + 15) >> 4));
                    if constexpr (kPublish) arrive(kBPub, f.at);
                } else {
                    arrive(kBGates, f.at);
                    if (++ends_done == 2) break;
                }
            }
            if (ends < 2) {
                if (more) pace(item);
                else ++ends;
                const Place<kProdInfos> f(k);
                ItemInfo& info = infos[f.at];
                wait(kBInfoFree, f.at, f.par ^ 1u);
                if (lane == 0) {
                    info.t0 = t0;
                    info.len = len;
                    info.hv = hv;
                    info.hqk = hv / p.by_group;
                    info.rec = rec_no;
                }
                arrive(kBItem, f.at);
                // (rows past the chunk's length: 0, and so nothing downstream changes by them)
                if (more) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int r = lane + 32 * h;
                        const size_t th = static_cast<size_t>(t0 + min(r, len - 1)) * p.Hv + hv;
                        cp_async_4(&info.nb2[r], p.g + th, r < len);
                        cp_async_4(&info.beta[r], p.beta + th, r < len);
                    }
                }
            }
            cp_async_commit();
            if (*reinterpret_cast<volatile int*>(&abort_flag) != 0) break;
        }
        cp_async_wait<0>();
    } else if (warp == kPLoadWarp) {
        // ===================== Q and K tiles
#pragma unroll 1
        for (uint32_t k = 0; item_at(kBItem, k); ++k) {
            const ItemInfo& info = infos[k % kProdInfos];
            const int t0 = info.t0, x = info.hqk * kD;
            const Place<kProdSlots> s(k);
            if (elect_one()) {          // towards L2 while the slot is taken
#pragma unroll 1
                for (int h = 0; h < kD; h += 64) {
                    tma_prefetch_2d(&maps.q, x + h, t0);
                    tma_prefetch_2d(&maps.k, x + h, t0);
                    tma_prefetch_2d(&maps.v, info.hv * kD + h, t0);
                }
            }
            __syncwarp();
            wait(kBSlot, s.at, s.par ^ 1u);
            if (elect_one()) {
                uint8_t* slot = smem + kPS_Slot + s.at * kPSlotBytes;
                uint64_t* bar = &bars[kBQk + s.at];
                armed[0] = k + 1;
                mbar_expect_tx(bar, 32768);
#pragma unroll 1
                for (int h = 0; h < 2; ++h, slot += 16384) {
                    tma_load_2d(slot, &maps.q, x + 64 * h, t0, bar);
                    tma_load_2d(slot + 8192, &maps.k, x + 64 * h, t0, bar);
                }
            }
            __syncwarp();
        }
    } else if (warp == kPLoadVWarp) {
        // ===================== P images out, V tiles in: both in Q's place
#pragma unroll 1
        for (uint32_t k = 0; item_at(kBItem, k); ++k) {
            const Place<kProdInfos> f(k);
            const ItemInfo& info = infos[f.at];
            // (read before the wait: should it run out, the item's place may be another's by then)
            const int t0 = info.t0, x = info.hv * kD;
            const uint32_t p_bytes = ((info.len + 15) >> 4) * kRecPBlock;
            uint8_t* const rec_p = ws + lay.records + static_cast<size_t>(info.rec) * kRecBytes + kRecP;
            const Place<kProdSlots> s(k);
            wait(kBP, s.at, s.par);
            if (lane == 0) {
                uint8_t* slot = smem + kPS_Slot + s.at * kPSlotBytes;
                uint64_t* bar = &bars[kBV + s.at];
                bulk_store(rec_p, slot, p_bytes);
                bulk_commit();
                bulk_wait_read_all();
                armed[1] = k + 1;
                mbar_expect_tx(bar, 16384);
                tma_load_2d(slot, &maps.v, x, t0, bar);
                tma_load_2d(slot + 16384, &maps.v, x + 64, t0, bar);
                mbar_arrive(&bars[kBInfoFree + f.at]);
                if constexpr (kPublish) {
                    bulk_wait_all();
                    mbar_arrive(&bars[kBPub + f.at]);
                }
            }
            __syncwarp();
        }
    } else if (warp == kPGramWarp) {
        // ===================== [Q;K] (128 x 128, K-major) times K^T: lanes 0-63 = q.k, lanes 64-127 = k.k
        const uint32_t idesc = make_idesc_bf16(128, 64, false, false);
        const uint64_t dA = make_sdesc_sw128(smem_u32(smem + kPS_Slot), 16, 1024);
#pragma unroll 1
        for (uint32_t k = 0; item_at(kBItem, k); ++k) {
            const Place<kProdSlots> s(k);
            const Place<2> b(k);
            wait(kBGramFree, b.at, b.par ^ 1u);
            wait(kBQk, s.at, s.par);
            tc_fence_after_sync();
            if (elect_one()) {
                const uint32_t tG = tmem + kPT_Gram + 64 * b.at;
                uint64_t a = sdesc_advance(dA, s.at * kPSlotBytes);
#pragma unroll 1
                for (int h = 0; h < 2; ++h, a = sdesc_advance(a, 16384))
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks)
                        mma_ss(tG, sdesc_advance(a, 32 * ks), sdesc_advance(a, 32 * ks + 8192), idesc, h + ks > 0);
                mma_commit(&bars[kBGram + b.at]);
            }
            __syncwarp();
        }
    } else if (warp == kPMmaWarp) {
        // ===================== U~^T (dv x r) = V^T T_u^T, T_u = hi + lo; W^T (dk x r) = K^T T_w^T: the raw V and K tiles
        // read MN-major, the images of T too
        const uint32_t s0 = smem_u32(smem);
        const uint64_t dV = make_sdesc_sw128(s0 + kPS_Slot, 16384, 1024), dT = make_sdesc_sw128(s0 + kPS_Img, 8192, 1024);
#pragma unroll 1
        for (uint32_t k = 0; item_at(kBItem, k); ++k) {
            const int nb = (infos[k % kProdInfos].len + 15) >> 4;       // 16-token blocks that hold tokens
            const Place<kProdSlots> s(k);
            const Place<2> b(k);
            wait(kBUwFree, b.at, b.par ^ 1u);
            wait(kBV, s.at, s.par);
            wait(kBImg, b.at, b.par);
            tc_fence_after_sync();
            if (elect_one()) {
                // T is lower triangular: k-step ks (columns 16 ks ..) has rows, here columns of the result, 16 ks .. only
                const uint32_t id0 = make_idesc_bf16(128, 64, true, true), id_step = make_idesc_bf16(0, 16, false, false) - make_idesc_bf16(0, 0, false, false);
                const uint32_t tU = tmem + kPT_U + 64 * b.at;
                const uint64_t v = sdesc_advance(dV, s.at * kPSlotBytes), t = sdesc_advance(dT, b.at * kPImgBytes);
#pragma unroll 1
                for (int h = 0; h < 2 * nb; ++h) {          // T_u's high parts, then the low ones
                    const int ks = h < nb ? h : h - nb;
                    mma_ss(tU + 16 * ks, sdesc_advance(v, 2048 * ks), sdesc_advance(t, 2080 * ks + (h < nb ? kPImgHi : kPImgLo)),
                           id0 - id_step * ks, h > 0);
                }
                mma_commit(&bars[kBU + b.at]);
#pragma unroll 1
                for (int ks = 0; ks < nb; ++ks)
                    mma_ss(tU + (kPT_W - kPT_U) + 16 * ks, sdesc_advance(v, 2048 * ks + 8192), sdesc_advance(t, 2080 * ks + kPImgW),
                           id0 - id_step * ks, ks > 0);
                mma_commit(&bars[kBW + b.at]);
            }
            __syncwarp();
        }
    } else if (warp >= kPStoreWarp0) {
        // ===================== U~ and W images out; where another kernel waits for them, records are published in order
#pragma unroll 1
        for (uint32_t k = warp - kPStoreWarp0; item_at(kBItem, k); k += 2) {
            const Place<kProdInfos> f(k);
            const Place<kProdSlots> s(k);
            const Place<2> b(k);
            const ItemInfo& info = infos[f.at];
            const int rec_no = info.rec;
            const uint32_t u_bytes = ((info.len + 15) >> 4) * kRecUBlock;
            uint8_t* rec = ws + lay.records + static_cast<size_t>(rec_no) * kRecBytes;
            const uint8_t* slot = smem + kPS_Slot + s.at * kPSlotBytes;
            wait(kBUStaged, b.at, b.par);
            if (lane == 0) {
                bulk_store(rec + kRecU + kRecUHalf, smem + kPS_Img + b.at * kPImgBytes + kPImgHi, u_bytes);
                bulk_commit();
                bulk_store(rec + kRecU, slot, min(u_bytes, 8192u));
                if (u_bytes > 8192) bulk_store(rec + kRecU + 8192, slot + 16384, u_bytes - 8192);
                bulk_commit();
            }
            __syncwarp();
            wait(kBStaged, s.at, s.par);
            if (lane == 0) {
                bulk_store(rec + kRecW, slot + 8192, 8192);
                bulk_store(rec + kRecW + 8192, slot + 24576, 8192);
                bulk_commit();
                bulk_wait_read<2>();
                mbar_arrive(&bars[kBImgFree + b.at]);
                bulk_wait_read<0>();
                mbar_arrive(&bars[kBSlot + s.at]);
            }
            __syncwarp();
            if constexpr (kPublish) {
                wait(kBPub, f.at, f.par);
                if (lane == 0) {
                    bulk_wait_all();
                    fence_proxy_async_all();
                    __threadfence();
                    st_release_u32(reinterpret_cast<uint32_t*>(ws + lay.flags) + rec_no, abort_flag == 0 ? 1u : 2u);     // 2 = after a timeout
                }
            }
            arrive(kBInfoFree, f.at);
        }
    } else if (warp < kPWriteWarp0 || warp == kPMaskWarpP || warp == kPMaskWarpA) {
        // ===================== masks.  Accumulator row of this thread: TMEM lane 32 (warp % 4) + lane; lanes 0-63 hold q.k
        // rows (-> P), lanes 64-127 k.k rows (-> A), either times e^{b_r - b_i}, which is one exponential everywhere (split
        // at b_31 the decay has a larger error, and outputs differ in their last bit).  Warps 0-3 take the 32 columns that
        // hold their rows' diagonal, the two others the columns 0-31 of rows 32-63.
        const bool below = warp >= kPWriteWarp0;
        const int half = warp & 1, r = 32 * half + lane, c0 = below ? 0 : 32 * half;
        const int last = lane - ((warp >> 1) & 1);               // keep columns i <= r of P, i < r of A
#pragma unroll 1
        for (uint32_t k = 0; item_at(kBGates, k); ++k) {
            int is_p = (warp & 2) == 0;                          // (opaque: two copies of what follows are too many)
            asm volatile("" : "+r"(is_p));
            const Place<kProdInfos> f(k);
            const Place<2> b(k);
            const ItemInfo& info = infos[f.at];
            const int len = info.len;
            const Place<kPAs> a(k);
            const float nbr2 = info.nb2[r];
            const float rowscale = is_p ? p.scale : info.beta[r];        // the output scale rides on P
            if (!is_p) wait(kBAFree, a.at, a.par ^ 1u);
            wait(kBGram, b.at, b.par);
            tc_fence_after_sync();
            if (32 * half < len) {       // (rows of a half without tokens are not read)
                uint8_t* const sP = smem + kPS_Slot + (k % kProdSlots) * kPSlotBytes;      // P is staged over Q
                float* const rowA = reinterpret_cast<float*>(smem + kPS_A + a.at * kPABytes) +
                                    (half ? kPLow + lane * kPLdLow : lane * kPLdTop);
                const uint32_t tG = tmem + kPT_Gram + 64 * b.at + (static_cast<uint32_t>((warp & 3) * 32) << 16);
#pragma unroll 1
                for (int c = c0; c < c0 + 32; c += 16) {
                    uint32_t x[16];
                    tmem_ld16(tG + c, x);
                    tmem_wait_ld();
                    float2 val[8];
#pragma unroll
                    for (int q4 = 0; q4 < 4; ++q4) {
                        const float4 f4 = *reinterpret_cast<const float4*>(info.nb2 + c + 4 * q4);
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            float2 z = add2(make_float2(-nbr2, -nbr2), e ? make_float2(f4.z, f4.w) : make_float2(f4.x, f4.y));
                            z = make_float2(ex2_approx(z.x), ex2_approx(z.y));
                            const int i = 4 * q4 + 2 * e;
                            val[2 * q4 + e] = mul2(mul2(make_float2(rowscale, rowscale), make_float2(__uint_as_float(x[i]), __uint_as_float(x[i + 1]))), z);
                        }
                    }
                    if (below) {
                        if (!is_p) {         // (operands of tf32 products alone)
#pragma unroll
                            for (int e = 0; e < 8; ++e) val[e] = make_float2(round_tf32(val[e].x), round_tf32(val[e].y));
                        }
                    } else {                 // what lies above the diagonal is discarded
                        const int keep = last - (c - c0);
#pragma unroll
                        for (int e = 0; e < 8; ++e) val[e] = make_float2(2 * e <= keep ? val[e].x : 0.f, 2 * e < keep ? val[e].y : 0.f);
                    }
                    if (is_p) {
#pragma unroll
                        for (int h = 0; h < 2; ++h)
                            *reinterpret_cast<uint4*>(sP + sw128_offset(r, (c >> 3) + h)) =
                                make_uint4(pack_bf16(val[4 * h].x, val[4 * h].y), pack_bf16(val[4 * h + 1].x, val[4 * h + 1].y),
                                           pack_bf16(val[4 * h + 2].x, val[4 * h + 2].y), pack_bf16(val[4 * h + 3].x, val[4 * h + 3].y));
                    } else {
#pragma unroll
                        for (int q4 = 0; q4 < 4; ++q4)
                            *reinterpret_cast<float4*>(rowA + c + 4 * q4) =
                                make_float4(val[2 * q4].x, val[2 * q4].y, val[2 * q4 + 1].x, val[2 * q4 + 1].y);
                    }
                }
                if (is_p && half == 0) {     // columns 32-63 of rows 0-31
#pragma unroll
                    for (int h = 4; h < 8; ++h) *reinterpret_cast<uint4*>(sP + sw128_offset(r, h)) = make_uint4(0u, 0u, 0u, 0u);
                }
            }
            tc_fence_before_sync();
            if (is_p) fence_proxy_async_smem();
            arrive(kBGramFree, b.at);
            if (lane == 0) mbar_arrive(&bars[is_p ? kBP + k % kProdSlots : kBA + a.at]);
        }
    } else if (warp >= kPSolveWarp0) {
        // ===================== solves.  Two warps of a group take the diagonal 32x32 blocks, all four the last step.
        const int group = (warp - kPSolveWarp0) >> 2, part = warp & 1, helper = (warp >> 1) & 1;
        const SolveImages im = {smem + kPS_Img + group * kPImgBytes};
        uint32_t half_par = 0;          // of items of more than 32 tokens
#pragma unroll 1
        for (uint32_t k = group; item_at(kBGates, k); k += 2) {
            const Place<2> b(k);
            const ItemInfo& info = infos[k % kProdInfos];
            const int len = info.len;
            const Place<kPAs> a(k);
            float* const sA = reinterpret_cast<float*>(smem + kPS_A + a.at * kPABytes);
            wait(kBA, a.at, a.par);
            if (32 * part < len && !helper) {
                const int j = lane & 15, I = 2 * part + (lane >> 4), i = 16 * I + j;
                float t[16];
                // the 32x32 block of this warp, and a lane's 16x16 one
                float* const L = part ? sA + kPLow + 32 : sA;
                const int ld = part ? kPLdLow : kPLdTop;
                float* const D = L + (lane & 16) * (ld + 1);
                invert_column(D, ld, j, t);
                wait(kBImgFree, group, b.par ^ 1u);      // (and every column of the block has read A_II)
#pragma unroll
                for (int q4 = 0; q4 < 4; ++q4)
                    *reinterpret_cast<float4*>(D + j * ld + 4 * q4) =
                        make_float4(round_tf32(t[4 * q4]), round_tf32(t[4 * q4 + 1]), round_tf32(t[4 * q4 + 2]), round_tf32(t[4 * q4 + 3]));
                const float fb = info.beta[i], fg = info.bg[i];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint32_t w[4], hi[4], lo[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) im.pair(make_float2(t[8 * h + 2 * e], t[8 * h + 2 * e + 1]), fb, fg, w[e], hi[e], lo[e]);
                    uint8_t* at = im.img + sw128_offset(i, 2 * I + h);
                    *reinterpret_cast<uint4*>(at + kPImgW) = make_uint4(w[0], w[1], w[2], w[3]);
                    *reinterpret_cast<uint4*>(at + kPImgHi) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                    *reinterpret_cast<uint4*>(at + kPImgLo) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                }
                __syncwarp();
                if (len > 32 * part + 16) join_blocks(L, ld, 32 * part, lane, im, info);
            } else {
                wait(kBImgFree, group, b.par ^ 1u);      // (no arrival below before the last round's all are in)
            }
            if (len > 32) {
                if (!helper) arrive(kBHalf, group);
                wait(kBHalf, group, half_par);
                half_par ^= 1u;
                merge_blocks(sA, part, 2 * helper, 2 * helper + 2, lane, im, info);
            }
            fence_proxy_async_smem();
            arrive(kBImg, group);
            if (lane == 0) mbar_arrive(&bars[kBAFree + a.at]);
        }
    } else {
        // ===================== write-out.  TMEM lane of this thread: 32 (warp % 4) + lane, a dv / dk index.
        const int q = warp & 3, d = 32 * q + lane;
        const uint32_t lane_base = static_cast<uint32_t>(q * 32) << 16;
#pragma unroll 1
        for (uint32_t k = 0; item_at(kBItem, k); ++k) {
            const Place<kProdInfos> f(k);
            const Place<kProdSlots> s(k);
            const Place<2> b(k);
            const int len = infos[f.at].len;
            const uint32_t tU = tmem + kPT_U + 64 * b.at + lane_base;
            uint8_t* const slot = smem + kPS_Slot + s.at * kPSlotBytes;
            wait(kBU, b.at, b.par);
            tc_fence_after_sync();
            {   // U~^T[d][64 tokens] -> [half of dv][token group][dv][4 tokens] fp32, staged over the (now dead) V tile (dv
                // 0-63, eight token groups in either part of it) and the images of T_u (dv 64-127); blocks without tokens
                // are neither written nor read
                uint8_t* sU = q < 2 ? slot : smem + kPS_Img + b.at * kPImgBytes + kPImgHi;
#pragma unroll 1
                for (int cb = 0; 16 * cb < len; ++cb) {
                    uint32_t y[16];
                    tmem_ld16(tU + 16 * cb, y);
                    tmem_wait_ld();
                    if (q < 2 && cb == 2) sU += 8192;        // (the K tile lies between the parts)
#pragma unroll
                    for (int q4 = 0; q4 < 4; ++q4)
                        reinterpret_cast<float4*>(sU)[rec_u_index(4 * cb + q4, d & 63)] =
                            make_float4(__uint_as_float(y[4 * q4]), __uint_as_float(y[4 * q4 + 1]),
                                        __uint_as_float(y[4 * q4 + 2]), __uint_as_float(y[4 * q4 + 3]));
                }
            }
            fence_proxy_async_smem();
            arrive(kBUStaged, b.at);
            wait(kBW, b.at, b.par);
            tc_fence_after_sync();
            {   // W^T[d][64 tokens] -> bf16, staged over the (now dead) K tile.  MN-major for the state pass's product
                // S W^T: one 128-byte row of 64 tokens per dk index.
                uint8_t* sW = slot + 8192 + (q >> 1) * 16384 + (q & 1) * 4096;
#pragma unroll 1
                for (int cb = 0; cb < 4; ++cb) {
                    uint32_t x[16] = {};            // (no tokens: W is zero there, and so U)
                    if (16 * cb < len) {
                        tmem_ld16(tU + (kPT_W - kPT_U) + 16 * cb, x);
                        tmem_wait_ld();
                    }
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        *reinterpret_cast<uint4*>(sW + sw128_offset(lane, 2 * cb + h)) =
                            make_uint4(pack_bf16(__uint_as_float(x[8 * h + 0]), __uint_as_float(x[8 * h + 1])),
                                       pack_bf16(__uint_as_float(x[8 * h + 2]), __uint_as_float(x[8 * h + 3])),
                                       pack_bf16(__uint_as_float(x[8 * h + 4]), __uint_as_float(x[8 * h + 5])),
                                       pack_bf16(__uint_as_float(x[8 * h + 6]), __uint_as_float(x[8 * h + 7])));
                }
            }
            tc_fence_before_sync();
            fence_proxy_async_smem();
            arrive(kBUwFree, b.at);
            if (lane == 0) mbar_arrive(&bars[kBStaged + s.at]);
        }
    }

    __syncwarp();
    tc_fence_before_sync();
    __syncthreads();
    if (abort_flag != 0) {
        // products still running read shared memory and write TMEM that the CTA is about to give back
        if (warp == kPGramWarp || warp == kPMmaWarp) {
            if (elect_one()) mma_commit(&bars[kBDrain + (warp == kPMmaWarp)]);
            mbar_wait(&bars[kBDrain + (warp == kPMmaWarp)], 0u, 1u << 12);
        }
        if (tid == 0) {
            report(p.dev_status, kDevTimeout);
            // copies already in flight land before the CTA's shared memory goes away
            for (uint32_t back = 1; back <= kProdSlots; ++back) {
                const uint32_t n = armed[0], m = armed[1];
                if (back <= n) mbar_wait(&bars[kBQk + (n - back) % kProdSlots], ((n - back) / kProdSlots) & 1u, 1u << 12);
                if (back <= m) mbar_wait(&bars[kBV + (m - back) % kProdSlots], ((m - back) / kProdSlots) & 1u, 1u << 12);
            }
        }
        __syncwarp();
    }
}

// A kernel's body: TMEM, the role, TMEM back.
template <ItemSource kSource>
__device__ __forceinline__ void produce_cta(const TensorMaps& maps, const PrefillParams& p, uint8_t* ws, const WorkspaceLayout& lay) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align_1024(smem_raw);
    __shared__ uint32_t tmem_base_s;
    const int warp = threadIdx.x >> 5;
    if (warp == kPMmaWarp) {
        tmem_alloc(&tmem_base_s, kProdTmemCols);
        tmem_relinquish();
    }
    produce_role<kSource>(maps, p, ws, lay, smem, &tmem_base_s);
    __syncthreads();
    if (warp == kPMmaWarp) tmem_dealloc(tmem_base_s, kProdTmemCols);
}

}  // namespace gdn
