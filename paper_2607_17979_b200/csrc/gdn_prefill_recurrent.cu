// Prefill of short prompts: blocks of up to 16 tokens on a state tile held in registers, no chunk
// records and no workspace (gdn_token_block.cuh describes a block's algebra and its layout).
//
// The rows of a state tile evolve independently under the gated delta rule, so a (sequence,
// v-head) tile is spread over four CTAs of 32 rows, which two warps carry through the blocks of the
// sequence.  kPipelined: two more warps load and stage the next block (tokens, decays, coefficients)
// meanwhile, in the other half of a double buffer.  Without (prompts of one block, where there may be
// thousands of them and occupancy counts) the two warps do both.  Bound by latency: the token-by-token loop this
// replaces took 0.43 us a token (one L2 round trip each).  One sequence, device time per call: 6 tokens
// 4.9 -> 4.1 us, 12 tokens 7.8 -> 6.1 us; longer prompts: see the routing rule.
#include "gdn_token_block.cuh"
#include "gdn_sm100.cuh"

namespace gdn {

constexpr int kRecWarps = 2;                  // that apply blocks

// CTAs an SM: what the registers allow.  8 tokens: 128 registers whether 7 or 8 are asked for, but the compiler
// spills less for 7 (6 tokens at 8 v-heads 4.58 against 4.72 us, 40 prompts of 8 at 32 v-heads 31.5 against 32.4).
template <int kMax, bool kPipelined>
__global__ void __launch_bounds__(kRecWarps * (kPipelined ? 64 : 32),
                                  kPipelined ? 2 : kMax == 16 ? 6 : kMax == 8 ? 7 : 8)
prefill_recurrent_kernel(const PrefillParams p) {
    using Block = TokenBlock<false, kRecWarps, kMax>;
    __shared__ __align__(16) Block st[kPipelined ? 2 : 1];
    constexpr int kThreads = kRecWarps * (kPipelined ? 64 : 32);
    constexpr int kSplit = kD / Block::kRows;
    const int unit = blockIdx.x / kSplit;
    const int row_base = (blockIdx.x - unit * kSplit) * Block::kRows;
    // (at 16 tokens the compiler spills four times as much around the multiplication: 20 sequences of 16 tokens at 32
    // heads 31.7 -> 32.4 us; elsewhere it is ahead, 6 tokens at 8 heads 4.50 -> 4.17)
    const int n = kMax == 16 && !kPipelined ? unit / p.Hv : unit / p.by_hv;
    const int hv = unit - n * p.Hv;
    const int hqk = hv / p.by_group;
    const int tid = threadIdx.x;
    sm100::pdl_launch_dependents();
    sm100::pdl_wait();

    const int t0 = p.cu_seqlens[n];
    const int t1 = p.cu_seqlens[n + 1];
    const int slot = p.slot_idx ? p.slot_idx[n] : n;
    const bool first_ok = (n != 0) || (t0 == 0);
    const bool last_ok = (n != p.N - 1) || (t1 == p.T);
    if (t0 < 0 || t1 < t0 || t1 > p.T || !first_ok || !last_ok) {
        if (tid == 0) report(p.dev_status, kDevBadCuSeqlens);
        return;
    }
    if (slot < 0 || slot >= p.num_slots) {
        if (slot >= p.num_slots && tid == 0) report(p.dev_status, kDevBadSlot);
        for (int idx = tid; idx < (t1 - t0) * (Block::kRows / 8); idx += kThreads) {
            const int t = t0 + idx / (Block::kRows / 8), c = (idx % (Block::kRows / 8)) * 8;
            *reinterpret_cast<uint4*>(p.o + (static_cast<size_t>(t) * p.Hv + hv) * kD + row_base + c) =
                make_uint4(0u, 0u, 0u, 0u);
        }
        return;
    }

    TokenRows t;
    t.qk_stride = static_cast<size_t>(p.Hqk) * kD;
    t.v_stride = static_cast<size_t>(p.Hv) * kD;
    t.g_stride = p.Hv;
    t.scale = p.scale;
    auto block_at = [&](int tok) {
        const size_t tq = (static_cast<size_t>(tok) * p.Hqk + hqk) * kD, tv = static_cast<size_t>(tok) * p.Hv + hv;
        t.q = p.q + tq;
        t.k = p.k + tq;
        t.v = p.v + tv * kD;
        t.o = p.o + tv * kD;
        t.g = p.g + tv;
        t.beta = p.beta + tv;
        t.count = min(kMax, t1 - tok);
    };
    const size_t tile = (static_cast<size_t>(slot) * p.Hv + hv) * (kD * kD);
    const int blocks = (t1 - t0 + kMax - 1) / kMax;

    if (kPipelined && tid >= kRecWarps * 32) {           // staging warps: block i + 1 while block i is applied
        const int stid = tid - kRecWarps * 32;
        auto stage_sync = [] { asm volatile("bar.sync 1, %0;" ::"n"(kRecWarps * 32) : "memory"); };
        TokenLoads<false, kRecWarps, kMax> ld;
        block_at(t0);
        if (blocks > 0) load_tokens(ld, t, row_base, stid);
        for (int i = 0; i < blocks; ++i) {
            stage_block(t, st[kPipelined ? i & 1 : 0], ld, stid, stage_sync);
            if (i + 1 < blocks) {          // on their way while the others apply this block
                block_at(t0 + (i + 1) * kMax);
                load_tokens(ld, t, row_base, stid);
            }
            __syncthreads();               // block i is staged, block i - 1 has been applied
        }
        return;
    }
    TokenLoads<false, kRecWarps, kMax> ld;
    block_at(t0);
    if (!kPipelined && blocks > 0) load_tokens(ld, t, row_base, tid);
    State<false> s;
    if (p.init_state) {
        load_state<false>(s, p.init_state + tile, row_base);
    } else {
#pragma unroll
        for (auto& c : s[0]) c[0] = c[1] = c[2] = c[3] = 0.f;
    }
    for (int i = 0; i < blocks; ++i) {
        block_at(t0 + i * kMax);
        if constexpr (!kPipelined) {
            if (i > 0) {
                load_tokens(ld, t, row_base, tid);
                __syncthreads();           // the staged block has been read
            }
            stage_block(t, st[0], ld, tid, [] { __syncthreads(); });
        }
        __syncthreads();
        apply_block(t, st[kPipelined ? i & 1 : 0], s, row_base);
    }
    store_state<false>(s, p.final_state + tile, row_base);
}

cudaError_t launch_prefill_recurrent(const PrefillParams& p, int longest, cudaStream_t stream) {
    const long long ctas = static_cast<long long>(p.N) * p.Hv * (8 / kRecWarps);
    if (ctas == 0 || p.T == 0) return cudaSuccess;
    // a bound on the longest sequence picks the variant; longer sequences take more blocks
    auto kernel = longest <= 4    ? prefill_recurrent_kernel<4, false>
                  : longest <= 8  ? prefill_recurrent_kernel<8, false>
                  : longest <= 16 ? prefill_recurrent_kernel<16, false>
                                  : prefill_recurrent_kernel<16, true>;
    return launch_dependent(kernel, dim3(static_cast<unsigned>(ctas)),
                            dim3(kRecWarps * (longest <= 16 ? 32 : 64)), 0, stream, p);
}

}  // namespace gdn
