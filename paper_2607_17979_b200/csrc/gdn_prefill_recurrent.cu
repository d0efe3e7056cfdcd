// Prefill of short prompts: blocks of up to 16 tokens on a state tile held in registers, no chunk
// records and no workspace (gdn_token_block.cuh describes a block's algebra and its layout).
//
// The rows of a state tile evolve independently under the gated delta rule, so a (sequence,
// v-head) tile is spread over four CTAs of two warps; a CTA carries its 32 rows through all
// blocks of its sequence.  Bound by latency: the token-by-token loop this replaces took 0.43 us a
// token (one L2 round trip each), a block of 16 takes about 3.7 us.  One sequence, device time per
// call: 6 tokens 4.9 -> 4.1 us, 12 tokens 7.8 -> 6.1 us, 128 tokens 57 -> 38 us.
#include "gdn_token_block.cuh"
#include "gdn_sm100.cuh"

namespace gdn {

constexpr int kRecWarps = 2;

template <int kMax>
__global__ void __launch_bounds__(kRecWarps * 32, kMax == 16 ? 6 : 8)
prefill_recurrent_kernel(const PrefillParams p) {
    using Block = TokenBlock<false, kRecWarps, kMax>;
    __shared__ __align__(16) Block st;
    constexpr int kSplit = kD / Block::kRows;
    const int unit = blockIdx.x / kSplit;
    const int row_base = (blockIdx.x - unit * kSplit) * Block::kRows;
    const int n = unit / p.Hv;
    const int hv = unit - n * p.Hv;
    const int hqk = hv / (p.Hv / p.Hqk);
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
        for (int idx = tid; idx < (t1 - t0) * (Block::kRows / 8); idx += kRecWarps * 32) {
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
    TokenLoads<false, kRecWarps, kMax> ld;
    block_at(t0);
    load_tokens(ld, t, row_base);
    State<false> s;
    if (p.init_state) {
        load_state<false>(s, p.init_state + tile, row_base);
    } else {
#pragma unroll
        for (auto& c : s[0]) c[0] = c[1] = c[2] = c[3] = 0.f;
    }
    for (int tok = t0; tok < t1;) {
        stage_block(t, st, ld);
        apply_block(t, st, s, row_base);
        tok += kMax;
        if (tok < t1) {
            block_at(tok);
            load_tokens(ld, t, row_base);
            __syncthreads();               // the staged block has been read
        }
    }
    store_state<false>(s, p.final_state + tile, row_base);
}

cudaError_t launch_prefill_recurrent(const PrefillParams& p, int longest, cudaStream_t stream) {
    const long long ctas = static_cast<long long>(p.N) * p.Hv * (8 / kRecWarps);
    if (ctas == 0 || p.T == 0) return cudaSuccess;
    // a bound on the longest sequence picks the block size; longer sequences take more blocks
    auto kernel = longest <= 4   ? prefill_recurrent_kernel<4>
                  : longest <= 8 ? prefill_recurrent_kernel<8>
                                 : prefill_recurrent_kernel<16>;
    return launch_dependent(kernel, dim3(static_cast<unsigned>(ctas)), dim3(kRecWarps * 32), 0, stream, p);
}

}  // namespace gdn
