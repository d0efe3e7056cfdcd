// Decode of L >= 1 new tokens per sequence with the state tile held in registers across the
// tokens, for either orientation of the tile in memory.
//
//   per token:  S <- exp(g) S ;  u = S k ;  S <- S + beta (v - u) k^T ;  o = scale S q
//
// A tile is read once and written once however many tokens are applied, so the 128 KiB of
// traffic per (sequence, v-head) is amortised over L tokens.  The tokens are applied as one block
// (gdn_token_block.cuh); the tile's loads are issued first and the tokens are staged in their shadow.
#include "gdn_token_block.cuh"
#include "gdn_sm100.cuh"

namespace gdn {

// A CTA of kWarps warps takes 16 kWarps of the tile's 128 dv rows (see the launcher), 16 warps an SM.  Tiles [dk][dv],
// 8 tokens: 128 registers whether 14 or 16 warps are asked for, but the compiler spills less for 14 (B = 23, L = 7
// 24.0 against 24.6 us, B = 64 58.0 / 58.5).
template <bool kTransposed, int kWarps, int kMax>
__global__ void __launch_bounds__(kWarps * 32, kTransposed && kWarps == 2 && kMax == 8 ? 7 : 16 / kWarps)
decode_multi_kernel(const DecodeMultiParams mp) {
    using Block = TokenBlock<kTransposed, kWarps, kMax>;
    __shared__ __align__(16) Block st;
    const DecodeParams& p = mp.d;
    constexpr int kSplit = kD / Block::kRows;
    const int unit = blockIdx.x / kSplit;
    const int row_base = (blockIdx.x - unit * kSplit) * Block::kRows;
    const int i = unit / p.Hv;
    const int hv = unit - i * p.Hv;
    const int hqk = hv / (p.Hv / mp.Hqk);
    sm100::pdl_launch_dependents();
    sm100::pdl_wait();

    const size_t tok0 = static_cast<size_t>(i) * mp.L;
    TokenRows t;
    t.q = p.q + (tok0 * mp.Hqk + hqk) * kD;
    t.k = p.k + (tok0 * mp.Hqk + hqk) * kD;
    t.v = p.v + (tok0 * p.Hv + hv) * kD;
    t.g = p.g + tok0 * p.Hv + hv;
    t.beta = p.beta + tok0 * p.Hv + hv;
    t.o = p.o + (tok0 * p.Hv + hv) * kD;
    t.qk_stride = static_cast<size_t>(mp.Hqk) * kD;
    t.v_stride = static_cast<size_t>(p.Hv) * kD;
    t.g_stride = p.Hv;
    t.count = mp.L;
    t.scale = p.scale;

    const int slot = p.slot_idx ? p.slot_idx[i] : i;
    if (slot < 0 || slot >= p.num_slots) {          // padding entry: zero o rows, no state
        if (slot >= p.num_slots && threadIdx.x == 0 && row_base == 0) report(p.dev_status, kDevBadSlot);
        for (int idx = threadIdx.x; idx < mp.L * Block::kRows; idx += kWarps * 32) {
            const int tok = idx / Block::kRows;
            t.o[tok * t.v_stride + row_base + idx - tok * Block::kRows] = __float2bfloat16(0.f);
        }
        return;
    }
    float* tile = p.pool + (static_cast<size_t>(slot) * p.Hv + hv) * (kD * kD);
    TokenLoads<kTransposed, kWarps, kMax> ld;
    load_tokens(ld, t, row_base, threadIdx.x);
    State<kTransposed> s;
    load_state<kTransposed>(s, tile, row_base);
    // (both barriers are passed while the tile's loads are in flight)
    stage_block(t, st, ld, threadIdx.x, [] { __syncthreads(); });
    __syncthreads();
    apply_block(t, st, s, row_base);
    store_state<kTransposed>(s, tile, row_base);
}

namespace {
template <bool kTransposed, int kWarps>
cudaError_t launch_shape(const DecodeMultiParams& mp, int32_t B, cudaStream_t stream) {
    const unsigned grid = static_cast<unsigned>(static_cast<long long>(B) * mp.d.Hv * (8 / kWarps));
    auto kernel = mp.L <= 4   ? decode_multi_kernel<kTransposed, kWarps, 4>
                  : mp.L <= 8 ? decode_multi_kernel<kTransposed, kWarps, 8>
                              : decode_multi_kernel<kTransposed, kWarps, 16>;
    return launch_dependent(kernel, dim3(grid), dim3(kWarps * 32), 0, stream, mp);
}
}  // namespace

cudaError_t launch_decode_multi(const DecodeMultiParams& mp, int32_t B, cudaStream_t stream) {
    const long long units = static_cast<long long>(B) * mp.d.Hv;
    if (units == 0) return cudaSuccess;
    DeviceInfo di;
    const int sms = device_info(&di) == cudaSuccess ? di.sms : 148;
    // Four CTAs of two warps per tile, or two of four, with 16 warps an SM either way.  Up to four tokens
    // a CTA lives little longer than its tile's loads and more, smaller CTAs overlap better; beyond,
    // what every CTA does for its tokens counts.  B = 64, 32 v-heads, two / four warps, us: L = 2 43.0 /
    // 43.8, L = 4 44.8 / 45.5, L = 8 55.7 / 53.8, L = 16 86.5 / 74.0; tiles [dk][dv] L = 2 46.3 / 47.9,
    // L = 8 58.7 / 59.0, L = 16 99.2 / 82.1.  With too few tiles to fill the SMs, two: B = 1, L = 8, 8
    // v-heads 4.0 / 4.3.
    const bool two = mp.L <= 4 || (mp.L <= 8 && (mp.layout != 0 || units * 4 <= 2LL * sms));
    if (mp.layout == 0) return two ? launch_shape<false, 2>(mp, B, stream) : launch_shape<false, 4>(mp, B, stream);
    return two ? launch_shape<true, 2>(mp, B, stream) : launch_shape<true, 4>(mp, B, stream);
}

}  // namespace gdn

// ---- in-place transpose of state tiles ([dv][dk] <-> [dk][dv]) ---------------------------------
// One CTA per (entry, v-head) tile.  The 128x128 tile is walked as 4x4 blocks of 32x32; a block
// pair (a, b) and (b, a) is read into two padded shared tiles and written back swapped and
// transposed, so the tile never needs a second copy in memory.
namespace gdn {

__global__ void __launch_bounds__(256)
state_transpose_kernel(float* pool, const int32_t* slot_idx, int32_t Hv, int32_t num_slots,
                       int32_t* dev_status) {
    __shared__ float ta[32][33], tb[32][33];
    const int i = blockIdx.x / Hv, hv = blockIdx.x - i * Hv;
    const int slot = slot_idx ? slot_idx[i] : i;
    if (slot < 0 || slot >= num_slots) {
        if (slot >= num_slots && threadIdx.x == 0) report(dev_status, kDevBadSlot);
        return;
    }
    float* tile = pool + (static_cast<size_t>(slot) * Hv + hv) * (kD * kD);
    const int c = threadIdx.x & 31, r0 = threadIdx.x >> 5;   // 8 rows per sweep
    for (int a = 0; a < 4; ++a)
        for (int b = a; b < 4; ++b) {
#pragma unroll
            for (int r = r0; r < 32; r += 8) {
                ta[r][c] = tile[(a * 32 + r) * kD + b * 32 + c];
                tb[r][c] = tile[(b * 32 + r) * kD + a * 32 + c];
            }
            __syncthreads();
#pragma unroll
            for (int r = r0; r < 32; r += 8) {
                tile[(b * 32 + r) * kD + a * 32 + c] = ta[c][r];
                if (a != b) tile[(a * 32 + r) * kD + b * 32 + c] = tb[c][r];
            }
            __syncthreads();
        }
}

cudaError_t launch_state_transpose(float* pool, const int32_t* slot_idx, int32_t n, int32_t Hv,
                                   int32_t num_slots, int32_t* dev_status, cudaStream_t stream) {
    const long long units = static_cast<long long>(n) * Hv;
    if (units == 0) return cudaSuccess;
    state_transpose_kernel<<<static_cast<unsigned>(units), 256, 0, stream>>>(pool, slot_idx, Hv,
                                                                             num_slots, dev_status);
    return cudaGetLastError();
}

}  // namespace gdn
