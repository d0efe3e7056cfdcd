// The persistent state pass as a kernel of its own (after the intra-chunk kernel); the role itself
// is in gdn_prefill_stream.cuh.
#include "gdn_prefill_half.cuh"
#include <algorithm>

namespace gdn {

__global__ void __launch_bounds__(kStreamThreads, 1)
prefill_state_stream_kernel(const __grid_constant__ TensorMaps maps, const PrefillParams p,
                            uint8_t* ws, const WorkspaceLayout lay) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align_1024(smem_raw);
    __shared__ uint32_t tmem_base_s;
    const int warp = threadIdx.x >> 5;
    if (warp == kSIssueWarp) {
        tmem_alloc(&tmem_base_s, kStateTmemCols);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = tmem_base_s;
    state_stream_role<false>(maps, p, ws, lay, smem, tmem, blockIdx.x, gridDim.x);
    __syncwarp();
    if (warp == kSIssueWarp) tmem_dealloc(tmem, kStateTmemCols);
}

// The same with two CTAs per unit (gdn_prefill_half.cuh).
__global__ void __launch_bounds__(kStreamThreads, 1)
prefill_state_half_kernel(const __grid_constant__ TensorMaps maps, const PrefillParams p, uint8_t* ws,
                          const WorkspaceLayout lay) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align_1024(smem_raw);
    __shared__ uint32_t tmem_base_s;
    const int warp = threadIdx.x >> 5;
    if (warp == kSIssueWarp) {
        tmem_alloc(&tmem_base_s, kStateTmemCols);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = tmem_base_s;
    state_half_role<kHalfAll>(maps, p, ws, lay, smem, tmem, blockIdx.x, gridDim.x);
    __syncwarp();
    if (warp == kSIssueWarp) tmem_dealloc(tmem, kStateTmemCols);
}

// Whether the state pass runs two CTAs per unit.  A half unit's chunk step takes about 1.0 us against 1.40 of a whole
// unit's, so half units win where the longest chain decides: always while every one of them has an SM of its own (32
// units of 64 chunks 135.8 us whole, 109.3 half), and for more units if the longest chain is at least twice what an SM has
// to do on average, set-up of the units included (us whole / half, 32 heads: 2.5 times the average 166.9 / 142.9, just
// below twice 162.2 / 152.5, 1.7 times 152.0 / 157.0, 1.5 times 156.5 / 196.5, once 139.9 / 155.6).  The longest chain is the
// caller's word.  If that bound is far too large, whole units would have been faster by up to 26 % (57 x 144 tokens at 32 heads 186
// us, half 220; 3 x 3000).  The device knows better, but a kernel that holds both forms and chooses costs every call of
// more units 2 us (1337 + 512 + 199 tokens 57.4 -> 59.8).
static bool half_units(int32_t T, int32_t N, int32_t Hv, int32_t longest, int sms) {
    const long long units = static_cast<long long>(N) * Hv;
    if (2 * units <= sms) return true;
    if (longest <= 0) return false;
    const long long chain = (longest + kChunk - 1) / kChunk;
    // about, half a chunk lost per sequence
    const long long items = std::max((2ll * (T / kChunk) + N) * Hv / 2, units);
    return chain * sms >= 2 * items + units;
}

// Prep (chunk table + sequences ranked by chunk count) is the fused path's; then the intra-chunk
// kernel over all items; then the state pass on at most as many CTAs as there are SMs.
cudaError_t launch_prefill_stream(const ChunkedParams& cp, cudaStream_t stream) {
    const PrefillParams& p = cp.p;
    DeviceInfo di;
    cudaError_t e = device_info(&di);
    if (e != cudaSuccess) return e;
    const int sms = di.sms;
    const long long units = static_cast<long long>(p.N) * p.Hv;
    e = ensure_dynamic_smem(prefill_state_stream_kernel, kStreamSmem);
    if (e != cudaSuccess) return e;
    e = ensure_dynamic_smem(prefill_state_half_kernel, kHalfSmem);
    if (e != cudaSuccess) return e;
    TensorMaps maps;
    if (!make_prefill_tensor_maps(&maps, p)) return cudaErrorInvalidValue;
    const bool inline_tables = prefill_tables_inline(cp);
    if (!inline_tables) {
        e = launch_prefill_ranked_prep(cp, stream, 0);
        if (e != cudaSuccess) return e;
    }
    if (cp.lay.max_chunks > 0) {
        e = launch_prefill_intra(maps, cp, stream, inline_tables);
        if (e != cudaSuccess) return e;
    }
    if (half_units(p.T, p.N, p.Hv, cp.longest, sms)) {
        const int grid = static_cast<int>(2 * units < sms ? 2 * units : sms);
        return launch_dependent(prefill_state_half_kernel, dim3(grid), dim3(kStreamThreads), kHalfSmem, stream, maps, p,
                                cp.ws, cp.lay);
    }
    const int grid = static_cast<int>(units < sms ? units : sms);
    return launch_dependent(prefill_state_stream_kernel, dim3(grid), dim3(kStreamThreads), kStreamSmem,
                            stream, maps, p, cp.ws, cp.lay);
}

}  // namespace gdn
