// The persistent state pass as a kernel of its own (after the intra-chunk kernel); the role itself
// is in gdn_prefill_stream.cuh.
#include "gdn_prefill_half.cuh"
#include <algorithm>

namespace gdn {

__global__ void __launch_bounds__(kStreamThreads, 1)
prefill_state_stream_kernel(const __grid_constant__ TensorMaps maps, const PrefillParams p,
                            uint8_t* ws, const WorkspaceLayout lay) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                               ~static_cast<uintptr_t>(1023));
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
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                               ~static_cast<uintptr_t>(1023));
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

// Whether the state pass runs two CTAs per unit.  A half unit's chunk step takes 1.06 us against 1.40 of a whole unit's, so
// half units win where the longest chain decides: always while every one of them has an SM of its own, and for more units
// if the longest chain (known from the caller) is at least twice what an SM has to do on average, set-up of the units
// included.  On 148 SMs (sustained, us, whole / half; ratio of the longest chain to the average of an SM): 32 units of 64 chunks
// 144 / 126; 96 units up to 64 chunks (3.1) 171 / 151; 136 up to 37 (8.7) 80 / 66; 128 up to 4 (3.1) 22.8 / 19.7; 336 up to 32 (3.7)
// 98 / 90.5; 256 up to 53 (2.0) 183 / 179.5; 544 up to 24 (1.75) 106.7 / 106.5; 448 up to 17 (1.4) 87 / 91; 440 up to 17 (1.3)
// 96 / 99; 480 up to 31 (1.0) 205 / 217; 448 units of which most have one chunk, up to 9 (2.6), 41.9 / 44.6.
static bool half_units(const ChunkedParams& cp, long long units, int sms) {
    if (2 * units <= sms) return true;
    if (cp.longest <= 0) return false;
    const long long chain = (cp.longest + kChunk - 1) / kChunk;
    // about, half a chunk lost per sequence
    const long long items = std::max((2ll * (cp.p.T / kChunk) + cp.p.N) * cp.p.Hv / 2, units);
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
    if (half_units(cp, units, sms)) {
        const int grid = static_cast<int>(2 * units < sms ? 2 * units : sms);
        return launch_dependent(prefill_state_half_kernel, dim3(grid), dim3(kStreamThreads), kHalfSmem, stream, maps, p,
                                cp.ws, cp.lay);
    }
    const int grid = static_cast<int>(units < sms ? units : sms);
    return launch_dependent(prefill_state_stream_kernel, dim3(grid), dim3(kStreamThreads), kStreamSmem,
                            stream, maps, p, cp.ws, cp.lay);
}

}  // namespace gdn
