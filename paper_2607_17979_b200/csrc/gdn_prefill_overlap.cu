// Chunked prefill with the record production in two parts around the persistent state pass.
//
// With few (sequence, v-head) units of unequal length the state pass is a handful of long serial chains: most SMs hold
// a short chain that ends early, or none, while the intra-chunk kernel before it needs the whole machine.  Here the
// intra-chunk work is cut in two along the order in which the chains consume the records (by position inside the
// sequence first): the first part runs alone, then the state pass starts, two CTAs per unit (gdn_prefill_half.cuh),
// and the second part runs beside it on the SMs that have no live chain, each record published through a flag
// (release) that the state pass's loading warp waits for (acquire, bounded).
//
// Five launches in one stream, the first four each a programmatic dependent of the one before:
//   prep          chunk table, ranking, processing order, cleared flags and done table, the cut
//   first part    waits for prep; items [0, cut) of the order, a CTA per SM
//   state pass    waits for the first part, THEN lets its dependent start, so the second part's
//                 CTAs are scheduled only once every state-pass CTA is resident: they can never
//                 take the SMs the chains need, and every chain that waits for a record is
//                 resident while the producers still have SMs of their own (the launcher keeps
//                 2 units <= SMs - kOverlapSpareSms, so every CTA has one half unit)
//   second part   does not wait for the state pass (it only feeds it); items [cut, total), pulled
//                 from a queue by a CTA per SM that is, or becomes, free, no further ahead of the
//                 chains than what stays in L2.  Its CTA 0 waits for the state pass at its very end,
//                 so that the completion of this launch implies the state pass's.
//   rest          an ordinary launch.  CUDA lets a programmatic dependent start early, it does not
//                 promise to; if the second part has not started when a chain has waited for a record for 0.2 ms,
//                 the chain gives up (without an error: a half unit's final state is written only after
//                 its last record has been loaded, so an unfinished one has left its initial state
//                 alone), the half units that were finished are marked, and this launch runs the others now that
//                 every record exists.  Normally every CTA finds its half unit done and returns at
//                 once.
#include "gdn_prefill_half.cuh"
#include "gdn_prefill_intra.cuh"
#include <algorithm>
#include <cstdlib>

namespace gdn {

// First part: the items [0, cut) of the processing order.
__global__ void __launch_bounds__(kProdThreads, 1)
prefill_intra_first_kernel(const __grid_constant__ TensorMaps maps, const PrefillParams p,
                           uint8_t* ws, const WorkspaceLayout lay) {
    pdl_launch_dependents();
    produce_cta<kItemsFirst>(maps, p, ws, lay);
}

// Second part: the items [cut, total) from a queue, in the order the chains consume them; each record is published
// through its flag.  No wait for the state pass (this kernel feeds it): every state-pass CTA has passed its own wait for
// the first part, hence for prep, before this kernel's CTAs are scheduled.
__global__ void __launch_bounds__(kProdThreads, 1)
prefill_intra_second_kernel(const __grid_constant__ TensorMaps maps, const PrefillParams p,
                            uint8_t* ws, const WorkspaceLayout lay) {
    int32_t* hdr = reinterpret_cast<int32_t*>(ws);
    if (blockIdx.x == 0 && threadIdx.x == 0) st_release_u32(reinterpret_cast<uint32_t*>(hdr + kHdrStarted), 1u);
    if (hdr[kHdrSplit] < hdr[kHdrTotalItems]) produce_cta<kItemsQueue>(maps, p, ws, lay);
    if (blockIdx.x == 0) pdl_wait();        // the call is complete when this launch is
}

// The two halves of a unit run as a cluster, which puts them on the two SMs of one TPC: a chain whose neighbour in the
// TPC is a producer takes 1.65 us a step instead of 1.2 (32768 tokens at 32 heads: 650 to 1000 us a call, by where the
// CTAs happened to land; as pairs 617).
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kStreamThreads, 1)
prefill_state_half_gated_kernel(const __grid_constant__ TensorMaps maps, const PrefillParams p,
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
    pdl_wait();                     // tables, cleared flags and the first part's records
    pdl_launch_dependents();        // now the second part may take the SMs that are left
    state_half_role<kHalfGated>(maps, p, ws, lay, smem, tmem, blockIdx.x, gridDim.x);
    __syncwarp();
    if (warp == kSIssueWarp) tmem_dealloc(tmem, kStateTmemCols);
}

// Last launch: the plain persistent pass over the units the gated pass did not finish (none, when
// the producers ran beside it as intended: then every CTA finds its units done and returns).
__global__ void __launch_bounds__(kStreamThreads, 1)
prefill_state_half_rest_kernel(const __grid_constant__ TensorMaps maps, const PrefillParams p,
                                 uint8_t* ws, const WorkspaceLayout lay) {
    // nothing left for this CTA: leave before any set-up
    {
        // (one half unit per CTA)
        if (reinterpret_cast<const uint16_t*>(ws + lay.done)[blockIdx.x] != 0) return;
    }
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
    state_half_role<kHalfRest>(maps, p, ws, lay, smem, tmem, blockIdx.x, gridDim.x);
    __syncwarp();
    if (warp == kSIssueWarp) tmem_dealloc(tmem, kStateTmemCols);
}

cudaError_t launch_prefill_overlap(const ChunkedParams& cp, cudaStream_t stream, int split_permille) {
    DeviceInfo di;
    cudaError_t e = device_info(&di);
    if (e != cudaSuccess) return e;
    const int sms = di.sms;
    const PrefillParams& p = cp.p;
    e = ensure_dynamic_smem(prefill_state_half_gated_kernel, kHalfSmem);
    if (e != cudaSuccess) return e;
    e = ensure_dynamic_smem(prefill_state_half_rest_kernel, kHalfSmem);
    if (e != cudaSuccess) return e;
    e = ensure_dynamic_smem(prefill_intra_first_kernel, kProdSmem);
    if (e != cudaSuccess) return e;
    e = ensure_dynamic_smem(prefill_intra_second_kernel, kProdSmem);
    if (e != cudaSuccess) return e;
    TensorMaps maps;
    if (!make_prefill_tensor_maps(&maps, p)) return cudaErrorInvalidValue;

    // The second part needs SMs of its own for as long as a chain may wait for it: with (nearly) as many half units as
    // SMs everything is produced before the state pass starts.  So it is where launches are known to be serialised:
    // the state pass waits for a launch that comes after it in the stream, the two must be able to run at the same
    // time.  A profiler that replays kernels one at a time cannot be seen from here: under it the state pass gives up
    // after 0.2 ms and the last launch does the work (2560 tokens at 32 heads 78 us, serialised 343; with waits that
    // ran out by themselves only, 4800); profile gdn_prefill_stream instead, which runs the same kernels' arithmetic.
    const long long units = static_cast<long long>(p.N) * p.Hv;
    const char* blocking = std::getenv("CUDA_LAUNCH_BLOCKING");
    if (2 * units > sms - kOverlapSpareSms || (blocking && blocking[0] != '\0' && blocking[0] != '0'))
        return launch_prefill_stream(cp, stream);
    // split_permille == -2 (for tests): the second part is launched as an ordinary successor of
    // the state pass, i.e. the launches are serialised on purpose
    const bool serialised = split_permille == -2;
    if (split_permille > 1000) split_permille = 1000;

    e = launch_prefill_ranked_prep(cp, stream, 2, split_permille, sms);
    if (e != cudaSuccess) return e;
    const dim3 items(static_cast<unsigned>(cp.lay.max_chunks) * static_cast<unsigned>(p.Hv));
    const dim3 resident_first(std::min(items.x, static_cast<unsigned>(sms)));
    e = launch_dependent(prefill_intra_first_kernel, resident_first, dim3(kProdThreads), kProdSmem,
                         stream, maps, p, cp.ws, cp.lay);
    if (e != cudaSuccess) return e;
    const int grid = static_cast<int>(2 * units);
    e = launch_dependent(prefill_state_half_gated_kernel, dim3(grid), dim3(kStreamThreads),
                         kHalfSmem, stream, maps, p, cp.ws, cp.lay);
    if (e != cudaSuccess) return e;
    const unsigned resident = static_cast<unsigned>(sms);
    const dim3 producers(items.x < resident ? items.x : resident);
    if (serialised) {
        prefill_intra_second_kernel<<<producers, kProdThreads, kProdSmem, stream>>>(maps, p, cp.ws, cp.lay);
        e = cudaGetLastError();
    } else {
        e = launch_dependent(prefill_intra_second_kernel, producers, dim3(kProdThreads), kProdSmem,
                             stream, maps, p, cp.ws, cp.lay);
    }
    if (e != cudaSuccess) return e;
    // an ordinary launch: it starts when the second part has ended, and the second part's first
    // CTA ends only after the state pass
    prefill_state_half_rest_kernel<<<grid, kStreamThreads, kHalfSmem, stream>>>(maps, p, cp.ws, cp.lay);
    return cudaGetLastError();
}

}  // namespace gdn
