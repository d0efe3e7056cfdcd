// Chunked prefill in ONE cooperative launch: the record producers and the state pass overlap.
//
// The grid has one CTA of 512 threads per SM.  The first `n_state` CTAs run the serial state pass
// (the role of the persistent state pass, gdn_prefill_stream.cuh: 8 chain warps, 4 output warps, an
// issuing warp and 3 loading warps), CTA b over the units b, b + n_state, ... of the list that has
// the longest sequences first.  The other CTAs run two independent groups of 256 threads that pull
// (chunk, v-head) items from a queue and write their records (the intra-chunk routine of
// gdn_prefill_device.cuh), in the order the state pass consumes them: by position inside the
// sequence first, by sequence rank second.  A record is published through a flag in global
// memory (release) and the state pass waits for the flag (acquire, bounded) before it copies the
// record in.  Producers never wait for consumers, every CTA is resident (cooperative launch with
// grid <= SM count), so the consumers' waits always end.
#include "gdn_prefill_stream.cuh"

namespace gdn {

// =============================================================================================
// Prep: chunk table, processing order, cleared queues and flags.  One CTA.
// =============================================================================================
constexpr int kFPrepThreads = 256;
// model of the two-part production (see the kernel): items per SM and chunk step, start-up lag of the second part in
// chunk steps, and a safety margin in items.  (The time is flat around these: 32 chains of 512 chunks 616 us with a lead
// of 8 steps, 617 of 4; of 41 80.5 and 82.1; 48 chains of 96, 32 and 15 chunks 152 and 153.)
constexpr int kSplitProdPermille = 385;
constexpr int kSplitLeadSteps = 8;
constexpr int kSplitMarginItems = 64;
// How many items in processing order the producers of the second part may be ahead of the first chain.  500 records are
// 29 MB, half of what one die's L2 holds; 32 chains of 512 chunks: 617 us, no bound 727 (the records have left L2 when
// they are read), 300 more (84 CTAs work on four items each).
constexpr int kPaceItems = 500;
// And the items that one of them makes in a chain's chunk step (2.3 and 1.07 us): where all of them together make fewer
// than the chains read, they have to be further ahead to be done in time.  (The cut reckons with less: it must hold.)
constexpr float kPaceRate = 0.45f;

// The model of the two-part production, in items of the processing order.  In step j the chains need the Hv pos[j + 1]
// first ones; a unit holds two SMs, and what the second part has begun kSplitLeadSteps before is ready.
struct SplitModel {
    const int32_t* pos;
    int32_t Hv, sms;
    // SMs without a half unit, summed over the steps before m
    __device__ __forceinline__ long long work(int m) const {
        const long long w = static_cast<long long>(m) * sms - 2ll * Hv * pos[m];
        return w < 0 ? 0 : w;
    }
    __device__ __forceinline__ long long ready_work(int j) const { return work(j > kSplitLeadSteps ? j - kSplitLeadSteps : 0); }
    __device__ __forceinline__ long long needed(int j) const { return static_cast<long long>(Hv) * pos[j + 1]; }
    // what step j lacks without a first part: by the cut's cautious rate, and by the producers' own
    __device__ __forceinline__ long long cut_for(int j) const { return needed(j) - ready_work(j) * kSplitProdPermille / 1000; }
    __device__ __forceinline__ long long short_of(int j) const {
        return needed(j) - static_cast<long long>(kPaceRate * ready_work(j));
    }
    // How far the producers may go with the first chain at chunk j: the window, and up to the step that lacks most at
    // least as far as that they are done in time.  (Held to the window there, 64 chains of 128 chunks take 358 us instead
    // of 290, 48 of 100 220 instead of 203, for the first part alone reaches far beyond it: the producers stood idle first
    // and were late then.  Not held at all beyond a large first part: 30000 and 1000 tokens at 32 heads 652 instead of 580.)
    __device__ __forceinline__ int32_t bound(int j, long long short_max, int short_step) const {
        const long long window = static_cast<long long>(Hv) * pos[j] + kPaceItems;
        const long long in_time = j <= short_step ? short_max + static_cast<long long>(kPaceRate * work(j)) : 0;
        const long long b = window > in_time ? window : in_time;
        return static_cast<int32_t>(b < 0x7fffffff ? b : 0x7fffffff);
    }
};

__global__ void __launch_bounds__(kFPrepThreads)
prefill_fused_prep_kernel(const int32_t* __restrict__ cu, int32_t T, int32_t N, int32_t Hv,
                          uint8_t* ws, WorkspaceLayout lay, int32_t* dev_status,
                          const int for_fused,     // 0: only the chunk table and the ranking;
                                                   // 1: + processing order, cleared queues and flags;
                                                   // 2: + where the two-part production is cut
                          const int split_permille, const int sms) {
    int32_t* hdr = reinterpret_cast<int32_t*>(ws);
    int32_t* seq_first = reinterpret_cast<int32_t*>(ws + lay.seq_first);
    int32_t* seq_bad = reinterpret_cast<int32_t*>(ws + lay.seq_bad);
    ChunkInfo* chunks = reinterpret_cast<ChunkInfo*>(ws + lay.chunks);
    int32_t* seq_by_rank = reinterpret_cast<int32_t*>(ws + lay.seq_by_rank);
    int32_t* order = reinterpret_cast<int32_t*>(ws + lay.order);
    int32_t* hist = reinterpret_cast<int32_t*>(ws + lay.hist);
    int32_t* fill = reinterpret_cast<int32_t*>(ws + lay.fill);
    int32_t* cnt = reinterpret_cast<int32_t*>(ws + lay.cnt);     // #sequences with more than v chunks
    int32_t* pos = reinterpret_cast<int32_t*>(ws + lay.pos);     // #chunks at positions < j
    uint32_t* flags = reinterpret_cast<uint32_t*>(ws + lay.flags);
    __shared__ int32_t warp_sums[kFPrepThreads / 32];
    __shared__ int32_t ends[kFPrepThreads];
    __shared__ int32_t running, end_before;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    pdl_launch_dependents();        // the next kernel's CTAs may become resident (they wait for us)

    for (int i = tid; i < lay.max_nc + 2; i += kFPrepThreads) { hist[i] = 0; fill[i] = 0; }
    if (for_fused)
        for (size_t i = tid; i < static_cast<size_t>(lay.max_chunks) * Hv; i += kFPrepThreads)
            flags[i] = 0u;
    if (for_fused == 2) {
        int32_t* done = reinterpret_cast<int32_t*>(ws + lay.done);
        for (int i = tid; i < N * Hv; i += kFPrepThreads) done[i] = 0;
    }
    if (tid == 0) {
        running = 0;
        end_before = 0;
        hdr[kHdrItemHead] = 0;
        hdr[kHdrStarted] = 0;
        hdr[kHdrProgress] = 0;
        if (cu[0] != 0 || cu[N] != T) report(dev_status, kDevBadCuSeqlens);
    }
    __syncthreads();
    // chunk counts, prefix sums, chunk table (as in the three-launch path) + histogram of counts
    for (int base = 0; base < N; base += kFPrepThreads) {
        const int n = base + tid;
        int32_t nc = 0, t0 = 0, t1 = 0;
        if (n < N) {
            t0 = cu[n];
            t1 = cu[n + 1];
        }
        const bool ok = block_bounds_ok(n < N, t0, t1, T, end_before, ends, tid);
        if (n < N) {
            if (!ok) report(dev_status, kDevBadCuSeqlens);
            seq_bad[n] = ok ? 0 : 1;
            nc = ok ? (t1 - t0 + kChunk - 1) / kChunk : 0;
            atomicAdd(&hist[nc], 1);
        }
        int32_t incl = nc;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += y;
        }
        if (lane == 31) warp_sums[warp] = incl;
        __syncthreads();
        int32_t warp_off = 0;
        for (int w = 0; w < warp; ++w) warp_off += warp_sums[w];
        const int32_t first = running + warp_off + incl - nc;
        if (n < N) {
            seq_first[n] = first;
            for (int j = 0; j < nc; ++j) {
                ChunkInfo ci;
                ci.seq = n;
                ci.t0 = t0 + j * kChunk;
                ci.len = min(kChunk, t1 - ci.t0);
                ci.pad = 0;
                chunks[first + j] = ci;
            }
        }
        __syncthreads();
        if (tid == kFPrepThreads - 1) running = first + nc;
        if (base + kFPrepThreads < N) atomicMax(&end_before, ends[tid]);
        __syncthreads();
    }
    if (tid == 0) {
        seq_first[N] = running;
        hdr[kHdrTotalChunks] = running;
        hdr[kHdrTotalItems] = running * Hv;
        running = 0;
    }
    __syncthreads();
    // cnt[v] = number of sequences with more than v chunks: exclusive suffix sum of the histogram,
    // as a block scan over tiles of the reversed index u = max_nc - v
    for (int base = 0; base <= lay.max_nc; base += kFPrepThreads) {
        const int u = base + tid;
        const int32_t x = u <= lay.max_nc ? hist[lay.max_nc - u] : 0;
        int32_t incl = x;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += y;
        }
        if (lane == 31) warp_sums[warp] = incl;
        __syncthreads();
        int32_t warp_off = 0;
        for (int w = 0; w < warp; ++w) warp_off += warp_sums[w];
        const int32_t excl = running + warp_off + incl - x;
        if (u <= lay.max_nc) cnt[lay.max_nc - u] = excl;
        __syncthreads();
        if (tid == kFPrepThreads - 1) running = excl + x;
        __syncthreads();
    }
    if (tid == 0) running = 0;
    __syncthreads();
    // pos[j] = number of chunks at positions < j: exclusive prefix sum of cnt (fused launch only)
    for (int base = 0; for_fused != 0 && base <= lay.max_nc; base += kFPrepThreads) {
        const int j = base + tid;
        const int32_t x = j <= lay.max_nc ? cnt[j] : 0;
        int32_t incl = x;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += y;
        }
        if (lane == 31) warp_sums[warp] = incl;
        __syncthreads();
        int32_t warp_off = 0;
        for (int w = 0; w < warp; ++w) warp_off += warp_sums[w];
        const int32_t excl = running + warp_off + incl - x;
        if (j <= lay.max_nc) pos[j] = excl;
        __syncthreads();
        if (tid == kFPrepThreads - 1) running = excl + x;
        __syncthreads();
    }
    // Two-part production (mode 2).  The items of the processing order before the cut are
    // produced before the state pass starts, the others beside it, on the SMs it leaves free.
    // The cut is the smallest head start with which the chains never catch up with the producers by SplitModel.
    if (for_fused == 2) {
        __shared__ int32_t need_max, short_max, short_step;
        if (tid == 0) need_max = short_max = short_step = 0;
        __syncthreads();
        const long long total_items = hdr[kHdrTotalItems];
        const SplitModel model = {pos, Hv, sms};
        long long local = 0;
        int32_t short_local = 0, short_at = 0;
        for (int j = tid; j < lay.max_nc; j += kFPrepThreads) {
            const long long need = model.cut_for(j), lacks = model.short_of(j);
            local = need > local ? need : local;
            if (lacks > short_local) {
                short_local = static_cast<int32_t>(lacks);
                short_at = j;
            }
        }
        if (local > total_items) local = total_items;
        atomicMax(&need_max, static_cast<int32_t>(local));
        atomicMax(&short_max, short_local);
        __syncthreads();
        if (short_local == short_max) atomicMax(&short_step, short_at);
        __syncthreads();
        for (int j = tid; j < lay.max_nc; j += kFPrepThreads) hist[j] = model.bound(j, short_max, short_step);
        if (tid == 0) {
            long long cut = split_permille >= 0 ? total_items * split_permille / 1000
                                                : static_cast<long long>(need_max) + kSplitMarginItems;
            if (cut > total_items) cut = total_items;
            hdr[kHdrSplit] = static_cast<int32_t>(cut);
        }
    }
    // rank of a sequence = its place in the order "more chunks first"; chunk j of the sequence of
    // rank r is processed at place pos[j] + r (the sequences that have a chunk j are ranks < cnt[j])
    int32_t* rank_of = reinterpret_cast<int32_t*>(ws + lay.rank_of);
    for (int n = tid; n < N; n += kFPrepThreads) {
        const int32_t nc = seq_first[n + 1] - seq_first[n];
        const int32_t rank = cnt[nc] + atomicAdd(&fill[nc], 1);
        seq_by_rank[rank] = n;
        rank_of[n] = rank;
    }
    if (for_fused) {
        // one thread per chunk (a loop per sequence would be a chain of dependent loads as long
        // as the longest sequence)
        __syncthreads();
        const int32_t total_chunks = hdr[kHdrTotalChunks];
        for (int c = tid; c < total_chunks; c += kFPrepThreads) {
            const int32_t n = chunks[c].seq;
            order[pos[c - seq_first[n]] + rank_of[n]] = c;
        }
    }
}

// The same tables for a batch of at most kFPrepThreads sequences when only the chunk table and the
// ranking are wanted (mode 0): one thread per sequence, one block scan, the ranking by counting in
// shared memory; no histogram, no cleared arrays.  About half the time of the general kernel, which
// every three-launch call of such a batch waits for.
__global__ void __launch_bounds__(kFPrepThreads)
prefill_small_prep_kernel(const int32_t* __restrict__ cu, int32_t T, int32_t N, uint8_t* ws,
                          WorkspaceLayout lay, int32_t* dev_status) {
    int32_t* hdr = reinterpret_cast<int32_t*>(ws);
    int32_t* seq_first = reinterpret_cast<int32_t*>(ws + lay.seq_first);
    int32_t* seq_bad = reinterpret_cast<int32_t*>(ws + lay.seq_bad);
    ChunkInfo* chunks = reinterpret_cast<ChunkInfo*>(ws + lay.chunks);
    int32_t* seq_by_rank = reinterpret_cast<int32_t*>(ws + lay.seq_by_rank);
    int32_t* rank_of = reinterpret_cast<int32_t*>(ws + lay.rank_of);
    __shared__ int32_t warp_sums[kFPrepThreads / 32];
    __shared__ int32_t s_nc[kFPrepThreads];
    __shared__ int32_t ends[kFPrepThreads];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    pdl_launch_dependents();        // the next kernel's CTAs may become resident (they wait for us)
    const int n = tid;
    int32_t nc = 0, t0 = 0, t1 = 0;
    if (n < N) {
        t0 = cu[n];
        t1 = cu[n + 1];
    }
    const bool ok = block_bounds_ok(n < N, t0, t1, T, 0, ends, tid);
    if (n < N) {
        if (!ok) report(dev_status, kDevBadCuSeqlens);
        seq_bad[n] = ok ? 0 : 1;
        nc = ok ? (t1 - t0 + kChunk - 1) / kChunk : 0;
    }
    if (tid == 0 && (cu[0] != 0 || cu[N] != T)) report(dev_status, kDevBadCuSeqlens);
    s_nc[tid] = n < N ? nc : -1;
    int32_t incl = nc;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += y;
    }
    if (lane == 31) warp_sums[warp] = incl;
    __syncthreads();
    int32_t warp_off = 0, total = 0;
    for (int w = 0; w < kFPrepThreads / 32; ++w) {
        if (w < warp) warp_off += warp_sums[w];
        total += warp_sums[w];
    }
    const int32_t first = warp_off + incl - nc;
    if (n < N) {
        seq_first[n] = first;
        for (int j = 0; j < nc; ++j) {
            ChunkInfo ci;
            ci.seq = n;
            ci.t0 = t0 + j * kChunk;
            ci.len = min(kChunk, t1 - ci.t0);
            ci.pad = 0;
            chunks[first + j] = ci;
        }
        // rank = place in the order "more chunks first" (ties by index)
        int32_t rank = 0;
        for (int m = 0; m < N; ++m) {
            const int32_t nm = s_nc[m];
            rank += (nm > nc || (nm == nc && m < n)) ? 1 : 0;
        }
        seq_by_rank[rank] = n;
        rank_of[n] = rank;
    }
    if (tid == 0) {
        seq_first[N] = total;
        hdr[kHdrTotalChunks] = total;
        hdr[kHdrTotalItems] = 0;       // (the queues of the other modes are not used)
        hdr[kHdrItemHead] = 0;
    }
}

// =============================================================================================
// The fused kernel
// =============================================================================================
constexpr int kFusedThreads = 512;
constexpr int kFGroups = 2;                          // intra role: two groups of 256 threads
constexpr uint32_t kFGroupSmem = (kI_End + 1023u) & ~1023u;
constexpr uint32_t kFusedSmem =
    (kFGroups * kFGroupSmem > kStreamSmem - 1024 ? kFGroups * kFGroupSmem : kStreamSmem - 1024) + 1024;

template <int kId, int kCount> __device__ __forceinline__ void named_sync() {
    asm volatile("bar.sync %0, %1;" ::"n"(kId), "n"(kCount) : "memory");
}

// ------------------------------------------------------------------ intra role
__device__ __forceinline__ void fused_intra_role(const TensorMaps& maps, const PrefillParams& p,
                                                 uint8_t* ws, const WorkspaceLayout& lay,
                                                 uint8_t* smem, IntraStatics* statics,
                                                 const uint32_t* tmem_base) {
    const int group = threadIdx.x >> 8;
    const int gtid = threadIdx.x & 255;
    IntraStatics& st = statics[group];
    uint8_t* gsmem = smem + group * kFGroupSmem;
    const uint32_t tmem_off = group * kIntraTmemCols;
    int32_t* hdr = reinterpret_cast<int32_t*>(ws);
    const int32_t total_items = hdr[kHdrTotalItems];
    const int32_t* order = reinterpret_cast<const int32_t*>(ws + lay.order);
    const ChunkInfo* chunks = reinterpret_cast<const ChunkInfo*>(ws + lay.chunks);
    uint32_t* flags = reinterpret_cast<uint32_t*>(ws + lay.flags);

    auto gsync = [group] {
        if (group == 0) named_sync<1, 256>();
        else if (group == 1) named_sync<2, 256>();
        else named_sync<3, 256>();
    };
    uint32_t n_done = 0;
    for (;;) {
        if (gtid == 0) st.item = atomicAdd(&hdr[kHdrItemHead], 1);
        gsync();
        const int item = st.item;
        if (item >= total_items) break;
        const int k = item / p.by_hv;
        const int hv = item - k * p.Hv;
        const int c = order[k];
        const ChunkInfo ci = chunks[c];
        const size_t slot = static_cast<size_t>(c) * p.Hv + hv;
        uint8_t* rec = ws + lay.records + slot * kRecBytes;
        const bool ok = intra_item<true>(maps, p, rec, ci, hv / p.by_group, hv, gsmem, st, tmem_base, tmem_off, gtid, gsync, n_done);
        ++n_done;
        // publish: every thread's own stores first, then the bulk stores, then the flag
        __threadfence();
        tc_fence_before_sync();
        gsync();
        if (gtid == 0) {
            bulk_wait_all();
            fence_proxy_async_all();
            __threadfence();
            st_release_u32(&flags[slot], ok ? 1u : 2u);      // 2 = produced after a timeout
        }
        if (!ok) break;
    }
}

// ---------------------------------------------------------------------------------------------
// The kernel: 512 threads per CTA (128 registers).  State CTA b runs the persistent state pass's
// role over the units b, b + n_state, ... of the rank-sorted list, its loading warps waiting
// for each record's flag; the other CTAs run two producer groups.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kFusedThreads, 1)
prefill_fused_kernel(const __grid_constant__ TensorMaps maps, const PrefillParams p, uint8_t* ws,
                     const WorkspaceLayout lay, const int n_state) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align_1024(smem_raw);
    __shared__ IntraStatics intra_statics[kFGroups];
    __shared__ uint32_t tmem_base_s;
    const int warp = threadIdx.x >> 5;
    if (warp == 0) {
        tmem_alloc(&tmem_base_s, 512);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = tmem_base_s;
    if (static_cast<int>(blockIdx.x) < n_state) {
        state_stream_role<true>(maps, p, ws, lay, smem, tmem, blockIdx.x, n_state);
    } else {
        fused_intra_role(maps, p, ws, lay, smem, intra_statics, &tmem_base_s);
        tc_fence_before_sync();
        __syncthreads();
    }
    if (warp == 0) tmem_dealloc(tmem, 512);
}

// =============================================================================================
// host side
// =============================================================================================
cudaError_t launch_prefill_ranked_prep(const ChunkedParams& cp, cudaStream_t stream, int mode,
                                       int split_permille, int sms) {
    if (mode == 0 && cp.p.N <= kFPrepThreads) {
        prefill_small_prep_kernel<<<1, kFPrepThreads, 0, stream>>>(cp.p.cu_seqlens, cp.p.T, cp.p.N, cp.ws,
                                                                   cp.lay, cp.p.dev_status);
        return cudaGetLastError();
    }
    prefill_fused_prep_kernel<<<1, kFPrepThreads, 0, stream>>>(cp.p.cu_seqlens, cp.p.T, cp.p.N,
                                                               cp.p.Hv, cp.ws, cp.lay,
                                                               cp.p.dev_status, mode, split_permille, sms);
    return cudaGetLastError();
}

cudaError_t launch_prefill_fused(const ChunkedParams& cp, cudaStream_t stream) {
    const PrefillParams& p = cp.p;
    DeviceInfo di;
    cudaError_t e = device_info(&di);
    if (e != cudaSuccess) return e;
    const int sms = di.sms, coop = di.cooperative;
    if (!coop || sms < 2) return cudaErrorNotSupported;
    e = ensure_dynamic_smem(prefill_fused_kernel, kFusedSmem);
    if (e != cudaSuccess) return e;
    TensorMaps maps;
    if (!make_prefill_tensor_maps(&maps, p)) return cudaErrorInvalidValue;

    e = launch_prefill_ranked_prep(cp, stream, 1);
    if (e != cudaSuccess) return e;

    // How many CTAs run the state pass: one per unit when the units are few (the shapes routed
    // here), else about 0.43 of the SMs; always at least one producer CTA.
    const long long units = static_cast<long long>(p.N) * p.Hv;
    int n_state = (sms * 7) / 16;
    if (n_state > units) n_state = static_cast<int>(units);
    if (n_state < 1) n_state = 1;
    if (n_state > sms - 1) n_state = sms - 1;
    int grid = sms;
    uint8_t* ws = cp.ws;
    WorkspaceLayout lay = cp.lay;
    PrefillParams pp = p;
    void* args[] = {&maps, &pp, &ws, &lay, &n_state};
    return cudaLaunchCooperativeKernel(reinterpret_cast<void*>(prefill_fused_kernel), dim3(grid),
                                       dim3(kFusedThreads), args, kFusedSmem, stream);
}

}  // namespace gdn
