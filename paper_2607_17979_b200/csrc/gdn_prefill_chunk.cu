// Chunked prefill on the sm_100a tensor cores (tcgen05 + TMEM, operands staged by TMA): the
// intra-chunk kernel and the host side shared by the launchers.
// The algebra and the record layout are described in gdn_prefill_chunk.cuh.
#include "gdn_prefill_intra.cuh"

namespace gdn {

// =============================================================================================
// K1: intra-chunk quantities of every (chunk, v-head) item, one persistent CTA per SM; see gdn_prefill_intra.cuh.
// =============================================================================================
// kInlineTable: a batch of at most kSmallSeqs sequences needs no table-building launch in front: the warp that hands the
// items out finds their chunks from cu_seqlens, a sequence a lane.
template <bool kInlineTable>
__global__ void __launch_bounds__(kProdThreads, 1)
prefill_intra_kernel(const __grid_constant__ TensorMaps maps, const PrefillParams p, uint8_t* ws,
                     const WorkspaceLayout lay) {
    pdl_launch_dependents();
    produce_cta<kInlineTable ? kItemsInline : kItemsTable>(maps, p, ws, lay);
}

// The same for few items: a CTA of 256 threads per item, up to four to an SM.
// Order of the CTAs.  In a row (kRow) the heads of a chunk stand next to one another, so that the heads that share Q and K
// find them in L2, the last chunks come first, so that what the state pass opens with was written last, and the CTAs
// without a chunk (the host can only bound their number) come behind all others instead of between the heads: 32
// sequences of 64 tokens at 8 heads 21.3 us, as a grid 24.9; 576 tokens at 32 heads 23.8, 25.8.  Fewer items run all at
// once, find nothing that an earlier one fetched, and only ask for the same lines at the same time (200 tokens 16.5
// instead of 16.3), so those have a grid of chunks x heads.  Two kernels: testing for the form inside one costs 0.1 us a
// call.
template <bool kInlineTable, bool kRow>
__global__ void __launch_bounds__(kIntraThreads, 4)
prefill_intra_few_kernel(const __grid_constant__ TensorMaps maps, const PrefillParams p, uint8_t* ws,
                     const WorkspaceLayout lay) {
    const int at = static_cast<int>(blockIdx.x);
    int c = at, hv = blockIdx.y;
    // this CTA's item; false beyond the batch's chunks
    const auto place = [&](int chunks) {
        if constexpr (!kRow) return c < chunks;
        const int item = chunks * p.Hv - 1 - at;
        c = item / p.by_hv;
        hv = item - c * p.Hv;
        return item >= 0;
    };
    __shared__ uint32_t tmem_base_s;
    const int tid = threadIdx.x, warp = tid >> 5;
    pdl_launch_dependents();
    // what needs nothing of the previous kernel's comes before the wait for it
    if (warp == 0) {
        if (tid == 0) {
            prefetch_tensormap(&maps.q);
            prefetch_tensormap(&maps.k);
            prefetch_tensormap(&maps.v);
        }
        __syncwarp();
        tmem_alloc(&tmem_base_s, kIntraTmemCols);
        tmem_relinquish();
        tc_fence_before_sync();
    }
    pdl_wait();                     // the chunk table is the previous kernel's
    ChunkInfo ci;
    bool mine;
    if constexpr (kInlineTable) {
        const int lane = tid & 31;
        int32_t t0 = 0, t1 = 0;
        if (lane < p.N) {
            t0 = p.cu_seqlens[lane];
            t1 = p.cu_seqlens[lane + 1];
        }
        const bool ok = warp_bounds_ok(t0, t1, p.T, lane);
        const int nc = ok ? (t1 - t0 + kChunk - 1) / kChunk : 0;
        int incl = nc;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += y;
        }
        mine = place(__shfl_sync(0xffffffffu, incl, 31));
        if (at == 0 && blockIdx.y == 0 && warp == 0 &&
            (!ok || (lane == 0 && t0 != 0) || (lane == p.N - 1 && t1 != p.T)))
            report(p.dev_status, kDevBadCuSeqlens);
        const unsigned here = __ballot_sync(0xffffffffu, c < incl && c >= incl - nc);
        ci.seq = __ffs(here) - 1;
        ci.t0 = t0 + (c - (incl - nc)) * kChunk;
        ci.len = min(kChunk, t1 - ci.t0);
        ci.t0 = __shfl_sync(0xffffffffu, ci.t0, ci.seq & 31);
        ci.len = __shfl_sync(0xffffffffu, ci.len, ci.seq & 31);
        ci.pad = 0;
    } else {
        mine = place(*reinterpret_cast<const int32_t*>(ws));
        if (mine) ci = reinterpret_cast<const ChunkInfo*>(ws + lay.chunks)[c];
    }
    if (!mine) {
        if (warp == 0) tmem_dealloc(tmem_base_s, kIntraTmemCols);
        return;
    }
    const int hqk = hv / p.by_group;
    uint8_t* rec = ws + lay.records + (static_cast<size_t>(c) * p.Hv + hv) * kRecBytes;

    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align_1024(smem_raw);
    __shared__ IntraStatics st;
    intra_item<false>(maps, p, rec, ci, hqk, hv, smem, st, &tmem_base_s, 0, tid, [] { __syncthreads(); });
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem_base_s, kIntraTmemCols);
}

// =============================================================================================
// host side
// =============================================================================================
namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = []() -> EncodeTiledFn {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &q) !=
                cudaSuccess || q != cudaDriverEntryPointSuccess)
            return nullptr;
        return reinterpret_cast<EncodeTiledFn>(f);
    }();
    return fn;
}

// [rows][cols] bf16 row-major tensor, boxes of 64 rows x 64 columns (128 bytes), 128B swizzle,
// out-of-range rows read as zero.
bool make_token_map(CUtensorMap* m, const void* base, int64_t rows, int64_t cols) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) return false;
    const cuuint64_t dims[2] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(rows)};
    const cuuint64_t strides[1] = {static_cast<cuuint64_t>(cols) * 2};
    const cuuint32_t box[2] = {64, 64};
    const cuuint32_t elem[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box,
               elem, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

bool make_prefill_tensor_maps(TensorMaps* maps, const PrefillParams& p) {
    return make_token_map(&maps->q, p.q, p.T, static_cast<int64_t>(p.Hqk) * kD) &&
           make_token_map(&maps->k, p.k, p.T, static_cast<int64_t>(p.Hqk) * kD) &&
           make_token_map(&maps->v, p.v, p.T, static_cast<int64_t>(p.Hv) * kD) &&
           make_token_map(&maps->o, p.o, p.T, static_cast<int64_t>(p.Hv) * kD);
}

bool prefill_tables_inline(const ChunkedParams& cp) {
    return cp.p.N <= kSmallSeqs && cp.lay.max_chunks > 0;
}

cudaError_t launch_prefill_intra(const TensorMaps& maps, const ChunkedParams& cp, cudaStream_t stream,
                                 bool inline_tables) {
    DeviceInfo di;
    cudaError_t e = device_info(&di);
    if (e != cudaSuccess) return e;
    const int64_t items = static_cast<int64_t>(cp.lay.max_chunks) * cp.p.Hv;
    // Few items run all at once in either form, and there the shorter way through one item counts: a pipeline's warps
    // fetch eight pieces of code from L2 before the first item is through (us a call, CTA per item / pipeline: 64 items
    // 13.4 / 15.8, 512 35.8 / 37.2, 672 43.5 / 43.6, 832 51.1 / 51.2, 1024 61.9 / 61.0, 1280 in 40 sequences 61.8 / 59.7, 3840
    // 156.5 / 142.4).  `items` counts a ragged chunk for each sequence, up to twice what there are.  So a batch whose
    // sequences, were they of equal length, had at most four items an SM, all of which run at once, has few too (32 heads,
    // 13 x 64 tokens 26.9 / 28.4, 16 x 48 30.9 / 32.6, 8 x 128 28.2 / 29.5, 18 x 64 33.6 / 34.2; beyond it 20 x 64 40.3 /
    // 39.7, 8 x 130 36.2 / 35.8).
    const int64_t n = cp.p.N, equal = n * (1 + (cp.p.T - 1) / (n * kChunk)) * cp.p.Hv;
    if (items <= 5ll * di.sms || equal <= 4ll * di.sms) {
        const bool row = items > 2ll * di.sms;
        auto kernel = row ? inline_tables ? prefill_intra_few_kernel<true, true> : prefill_intra_few_kernel<false, true>
                          : inline_tables ? prefill_intra_few_kernel<true, false> : prefill_intra_few_kernel<false, false>;
        e = ensure_dynamic_smem(kernel, kIntraSmem);
        if (e != cudaSuccess) return e;
        const dim3 grid = row ? dim3(static_cast<unsigned>(items)) : dim3(cp.lay.max_chunks, cp.p.Hv);
        return launch_dependent(kernel, grid, dim3(kIntraThreads), kIntraSmem, stream, maps, cp.p, cp.ws, cp.lay);
    }
    auto kernel = inline_tables ? prefill_intra_kernel<true> : prefill_intra_kernel<false>;
    e = ensure_dynamic_smem(kernel, kProdSmem);
    if (e != cudaSuccess) return e;
    return launch_dependent(kernel, dim3(static_cast<unsigned>(di.sms)), dim3(kProdThreads), kProdSmem, stream, maps, cp.p, cp.ws, cp.lay);
}

// The three-launch path: table-building launch (none for small batches), the intra-chunk kernel
// over all items, the persistent state pass.
cudaError_t launch_prefill_chunked(const ChunkedParams& cp, cudaStream_t stream) {
    return launch_prefill_stream(cp, stream);
}

}  // namespace gdn
