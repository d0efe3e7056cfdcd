// Gate / beta preprocessing in front of prefill and decode: raw per-token projections to the
// log-domain gate g = ln(alpha) and the write strength beta the recurrence takes.
//
//   g[t][h]    = -exp(A_log[h]) * softplus(a[t][h] + dt_bias[h])      (<= 0, so alpha in (0, 1])
//   beta[t][h] = sigmoid(b[t][h])
//
// The paper names such a helper but prints no formula; this is the parametrisation of the
// published Gated DeltaNet layer.  Element-wise, fp32, one thread per (token, head).
#include "gdn_common.cuh"
#include "gdn_sm100.cuh"

namespace gdn {

__global__ void __launch_bounds__(256)
gate_kernel(const __nv_bfloat16* __restrict__ a, const __nv_bfloat16* __restrict__ b,
            const float* __restrict__ A_log, const float* __restrict__ dt_bias,
            float* __restrict__ g, float* __restrict__ beta, int n, int Hv, FastDiv by_hv) {
    sm100::pdl_launch_dependents();
    sm100::pdl_wait();
    const int idx = blockIdx.x * 256 + threadIdx.x;
    if (idx >= n) return;
    const int h = idx - (idx / by_hv) * Hv;
    const float x = __bfloat162float(a[idx]) + dt_bias[h];
    const float softplus = fmaxf(x, 0.f) + log1pf(expf(-fabsf(x)));
    g[idx] = -expf(A_log[h]) * softplus;
    beta[idx] = 1.f / (1.f + expf(-__bfloat162float(b[idx])));
}

cudaError_t launch_gate(const __nv_bfloat16* a, const __nv_bfloat16* b, const float* A_log,
                        const float* dt_bias, float* g, float* beta, long long n, int Hv,
                        cudaStream_t stream) {
    if (n == 0) return cudaSuccess;
    // whole rows of at most 2^30 elements a launch: 32-bit indices (a 64-bit remainder stood in front of every load)
    const long long most = (1ll << 30) / Hv > 0 ? (1ll << 30) / Hv * Hv : Hv;
    cudaError_t e = cudaSuccess;
    for (long long at = 0; at < n && e == cudaSuccess; at += most) {
        const int m = static_cast<int>(n - at < most ? n - at : most);
        e = launch_dependent(gate_kernel, dim3(static_cast<unsigned>((m + 255) / 256)), dim3(256), 0, stream, a + at, b + at,
                             A_log, dt_bias, g + at, beta + at, m, Hv, fast_div(Hv));
    }
    return e;
}

}  // namespace gdn
