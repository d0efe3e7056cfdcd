// Shared declarations of the CUDA side of the gated delta rule library.
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include <stddef.h>

namespace gdn {

constexpr int kD = 128;          // dk == dv == 128 is the only supported head size
constexpr int kChunk = 64;       // prefill chunk length
constexpr int kDecodeMaxTokens = 16;  // most new tokens per sequence in one multi-token decode

// device status bits (mirror GDN_DEV_* of the public header)
constexpr int kDevBadSlot = 1;
constexpr int kDevBadCuSeqlens = 2;
constexpr int kDevTimeout = 4;

// Division of 0 <= x < 2^31 by a number known on the host: x * ceil(2^(31 + s) / d) >> 31 + s with 2^s >= d, exact
// because the product's error is below x / 2^31 of a unit.  In line a division by a kernel argument takes about 150
// cycles, and the three that map a CTA to its sequence and heads stand in front of its first load.
struct FastDiv {
    uint32_t mul;
    uint16_t shift;
};
inline FastDiv fast_div(uint32_t d) {
    uint32_t s = 0;
    while ((1ull << s) < d) ++s;
    return FastDiv{static_cast<uint32_t>(((1ull << (31 + s)) + d - 1) / d), static_cast<uint16_t>(31 + s)};
}
__host__ __device__ inline int32_t operator/(int32_t x, const FastDiv& d) {
    return static_cast<int32_t>(static_cast<uint64_t>(static_cast<uint32_t>(x)) * d.mul >> d.shift);
}

struct DecodeParams {
    const __nv_bfloat16* q;
    const __nv_bfloat16* k;
    const __nv_bfloat16* v;
    const float* g;
    const float* beta;
    float* pool;
    const int32_t* slot_idx;
    __nv_bfloat16* o;
    int32_t* dev_status;
    int32_t Hv, num_slots;
    // 96 bytes in all: a launch with 88 or 96 bytes of arguments takes 2.03 us of host time, with 80 or less and 104
    // or more 2.4-2.5, and the smallest calls are bound by it
    uint32_t mul_hv, mul_group;          // by_hv(), by_group(): division by Hv, by Hv / Hqk
    uint16_t shift_hv, shift_group;
    float scale;
    void set_heads(int32_t Hqk, int32_t Hv_) {
        Hv = Hv_;
        const FastDiv a = fast_div(Hv), b = fast_div(Hv / Hqk);
        mul_hv = a.mul; shift_hv = a.shift;
        mul_group = b.mul; shift_group = b.shift;
    }
    __device__ FastDiv by_hv() const { return FastDiv{mul_hv, shift_hv}; }
    __device__ FastDiv by_group() const { return FastDiv{mul_group, shift_group}; }
};
static_assert(sizeof(DecodeParams) == 96, "see above");

struct DecodeMultiParams {
    DecodeParams d;      // q,k [B][L][Hqk][128]; v,o [B][L][Hv][128]; g,beta [B][L][Hv]
    int32_t Hqk;
    int32_t L;           // new tokens per sequence, 1..kDecodeMaxTokens
    int32_t layout;      // 0: tile [dv][dk];  1: tile [dk][dv]
};

struct PrefillParams {
    const __nv_bfloat16* q;
    const __nv_bfloat16* k;
    const __nv_bfloat16* v;
    const float* g;
    const float* beta;
    const int32_t* cu_seqlens;
    const float* init_state;
    float* final_state;
    const int32_t* slot_idx;
    __nv_bfloat16* o;
    int32_t T, N, Hqk, Hv, num_slots;
    FastDiv by_hv, by_group;      // division by Hv, by Hv / Hqk
    float scale;
    int32_t* dev_status;
};

// The current device's SM count and cooperative-launch support, queried once per device.
struct DeviceInfo {
    int device, sms, cooperative;
};
cudaError_t device_info(DeviceInfo* out);
// Raises a kernel's dynamic shared memory limit on the current device, once per device.
cudaError_t ensure_dynamic_smem(const void* kernel, int bytes);
template <class K> inline cudaError_t ensure_dynamic_smem(K* kernel, int bytes) {
    return ensure_dynamic_smem(reinterpret_cast<const void*>(kernel), bytes);
}

cudaError_t launch_decode(const DecodeParams& p, int32_t B, cudaStream_t stream);
cudaError_t launch_decode_multi(const DecodeMultiParams& mp, int32_t B, cudaStream_t stream);
cudaError_t launch_gate(const __nv_bfloat16* a, const __nv_bfloat16* b, const float* A_log,
                        const float* dt_bias, float* g, float* beta, long long n, int Hv,
                        cudaStream_t stream);
cudaError_t launch_state_transpose(float* pool, const int32_t* slot_idx, int32_t n, int32_t Hv,
                                   int32_t num_slots, int32_t* dev_status, cudaStream_t stream);
// longest: a bound on the longest sequence (picks the block size, never the results)
cudaError_t launch_prefill_recurrent(const PrefillParams& p, int longest, cudaStream_t stream);

__device__ __forceinline__ void report(int32_t* dev_status, int bit) {
    if (dev_status) atomicOr(dev_status, bit);
}

// four consecutive bf16 -> four floats (8-byte aligned source)
__device__ __forceinline__ float4 load_bf16x4(const __nv_bfloat16* p) {
    const uint2 raw = *reinterpret_cast<const uint2*>(p);
    float4 r;
    r.x = __uint_as_float(raw.x << 16);
    r.y = __uint_as_float(raw.x & 0xffff0000u);
    r.z = __uint_as_float(raw.y << 16);
    r.w = __uint_as_float(raw.y & 0xffff0000u);
    return r;
}

__device__ __forceinline__ float dot4(const float4& a, const float4& b, float acc) {
    acc = fmaf(a.x, b.x, acc);
    acc = fmaf(a.y, b.y, acc);
    acc = fmaf(a.z, b.z, acc);
    acc = fmaf(a.w, b.w, acc);
    return acc;
}

// Packed pair of fp32 multiply-adds (one issue slot for two): a * b + c.
__device__ __forceinline__ float2 fma2(const float2 a, const float2 b, const float2 c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;"
        : "=l"(d)
        : "l"(*reinterpret_cast<const unsigned long long*>(&a)),
          "l"(*reinterpret_cast<const unsigned long long*>(&b)),
          "l"(*reinterpret_cast<const unsigned long long*>(&c)));
    return *reinterpret_cast<float2*>(&d);
}

// The same for a product or a sum of pairs.
__device__ __forceinline__ float2 mul2(const float2 a, const float2 b) {
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;"
        : "=l"(d)
        : "l"(*reinterpret_cast<const unsigned long long*>(&a)), "l"(*reinterpret_cast<const unsigned long long*>(&b)));
    return *reinterpret_cast<float2*>(&d);
}
__device__ __forceinline__ float2 add2(const float2 a, const float2 b) {
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;"
        : "=l"(d)
        : "l"(*reinterpret_cast<const unsigned long long*>(&a)), "l"(*reinterpret_cast<const unsigned long long*>(&b)));
    return *reinterpret_cast<float2*>(&d);
}

// sum over the 8 lanes that share a state row (lanes differing in bits 0..2)
__device__ __forceinline__ float sum8(float x) {
    x += __shfl_xor_sync(0xffffffffu, x, 1);
    x += __shfl_xor_sync(0xffffffffu, x, 2);
    x += __shfl_xor_sync(0xffffffffu, x, 4);
    return x;
}

}  // namespace gdn
