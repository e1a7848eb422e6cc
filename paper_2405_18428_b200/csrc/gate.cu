// Gate transform of the key-channel decay (Eq. gate_gla): alpha = sigmoid(x)^(1/tau), produced
// directly as log(alpha) = logsigmoid(x)/tau, which is what the chunkwise operator consumes.
// Elementwise: 6 bytes (bf16) per element, but also an exponential and a polynomial, 30 instructions in scalar form with
// a division for the head, which kept the issue slots 80% busy at 60% of the bandwidth.  Hence packed arithmetic on
// channel pairs and a grid stride of whole token rows, so that a thread's head never changes.  12.6M elements in bf16
// 17.8 -> 14.8 us; 18.9M, where the writes reach memory, 22.5 -> 21.7 (5.2 TB/s).
#include "dig_common.cuh"

namespace dig {
namespace {

constexpr int kMaxHeads = 256;
constexpr int kPerSM = 8;        // one wave: twice as many CTAs take the same time, eight times as many 1.4 times as long
struct InvTau { float v[kMaxHeads]; };

__device__ __forceinline__ float2 both(float c) { return make_float2(c, c); }
__device__ __forceinline__ float2 log_sigmoid(float2 x)
{
    // log(1/(1+e^-x)) = min(x, 0) - log1p(t), t = e^-|x| in (0, 1], without overflow on either side.
    // t: 2^(-|x| log2 e) with the rounding error of the product carried along (the fast exponential
    // alone would lose |x| * 6e-8 of relative accuracy for large |x|).
    // log1p(t) = t (1 + t r(t)), r a degree-8 polynomial fitted at Chebyshev nodes of [0, 1]: relative
    // error 1.5e-7 in fp32 over the whole interval, and exact behaviour t - t^2/2 as t -> 0, so small
    // results (large positive x) keep their relative accuracy.  r is evaluated with its sign turned, which
    // leaves one multiply-add for the last line.
    const float2 ax = make_float2(-fabsf(x.x), -fabsf(x.y));
    const float2 hi = mul2(ax, both(1.44269502162933349609375f));
    const float2 lo = fma2(ax, both(1.925963033500011e-8f), fma2(ax, both(1.44269502162933349609375f), mul2(ax, both(-1.44269502162933349609375f))));
    float2 t;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(t.x) : "f"(hi.x));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(t.y) : "f"(hi.y));
    t = fma2(t, mul2(lo, both(0.693147182464599609375f)), t);
    float2 r = both(4.466211586e-03f);
    r = fma2(r, t, both(-2.522405428e-02f));
    r = fma2(r, t, both(6.675772493e-02f));
    r = fma2(r, t, both(-1.156184543e-01f));
    r = fma2(r, t, both(1.584756571e-01f));
    r = fma2(r, t, both(-1.985410623e-01f));
    r = fma2(r, t, both(2.498652617e-01f));
    r = fma2(r, t, both(-3.333284189e-01f));
    r = fma2(r, t, both(4.999999698e-01f));
    return fma2(t, fma2(t, r, both(-1.f)), make_float2(fminf(x.x, 0.f), fminf(x.y, 0.f)));
}

// stride: vectors of 4 elements from one of a thread's to the next, a multiple of a token's unless every thread has one
// vector at most; threads from there on have none.  Four elements, so that a warp's stores fill whole sectors.
template <typename T>
__global__ void __launch_bounds__(256, 8)
gate_logsigmoid(const T *__restrict__ g, float *__restrict__ gate, size_t n4, uint32_t stride, int H, int dk, InvTau inv_tau)
{
    const uint32_t first = blockIdx.x * blockDim.x + threadIdx.x;
    const float2 it = both(inv_tau.v[first / (dk >> 2) % H]);
    pdl_wait();
    auto put = [&](size_t i, float4 x) {
        const float2 a = mul2(log_sigmoid(make_float2(x.x, x.y)), it), b = mul2(log_sigmoid(make_float2(x.z, x.w)), it);
        store4(gate + i * 4, make_float4(a.x, a.y, b.x, b.y));
    };
    if (first < stride) {
        size_t i = first;
        for (; i + stride < n4; i += 2 * (size_t)stride) {
            const float4 x = load4(g + i * 4), y = load4(g + (i + stride) * 4);
            put(i, x);
            put(i + stride, y);
        }
        if (i < n4) put(i, load4(g + i * 4));
    }
    pdl_launch_dependents();
}

}  // namespace

dig_status launch_gate(const void *g, const float *tau_host, float *gate, int B, int L, int H,
                       int dk, int dtype, cudaStream_t stream)
{
    if (H > kMaxHeads) return DIG_ERR_UNSUPPORTED;
    InvTau it;
    for (int h = 0; h < H; ++h) {
        if (!(tau_host[h] > 0.f)) return DIG_ERR_INVALID_ARG;
        it.v[h] = 1.0f / tau_host[h];
    }
    const size_t n4 = (size_t)B * L * H * dk / 4;
    const int sms = device_sm_count();
    if (sms <= 0) return DIG_ERR_CUDA;
    // kPerSM CTAs per SM, less what is over after whole token rows
    const uint32_t most = (uint32_t)sms * kPerSM * 256, row = (uint32_t)(H * dk / 4);
    const uint32_t stride = n4 <= most ? (uint32_t)n4 : most - most % row, blocks = (stride + 255) / 256;
    KernelTimer t(KID_GATE, stream);
    if (dtype == DIG_F32)
        launch_pdl(gate_logsigmoid<float>, dim3(blocks), dim3(256), 0, stream, (const float *)g, gate, n4, stride, H, dk, it);
    else
        launch_pdl(gate_logsigmoid<__nv_bfloat16>, dim3(blocks), dim3(256), 0, stream, (const __nv_bfloat16 *)g, gate, n4, stride, H, dk, it);
    return cuda_ok(cudaGetLastError());
}

}  // namespace dig
