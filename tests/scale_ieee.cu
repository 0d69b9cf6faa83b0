// Compares the branch-free group scale with the IEEE operations it stands for, over whole binades; prints the number of
// differences of each kind.  Compiled and run by test_gpu_scale.py.
#include <cstdio>

#include "pq_common.cuh"

__device__ unsigned long long bad[3];

__device__ uint32_t mix(uint32_t x) {
    x = (x ^ (x >> 16)) * 0x7feb352du;
    x = (x ^ (x >> 15)) * 0x846ca68bu;
    return x ^ (x >> 16);
}
__device__ float with(uint32_t exponent, uint32_t mantissa) { return __uint_as_float((exponent << 23) | (mantissa & 0x7FFFFFu)); }

// every mantissa (blockIdx.x, threadIdx.x), one exponent or divisor per blockIdx.y
__global__ void reciprocals() {
    const uint32_t m = blockIdx.x * 1024u + threadIdx.x;
    const uint32_t e = blockIdx.y == 0 ? 127u : blockIdx.y == 1 ? 58u : 195u;
    const float d = with(e, m);
    if (__float_as_uint(pq::reciprocal_of(d)) != __float_as_uint(__frcp_rn(d))) atomicAdd(&bad[0], 1ull);
}
__global__ void quotients() {
    const uint32_t m = blockIdx.x * 1024u + threadIdx.x, k = blockIdx.y;
    const uint32_t edge[8] = {0u, 1u, 0x7FFFFFu, 0x7FFFFEu, 0x400000u, 0x3FFFFFu, 0x555555u, 0x2AAAABu};
    const float c = with(100u + mix(k) % 60u, k < 8 ? edge[k] : mix(k + 77u));
    const float a = with(100u + mix(k + 5u) % 60u, m);
    if (__float_as_uint(pq::quotient_by(a, c, pq::reciprocal_of(c))) != __float_as_uint(__fdiv_rn(a, c))) atomicAdd(&bad[1], 1ull);
}
__global__ void scales() {
    const uint32_t i = (blockIdx.y * gridDim.x + blockIdx.x) * 1024u + threadIdx.x;
    const float ts = with(67u + mix(i) % 120u, mix(i + 1u));  // 2^-60 .. 2^60
    const pq::Nvfp4Scaler s = pq::nvfp4_scaler(ts);
    float amax = with(mix(i + 2u) % 255u, mix(i + 3u));
    if (i % 16u < 12u) amax = __fmul_rn(ts, with(115u + mix(i + 4u) % 24u, mix(i + 3u)));  // quotients around the format's range
    if (i % 64u == 13u) amax = 0.0f;
    if (i % 64u == 29u) amax = __uint_as_float(0x7F800000u);
    if (i % 64u == 45u) amax = __uint_as_float(0x7FFFFFFFu);
    if (i % 64u == 61u) amax = __uint_as_float(mix(i + 6u) & 0x7FFFFFu);
    uint32_t f, g;
    float rf, rg, d;
    pq::nvfp4_scale<true>(amax, s, f, rf);
    pq::nvfp4_scale(amax, ts, g, d, rg);
    if (f != g || __float_as_uint(rf) != __float_as_uint(rg) || !s.fast) atomicAdd(&bad[2], 1ull);
}

int main() {
    reciprocals<<<dim3(8192, 3), 1024>>>();
    quotients<<<dim3(8192, 64), 1024>>>();
    scales<<<dim3(8192, 32), 1024>>>();
    unsigned long long host[3] = {1, 1, 1};
    if (cudaMemcpyFromSymbol(host, bad, sizeof(host)) != cudaSuccess) return 2;
    printf("%llu %llu %llu\n", host[0], host[1], host[2]);
    return 0;
}
