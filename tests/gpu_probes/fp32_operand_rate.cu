// Cycles that an SM sub-partition takes per FP32 multiply-add of a warp, by the number of
// distinct registers it reads: c += a * a (two) and c += a * b (three), scalar FFMA and
// packed FFMA2. One CTA of 512 threads per SM, so four warps a sub-partition, each with
// independent multiply-adds into eight sums (of pairs); every CTA reads its SM's cycle
// counter around the loop. Prints, per form, the median cycles per warp instruction.
#include <algorithm>
#include <cstdio>
#include <cuda_runtime.h>
#include <vector>

constexpr int kThreads = 512, kIters = 2048, kUnroll = 4, kSums = 8;

template <bool PACKED, bool THREE>
__global__ void __launch_bounds__(kThreads, 1) sums(float seed, long long *cyc, float *sink) {
    float2 a[kSums], b[kSums], c[kSums];
#pragma unroll
    for (int k = 0; k < kSums; ++k) {
        a[k] = make_float2(seed * (k + 1) + threadIdx.x * 1e-9f, seed * (k + 2));
        b[k] = make_float2(seed - k * 1e-7f * threadIdx.x, seed * (k + 3));
        c[k] = make_float2(k, threadIdx.x);
    }
    __syncthreads();
    const long long t0 = clock64();
    for (int it = 0; it < kIters; ++it)
#pragma unroll
        for (int u = 0; u < kUnroll; ++u)
#pragma unroll
            for (int k = 0; k < kSums; ++k) {
                const float2 p = a[k], q = THREE ? b[(k + u) % kSums] : a[k];
                if (PACKED) c[k] = __ffma2_rn(p, q, c[k]);
                else c[k].x = __fmaf_rn(p.x, q.x, c[k].x);
            }
    __syncthreads();
    if (threadIdx.x == 0) cyc[blockIdx.x] = clock64() - t0;
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < kSums; ++k) s += c[k].x + c[k].y;
    if (s == 1234.5f) sink[0] = s;  // keeps the sums alive
}

template <bool PACKED, bool THREE>
bool run(const char *name, int sms) {
    long long *cyc;
    float *sink;
    if (cudaMalloc(&cyc, sms * sizeof(long long)) != cudaSuccess || cudaMalloc(&sink, 4) != cudaSuccess) return false;
    for (int rep = 0; rep < 3; ++rep) sums<PACKED, THREE><<<sms, kThreads>>>(1e-3f, cyc, sink);
    std::vector<long long> h(sms);
    if (cudaMemcpy(h.data(), cyc, sms * sizeof(long long), cudaMemcpyDeviceToHost) != cudaSuccess) return false;
    std::nth_element(h.begin(), h.begin() + sms / 2, h.end());
    const double instructions = (double)kIters * kUnroll * kSums * (kThreads / 32 / 4);  // per sub-partition
    std::printf("%s %.3f\n", name, h[sms / 2] / instructions);
    cudaFree(cyc);
    cudaFree(sink);
    return true;
}

int main() {
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, 0) != cudaSuccess) return 1;
    const bool ok = run<false, false>("ffma_two", sms) && run<false, true>("ffma_three", sms) &&
                    run<true, false>("ffma2_two", sms) && run<true, true>("ffma2_three", sms);
    return ok ? 0 : 1;
}
