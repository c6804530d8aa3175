// rewl_probe.cu -- rewl_measure_pipes: issue rates of the pipes the WL step
// uses, measured on the current device, for the per-flip roofline of the
// benchmark (published peaks cover HBM and the tensor types only).
//
// Throughput: one CTA of 1024 threads per SM (its dynamic shared memory keeps
// a second CTA off the SM), each thread running 8 independent chains of one
// operation written as inline PTX (so that the compiler neither fuses nor
// removes it); lane-operations per clock per SM = operations of the CTA /
// clock64 cycles it took.  Latency: one thread, one dependent chain.
#include <cstdint>

#include "rewl.h"
#include "rewl_host_internal.hpp"

namespace {

enum : int { OP_DADD = 0, OP_IMAD = 1, OP_IMADHI = 2, OP_LOP3 = 3, OP_IADD = 4, OP_LDS = 5, OP_COUNT = 6 };
constexpr int kThreads = 1024, kChains = 8, kIters = 2048;
constexpr size_t kSmem = 120 * 1024;  // more than half an SM's shared memory

template <int OP>
__device__ __forceinline__ void step(double *d, uint32_t *a, uint32_t b, uint32_t c, double y, uint32_t sbase) {
#pragma unroll
    for (int j = 0; j < kChains; ++j) {
        if (OP == OP_DADD) asm volatile("add.rn.f64 %0, %0, %1;" : "+d"(d[j]) : "d"(y));
        if (OP == OP_IMAD) asm volatile("mad.lo.u32 %0, %0, %1, %2;" : "+r"(a[j]) : "r"(b), "r"(c));
        if (OP == OP_IMADHI) asm volatile("mul.hi.u32 %0, %0, %1;" : "+r"(a[j]) : "r"(b | 0x80000000u));
        if (OP == OP_LOP3) asm volatile("lop3.b32 %0, %0, %1, %2, 0x96;" : "+r"(a[j]) : "r"(b), "r"(c));
        if (OP == OP_IADD) asm volatile("add.u32 %0, %0, %1;" : "+r"(a[j]) : "r"(b));
        if (OP == OP_LDS) {
            uint32_t v;
            // word lane + 32 (a[j] & 7): one bank per lane, inside the 1 KB the CTA zeroed
            const uint32_t w = (threadIdx.x & 31u) + ((a[j] & 7u) << 5);
            asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(sbase + (w << 2)));
            a[j] += v + 1u;
        }
    }
}

template <int OP>
__global__ void __launch_bounds__(kThreads) throughput_kernel(unsigned long long *cycles, uint32_t *sink) {
    extern __shared__ uint32_t s[];
    for (int i = threadIdx.x; i < 256; i += blockDim.x) s[i] = 0u;
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(s);
    double d[kChains];
    uint32_t a[kChains];
#pragma unroll
    for (int j = 0; j < kChains; ++j) {
        d[j] = 1.0 + j * 1e-3 + threadIdx.x * 1e-7;
        a[j] = threadIdx.x * 2654435761u + (uint32_t)j;
    }
    const uint32_t b = threadIdx.x | 1u, c = blockIdx.x + 7u;
    const double y = 1e-9;
    __syncthreads();
    const long long t0 = clock64();
    for (int it = 0; it < kIters; ++it) step<OP>(d, a, b, c, y, sbase);
    __syncthreads();
    const long long t1 = clock64();
    uint32_t acc = 0u;
#pragma unroll
    for (int j = 0; j < kChains; ++j) acc ^= a[j] ^ (uint32_t)__double_as_longlong(d[j]);
    if (acc == 0x12345678u) sink[0] = acc;  // keeps the chains alive
    if (threadIdx.x == 0) cycles[blockIdx.x] = (unsigned long long)(t1 - t0);
}

template <int OP>
__global__ void latency_kernel(unsigned long long *cycles, uint32_t *sink) {
    __shared__ uint32_t s[256];
    for (int i = threadIdx.x; i < 256; i += blockDim.x) s[i] = 0u;
    __syncthreads();
    if (threadIdx.x != 0) return;
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(s);
    double d = 1.0;
    uint32_t a = 12345u;
    const long long t0 = clock64();
#pragma unroll 16
    for (int it = 0; it < kIters; ++it) {
        if (OP == OP_DADD) asm volatile("add.rn.f64 %0, %0, %1;" : "+d"(d) : "d"(1e-9));
        if (OP == OP_IMAD) asm volatile("mad.lo.u32 %0, %0, %1, %2;" : "+r"(a) : "r"(3u), "r"(1u));
        if (OP == OP_LDS) asm volatile("ld.shared.u32 %0, [%1];" : "=r"(a) : "r"(sbase + ((a & 255u) << 2)));
    }
    const long long t1 = clock64();
    if ((a ^ (uint32_t)__double_as_longlong(d)) == 0x12345678u) sink[0] = a;
    cycles[0] = (unsigned long long)(t1 - t0);
}

template <int OP>
cudaError_t run_throughput(int sms, unsigned long long *d_cyc, uint32_t *d_sink, double *rate) {
    cudaError_t e = cudaFuncSetAttribute(throughput_kernel<OP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
    if (e != cudaSuccess) return e;
    for (int rep = 0; rep < 2; ++rep) {  // the first launch warms up
        throughput_kernel<OP><<<sms, kThreads, kSmem>>>(d_cyc, d_sink);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    std::vector<unsigned long long> cyc((size_t)sms);
    e = cudaMemcpy(cyc.data(), d_cyc, cyc.size() * 8, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return e;
    double sum = 0.0;
    for (unsigned long long c : cyc) sum += (double)kThreads * kChains * kIters / (double)c;
    *rate = sum / sms;
    return cudaSuccess;
}

template <int OP>
cudaError_t run_latency(unsigned long long *d_cyc, uint32_t *d_sink, double *lat) {
    unsigned long long c = 0;
    for (int rep = 0; rep < 2; ++rep) {
        latency_kernel<OP><<<1, 32>>>(d_cyc, d_sink);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    cudaError_t e = cudaMemcpy(&c, d_cyc, 8, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return e;
    *lat = (double)c / kIters;
    return cudaSuccess;
}

}  // namespace

extern "C" rewl_status rewl_measure_pipes(rewl_pipe_rates *out) {
    REWL_API_TRY
    if (!out) return rewl::host::fail(REWL_ERR_ARG, "NULL argument");
    int dev = 0, sms = 0, khz = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&khz, cudaDevAttrClockRate, dev);
    if (e != cudaSuccess) return rewl::host::fail(REWL_ERR_CUDA, "device query: %s", cudaGetErrorString(e));
    unsigned long long *d_cyc = nullptr;
    uint32_t *d_sink = nullptr;
    e = cudaMalloc((void **)&d_cyc, (size_t)sms * 8);
    if (e == cudaSuccess) e = cudaMalloc((void **)&d_sink, 64);
    if (e == cudaSuccess) e = run_throughput<OP_DADD>(sms, d_cyc, d_sink, &out->dadd);
    if (e == cudaSuccess) e = run_throughput<OP_IMAD>(sms, d_cyc, d_sink, &out->imad);
    if (e == cudaSuccess) e = run_throughput<OP_IMADHI>(sms, d_cyc, d_sink, &out->imad_hi);
    if (e == cudaSuccess) e = run_throughput<OP_LOP3>(sms, d_cyc, d_sink, &out->lop3);
    if (e == cudaSuccess) e = run_throughput<OP_IADD>(sms, d_cyc, d_sink, &out->iadd);
    if (e == cudaSuccess) e = run_throughput<OP_LDS>(sms, d_cyc, d_sink, &out->lds);
    if (e == cudaSuccess) e = run_latency<OP_DADD>(d_cyc, d_sink, &out->dadd_latency);
    if (e == cudaSuccess) e = run_latency<OP_IMAD>(d_cyc, d_sink, &out->imad_latency);
    if (e == cudaSuccess) e = run_latency<OP_LDS>(d_cyc, d_sink, &out->lds_latency);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    cudaFree(d_cyc);
    cudaFree(d_sink);
    if (e != cudaSuccess) return rewl::host::fail(REWL_ERR_CUDA, "pipe probe: %s", cudaGetErrorString(e));
    out->sms = sms;
    out->max_clock_mhz = khz / 1000.0;
    return REWL_OK;
    REWL_API_CATCH
}
