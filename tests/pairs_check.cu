// Compares the branch-free reciprocals, quotients and square roots of
// csrc/pairs.cuh with CUDA's correctly rounded intrinsics; each entry returns
// the number of differences (or -1 on a CUDA error).
#include <cuda_runtime.h>
#include <stdint.h>

#include "pairs.cuh"

namespace {

typedef unsigned long long u64;

// Every float of [lo, hi] (positive, by bits), and its negative for reciprocals.
__global__ void unary_kernel(uint32_t lo, uint32_t hi, bool roots, u64* bad) {
    for (u64 u = lo + blockIdx.x * (u64)blockDim.x + threadIdx.x; u <= hi; u += (u64)gridDim.x * blockDim.x) {
        const float x = __uint_as_float((uint32_t)u);
        bool same;
        if (roots) {
            const float e = __fsqrt_rn(x);
            const float2 p = ps::sqrt_rn2(make_float2(x, x));
            same = ps::sqrt_rn(x) == e && p.x == e && p.y == e;
        } else {
            const float e = __frcp_rn(x);
            const float2 p = ps::rcp_rn2(make_float2(x, -x));
            same = ps::rcp_rn(x) == e && p.x == e && p.y == -e;
        }
        if (!same) atomicAdd(bad, 1ull);
    }
}

// Every float of [lo, hi] divided by the constant c.
__global__ void constant_kernel(uint32_t lo, uint32_t hi, float c, u64* bad) {
    const float inv = 1.0f / c;
    for (u64 u = lo + blockIdx.x * (u64)blockDim.x + threadIdx.x; u <= hi; u += (u64)gridDim.x * blockDim.x) {
        const float a = __uint_as_float((uint32_t)u), e = __fdiv_rn(a, c);
        const float2 p = ps::div_rn2(make_float2(a, -a), ps::dup2(c), ps::dup2(inv));
        if (!(ps::div_rn(a, c, inv) == e && p.x == e && p.y == -e)) atomicAdd(bad, 1ull);
    }
}

__device__ uint32_t next(u64& s) {  // xorshift
    s ^= s << 13;
    s ^= s >> 7;
    s ^= s << 17;
    return (uint32_t)(s >> 16);
}

// Random quotients a / b, exponents of a in [a0, a1] and of b in [b0, b1].
__global__ void quotient_kernel(int a0, int a1, int b0, int b1, u64* bad) {
    u64 s = 0x9E3779B97F4A7C15ull * (blockIdx.x * (u64)blockDim.x + threadIdx.x + 1);
    for (int i = 0; i < 4000; ++i) {
        const float a = __uint_as_float((next(s) & 0x807fffffu) | (uint32_t)(127 + a0 + (int)(next(s) % (a1 - a0 + 1))) << 23);
        const float b = __uint_as_float((next(s) & 0x807fffffu) | (uint32_t)(127 + b0 + (int)(next(s) % (b1 - b0 + 1))) << 23);
        const float e = __fdiv_rn(a, b);
        const float2 bb = make_float2(b, -b), p = ps::div_rn2(ps::dup2(a), bb, ps::rcp_rn2(bb));
        if (!(ps::div_rn(a, b, ps::rcp_rn(b)) == e && p.x == e && p.y == -e)) atomicAdd(bad, 1ull);
    }
}

template <class F>
long long count(F launch) {
    u64 *d = nullptr, h = 0;
    if (cudaMalloc(&d, sizeof(h)) != cudaSuccess) return -1;
    cudaMemset(d, 0, sizeof(h));
    launch(d);
    const bool ok = cudaGetLastError() == cudaSuccess && cudaMemcpy(&h, d, sizeof(h), cudaMemcpyDeviceToHost) == cudaSuccess;
    cudaFree(d);
    return ok ? (long long)h : -1;
}

}  // namespace

extern "C" long long check_unary(uint32_t lo, uint32_t hi, int roots) {
    return count([&](u64* d) { unary_kernel<<<2048, 256>>>(lo, hi, roots != 0, d); });
}
extern "C" long long check_constant(uint32_t lo, uint32_t hi, float c) {
    return count([&](u64* d) { constant_kernel<<<2048, 256>>>(lo, hi, c, d); });
}
extern "C" long long check_quotients(int a0, int a1, int b0, int b1) {
    return count([&](u64* d) { quotient_kernel<<<1024, 256>>>(a0, a1, b0, b1, d); });
}
