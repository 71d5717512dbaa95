// Device helpers shared by the convolution kernels: packed fp32 arithmetic, asynchronous copies into shared memory,
// division by a launch constant.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace distdl {

constexpr int kConvMaxWorkers = 64;

// n / d == umulhi(n, magic) >> shift for any n < 2^31 (magic 0 stands for d = 1): magic = ceil(2^(31+s) / d) with
// s = ceil(log2 d) is below 2^32 and divides exactly.
struct FastDiv {
    uint32_t d, magic, shift;
};
inline FastDiv make_fast_div(uint32_t d) {
    FastDiv f = {d, 0, 0};
    if (d < 2) return f;
    uint32_t sh = 0;
    while ((1u << sh) < d) ++sh;
    const uint64_t num = (uint64_t)1 << (31 + sh);
    f.magic = (uint32_t)((num + d - 1) / d);
    f.shift = sh - 1;
    return f;
}

#ifdef __CUDACC__
__device__ __forceinline__ uint32_t fast_quot(const FastDiv &f, uint32_t n) {
    return f.magic ? __umulhi(n, f.magic) >> f.shift : n;
}
// n = q * d + r: returns r and leaves q in n
__device__ __forceinline__ uint32_t fast_rem(const FastDiv &f, uint32_t &n) {
    const uint32_t q = fast_quot(f, n), r = n - q * f.d;
    n = q;
    return r;
}

// Packed fp32 pair arithmetic (two FMAs per instruction on sm_100).
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}
__device__ __forceinline__ void unpack2(uint64_t v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

// x itself, as the result of an instruction: `zero` is a kernel parameter that holds 0.  A pair that is only put together by
// register moves is put together again at every use when registers are short; the result of an exclusive-or is kept.
__device__ __forceinline__ float fresh(float x, uint32_t zero) { return __uint_as_float(__float_as_uint(x) ^ zero); }

// Coordinate i of a tile cell along one dimension -> owning worker coordinate (w - 1, w or w + 1) and index in its bulk;
// false outside the tensor.
__device__ __forceinline__ bool conv_owner(const int32_t *b, int workers, int w, int i, int &owner, int &index) {
    owner = w;
    index = i;
    if (i < 0) {
        owner = w - 1;
        if (owner < 0) return false;
        index = i + b[owner];
        return index >= 0;
    }
    if (i >= b[w]) {
        owner = w + 1;
        if (owner >= workers) return false;
        index = i - b[w];
        return index < b[owner];
    }
    return true;
}

__device__ __forceinline__ void cp_async4_to(uint32_t smem, const float *gmem) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async16_to(uint32_t smem, const float *gmem) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait_group() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
#endif

}  // namespace distdl
