// Double-float values: the unevaluated sum hi + lo of two FP32 numbers, about 48
// significant bits (error-free transformations of Knuth and Dekker, FMA-based exact
// products). Used for the forward blur b = psi * P_v, whose FP32 FFT rounding
// (absolute, scaled by the whole volume's norm) would swamp dim voxels of b. The
// arithmetic is in adf.cuh (scalar) and adp.cuh (packed pairs); here are the types,
// the constants and the asynchronous copies.
#pragma once

#include "fft.cuh"

namespace mvd {

struct dd {
    float hi, lo;
};

// complex double-float, 16 bytes. In device memory (global and shared) the order is
// re.hi, im.hi, re.lo, im.lo (adp.cuh), read and written through cdp_load / cdp_store.
struct __align__(16) cdd {
    dd re, im;
};

// 16-byte asynchronous global -> shared copy (L2 only); with !valid nothing is
// read and the 16 bytes are zero-filled (src then only needs to be a valid
// address)
__device__ __forceinline__ void cp_async16(void* dst_smem, const void* src, bool valid) {
    const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(dst_smem));
    const int n = valid ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async8(void* dst_smem, const void* src, bool valid) {
    const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(dst_smem));
    const int n = valid ? 8 : 0;
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(d), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}

// constant (cos, S sin) pairs as double-float: hi = fl32(c), lo = fl32(c - hi)
#define MVD_DD(c) dd{(float)(c), (float)((c) - (double)(float)(c))}

}  // namespace mvd
