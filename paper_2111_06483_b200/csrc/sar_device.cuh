// Device helpers shared by the gather kernels (internal): packed float32 pairs, shared-memory accesses, asynchronous copies.
#pragma once

#include "sar_common.cuh"

namespace sar {

// order-preserving float -> unsigned key (for shared-memory atomicMax)
__device__ __forceinline__ unsigned fkey(float x) {
    const unsigned b = __float_as_uint(x);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float fkey_inv(unsigned k) {
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}
constexpr unsigned kKeyNegInf = 0x007fffffu;  // fkey(-inf)

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// shared-memory accesses through 32-bit shared-window addresses (no 64-bit pointer arithmetic)
__device__ __forceinline__ uint4 lds128(unsigned addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];\n" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}
__device__ __forceinline__ float lds_f32(unsigned addr) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];\n" : "=f"(v) : "r"(addr));
    return v;
}
// packed pairs of float32 (Blackwell's two-wide FP32 pipe: one instruction, two fused multiply-adds)
typedef float2 f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) { return make_float2(lo, hi); }
__device__ __forceinline__ void unpack2(f32x2 p, float &lo, float &hi) {
    lo = p.x;
    hi = p.y;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) { return __ffma2_rn(a, b, c); }  // a*b + c, element-wise
__device__ __forceinline__ f32x2 zero2() { return make_float2(0.f, 0.f); }
// 16 bytes of storage type T -> EPV/2 packed float32 pairs
template <typename T>
struct Pairs;
template <>
struct Pairs<float> {
    __device__ __forceinline__ static void get(const uint4 &d, f32x2 (&p)[2]) {
        p[0] = pack2(__uint_as_float(d.x), __uint_as_float(d.y));
        p[1] = pack2(__uint_as_float(d.z), __uint_as_float(d.w));
    }
};
template <>
struct Pairs<__nv_bfloat16> {
    __device__ __forceinline__ static void get(const uint4 &d, f32x2 (&p)[4]) {
        p[0] = pack2(__uint_as_float(d.x << 16), __uint_as_float(d.x & 0xffff0000u));
        p[1] = pack2(__uint_as_float(d.y << 16), __uint_as_float(d.y & 0xffff0000u));
        p[2] = pack2(__uint_as_float(d.z << 16), __uint_as_float(d.z & 0xffff0000u));
        p[3] = pack2(__uint_as_float(d.w << 16), __uint_as_float(d.w & 0xffff0000u));
    }
};

}  // namespace sar
