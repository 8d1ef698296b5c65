// Per-lane vectors of the gather kernels (16-byte or scalar loads of fp32 / bf16 features, widened to
// fp32) and the element store shared by them.
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

namespace gnnfd {

// ---- per-lane vectors: VECN elements of T, widened to fp32

// plain loads from global memory: what they read may have been written by the launch before (see grid_dependency)
__device__ __forceinline__ uint4 load16(const void* p)
{
    uint4 v;
    asm("ld.global.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ float load4(const float* p)
{
    float v;
    asm("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}

template <typename T, int VECN> struct Vec;

template <> struct Vec<float, 4> {
    float4 v;
    __device__ __forceinline__ void load(const float* p)
    {
        const uint4 w = load16(p);
        v = make_float4(__uint_as_float(w.x), __uint_as_float(w.y), __uint_as_float(w.z), __uint_as_float(w.w));
    }
    __device__ __forceinline__ void zero() { v = make_float4(0.f, 0.f, 0.f, 0.f); }
    __device__ __forceinline__ float get(int i) const { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }
};
template <> struct Vec<float, 1> {
    float v;
    __device__ __forceinline__ void load(const float* p) { v = load4(p); }
    __device__ __forceinline__ void zero() { v = 0.f; }
    __device__ __forceinline__ float get(int) const { return v; }
};
template <> struct Vec<__nv_bfloat16, 8> {
    uint4 v;
    __device__ __forceinline__ void load(const __nv_bfloat16* p) { v = load16(p); }
    __device__ __forceinline__ void zero() { v = make_uint4(0u, 0u, 0u, 0u); }
    __device__ __forceinline__ uint32_t word(int i) const { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }
    __device__ __forceinline__ float get(int i) const
    {
        const uint32_t w = word(i >> 1);
        return __uint_as_float((i & 1) ? (w & 0xffff0000u) : (w << 16));   // bf16 -> fp32 is exact
    }
};
// (x, y) += the two bf16 values of a word, widened in the addition: the same rounding as widening first, in half the instructions.
// SAGE, 64 columns on 40 M entries 412 -> 379 us, 100 on 18 M 279 -> 259, 301 on 6 M 308 -> 265, 256 on 40 M 1150 -> 1053, on 3 M 129 -> 113,
// 512 on 8 M 543 -> 480.
__device__ __forceinline__ void add_widened(float& x, float& y, uint32_t w)
{
    asm("{\n\t.reg .b16 lo, hi;\n\tmov.b32 {lo, hi}, %2;\n\tadd.rn.f32.bf16 %0, lo, %0;\n\tadd.rn.f32.bf16 %1, hi, %1;\n\t}"
        : "+f"(x), "+f"(y) : "r"(w));
}
template <> struct Vec<__nv_bfloat16, 1> {
    unsigned short v;
    __device__ __forceinline__ void load(const __nv_bfloat16* p) { asm("ld.global.b16 %0, [%1];" : "=h"(v) : "l"(p)); }
    __device__ __forceinline__ void zero() { v = 0; }
    __device__ __forceinline__ float get(int) const { return __uint_as_float((uint32_t)v << 16); }
};

// Two adjacent 16-byte vectors with one 32-byte load (p must be 32-byte aligned): half the load
// instructions and, when a lane's two vectors sit next to each other, half the cache lines touched
// per instruction.
__device__ __forceinline__ void load_pair(Vec<float, 4>& a, Vec<float, 4>& b, const float* p)
{
    uint32_t r[8];
    asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "l"(p));
    a.v = make_float4(__uint_as_float(r[0]), __uint_as_float(r[1]), __uint_as_float(r[2]), __uint_as_float(r[3]));
    b.v = make_float4(__uint_as_float(r[4]), __uint_as_float(r[5]), __uint_as_float(r[6]), __uint_as_float(r[7]));
}
__device__ __forceinline__ void load_pair(Vec<__nv_bfloat16, 8>& a, Vec<__nv_bfloat16, 8>& b, const __nv_bfloat16* p)
{
    asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(a.v.x), "=r"(a.v.y), "=r"(a.v.z), "=r"(a.v.w), "=r"(b.v.x), "=r"(b.v.y), "=r"(b.v.z), "=r"(b.v.w)
                 : "l"(p));
}
// scalar vectors have no pair form; never called (the callers test the vector width first)
template <typename T>
__device__ __forceinline__ void load_pair(Vec<T, 1>& a, Vec<T, 1>& b, const T* p) { a.load(p); b.load(p + 1); }

// (x, y) += w * (a, b), (x, y) += (a, b) and (x, y) *= (a, b), each in one instruction: the same roundings as two scalar ones
// for half the issue slots.
__device__ __forceinline__ void fma_pair(float& x, float& y, float w, float a, float b)
{
    asm("{\n\t.reg .b64 p, q, r;\n\tmov.b64 p, {%2, %2};\n\tmov.b64 q, {%3, %4};\n\tmov.b64 r, {%0, %1};\n\t"
        "fma.rn.f32x2 r, p, q, r;\n\tmov.b64 {%0, %1}, r;\n\t}" : "+f"(x), "+f"(y) : "f"(w), "f"(a), "f"(b));
}
__device__ __forceinline__ void add_pair(float& x, float& y, float a, float b)
{
    asm("{\n\t.reg .b64 q, r;\n\tmov.b64 q, {%2, %3};\n\tmov.b64 r, {%0, %1};\n\t"
        "add.rn.f32x2 r, q, r;\n\tmov.b64 {%0, %1}, r;\n\t}" : "+f"(x), "+f"(y) : "f"(a), "f"(b));
}
__device__ __forceinline__ void mul_pair(float& x, float& y, float a, float b)
{
    asm("{\n\t.reg .b64 q, r;\n\tmov.b64 q, {%2, %3};\n\tmov.b64 r, {%0, %1};\n\t"
        "mul.rn.f32x2 r, q, r;\n\tmov.b64 {%0, %1}, r;\n\t}" : "+f"(x), "+f"(y) : "f"(a), "f"(b));
}

__device__ __forceinline__ void store_elem(void* out, int out_bf16, int64_t idx, float val)
{
    if (out_bf16) static_cast<__nv_bfloat16*>(out)[idx] = __float2bfloat16_rn(val);
    else __stcs(static_cast<float*>(out) + idx, val);
}

}  // namespace gnnfd
