// Packed pair of FP32 lanes for the paired-node fused kernels.
//
// Blackwell executes FP32 multiply, add and fused multiply-add on pairs of
// values in one instruction (__fmul2_rn, __fadd2_rn, __ffma2_rn).  `f2`
// carries the same quantity of two neighbouring lattice nodes; the node
// arithmetic of lbm_node.cuh is instantiated with R = f2 unchanged.  Every
// lane rounds exactly like the scalar FP32 operation it replaces, and the
// node arithmetic names each fused multiply-add (mad) while the compiler's
// own contraction is off; what the assembler contracts in the packed form
// all the same is named in lbm_node.cuh.
#pragma once

#include <cuda_runtime.h>

#include "lbm_node.cuh"

namespace lbm {

struct f2 {
    float2 v;
    __device__ __forceinline__ f2() {}
    __device__ __forceinline__ f2(float a) : v(make_float2(a, a)) {}
    __device__ __forceinline__ f2(double a) : v(make_float2((float)a, (float)a)) {}
    __device__ __forceinline__ f2(int a) : v(make_float2((float)a, (float)a)) {}
    __device__ __forceinline__ f2(float2 x) : v(x) {}
};

__device__ __forceinline__ float2 neg2(float2 x) { return make_float2(-x.x, -x.y); }

__device__ __forceinline__ f2 operator*(const f2& a, const f2& b) { return f2(__fmul2_rn(a.v, b.v)); }
__device__ __forceinline__ f2 operator+(const f2& a, const f2& b) { return f2(__fadd2_rn(a.v, b.v)); }
__device__ __forceinline__ f2 operator-(const f2& a, const f2& b) { return f2(__fadd2_rn(a.v, neg2(b.v))); }
__device__ __forceinline__ f2 operator-(const f2& a) { return f2(neg2(a.v)); }

__device__ __forceinline__ f2& operator+=(f2& a, const f2& b) { return a = a + b; }
__device__ __forceinline__ f2& operator-=(f2& a, const f2& b) { return a = a - b; }

__device__ __forceinline__ f2 mad(const f2& a, const f2& b, const f2& c) { return f2(__ffma2_rn(a.v, b.v, c.v)); }

// Per-lane operations without a packed form.
__device__ __forceinline__ f2 fdiv(const f2& a, const f2& b) {
    return f2(make_float2(__fdividef(a.v.x, b.v.x), __fdividef(a.v.y, b.v.y)));
}
__device__ __forceinline__ f2 recip(const f2& b) { return fdiv(f2(1.0f), b); }
__device__ __forceinline__ f2 root(const f2& a) { return f2(make_float2(sqrtf(a.v.x), sqrtf(a.v.y))); }

__device__ __forceinline__ f2 cs_dev(const f2* c, const f2* lo, const f2& rho_d, const f2& T, const f2& T_d) {
    float k[7], l[7];
#pragma unroll
    for (int i = 0; i < 7; ++i) {
        k[i] = c[i].v.x;
        l[i] = lo[i].v.x;
    }
    return f2(make_float2(cs_dev(k, l, rho_d.v.x, T.v.x, T_d.v.x), cs_dev(k, l, rho_d.v.y, T.v.y, T_d.v.y)));
}

}  // namespace lbm
