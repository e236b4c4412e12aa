// FP64 sums of a node's populations for the readers of the state.
#pragma once

#include <cuda_runtime.h>

#include "lbm_node.cuh"

namespace lbm {

// FP64 sums over the populations of a node stored in FP32.  An FP64 addition
// or FP32-to-FP64 conversion issues once per 76 cycles and scheduler, and 18
// conversions and 24 additions were most of what the readers of the state
// spent.  Instead the sums are formed exactly in 64-bit integers: with the
// largest exponent emax of the nine values, each is its signed 24-bit
// mantissa times 2^(e - emax + 30), one wide multiply-add per term, and the
// sum is converted, and so rounded, once.  Values more than 30 binades below
// the largest, denormals, infinities and NaN take the FP64 additions.
// k_macros with its consumer's passes, 39.2M nodes: 6.3 -> 3.5 ms; with the
// conversion of the sums in integers too, k_macros at 4096^2 0.89 -> 0.76 ms.
struct Fixed9 {
    int m[9], p[9];  // mantissa with sign, power of two
    int emax;
    __device__ __forceinline__ bool set(const float* f) {
        int e[9];
        emax = 0;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            e[i] = (__float_as_int(f[i]) >> 23) & 255;
            emax = max(emax, e[i]);
        }
        bool ok = emax != 255;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const int b = __float_as_int(f[i]), s = b >> 31;
            const bool zero = (b & 0x7fffffff) == 0;
            const int sh = e[i] - emax + 30;
            ok = ok && (zero || (e[i] != 0 && sh >= 0));
            m[i] = zero ? 0 : ((((b & 0x007fffff) | 0x00800000) ^ s) - s);
            p[i] = 1 << (sh & 31);
        }
        return ok;
    }
    __device__ __forceinline__ long long at(int i) const { return (long long)m[i] * p[i]; }
    // the sum v of terms at(i) times 2^(emax - 180), rounded to nearest even
    // as (double)v is, in integers: that conversion takes an FP64 issue slot.
    // |v| < 9 * 2^54, so its leading bit moves up to bit 62, and the ten bits
    // below the 53 round it; a carry out of them raises the exponent.
    __device__ __forceinline__ double value(long long v) const {
        const unsigned long long u = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
        const int up = __clzll((long long)u) - 1;
        const unsigned long long n = u << (up & 63), r = (n + 0x1ff + ((n >> 10) & 1)) >> 10;
        const long long bits = (long long)(r + ((unsigned long long)(1022 + 62 - up + emax - 180) << 52));
        return __longlong_as_double(v == 0 ? 0 : bits | (v & (long long)0x8000000000000000ull));
    }
};

__device__ __forceinline__ void node_sums_fp64(const double* v, double& rd, double& jx, double& jy, double& sg) {
    node_sums(v, v + 9, rd, jx, jy, sg);
}
__device__ __forceinline__ void node_sums_fp64(const float* v, double& rd, double& jx, double& jy, double& sg) {
    Fixed9 f, g;
    const bool okf = f.set(v), okg = g.set(v + 9);
    if (okf && okg) {
        const long long d1 = f.at(5) - f.at(7), d2 = f.at(6) - f.at(8);
        long long r = f.at(0), s = g.at(0);
#pragma unroll
        for (int i = 1; i < 9; ++i) {
            r += f.at(i);
            s += g.at(i);
        }
        rd = f.value(r);
        jx = f.value(f.at(1) - f.at(3) + (d1 - d2));
        jy = f.value(f.at(2) - f.at(4) + (d1 + d2));
        sg = g.value(s);
    } else {
        double w[18];
#pragma unroll
        for (int q = 0; q < 18; ++q) w[q] = (double)v[q];
        node_sums(w, w + 9, rd, jx, jy, sg);
    }
}

}  // namespace lbm
