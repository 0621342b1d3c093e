// Vector loads and stores of V consecutive members (16-byte accesses for
// float4 / double2) shared by the lattice kernels. Internal header.
#pragma once
#include <cuda_runtime.h>

namespace lbmgpu {

template <typename T, int V>
struct Vec;
template <>
struct Vec<double, 1> {
    static __device__ __forceinline__ void ld(const double* p, double (&v)[1]) { v[0] = __ldg(p); }
    static __device__ __forceinline__ void st(double* p, const double (&v)[1]) { p[0] = v[0]; }
};
template <>
struct Vec<double, 2> {
    static __device__ __forceinline__ void ld(const double* p, double (&v)[2]) {
        double2 t = __ldg(reinterpret_cast<const double2*>(p));
        v[0] = t.x;
        v[1] = t.y;
    }
    static __device__ __forceinline__ void st(double* p, const double (&v)[2]) {
        *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
    }
};
template <>
struct Vec<float, 1> {
    static __device__ __forceinline__ void ld(const float* p, float (&v)[1]) { v[0] = __ldg(p); }
    static __device__ __forceinline__ void st(float* p, const float (&v)[1]) { p[0] = v[0]; }
};
template <>
struct Vec<float, 2> {
    static __device__ __forceinline__ void ld(const float* p, float (&v)[2]) {
        float2 t = __ldg(reinterpret_cast<const float2*>(p));
        v[0] = t.x;
        v[1] = t.y;
    }
    static __device__ __forceinline__ void st(float* p, const float (&v)[2]) {
        *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
    }
};
template <>
struct Vec<float, 4> {
    static __device__ __forceinline__ void ld(const float* p, float (&v)[4]) {
        float4 t = __ldg(reinterpret_cast<const float4*>(p));
        v[0] = t.x;
        v[1] = t.y;
        v[2] = t.z;
        v[3] = t.w;
    }
    static __device__ __forceinline__ void st(float* p, const float (&v)[4]) {
        *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    }
};

// (double)x without the FP64 pipe, on which a conversion costs as much as an
// addition (two per SM cycle on GB300): a normal binary32 number's bits are
// its binary64 number's, the exponent rebiased.
__device__ __forceinline__ double widen(float x) {
    const unsigned b = __float_as_uint(x), e = b & 0x7f800000u;
    if (e == 0u || e == 0x7f800000u) return (double)x;  // zero, subnormal, infinity, NaN
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(b << 29));
}
__device__ __forceinline__ double widen(double x) { return x; }

// (float)x, rounded to nearest even, likewise on the integer units: the
// value's low 29 bits decide. Outside the range of normal binary32 numbers
// the conversion instruction.
__device__ __forceinline__ float narrow(double x) {
    const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
    const unsigned m = h & 0x7fffffffu;
    if (m < 0x38100000u || m >= 0x47e00000u) return __double2float_rn(x);
    unsigned r = ((m - 0x38000000u) << 3) | (l >> 29);
    const unsigned rest = l << 3;
    r += (rest > 0x80000000u || (rest == 0x80000000u && (r & 1u))) ? 1u : 0u;
    return __uint_as_float((h & 0x80000000u) | r);
}
__device__ __forceinline__ void narrow_to(float& d, double x) { d = narrow(x); }
__device__ __forceinline__ void narrow_to(double& d, double x) { d = x; }

// Density and velocity of one member's f (g = f - w with SHIFT), FP64: 16
// additions and two divisions (one division and two products took 0.1 ms less
// per pass at 256^2 x 64 and left u and v an ulp off in a quarter of the cells).
template <bool SHIFT>
__device__ __forceinline__ void moments_of(const double (&g)[9], double& r, double& ux, double& uy) {
    const double d56 = g[5] - g[6], d78 = g[7] - g[8];
    const double jx = (g[1] - g[2]) + (d56 + d78), jy = (g[3] - g[4]) + (d56 - d78);
    r = ((g[0] + g[1]) + (g[2] + g[3])) + ((g[4] + g[5]) + (g[6] + g[7])) + g[8];
    if (SHIFT) r += 1.0;
    ux = jx / r;
    uy = jy / r;
}

// Work item t of a lattice kernel -> member group mv (of kv per cell), cell,
// and its coordinates (x, y). The divisions run in 32 bits while t fits
// (64-bit integer division is emulated and costs several times more).
__device__ __forceinline__ void split_item(long long t, int kv, int nx, int& mv, long long& cell, int& x,
                                           int& y) {
    if (t < 0x100000000LL) {
        const unsigned tt = (unsigned)t, ukv = (unsigned)kv, unx = (unsigned)nx;
        const unsigned c = tt / ukv;
        mv = (int)(tt - c * ukv);
        cell = c;
        const unsigned yy = c / unx;
        y = (int)yy;
        x = (int)(c - yy * unx);
    } else {
        mv = (int)(t % kv);
        cell = t / kv;
        x = (int)(cell % nx);
        y = (int)(cell / nx);
    }
}

}  // namespace lbmgpu
