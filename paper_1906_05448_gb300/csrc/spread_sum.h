// Sums of spread forces in 32-bit integers (FP32 storage, particles.cu),
// without CUDA, so that their error is checked on the CPU.
//
// Each component of a particle's marker forces has a scale of its own: the
// power of two that puts its largest |F_l dV_l| at 2^29 .. 2^30. The weights
// of a cell over the markers of a sphere (about one per unit of surface) add
// up to 0.91 at most, at a radius of 1.1, and to 0.5 .. 0.6 beyond 2, so a sum
// stays below 2^30; its terms are rounded at 2^-30 or less of the largest
// force, finer than FP32 sums of that size. One scale for the three
// components left a force that is much weaker across the flow than along it
// 2^-28 of the stronger one: at a hundredth of it 8e-6 of itself, where FP32
// sums have 8e-8 and these 6e-8.
// Spheres of fewer than six markers are summed in FP32: a cell takes a term or
// two there, which FP32 rounds once and the integers twice.
#pragma once

#include <math.h>
#include <string.h>

#ifndef LBM_HD
#ifdef __CUDACC__
#define LBM_HD __host__ __device__ __forceinline__
#else
#define LBM_HD inline
#endif
#endif

namespace lbmgb {

LBM_HD bool spread_few(int markers) { return markers < 6; }

// m >= 0: the largest |F_l dV_l| of a component
LBM_HD float spread_scale(float m) {  // 2^(29 - exponent of m)
    unsigned u;
    memcpy(&u, &m, 4);
    const int e = (int)(u >> 23) - 127;
    return m > 0.f ? exp2f((float)(29 - e < 120 ? 29 - e : 120)) : 1.f;
}
LBM_HD int spread_term(float v, float s) {
#ifdef __CUDA_ARCH__
    return __float2int_rn(v * s);
#else
    return (int)lrintf(v * s);
#endif
}
LBM_HD float spread_value(int v, float s) { return (float)v / s; }

}  // namespace lbmgb
