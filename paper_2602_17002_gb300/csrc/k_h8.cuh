// Point work of the FP32 affine H8 elements, one lane per element.
//
// A trilinear field is a sum of eight products of the parent coordinates; its
// coefficients C_m (bit 0, 1, 2 of m: the coordinate xi, eta, zeta is a factor
// of the product) are sums of the nodal values with signs. At a Gauss point
// (s_x, s_y, s_z) / sqrt 3, with the powers of 1/sqrt 3 folded into the C_m,
//   d/dxi   = C1 + s_y C3 + s_z C5 + s_y s_z C7
//   d/deta  = C2 + s_x C3 + s_z C6 + s_x s_z C7
//   d/dzeta = C4 + s_x C5 + s_y C6 + s_x s_y C7
// so the two points of one (s_y, s_z) share the xi derivative and differ in a
// sign elsewhere: 9 operations a component for both where the sums over the
// eight nodes take 48. The points are evaluated two at a time in packed
// arithmetic (F2); their operators are accumulated on the C_m (the transposed
// map), and the element vector is formed once from those. The normalised
// consistent mass is diagonal on the C_m: 1/2 per coordinate that is not a
// factor, 1/6 per one that is.
#pragma once

#include "k_t10.cuh"

namespace tlfe {

// the signed sums over the corners (its own transpose): y[m] = sum_n (-1)^(bits of m not set in n) x[n]
__device__ __forceinline__ void h8_transform(V3f x[8])
{
#pragma unroll
    for (int d = 1; d < 8; d *= 2)
#pragma unroll
        for (int n = 0; n < 8; ++n)
            if (!(n & d)) {
                const V3f a = x[n], b = x[n + d];
                x[n] = a + b;
                x[n + d] = b - a;
            }
}
// transpose of h8_transform
__device__ __forceinline__ void h8_transform_t(V3f x[8])
{
#pragma unroll
    for (int d = 1; d < 8; d *= 2)
#pragma unroll
        for (int n = 0; n < 8; ++n)
            if (!(n & d)) {
                const V3f a = x[n], b = x[n + d];
                x[n] = a - b;
                x[n + d] = a + b;
            }
}
// 1/8 (1/sqrt 3)^(factors - 1) of coefficient m = 1..7
__host__ __device__ constexpr float h8_scale(int m)
{
    const int f = (m & 1) + ((m >> 1) & 1) + ((m >> 2) & 1);
    return f == 1 ? 0.125f : (f == 2 ? float(0.125 * 0.57735026918962576451) : float(0.125 / 3.0));
}
// the normalised consistent mass on the transformed values: 1/8 of its
// eigenvalue for m (the transform times its transpose is 8)
__host__ __device__ constexpr double h8_mass(int m)
{
    const int f = (m & 1) + ((m >> 1) & 1) + ((m >> 2) & 1);
    return f == 0 ? 1.0 / 64 : (f == 1 ? 1.0 / 192 : (f == 2 ? 1.0 / 576 : 1.0 / 1728));
}

// gradients of one field at the point (sx, sy, sz) or, with V = F2, at both
// points of (sy, sz); J^{-1} applied. c[((m - 1) * 3 + row) * 32]: the scaled
// coefficients
template <typename V>
__device__ __forceinline__ void h8_gradients(const float *c, V sx, float sy, float sz, const float Ji[9], V G[9])
{
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        float C[8];
#pragma unroll
        for (int m = 1; m < 8; ++m) C[m] = c[((m - 1) * 3 + a) * 32];
        const float u = fmaf(sz, C[7], C[3]), v = fmaf(sy, C[7], C[5]);
        const float gx = fmaf(sy, u, fmaf(sz, C[5], C[1]));
        const V gy = u * sx + V(fmaf(sz, C[6], C[2])), gz = v * sx + V(fmaf(sy, C[6], C[4]));
#pragma unroll
        for (int b = 0; b < 3; ++b) G[a * 3 + b] = gy * Ji[3 + b] + V(gx * Ji[b]) + gz * Ji[6 + b];
    }
}

// adds the operators of the point(s) to the coefficients' accumulators (the
// transpose of h8_gradients): T row-major, Aj the lane's J^{-1}
template <typename V>
__device__ __forceinline__ void h8_accumulate(const V T[9], V sx, float sy, float sz, const float *Aj, float detJ,
                                              V3f C[8])
{
    float t[3][5];  // component: sums of the xi, eta, zeta parts, those of the eta, zeta parts times sx
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float j0 = detJ * Aj[(k * 3) * 32], j1 = detJ * Aj[(k * 3 + 1) * 32], j2 = detJ * Aj[(k * 3 + 2) * 32];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const V h = T[a * 3] * j0 + T[a * 3 + 1] * j1 + T[a * 3 + 2] * j2;
            t[a][k] = sum_of(h);
            if (k > 0) t[a][2 + k] = sum_of(V(h * sx));
        }
    }
    auto part = [&](int k) { return V3f{make_float2(t[0][k], t[1][k]), t[2][k]}; };
    const V3f hx = part(0), hy = part(1), hz = part(2), dy = part(3), dz = part(4);
    C[1] = C[1] + hx;
    C[2] = C[2] + hy;
    C[4] = C[4] + hz;
    C[6] = C[6].fma(sz, hy).fma(sy, hz);
    C[3] = (C[3] + dy).fma(sy, hx);
    C[5] = (C[5] + dz).fma(sz, hx);
    C[7] = C[7].fma(sy * sz, hx).fma(sz, dy).fma(sy, dz);
}

}  // namespace tlfe
