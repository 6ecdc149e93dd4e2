// Point work of the FP32 affine T10 elements, one lane per element.
//
// The gradient of a quadratic field on a straight-sided tetrahedron is linear
// in the barycentric coordinates. With E_aj the value at the mid-edge node of
// edge (a, j) (E_jj: at corner j) and Delta_k = x_{k+1} - x_0, the parent
// gradient at corner j is 4 (E_{k+1,j} - E_{0,j}) - Delta_k, so that
//   at the centroid             G0_k = sum_j (E_{k+1,j} - E_{0,j}) - Delta_k,
//   at (a, b, b, b), a at j     base_k + 4 (a - b) (E_{k+1,j} - E_{0,j}),
//                               base_k = 4 b G0_k - (a - b) Delta_k:
// 6 operations a component, direction and point where the sum over the ten
// nodes takes 21. So
//   - the gradients of every field at the four points (a, b, b, b) are formed
//     once per element and kept in the lane's own column of shared memory, two
//     points side by side;
//   - the points are evaluated two at a time in packed arithmetic (F2), which
//     halves their instructions, and their operators overwrite the gradients;
//     the centroid of the 5-point rule comes first, on its own;
//   - the element vectors are the transposed map of the four operators. The
//     centroid has the mean of the other points' shape-function gradients, so
//     its operator is added to theirs in the ratio of the weights.
#pragma once

#include "tlfe_elem.cuh"
#include "tlfe_internal.h"

namespace tlfe {

// 3-vector of a node, (x, y) paired
struct V3f {
    float2 xy;
    float z;
    __device__ __forceinline__ V3f operator+(const V3f &o) const { return {__fadd2_rn(xy, o.xy), z + o.z}; }
    __device__ __forceinline__ V3f operator-(const V3f &o) const { return {__fadd2_rn(xy, neg2(o.xy)), z - o.z}; }
    __device__ __forceinline__ V3f operator*(float s) const { return {__fmul2_rn(xy, make_float2(s, s)), z * s}; }
    // this + s v
    __device__ __forceinline__ V3f fma(float s, const V3f &v) const
    {
        return {__ffma2_rn(v.xy, make_float2(s, s), xy), fmaf(v.z, s, z)};
    }
};

// node holding E_pj (no recursion: it has to fold to a constant in unrolled loops)
__host__ __device__ __forceinline__ constexpr int t10_node(int p, int j)
{
    const int lo = p < j ? p : j, hi = p < j ? j : p;
    return lo == hi ? lo : (lo == 0 ? (hi == 1 ? 4 : (hi == 2 ? 6 : 7)) : (lo == 1 ? (hi == 2 ? 5 : 8) : 9));
}

// the four points (a, b, b, b) of the rule, their weight, and the centroid's
template <int NQ> struct T10Rule {
    static constexpr double a = NQ == 5 ? 0.5 : 0.58541019662496845446;
    static constexpr double b = NQ == 5 ? 1.0 / 6.0 : 0.13819660112501051518;
    static constexpr double w = NQ == 5 ? 3.0 / 40.0 : 1.0 / 24.0;
    static constexpr double w0 = NQ == 5 ? -2.0 / 15.0 : 0.0;
};

// gradients of one field at the four points, J^{-1} applied, into the lane's
// records: entry (row, col) of points 2h and 2h + 1 at rec[(h * NV + row * 3 +
// col) * 32]; g0 receives the centroid's (row-major) when the rule has it
template <int NQ, int NV>
__device__ __forceinline__ void t10_gradients(const V3f x[10], const float Ji[9], float2 *rec, float g0[9])
{
    using Q = T10Rule<NQ>;
    V3f S[3], base[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const V3f D = x[k + 1] - x[0];
        S[k] = (((x[t10_node(k + 1, 0)] - x[0]) + (x[t10_node(k + 1, 1)] - x[t10_node(0, 1)])) +
                ((x[t10_node(k + 1, 2)] - x[t10_node(0, 2)]) + (x[t10_node(k + 1, 3)] - x[t10_node(0, 3)]))) -
               D;
        base[k] = (S[k] * float(4.0 * Q::b)).fma(float(Q::b - Q::a), D);
    }
    auto column = [&](const V3f g[3], int c) {  // column c of (g_0 g_1 g_2) J^{-1}
        return (g[0] * Ji[c]).fma(Ji[3 + c], g[1]).fma(Ji[6 + c], g[2]);
    };
    if constexpr (NQ == 5) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const V3f v = column(S, c);
            g0[c] = v.xy.x;
            g0[3 + c] = v.xy.y;
            g0[6 + c] = v.z;
        }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        V3f g[2][3];
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int j = 2 * h + r;
                g[r][k] = base[k].fma(float(4.0 * (Q::a - Q::b)), x[t10_node(k + 1, j)] - x[t10_node(0, j)]);
            }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const V3f v = column(g[0], c), w = column(g[1], c);
            rec[(h * NV + c) * 32] = make_float2(v.xy.x, w.xy.x);
            rec[(h * NV + 3 + c) * 32] = make_float2(v.xy.y, w.xy.y);
            rec[(h * NV + 6 + c) * 32] = make_float2(v.z, w.z);
        }
    }
}

// element vector of one output field from its operators at the four points
// (laid out as t10_gradients writes them): the transposed map.
// Jw = (point weight) det J J^{-1}
template <int NQ, int NV> __device__ __forceinline__ void t10_vectors(const float2 *rec, const float Jw[9], V3f F[10])
{
    using Q = T10Rule<NQ>;
    V3f T[4][3], U[3];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float2 x = rec[(h * NV + c) * 32], y = rec[(h * NV + 3 + c) * 32], z = rec[(h * NV + 6 + c) * 32];
            T[2 * h][c] = {make_float2(x.x, y.x), z.x};
            T[2 * h + 1][c] = {make_float2(x.y, y.y), z.y};
        }
    {
        V3f s[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) s[c] = (T[0][c] + T[1][c]) + (T[2][c] + T[3][c]);
#pragma unroll
        for (int k = 0; k < 3; ++k) U[k] = (s[0] * Jw[k * 3]).fma(Jw[k * 3 + 1], s[1]).fma(Jw[k * 3 + 2], s[2]);
    }
    F[0] = (U[0] + U[1]) + U[2];  // the -Delta parts: 4 b + (a - b) = 1
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        F[k + 1] = U[k] * -1.f;
        U[k] = U[k] * float(4.0 * Q::b);
    }
    bool first[10] = {false, false, false, false, true, true, true, true, true, true};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        V3f s;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const V3f y = (T[j][0] * Jw[k * 3]).fma(Jw[k * 3 + 1], T[j][1]).fma(Jw[k * 3 + 2], T[j][2]);
            const V3f Y = U[k].fma(float(4.0 * (Q::a - Q::b)), y);
            const int i = t10_node(k + 1, j);
            F[i] = first[i] ? Y : F[i] + Y;
            first[i] = false;
            s = k == 0 ? Y : s + Y;
        }
        const int i = t10_node(0, j);
        F[i] = first[i] ? s * -1.f : F[i] - s;
        first[i] = false;
    }
}

// consistent mass of a straight-sided T10 (mass_hat): y = c Mhat x, from the
// sums over corners and edges (entries in units of 1/420: corner-corner 6 or
// 1, corner-edge -4 with and -6 without the corner, edge-edge 32, 16 or 8)
__device__ __forceinline__ void t10_mass(const V3f x[10], float c, V3f y[10])
{
    const float s = c * float(1.0 / 420.0);
    const V3f sc = (x[0] + x[1]) + (x[2] + x[3]);
    const V3f se = ((x[4] + x[5]) + (x[6] + x[7])) + (x[8] + x[9]);
    const V3f bc = sc.fma(-6.f, se), be = (se * 16.f).fma(-6.f, sc);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const V3f e = (x[t10_node(i, (i + 1) & 3)] + x[t10_node(i, (i + 2) & 3)]) + x[t10_node(i, (i + 3) & 3)];
        y[i] = bc.fma(5.f, x[i]).fma(2.f, e) * s;
    }
    constexpr int opp[6] = {9, 7, 8, 5, 6, 4};  // edge opposite to edge node 4 + e
#pragma unroll
    for (int e = 0; e < 6; ++e)
        y[4 + e] = be.fma(2.f, x[t10_ea(e)] + x[t10_eb(e)]).fma(16.f, x[4 + e]).fma(-8.f, x[opp[e]]) * s;
}

}  // namespace tlfe
