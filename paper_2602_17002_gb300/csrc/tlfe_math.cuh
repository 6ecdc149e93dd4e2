// Device-side element and constitutive math of the TL-FEA hot path.
//
// Everything works in the displacement form of the kinematics: with the
// nodal unknowns x_i = X_i + u_i and U H = I (Sec. 6, H = Hp (U Hp)^{-1}),
// the deformation gradient F = sum_i x_i h_i^T (Sec. 2.1) equals I + G with
// G = sum_i u_i h_i^T. Strain-like quantities are formed from G directly so
// that FP32 keeps its relative accuracy at small strain:
//   B     = C - I = G + G^T + G^T G  (twice the Green strain)
//   J - 1 = tr G + I2(G) + det G     (expansion of det(I + G))
// Every law is evaluated through its second Piola-Kirchhoff stress S, P = F S:
// S and its derivative are symmetric (6 entries), the elastic and the viscous
// part share one product with F, and the derivative along dF needs two 3x3
// products, dP = dF S + F dS, with dS linear in dE = sym(F^T dF); F enters as
// I + G term by term, so that its unit diagonal is never rounded. With
// P = A cof(F) (first Piola-Kirchhoff form) the neo-Hookean + Kelvin-Voigt
// stress and its derivative took about 515 multiply-adds a point instead of
// about 350.
// Mooney-Rivlin (App. C, Eq. mr_first_piola; neo-Hookean is mu01 = 0):
//   S = 2 mu10 J^{-2/3} (I - I1/3 C^{-1}) + 2 mu01 J^{-4/3} (I1 I - C - 2/3 I2 C^{-1})
//       + k (J - 1) J C^{-1}
// with C^{-1} = Q / J^2, Q = cof(C) = (1 + t) I - B + cof(B), t = tr B. The
// isochoric brackets vanish at C = I; written in B they lose no digits there
// (I2, I3: invariants of B; J^2 = 1 + t + I2 + I3):
//   J^2 (I - I1/3 C^{-1}) = M = (1 + t/3) (B - cof B) - (t/3 + t^2/3 - I2 - I3) I
//   J^2 (I1 I - C - 2/3 I2(C) C^{-1}) = M2
//     = (1 + t/3 - I2/3 - I3) B - 2/3 (3 + 2t + I2) cof B
//       + ((I2 + I3)(2 + t) - t/3 - t^2/3 - 2/3 I2 (1 + t)) I
// so that S = alpha M + alpha2 M2 + beta Q with alpha = 2 mu10 J^{-8/3},
// alpha2 = 2 mu01 J^{-10/3}, beta = k (J - 1) / J. M and Q are both sums of I
// and N = B - cof(B): with s = 1 + t/3 and i = I2 + I3 - t (1 + t)/3,
//   M = s N + i I, Q = (1 + t) I - N,
//   S = (alpha s - beta) N + (alpha i + beta (1 + t)) I      (+ alpha2 M2):
// neither is formed, and dS is the derivative of this form.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace tlfe {

enum { ET_T4 = 0, ET_T10 = 1, ET_H8 = 2, ET_Q27 = 3 };
enum { MODEL_SVK = 0, MODEL_NH = 1, MODEL_MR = 2 };

template <int ET> struct Elem;
template <> struct Elem<ET_T4> { static constexpr int NPE = 4; };
template <> struct Elem<ET_T10> { static constexpr int NPE = 10; };
template <> struct Elem<ET_H8> { static constexpr int NPE = 8; };
template <> struct Elem<ET_Q27> { static constexpr int NPE = 27; };

__host__ __device__ inline int nodes_per_elem(int et)
{
    return et == ET_T4 ? 4 : (et == ET_T10 ? 10 : (et == ET_H8 ? 8 : (et == ET_Q27 ? 27 : -1)));
}

// Material record as the kernels see it (Lame constants, Kelvin-Voigt
// constants, density, Mooney-Rivlin mu01 with mu10 = mu/2 - mu01; mu01 = 0
// unless model == MODEL_MR) in the arithmetic type R.
template <typename R> struct Mat {
    int model;
    R mu, lam, mu_v, lam_v, rho, mu01;
};

// ---------------------------------------------------------------------------
// Two quadrature points of one element in one FP32x2 register pair: every
// operation below is one packed instruction for both (negated, swapped and
// broadcast operands cost nothing). A product is kept open until it is used,
// so that sums of products become packed multiply-adds, as the compiler makes
// them of the scalar types.
// ---------------------------------------------------------------------------
struct F2 {
    float2 v;
    __device__ __forceinline__ F2() {}
    __device__ __forceinline__ F2(float x) : v(make_float2(x, x)) {}
    __device__ __forceinline__ F2(float2 x) : v(x) {}
};
struct F2Prod {
    float2 a, b;
    __device__ __forceinline__ operator F2() const { return __fmul2_rn(a, b); }
};
__device__ __forceinline__ float2 neg2(float2 x) { return make_float2(-x.x, -x.y); }
__device__ __forceinline__ F2 operator-(F2 x) { return neg2(x.v); }
__device__ __forceinline__ F2Prod operator-(F2Prod p) { return {neg2(p.a), p.b}; }
__device__ __forceinline__ F2Prod operator*(F2 a, F2 b) { return {a.v, b.v}; }
__device__ __forceinline__ F2Prod operator*(F2 a, float b) { return {a.v, make_float2(b, b)}; }
__device__ __forceinline__ F2Prod operator*(float a, F2 b) { return {make_float2(a, a), b.v}; }
__device__ __forceinline__ F2 operator+(F2 a, F2 b) { return __fadd2_rn(a.v, b.v); }
__device__ __forceinline__ F2 operator-(F2 a, F2 b) { return __fadd2_rn(a.v, neg2(b.v)); }
__device__ __forceinline__ F2 operator+(F2Prod p, F2 c) { return __ffma2_rn(p.a, p.b, c.v); }
__device__ __forceinline__ F2 operator+(F2 c, F2Prod p) { return __ffma2_rn(p.a, p.b, c.v); }
__device__ __forceinline__ F2 operator+(F2Prod p, F2Prod q) { return __ffma2_rn(q.a, q.b, __fmul2_rn(p.a, p.b)); }
__device__ __forceinline__ F2 operator-(F2Prod p, F2 c) { return __ffma2_rn(p.a, p.b, neg2(c.v)); }
__device__ __forceinline__ F2 operator-(F2 c, F2Prod p) { return __ffma2_rn(neg2(p.a), p.b, c.v); }
__device__ __forceinline__ F2 operator-(F2Prod p, F2Prod q) { return __ffma2_rn(neg2(q.a), q.b, __fmul2_rn(p.a, p.b)); }
template <typename T> __device__ __forceinline__ F2 &operator+=(F2 &a, const T &b) { return a = a + b; }

// the scalar type of a value type, and per-point truth values
template <typename V> struct ValueOf {
    using S = V;
    using Mask = bool;
};
struct Mask2 {
    bool x, y;
};
template <> struct ValueOf<F2> {
    using S = float;
    using Mask = Mask2;
};
__device__ __forceinline__ bool positive(float x) { return x > 0.f; }
__device__ __forceinline__ bool positive(double x) { return x > 0.0; }
__device__ __forceinline__ Mask2 positive(F2 x) { return {x.v.x > 0.f, x.v.y > 0.f}; }
__device__ __forceinline__ bool all_of(bool m) { return m; }
__device__ __forceinline__ bool all_of(Mask2 m) { return m.x && m.y; }
__device__ __forceinline__ int count_not(bool m) { return m ? 0 : 1; }
__device__ __forceinline__ int count_not(Mask2 m) { return (m.x ? 0 : 1) + (m.y ? 0 : 1); }
template <typename R> __device__ __forceinline__ R where(bool m, R a, R b) { return m ? a : b; }
__device__ __forceinline__ F2 where(Mask2 m, F2 a, F2 b)
{
    return make_float2(m.x ? a.v.x : b.v.x, m.y ? a.v.y : b.v.y);
}
__device__ __forceinline__ float sum_of(float x) { return x; }  // over the points of the value
__device__ __forceinline__ float sum_of(F2 x) { return x.v.x + x.v.y; }
__device__ __forceinline__ void set_true(bool &m) { m = true; }
__device__ __forceinline__ void set_true(Mask2 &m) { m.x = m.y = true; }

// ---------------------------------------------------------------------------
// 3x3 helpers on row-major register arrays
// ---------------------------------------------------------------------------

// R = A B
template <typename R> __device__ __forceinline__ void mm3(const R A[9], const R B[9], R C[9])
{
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b)
            C[a * 3 + b] = A[a * 3] * B[b] + A[a * 3 + 1] * B[3 + b] + A[a * 3 + 2] * B[6 + b];
}

// FP32 products with rows 0 and 1 paired in packed FP32x2 operations (one
// instruction for two lanes of work; the same operations in the same order
// as the scalar form)
__device__ __forceinline__ void mm3(const float A[9], const float B[9], float C[9])
{
    const float2 a0 = make_float2(A[0], A[3]), a1 = make_float2(A[1], A[4]), a2 = make_float2(A[2], A[5]);
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        float2 q = __fmul2_rn(a0, make_float2(B[b], B[b]));
        q = __ffma2_rn(a1, make_float2(B[3 + b], B[3 + b]), q);
        q = __ffma2_rn(a2, make_float2(B[6 + b], B[6 + b]), q);
        C[b] = q.x;
        C[3 + b] = q.y;
        C[6 + b] = fmaf(A[8], B[6 + b], fmaf(A[7], B[3 + b], A[6] * B[b]));
    }
}

// Symmetric 3x3 matrices as 6 entries xx yy zz xy xz yz. Strain-like ones
// (B, dE of a direction) that are summed with their transpose keep the
// off-diagonal sums unhalved ("engineering" shear): entry xy of eng(A, B)
// is (A^T B)_xy + (A^T B)_yx, the diagonal is that of A^T B.
template <typename V> __device__ __forceinline__ void sym_eng(const V A[9], const V B[9], V e[6])
{
#pragma unroll
    for (int a = 0; a < 3; ++a) e[a] = A[a] * B[a] + A[3 + a] * B[3 + a] + A[6 + a] * B[6 + a];
    e[3] = A[0] * B[1] + A[3] * B[4] + A[6] * B[7] + A[1] * B[0] + A[4] * B[3] + A[7] * B[6];
    e[4] = A[0] * B[2] + A[3] * B[5] + A[6] * B[8] + A[2] * B[0] + A[5] * B[3] + A[8] * B[6];
    e[5] = A[1] * B[2] + A[4] * B[5] + A[7] * B[8] + A[2] * B[1] + A[5] * B[4] + A[8] * B[7];
}

// eng(F, D) for F = I + G from G: no rounding of F's unit diagonal
template <typename V> __device__ __forceinline__ void sym_eng_ig(const V G[9], const V D[9], V e[6])
{
#pragma unroll
    for (int a = 0; a < 3; ++a) e[a] = D[4 * a] + G[a] * D[a] + G[3 + a] * D[3 + a] + G[6 + a] * D[6 + a];
    e[3] = D[1] + D[3] + G[0] * D[1] + G[3] * D[4] + G[6] * D[7] + G[1] * D[0] + G[4] * D[3] + G[7] * D[6];
    e[4] = D[2] + D[6] + G[0] * D[2] + G[3] * D[5] + G[6] * D[8] + G[2] * D[0] + G[5] * D[3] + G[8] * D[6];
    e[5] = D[5] + D[7] + G[1] * D[2] + G[4] * D[5] + G[7] * D[8] + G[2] * D[1] + G[5] * D[4] + G[8] * D[7];
}

// S : e for a symmetric S and an engineering e (the doubled off-diagonals are in e)
template <typename V> __device__ __forceinline__ V dot6(const V S[6], const V e[6])
{
    return S[0] * e[0] + S[1] * e[1] + S[2] * e[2] + S[3] * e[3] + S[4] * e[4] + S[5] * e[5];
}

// cofactors of a symmetric matrix
template <typename V> __device__ __forceinline__ void cof6(const V B[6], V c[6])
{
    c[0] = B[1] * B[2] - B[5] * B[5];
    c[1] = B[0] * B[2] - B[4] * B[4];
    c[2] = B[0] * B[1] - B[3] * B[3];
    c[3] = B[4] * B[5] - B[3] * B[2];
    c[4] = B[3] * B[5] - B[4] * B[1];
    c[5] = B[3] * B[4] - B[5] * B[0];
}

// derivative of cof6 at C along dC = 2 sym, given e = eng(F, dF) = (dE_xx, .., 2 dE_xy, ..):
// diagonal entries halved (d/2), off-diagonal ones whole
template <typename V> __device__ __forceinline__ void dcof6(const V C[6], const V e[6], V d[6])
{
    const V t0 = e[0] + e[0], t1 = e[1] + e[1], t2 = e[2] + e[2];
    d[0] = C[1] * e[2] + C[2] * e[1] - C[5] * e[5];
    d[1] = C[0] * e[2] + C[2] * e[0] - C[4] * e[4];
    d[2] = C[0] * e[1] + C[1] * e[0] - C[3] * e[3];
    d[3] = C[4] * e[5] + C[5] * e[4] - C[2] * e[3] - C[3] * t2;
    d[4] = C[3] * e[5] + C[5] * e[3] - C[1] * e[4] - C[4] * t1;
    d[5] = C[3] * e[4] + C[4] * e[3] - C[0] * e[5] - C[5] * t0;
}

// Products with a symmetric S (6 entries): P = A S, P += A S, and P = F S for
// F = I + G, as S + G S (no rounding of F's unit diagonal)
template <typename V> __device__ __forceinline__ void full6(const V S[6], V M[9])
{
    M[0] = S[0], M[4] = S[1], M[8] = S[2];
    M[1] = M[3] = S[3];
    M[2] = M[6] = S[4];
    M[5] = M[7] = S[5];
}
template <typename V> __device__ __forceinline__ void mm6(const V A[9], const V S[6], V P[9])
{
    V M[9];
    full6(S, M);
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) P[a * 3 + b] = A[a * 3] * M[b] + A[a * 3 + 1] * M[3 + b] + A[a * 3 + 2] * M[6 + b];
}
template <typename V> __device__ __forceinline__ void mm6_acc(const V A[9], const V S[6], V P[9])
{
    V M[9];
    full6(S, M);
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b)
            P[a * 3 + b] = P[a * 3 + b] + A[a * 3] * M[b] + A[a * 3 + 1] * M[3 + b] + A[a * 3 + 2] * M[6 + b];
}
// FP32: rows 0 and 1 paired in packed FP32x2 operations (one issue slot for
// two multiply-adds; broadcast and swapped operands are free)
__device__ __forceinline__ void mm6(const float A[9], const float S[6], float P[9])
{
    const float2 a0 = make_float2(A[0], A[3]), a1 = make_float2(A[1], A[4]), a2 = make_float2(A[2], A[5]);
    float M[9];
    full6(S, M);
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        float2 q = __fmul2_rn(a0, make_float2(M[b], M[b]));
        q = __ffma2_rn(a1, make_float2(M[3 + b], M[3 + b]), q);
        q = __ffma2_rn(a2, make_float2(M[6 + b], M[6 + b]), q);
        P[b] = q.x;
        P[3 + b] = q.y;
        P[6 + b] = fmaf(A[8], M[6 + b], fmaf(A[7], M[3 + b], A[6] * M[b]));
    }
}
__device__ __forceinline__ void mm6_acc(const float A[9], const float S[6], float P[9])
{
    const float2 a0 = make_float2(A[0], A[3]), a1 = make_float2(A[1], A[4]), a2 = make_float2(A[2], A[5]);
    float M[9];
    full6(S, M);
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        float2 q = __ffma2_rn(a0, make_float2(M[b], M[b]), make_float2(P[b], P[3 + b]));
        q = __ffma2_rn(a1, make_float2(M[3 + b], M[3 + b]), q);
        q = __ffma2_rn(a2, make_float2(M[6 + b], M[6 + b]), q);
        P[b] = q.x;
        P[3 + b] = q.y;
        P[6 + b] = fmaf(A[8], M[6 + b], fmaf(A[7], M[3 + b], fmaf(A[6], M[b], P[6 + b])));
    }
}
template <typename V> __device__ __forceinline__ void mm6_ig(const V G[9], const V S[6], V P[9])
{
    full6(S, P);
    mm6_acc(G, S, P);
}

// ---------------------------------------------------------------------------
// Constitutive state at one quadrature point
// ---------------------------------------------------------------------------

// Per-point quantities kept between the stress and its derivatives (V: one
// point, or two of one element in F2).
template <typename V> struct QP {
    V G[9];    // sum u_i h_i^T; F = I + G
    V Fd[9];   // sum udot_i h_i^T (valid when visc)
    V S[6];    // elastic second Piola-Kirchhoff stress
    V Sv[6];   // viscous second Piola-Kirchhoff stress (valid when visc)
    V B[6];    // C - I
    V N[6];    // MR / NH: B - cof(B)
    // MR / NH: alpha, alpha s - beta, and the scalars of the header comment
    V al, c1, s, i, t1;   // t1 = 1 + t
    V rD, rJ, r1;         // J^{-2}, 1/J, J^{-1/3}
    V Jm1r;               // (J - 1) / J
    typename ValueOf<V>::Mask ok;
};

__device__ __forceinline__ float rcbrt_(float x) { return rcbrtf(x); }
__device__ __forceinline__ double rcbrt_(double x) { return rcbrt(x); }
__device__ __forceinline__ F2 rcbrt_(F2 x) { return make_float2(rcbrtf(x.v.x), rcbrtf(x.v.y)); }

// factors of M2 = x1 B - x2 cof(B) + x0 I (see the header comment)
template <typename R, typename V>
__device__ __forceinline__ void mr_factors(V t, V I2, V I3, V &x0, V &x1, V &x2)
{
    const R third = R(1.0 / 3.0);
    const V t1 = t + V(R(1));
    x1 = third * (t - I2) - I3 + V(R(1));
    x2 = (R(2) * third) * (R(2) * t + I2 + V(R(3)));
    x0 = (I2 + I3) * (t + V(R(2))) - V(third * t) * t1 - V((R(2) * third) * I2) * t1;
}

// Elastic and viscous stress state. visc: whether Fd is meaningful and the
// material damped. Clears q.ok (and leaves no elastic part) where the
// neo-Hookean law meets J <= 0 or a J that is not a number.
template <typename R, typename V> __device__ __forceinline__ void stress_state(const Mat<R> &m, QP<V> &q, bool visc)
{
    const V *G = q.G;
    set_true(q.ok);
    if (visc) {
        // Edot = sym(Fd^T F); S^v = 2 mu_v Edot + lam_v tr(Edot) I  (Sec. 3.2.3)
        V e[6];
        sym_eng_ig<V>(G, q.Fd, e);
        const V i = m.lam_v * (e[0] + e[1] + e[2]);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            q.Sv[k] = (R(2) * m.mu_v) * e[k] + i;
            q.Sv[3 + k] = m.mu_v * e[3 + k];
        }
    }
    // B = G + G^T + G^T G
#pragma unroll
    for (int a = 0; a < 3; ++a) q.B[a] = R(2) * G[4 * a] + G[a] * G[a] + G[3 + a] * G[3 + a] + G[6 + a] * G[6 + a];
    q.B[3] = G[1] + G[3] + G[0] * G[1] + G[3] * G[4] + G[6] * G[7];
    q.B[4] = G[2] + G[6] + G[0] * G[2] + G[3] * G[5] + G[6] * G[8];
    q.B[5] = G[5] + G[7] + G[1] * G[2] + G[4] * G[5] + G[7] * G[8];
    const V t = q.B[0] + q.B[1] + q.B[2];
    if (m.model == MODEL_SVK) {
        // S = lam tr(E) I + 2 mu E  (App. C SVK)
        const V i = (R(0.5) * m.lam) * t;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            q.S[k] = m.mu * q.B[k] + i;
            q.S[3 + k] = m.mu * q.B[3 + k];
        }
        return;
    }
    // neo-Hookean: mu10 = mu/2, k = lam + 2 mu / 3
    const R third = R(1.0 / 3.0);
    const V c0 = G[4] * G[8] - G[5] * G[7], c1 = G[5] * G[6] - G[3] * G[8], c2 = G[3] * G[7] - G[4] * G[6];
    const V dG = G[0] * c0 + G[1] * c1 + G[2] * c2;
    const V I2G = c0 + (G[0] * G[4] - G[1] * G[3]) + (G[0] * G[8] - G[2] * G[6]);
    const V Jm1 = (G[0] + G[4] + G[8]) + I2G + dG;
    q.ok = positive(Jm1 + V(R(1)));
    const V jm = where(q.ok, Jm1, V(R(0))), J = jm + V(R(1));
    // J^{-1/3} and 1/J to the last bit of 1 + (J - 1): alpha holds the eighth
    // power of J^{-1/3}, whose rounding (and that of J) would otherwise be most
    // of the FP32 error of the operator product. err = 1 - r^3 (J + jl).
    const V r0 = rcbrt_(J), rJ0 = V(r0 * r0) * r0;
    const V jl = jm - (J - V(R(1)));
    const V err = V(V(R(1)) - rJ0 * J) - rJ0 * jl;
    const V r = r0 + V(third * r0) * err, r2 = r * r;
    q.r1 = r;
    q.rJ = rJ0 + rJ0 * err;
    q.rD = q.rJ * q.rJ;
    q.Jm1r = jm * q.rJ;
    q.al = (m.mu - R(2) * m.mu01) * V(q.rD * r2);
    const V be = (m.lam + R(2) * third * m.mu) * q.Jm1r;
    V cB[6];
    cof6<V>(q.B, cB);
    const V I2 = cB[0] + cB[1] + cB[2];
    const V I3 = q.B[0] * cB[0] + q.B[3] * cB[3] + q.B[4] * cB[4];
    q.t1 = t + V(R(1));
    q.s = third * t + V(R(1));
    q.i = (I2 + I3) - V(third * t) * q.t1;
    q.c1 = q.al * q.s - be;
    const V iso = q.al * q.i + be * q.t1;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        q.N[k] = q.B[k] - cB[k];
        q.S[k] = k < 3 ? V(q.c1 * q.N[k] + iso) : V(q.c1 * q.N[k]);
    }
    if (m.model == MODEL_MR) {
        const V a2 = (R(2) * m.mu01) * V(V(q.rD * q.rJ) * r);  // 2 mu01 J^{-10/3}
        V x0, x1, x2;
        mr_factors<R, V>(t, I2, I3, x0, x1, x2);
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const V M2 = x1 * q.B[k] - x2 * cB[k] + (k < 3 ? x0 : V(R(0)));
            q.S[k] += a2 * M2;
        }
    }
    if (!all_of(q.ok)) {
        const V z = V(R(0));
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            q.S[k] = where(q.ok, q.S[k], z);
            q.N[k] = where(q.ok, q.N[k], z);
            q.B[k] = where(q.ok, q.B[k], z);
        }
        q.al = where(q.ok, q.al, z);
        q.c1 = where(q.ok, q.c1, z);
        q.s = where(q.ok, q.s, z);
        q.i = where(q.ok, q.i, z);
        q.t1 = where(q.ok, q.t1, z);
        q.rD = where(q.ok, q.rD, z);
        q.Jm1r = where(q.ok, q.Jm1r, z);
    }
}

// first Piola-Kirchhoff stress of the state: F (S + S^v)
template <typename V> __device__ __forceinline__ void first_piola(const QP<V> &q, bool visc, V P[9])
{
    using R = typename ValueOf<V>::S;
    V St[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) St[k] = visc ? q.S[k] + q.Sv[k] : q.S[k];
    mm6_ig(q.G, St, P);
    if (!all_of(q.ok) && !visc)  // an F that is not a number leaves no trace
#pragma unroll
        for (int k = 0; k < 9; ++k) P[k] = where(q.ok, P[k], V(R(0)));
}

template <typename R, typename V>
__device__ __forceinline__ void stress(const Mat<R> &m, QP<V> &q, bool visc, V P[9])
{
    stress_state<R, V>(m, q, visc);
    first_piola<V>(q, visc, P);
}

// c times the elastic derivative dS along e = eng(F, dF)
template <typename R, typename V>
__device__ __forceinline__ void dS_elastic(const Mat<R> &m, const QP<V> &q, const V e[6], R c, V dS[6])
{
    const V trE = e[0] + e[1] + e[2];
    if (m.model == MODEL_SVK) {
        const R a = c * m.mu;
        const V i = (c * m.lam) * trE;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            dS[k] = (R(2) * a) * e[k] + i;
            dS[3 + k] = a * e[3 + k];
        }
        return;
    }
    // derivative of S = c1 N + c0 I, c1 = alpha s - beta, c0 = alpha i + beta (1 + t), along dB = 2 dE
    // (j = dJ / J = Q : dE / J^2, dt = 2 tr dE; dalpha = -8/3 alpha j, dbeta = k j / J):
    //   dN = dB - dcof(B), ds = dt / 3, di = dt (t - 1) / 3 - 2 N : dE
    // No term is larger than the derivative itself (formed from M, Q and dcof(C), whose identity parts
    // cancel, the FP32 error is 1.4 times as large).
    const R third = R(1.0 / 3.0);
    const R kb = m.lam + R(2) * third * m.mu;
    const V NE = dot6<V>(q.N, e);
    const V dt = trE + trE;
    const V j = (q.t1 * trE - NE) * q.rD;
    const V da = V((R(-8) * third) * q.al) * j;   // dalpha
    const V db = V(kb * j) * q.rJ;                // dbeta
    const V adt = V(third * q.al) * dt;           // alpha dt / 3
    const V be = q.al * q.s - q.c1;
    const V dc1 = c * V(da * q.s + adt - db);
    const V dc0 = c * V(da * q.i + adt * (q.t1 - V(R(2))) - V(q.al * (NE + NE)) + db * q.t1 + be * dt);
    const V cc = c * q.c1, cc2 = cc + cc;
    V d[6];
    dcof6<V>(q.B, e, d);
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const V u = e[k] - d[k];
        dS[k] = k < 3 ? V(cc2 * u + V(dc1 * q.N[k] + dc0)) : V(cc * u + dc1 * q.N[k]);
    }
    if (m.model == MODEL_MR) {
        // S2 = a2 M2, a2 = 2 mu01 J^{-10/3}: dS2 = -(10/3) j S2 + a2 dM2
        const V t = q.B[0] + q.B[1] + q.B[2];
        V cB[6];
        cof6<V>(q.B, cB);
        const V I2 = cB[0] + cB[1] + cB[2];
        const V I3 = q.B[0] * cB[0] + q.B[3] * cB[3] + q.B[4] * cB[4];
        V x0, x1, x2;
        mr_factors<R, V>(t, I2, I3, x0, x1, x2);
        const V a2 = (R(2) * m.mu01) * V(V(q.rD * q.rJ) * q.r1);  // 2 mu01 J^{-10/3}
        // invariants of B along dB = 2 dE
        V dcB[6];
        dcof6<V>(q.B, e, dcB);  // diagonal halved
        const V dI2 = R(2) * (dcB[0] + dcB[1] + dcB[2]);
        const V dI3 = R(2) * dot6<V>(cB, e);
        const V dx1 = third * (dt - dI2) - dI3;
        const V dx2 = (R(2) * third) * (R(2) * dt + dI2);
        const V dx0 = (dI2 + dI3) * (t + V(R(2))) + (I2 + I3) * dt - V(third * dt) * (R(2) * t + V(R(1))) -
                      V((R(2) * third) * dI2) * (t + V(R(1))) - V((R(2) * third) * I2) * dt;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const V M2 = x1 * q.B[k] - x2 * cB[k] + (k < 3 ? x0 : V(R(0)));
            const V dB = k < 3 ? e[k] + e[k] : e[k];
            const V dc = k < 3 ? dcB[k] + dcB[k] : dcB[k];
            const V dM2 = dx1 * q.B[k] + x1 * dB - dx2 * cB[k] - x2 * dc + (k < 3 ? dx0 : V(R(0)));
            dS[k] += V(c * a2) * (dM2 - V((R(10) * third) * j) * M2);
        }
    }
}

// Directional derivative of P along (dF, dFd):
//   dP = D_F P^e[dF] + (position-side viscous terms, if visc and not sym_only)
//        + D_Fd P^v[dFd]
// with dF = dFd the given direction; cK scales everything depending on dF, cC
// everything depending on dFd. sym_only drops the viscous stiffness K^v (the
// non-symmetric part).
template <typename R, typename V>
__device__ __forceinline__ void dstress(const Mat<R> &m, const QP<V> &q, bool visc, const V dF[9],
                                        R cK, R cC, bool sym_only, V dP[9])
{
    V e[6], T[6], Sk[6];
    sym_eng_ig<V>(q.G, dF, e);
#pragma unroll
    for (int k = 0; k < 6; ++k) T[k] = Sk[k] = V(R(0));
    if (cK != R(0)) {
        dS_elastic<R, V>(m, q, e, cK, T);
        const bool vk = visc && !sym_only;
        if (vk) {  // position-side viscous derivative: dEdot = sym(Fd^T dF)
            V ev[6];
            sym_eng<V>(q.Fd, dF, ev);
            const R a = cK * m.mu_v;
            const V i = (cK * m.lam_v) * (ev[0] + ev[1] + ev[2]);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                T[k] += (R(2) * a) * ev[k] + i;
                T[3 + k] += a * ev[3 + k];
            }
        }
#pragma unroll
        for (int k = 0; k < 6; ++k) Sk[k] = cK * (vk ? q.S[k] + q.Sv[k] : q.S[k]);
    }
    if (cC != R(0)) {  // velocity direction: dEdot = sym(F^T dFd)
        const R a = cC * m.mu_v;
        const V i = (cC * m.lam_v) * (e[0] + e[1] + e[2]);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            T[k] += (R(2) * a) * e[k] + i;
            T[3 + k] += a * e[3 + k];
        }
    }
    mm6_ig(q.G, T, dP);
    if (cK != R(0)) mm6_acc(dF, Sk, dP);
    if (!all_of(q.ok) && !(visc && !sym_only) && !(cC != R(0) && (m.mu_v != R(0) || m.lam_v != R(0))))
#pragma unroll
        for (int k = 0; k < 9; ++k) dP[k] = where(q.ok, dP[k], V(R(0)));
}

// Adjoint of the stress map at one point against a cotangent Gh (=sum r_i h_i^T):
//   gF  = (dP/dF)^T [Gh]  (elastic part self-adjoint; viscous part explicit)
//   gFd = (dP/dFd)^T [Gh]
//   gmu = dP/dmu : Gh, glam = dP/dlam : Gh, contracted as dS/dmu : sym(F^T Gh)
template <typename R, typename V>
__device__ __forceinline__ void astress(const Mat<R> &m, const QP<V> &q, bool visc, const V Gh[9],
                                        V gF[9], V gFd[9], V &gmu, V &glam)
{
    V e[6], T[6], St[6];
    sym_eng_ig<V>(q.G, Gh, e);
    dS_elastic<R, V>(m, q, e, R(1), T);
#pragma unroll
    for (int k = 0; k < 6; ++k) St[k] = visc ? q.S[k] + q.Sv[k] : q.S[k];
    mm6_ig(q.G, T, gF);
    mm6_acc(Gh, St, gF);
    const V trE = e[0] + e[1] + e[2];
    if (visc) {
        // L = (F S^v) : Gh, Ebar = 2 mu_v sym(F^T Gh) + lam_v tr I:
        // dL/dF = Gh S^v + Fd Ebar, dL/dFd = F Ebar
        V Eb[6];
        const V i = m.lam_v * trE;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            Eb[k] = (R(2) * m.mu_v) * e[k] + i;
            Eb[3 + k] = m.mu_v * e[3 + k];
        }
        mm6_acc(q.Fd, Eb, gF);
        mm6_ig(q.G, Eb, gFd);
    } else {
#pragma unroll
        for (int k = 0; k < 9; ++k) gFd[k] = V(R(0));
        if (!all_of(q.ok))
#pragma unroll
            for (int k = 0; k < 9; ++k) gF[k] = where(q.ok, gF[k], V(R(0)));
    }
    if (m.model == MODEL_SVK) {
        // dS/dlam = tr(E) I, dS/dmu = 2 E = B
        gmu = dot6<V>(q.B, e);
        glam = V(R(0.5) * (q.B[0] + q.B[1] + q.B[2])) * trE;
    } else {
        // dS/dmu = J^{-8/3} M + 2/3 (J - 1)/J Q (mu01 held fixed), dS/dlam = (J - 1)/J Q
        const V NE = dot6<V>(q.N, e);
        const V gq = q.Jm1r * (q.t1 * trE - NE);
        const V g = V(V(q.rD * q.r1) * q.r1) * (q.s * NE + q.i * trE) + R(2.0 / 3.0) * gq;
        gmu = where(q.ok, g, V(R(0)));
        glam = where(q.ok, gq, V(R(0)));
    }
}

}  // namespace tlfe
