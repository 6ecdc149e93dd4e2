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
// products, dP = dF S + F dS, with dS linear in dE = sym(F^T dF). With
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
//   S = (alpha s - beta) N + (alpha i + beta (1 + t)) I      (+ alpha2 M2),
// and the same holds for the parts of dS that M and Q enter: neither is formed.
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
// 3x3 helpers on row-major register arrays
// ---------------------------------------------------------------------------

template <typename R> __device__ __forceinline__ R tr3(const R A[9]) { return A[0] + A[4] + A[8]; }

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
template <typename R> __device__ __forceinline__ void sym_eng(const R A[9], const R B[9], R e[6])
{
#pragma unroll
    for (int a = 0; a < 3; ++a) e[a] = A[a] * B[a] + A[3 + a] * B[3 + a] + A[6 + a] * B[6 + a];
    e[3] = A[0] * B[1] + A[3] * B[4] + A[6] * B[7] + A[1] * B[0] + A[4] * B[3] + A[7] * B[6];
    e[4] = A[0] * B[2] + A[3] * B[5] + A[6] * B[8] + A[2] * B[0] + A[5] * B[3] + A[8] * B[6];
    e[5] = A[1] * B[2] + A[4] * B[5] + A[7] * B[8] + A[2] * B[1] + A[5] * B[4] + A[8] * B[7];
}

// S : e for a symmetric S and an engineering e (the doubled off-diagonals are in e)
template <typename R> __device__ __forceinline__ R dot6(const R S[6], const R e[6])
{
    return S[0] * e[0] + S[1] * e[1] + S[2] * e[2] + S[3] * e[3] + S[4] * e[4] + S[5] * e[5];
}

// cofactors of a symmetric matrix
template <typename R> __device__ __forceinline__ void cof6(const R B[6], R c[6])
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
template <typename R> __device__ __forceinline__ void dcof6(const R C[6], const R e[6], R d[6])
{
    const R t0 = e[0] + e[0], t1 = e[1] + e[1], t2 = e[2] + e[2];
    d[0] = C[1] * e[2] + C[2] * e[1] - C[5] * e[5];
    d[1] = C[0] * e[2] + C[2] * e[0] - C[4] * e[4];
    d[2] = C[0] * e[1] + C[1] * e[0] - C[3] * e[3];
    d[3] = C[4] * e[5] + C[5] * e[4] - C[2] * e[3] - C[3] * t2;
    d[4] = C[3] * e[5] + C[5] * e[3] - C[1] * e[4] - C[4] * t1;
    d[5] = C[3] * e[4] + C[4] * e[3] - C[0] * e[5] - C[5] * t0;
}

// P = A S with S symmetric (6 entries)
template <typename R> __device__ __forceinline__ void mm6(const R A[9], const R S[6], R P[9])
{
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        P[a * 3 + 0] = A[a * 3] * S[0] + A[a * 3 + 1] * S[3] + A[a * 3 + 2] * S[4];
        P[a * 3 + 1] = A[a * 3] * S[3] + A[a * 3 + 1] * S[1] + A[a * 3 + 2] * S[5];
        P[a * 3 + 2] = A[a * 3] * S[4] + A[a * 3 + 1] * S[5] + A[a * 3 + 2] * S[2];
    }
}
template <typename R> __device__ __forceinline__ void mm6_acc(const R A[9], const R S[6], R P[9])
{
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        P[a * 3 + 0] += A[a * 3] * S[0] + A[a * 3 + 1] * S[3] + A[a * 3 + 2] * S[4];
        P[a * 3 + 1] += A[a * 3] * S[3] + A[a * 3 + 1] * S[1] + A[a * 3 + 2] * S[5];
        P[a * 3 + 2] += A[a * 3] * S[4] + A[a * 3 + 1] * S[5] + A[a * 3 + 2] * S[2];
    }
}
// FP32: rows 0 and 1 paired in packed FP32x2 operations (one issue slot for
// two multiply-adds; broadcast and swapped operands are free)
__device__ __forceinline__ void mm6(const float A[9], const float S[6], float P[9])
{
    const float2 a0 = make_float2(A[0], A[3]), a1 = make_float2(A[1], A[4]), a2 = make_float2(A[2], A[5]);
    const float s[9] = {S[0], S[3], S[4], S[3], S[1], S[5], S[4], S[5], S[2]};
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        float2 q = __fmul2_rn(a0, make_float2(s[b], s[b]));
        q = __ffma2_rn(a1, make_float2(s[3 + b], s[3 + b]), q);
        q = __ffma2_rn(a2, make_float2(s[6 + b], s[6 + b]), q);
        P[b] = q.x;
        P[3 + b] = q.y;
        P[6 + b] = fmaf(A[8], s[6 + b], fmaf(A[7], s[3 + b], A[6] * s[b]));
    }
}
__device__ __forceinline__ void mm6_acc(const float A[9], const float S[6], float P[9])
{
    const float2 a0 = make_float2(A[0], A[3]), a1 = make_float2(A[1], A[4]), a2 = make_float2(A[2], A[5]);
    const float s[9] = {S[0], S[3], S[4], S[3], S[1], S[5], S[4], S[5], S[2]};
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        float2 q = __ffma2_rn(a0, make_float2(s[b], s[b]), make_float2(P[b], P[3 + b]));
        q = __ffma2_rn(a1, make_float2(s[3 + b], s[3 + b]), q);
        q = __ffma2_rn(a2, make_float2(s[6 + b], s[6 + b]), q);
        P[b] = q.x;
        P[3 + b] = q.y;
        P[6 + b] = fmaf(A[8], s[6 + b], fmaf(A[7], s[3 + b], fmaf(A[6], s[b], P[6 + b])));
    }
}

// ---------------------------------------------------------------------------
// Constitutive state at one quadrature point
// ---------------------------------------------------------------------------

// Per-point quantities kept between the stress and its derivatives.
template <typename R> struct QP {
    R F[9];    // I + G
    R G[9];    // sum u_i h_i^T
    R Fd[9];   // sum udot_i h_i^T (valid when visc)
    R S[6];    // elastic second Piola-Kirchhoff stress
    R Sv[6];   // viscous second Piola-Kirchhoff stress (valid when visc)
    R B[6];    // C - I
    R N[6];    // MR / NH: B - cof(B)
    // MR / NH: alpha, alpha s - beta, and the scalars of the header comment
    R al, c1, s, i, t1;   // t1 = 1 + t
    R rD, rJ, r1;         // J^{-2}, 1/J, J^{-1/3}
    R Jm1r;               // (J - 1) / J
    bool ok;
};

template <typename R> __device__ __forceinline__ R rcbrt_(R x);
template <> __device__ __forceinline__ float rcbrt_<float>(float x) { return rcbrtf(x); }
template <> __device__ __forceinline__ double rcbrt_<double>(double x) { return rcbrt(x); }

// Elastic and viscous stress state. visc: whether Fd is meaningful and the
// material damped. Sets q.ok = false (and no elastic part) when the
// neo-Hookean law meets J <= 0 or a J that is not a number.
template <typename R> __device__ __forceinline__ void stress_state(const Mat<R> &m, QP<R> &q, bool visc)
{
    const R *G = q.G;
#pragma unroll
    for (int k = 0; k < 9; ++k) q.F[k] = G[k] + ((k % 4 == 0) ? R(1) : R(0));
    q.ok = true;
    if (visc) {
        // Edot = sym(Fd^T F); S^v = 2 mu_v Edot + lam_v tr(Edot) I  (Sec. 3.2.3)
        R e[6];
        sym_eng(q.Fd, q.F, e);
        const R i = m.lam_v * (e[0] + e[1] + e[2]);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            q.Sv[k] = R(2) * m.mu_v * e[k] + i;
            q.Sv[3 + k] = m.mu_v * e[3 + k];
        }
    }
    // B = G + G^T + G^T G
#pragma unroll
    for (int a = 0; a < 3; ++a) q.B[a] = R(2) * G[4 * a] + G[a] * G[a] + G[3 + a] * G[3 + a] + G[6 + a] * G[6 + a];
    q.B[3] = G[1] + G[3] + G[0] * G[1] + G[3] * G[4] + G[6] * G[7];
    q.B[4] = G[2] + G[6] + G[0] * G[2] + G[3] * G[5] + G[6] * G[8];
    q.B[5] = G[5] + G[7] + G[1] * G[2] + G[4] * G[5] + G[7] * G[8];
    const R t = q.B[0] + q.B[1] + q.B[2];
    if (m.model == MODEL_SVK) {
        // S = lam tr(E) I + 2 mu E  (App. C SVK)
        const R i = R(0.5) * m.lam * t;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            q.S[k] = m.mu * q.B[k] + i;
            q.S[3 + k] = m.mu * q.B[3 + k];
        }
        return;
    }
    // neo-Hookean: mu10 = mu/2, k = lam + 2 mu / 3
    const R third = R(1.0 / 3.0);
    const R c0 = G[4] * G[8] - G[5] * G[7], c1 = G[5] * G[6] - G[3] * G[8], c2 = G[3] * G[7] - G[4] * G[6];
    const R dG = G[0] * c0 + G[1] * c1 + G[2] * c2;
    const R I2G = c0 + (G[0] * G[4] - G[1] * G[3]) + (G[0] * G[8] - G[2] * G[6]);
    const R Jm1 = tr3(G) + I2G + dG;
    const R J = R(1) + Jm1;
    if (!(J > R(0))) {
        q.ok = false;
#pragma unroll
        for (int k = 0; k < 6; ++k) q.S[k] = q.N[k] = q.B[k] = R(0);
        q.al = q.c1 = q.s = q.i = q.t1 = q.rD = q.rJ = q.r1 = q.Jm1r = R(0);
        return;
    }
    const R r = rcbrt_<R>(J), r2 = r * r;
    q.r1 = r;
    q.rJ = r2 * r;
    q.rD = q.rJ * q.rJ;
    q.Jm1r = Jm1 * q.rJ;
    q.al = (m.mu - R(2) * m.mu01) * (q.rD * r2);
    const R be = (m.lam + R(2) * third * m.mu) * q.Jm1r;
    R cB[6];
    cof6(q.B, cB);
    const R I2 = cB[0] + cB[1] + cB[2];
    const R I3 = q.B[0] * cB[0] + q.B[3] * cB[3] + q.B[4] * cB[4];
    q.t1 = R(1) + t;
    q.s = R(1) + third * t;
    q.i = (I2 + I3) - third * t * q.t1;
    q.c1 = q.al * q.s - be;
    const R iso = q.al * q.i + be * q.t1;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        q.N[k] = q.B[k] - cB[k];
        q.S[k] = k < 3 ? q.c1 * q.N[k] + iso : q.c1 * q.N[k];
    }
    if (m.model == MODEL_MR) {
        const R a2 = R(2) * m.mu01 * q.rD * q.rJ * r;  // 2 mu01 J^{-10/3}
        const R x1 = R(1) + third * (t - I2) - I3;
        const R x2 = R(2) * third * (R(3) + R(2) * t + I2);
        const R x0 = (I2 + I3) * (R(2) + t) - third * t * q.t1 - R(2) * third * I2 * q.t1;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const R M2 = x1 * q.B[k] - x2 * cB[k] + (k < 3 ? x0 : R(0));
            q.S[k] += a2 * M2;
        }
    }
}

// first Piola-Kirchhoff stress of the state: F (S + S^v)
template <typename R> __device__ __forceinline__ void first_piola(const QP<R> &q, bool visc, R P[9])
{
    R St[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) St[k] = visc ? q.S[k] + q.Sv[k] : q.S[k];
    mm6(q.F, St, P);
    if (!q.ok && !visc)  // an F that is not a number leaves no trace
#pragma unroll
        for (int k = 0; k < 9; ++k) P[k] = R(0);
}

template <typename R>
__device__ __forceinline__ void stress(const Mat<R> &m, QP<R> &q, bool visc, R P[9])
{
    stress_state<R>(m, q, visc);
    first_piola<R>(q, visc, P);
}

// c times the elastic derivative dS along e = eng(F, dF)
template <typename R>
__device__ __forceinline__ void dS_elastic(const Mat<R> &m, const QP<R> &q, const R e[6], R c, R dS[6])
{
    const R trE = e[0] + e[1] + e[2];
    if (m.model == MODEL_SVK) {
        const R i = c * m.lam * trE, a = c * m.mu;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            dS[k] = R(2) * a * e[k] + i;
            dS[3 + k] = a * e[3 + k];
        }
        return;
    }
    // S_iso = alpha M = mu J^{-2/3} (I - I1/3 C^{-1}), C^{-1} = Q / J^2, j = dJ / J = C^{-1} : dE:
    //   dS_iso = -(2/3) j S_iso - mu J^{-2/3}/3 (2 tr dE C^{-1} + I1 dC^{-1})
    //   d(k (J - 1) J C^{-1}) = k (2J - 1) J j C^{-1} + k (J - 1) J dC^{-1}
    //   dC^{-1} = (dQ - 2 j Q) / J^2
    const R third = R(1.0 / 3.0);
    const R kb = m.lam + R(2) * third * m.mu;
    const R as = q.al * q.s;  // alpha I1 / 3; beta = as - c1
    const R QE = q.t1 * trE - dot6(q.N, e);
    const R j = QE * q.rD;
    const R a23 = c * R(2) * third * q.al;
    const R xM = -a23 * j;
    const R xQ = c * j * (kb + as + q.c1) - a23 * trE;
    const R xd = -c * q.c1;
    const R y1 = xM * q.s - xQ, y0 = xM * q.i + xQ * q.t1;
    R C[6], dQ[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) C[k] = k < 3 ? R(1) + q.B[k] : q.B[k];
    dcof6(C, e, dQ);
#pragma unroll
    for (int k = 0; k < 6; ++k) dS[k] = k < 3 ? y1 * q.N[k] + (R(2) * xd * dQ[k] + y0) : y1 * q.N[k] + xd * dQ[k];
    if (m.model == MODEL_MR) {
        // S2 = a2 M2, a2 = 2 mu01 J^{-10/3}: dS2 = -(10/3) j S2 + a2 dM2
        const R t = q.B[0] + q.B[1] + q.B[2];
        R cB[6];
        cof6(q.B, cB);
        const R I2 = cB[0] + cB[1] + cB[2];
        const R I3 = q.B[0] * cB[0] + q.B[3] * cB[3] + q.B[4] * cB[4];
        const R x1 = R(1) + third * (t - I2) - I3;
        const R x2 = R(2) * third * (R(3) + R(2) * t + I2);
        const R x0 = (I2 + I3) * (R(2) + t) - third * t * (R(1) + t) - R(2) * third * I2 * (R(1) + t);
        const R a2 = R(2) * m.mu01 * q.rD * q.rJ * q.r1;  // 2 mu01 J^{-10/3}
        // invariants of B along dB = 2 dE
        R dcB[6];
        dcof6(q.B, e, dcB);  // diagonal halved
        const R dt = R(2) * trE;
        const R dI2 = R(2) * (dcB[0] + dcB[1] + dcB[2]);
        const R dI3 = R(2) * (cB[0] * e[0] + cB[1] * e[1] + cB[2] * e[2] + cB[3] * e[3] + cB[4] * e[4] + cB[5] * e[5]);
        const R dx1 = third * (dt - dI2) - dI3;
        const R dx2 = R(2) * third * (R(2) * dt + dI2);
        const R dx0 = (dI2 + dI3) * (R(2) + t) + (I2 + I3) * dt - third * dt * (R(1) + R(2) * t) -
                      R(2) * third * (dI2 * (R(1) + t) + I2 * dt);
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const R M2 = x1 * q.B[k] - x2 * cB[k] + (k < 3 ? x0 : R(0));
            const R dB = k < 3 ? R(2) * e[k] : e[k];
            const R dc = k < 3 ? R(2) * dcB[k] : dcB[k];
            const R dM2 = dx1 * q.B[k] + x1 * dB - dx2 * cB[k] - x2 * dc + (k < 3 ? dx0 : R(0));
            dS[k] += c * a2 * (dM2 - R(10) * third * j * M2);
        }
    }
}

// Directional derivative of P along (dF, dFd):
//   dP = D_F P^e[dF] + (position-side viscous terms, if visc and not sym_only)
//        + D_Fd P^v[dFd]
// with dF = dFd the given direction; cK scales everything depending on dF, cC
// everything depending on dFd. sym_only drops the viscous stiffness K^v (the
// non-symmetric part).
template <typename R>
__device__ __forceinline__ void dstress(const Mat<R> &m, const QP<R> &q, bool visc, const R dF[9],
                                        R cK, R cC, bool sym_only, R dP[9])
{
    R e[6], T[6];
    sym_eng(q.F, dF, e);
    if (cK != R(0)) {
        R Sk[6];
        dS_elastic<R>(m, q, e, cK, T);
        const bool vk = visc && !sym_only;
        if (vk) {  // position-side viscous derivative: dEdot = sym(Fd^T dF)
            R ev[6];
            sym_eng(q.Fd, dF, ev);
            const R a = cK * m.mu_v, i = cK * m.lam_v * (ev[0] + ev[1] + ev[2]);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                T[k] += R(2) * a * ev[k] + i;
                T[3 + k] += a * ev[3 + k];
            }
        }
#pragma unroll
        for (int k = 0; k < 6; ++k) Sk[k] = cK * (vk ? q.S[k] + q.Sv[k] : q.S[k]);
        mm6(dF, Sk, dP);
    } else {
#pragma unroll
        for (int k = 0; k < 6; ++k) T[k] = R(0);
#pragma unroll
        for (int k = 0; k < 9; ++k) dP[k] = R(0);
    }
    if (cC != R(0)) {  // velocity direction: dEdot = sym(F^T dFd)
        const R a = cC * m.mu_v, i = cC * m.lam_v * (e[0] + e[1] + e[2]);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            T[k] += R(2) * a * e[k] + i;
            T[3 + k] += a * e[3 + k];
        }
    }
    mm6_acc(q.F, T, dP);
    if (!q.ok && !(visc && !sym_only) && !(cC != R(0) && (m.mu_v != R(0) || m.lam_v != R(0))))
#pragma unroll
        for (int k = 0; k < 9; ++k) dP[k] = R(0);
}

// Adjoint of the stress map at one point against a cotangent Gh (=sum r_i h_i^T):
//   gF  = (dP/dF)^T [Gh]  (elastic part self-adjoint; viscous part explicit)
//   gFd = (dP/dFd)^T [Gh]
//   gmu = dP/dmu : Gh, glam = dP/dlam : Gh, contracted as dS/dmu : sym(F^T Gh)
template <typename R>
__device__ __forceinline__ void astress(const Mat<R> &m, const QP<R> &q, bool visc, const R Gh[9],
                                        R gF[9], R gFd[9], R &gmu, R &glam)
{
    R e[6], T[6], St[6];
    sym_eng(q.F, Gh, e);
    dS_elastic<R>(m, q, e, R(1), T);
#pragma unroll
    for (int k = 0; k < 6; ++k) St[k] = visc ? q.S[k] + q.Sv[k] : q.S[k];
    mm6(Gh, St, gF);
    mm6_acc(q.F, T, gF);
    const R trE = e[0] + e[1] + e[2];
    if (visc) {
        // L = (F S^v) : Gh, Ebar = 2 mu_v sym(F^T Gh) + lam_v tr I:
        // dL/dF = Gh S^v + Fd Ebar, dL/dFd = F Ebar
        R Eb[6];
        const R i = m.lam_v * trE;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            Eb[k] = R(2) * m.mu_v * e[k] + i;
            Eb[3 + k] = m.mu_v * e[3 + k];
        }
        mm6_acc(q.Fd, Eb, gF);
        mm6(q.F, Eb, gFd);
    } else {
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            gFd[k] = R(0);
            if (!q.ok) gF[k] = R(0);
        }
    }
    if (m.model == MODEL_SVK) {
        // dS/dlam = tr(E) I, dS/dmu = 2 E = B
        gmu = dot6(q.B, e);
        glam = R(0.5) * (q.B[0] + q.B[1] + q.B[2]) * trE;
    } else {
        // dS/dmu = J^{-8/3} M + 2/3 (J - 1)/J Q (mu01 held fixed), dS/dlam = (J - 1)/J Q
        const R NE = dot6(q.N, e);
        const R gq = q.Jm1r * (q.t1 * trE - NE);
        const R g = q.rD * q.r1 * q.r1 * (q.s * NE + q.i * trE) + R(2.0 / 3.0) * gq;
        gmu = q.ok ? g : R(0);
        glam = q.ok ? gq : R(0);
    }
}

}  // namespace tlfe
