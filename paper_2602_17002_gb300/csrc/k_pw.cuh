// FP64 element kernels with one CTA per tile and one warp per quadrature point
// (force, operator product, adjoint, and force + operator product of affine
// T10 blocks): lane = element, warp = point.
//
// FP64 arithmetic runs at 1/64 of the FP32 rate here, so what counts is the
// number of multiply-adds, and for small meshes how many SMs share them.
// Against one warp per tile (k_elem.cuh):
//   - what the points share of a gradient is formed once per element instead
//     of at every point (PW::base), and the element vectors are formed once
//     from the points' operators (PW::vectors): about 40 multiply-adds a point
//     and field where the sums over ten nodes take 90;
//   - a thread holds one point's state and nothing else, so 10 warps fit an SM
//     in 168 registers;
//   - a tile occupies the FP64 pipe of one SM on its own, where four tiles
//     used to share it: meshes with fewer tiles than SMs take a quarter of the
//     time; and the next tile's nodal values are gathered while this one's
//     element vectors are formed and scattered.
// Measured: force + operator product of 384 elements (4 points, SVK) 142 -> 47
// us as two passes, 35 us as one (OP_FM); force + operator product + adjoint
// of 60,000 damped neo-Hookean elements 1572 -> 1139 us, 963 with one pass for
// the first two. FP32 blocks stay with one warp per tile: there this layout
// executes 7,000 warp instructions a tile against 5,700 and waits at its
// barriers (beam step of 480,000 elements 345 us against 274).
//
// Per tile, with four CTA barriers:
//   1. the patch, gathered by cp.async during the previous tile, has landed;
//   2. warp f forms field f's part of the gradient that all points share;
//   3. warp q forms the gradients of point q, its stress and operators, and
//      stores the operators (9 values per output field and lane);
//   4. warp by (output field, component), the element vectors go to
//      node-sorted slots;
//   5. one thread per unique node sums its slots and adds them to the global
//      array (or stores them as the tile's partial: sorted scatter).
// Every wait on a bulk copy is bounded, as in k_elem.cuh.
#pragma once

#include "tlfe_elem.cuh"
#include "tlfe_internal.h"

namespace tlfe {

__host__ __device__ constexpr size_t up16(size_t x) { return (x + 15) / 16 * 16; }

// 3-vector of a node
struct V3 {
    double x, y, z;
    __device__ __forceinline__ V3 operator+(const V3 &o) const { return {x + o.x, y + o.y, z + o.z}; }
    __device__ __forceinline__ V3 operator-(const V3 &o) const { return {x - o.x, y - o.y, z - o.z}; }
    __device__ __forceinline__ V3 operator*(double s) const { return {x * s, y * s, z * s}; }
    // this + s v
    __device__ __forceinline__ V3 fma(double s, const V3 &v) const
    {
        return {::fma(s, v.x, x), ::fma(s, v.y, y), ::fma(s, v.z, z)};
    }
};

// field F (0 displacement, 1 velocity, 2 direction) of a patch record
template <int OP, int F> __device__ __forceinline__ V3 pw_value(const double *rec)
{
    using RC = Rec<OP, double>;
    V3 v;
    ld3c<F == 0 ? 0 : (F == 1 ? RC::OFF_UD : RC::OFF_V)>(rec, v.x, v.y, v.z);
    return v;
}

template <int ET, int NQ> struct PW;

// T10. The gradient of a quadratic field on a straight-sided tetrahedron is
// linear in the barycentric coordinates. With E_aj the value at the mid-edge
// node of edge (a, j) (E_jj: at corner j) and Delta_k = x_{k+1} - x_0, the
// parent gradient at corner j is 4 (E_{k+1,j} - E_{0,j}) - Delta_k, so that
//   at the centroid             G0_k = sum_j (E_{k+1,j} - E_{0,j}) - Delta_k,
//   at (a, b, b, b), a at j     base_k + 4 (a - b) (E_{k+1,j} - E_{0,j}),
//                               base_k = 4 b G0_k - (a - b) Delta_k:
// 6 operations a component, direction and point where the sum over the ten
// nodes takes 21. The element vector is the transposed map; the centroid
// (point 0 of the 5-point rule) has the mean of the other points'
// shape-function gradients, so its operator is added to theirs in the ratio
// of the weights.
template <int NQ> struct PW<ET_T10, NQ> {
    using R = double;
    static constexpr int NPE = 10;
    static constexpr double a = NQ == 5 ? 0.5 : 0.58541019662496845446;
    static constexpr double b = NQ == 5 ? 1.0 / 6.0 : 0.13819660112501051518;
    static constexpr double w = NQ == 5 ? 3.0 / 40.0 : 1.0 / 24.0;
    static constexpr double w0 = NQ == 5 ? -2.0 / 15.0 : 0.0;
    static constexpr int NB = NQ == 5 ? 18 : 9;  // base (and G0) values of a field

    __host__ __device__ __forceinline__ static constexpr int node(int p, int j)  // holds E_pj
    {
        const int lo = p < j ? p : j, hi = p < j ? j : p;
        return lo == hi ? lo : (lo == 0 ? (hi == 1 ? 4 : (hi == 2 ? 6 : 7)) : (lo == 1 ? (hi == 2 ? 5 : 8) : 9));
    }

    // base (and G0) of one field from its nodal values (x[0] subtracted or
    // not: only differences enter) into out[(k * 3 + component) * 32]
    __device__ __forceinline__ static void base(const V3 x[10], R *out)
    {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const V3 D = x[k + 1] - x[0];
            const V3 S = (((x[node(k + 1, 0)] - x[0]) + (x[node(k + 1, 1)] - x[node(0, 1)])) +
                             ((x[node(k + 1, 2)] - x[node(0, 2)]) + (x[node(k + 1, 3)] - x[node(0, 3)]))) - D;
            const V3 B = (S * R(4.0 * b)).fma(R(b - a), D);
            out[(k * 3) * 32] = B.x;
            out[(k * 3 + 1) * 32] = B.y;
            out[(k * 3 + 2) * 32] = B.z;
            if constexpr (NQ == 5) {
                out[(9 + k * 3) * 32] = S.x;
                out[(9 + k * 3 + 1) * 32] = S.y;
                out[(9 + k * 3 + 2) * 32] = S.z;
            }
        }
    }

    // element vector of one component from the points' operators:
    // T[q * stride] holds (row of the component) T_b at b * 32; Ji = J^{-1},
    // s = detJ
    __device__ __forceinline__ static void vectors(const R *T, int stride, const R Ji[9], R detJ, R F[10])
    {
        R t[4][3], sum[3], U[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const R t0 = NQ == 5 ? T[c * 32] * R(w0 / (4.0 * w)) : R(0);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                t[j][c] = T[(NQ == 5 ? j + 1 : j) * stride + c * 32];
                if (NQ == 5) t[j][c] += t0;
            }
            sum[c] = (t[0][c] + t[1][c]) + (t[2][c] + t[3][c]);
        }
        const R wd = R(w) * detJ;
        R J[9];
#pragma unroll
        for (int r = 0; r < 9; ++r) J[r] = wd * Ji[r];
#pragma unroll
        for (int k = 0; k < 3; ++k) U[k] = sum[0] * J[k * 3] + sum[1] * J[k * 3 + 1] + sum[2] * J[k * 3 + 2];
        F[0] = (U[0] + U[1]) + U[2];  // the -Delta parts: 4 b + (a - b) = 1
#pragma unroll
        for (int k = 0; k < 3; ++k) F[k + 1] = -U[k];
#pragma unroll
        for (int i = 4; i < 10; ++i) F[i] = R(0);
#pragma unroll
        for (int k = 0; k < 3; ++k) U[k] *= R(4.0 * b);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            R s = R(0);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const R y = t[j][0] * J[k * 3] + t[j][1] * J[k * 3 + 1] + t[j][2] * J[k * 3 + 2];
                const R Y = U[k] + R(4.0 * (a - b)) * y;
                F[node(k + 1, j)] += Y;
                s += Y;
            }
            F[node(0, j)] -= s;
        }
    }

    // consistent mass (mass_hat) of one component, added to F: from the sums
    // over corners and edges (units of 1/420: corner-corner 6 or 1,
    // corner-edge -4 with and -6 without the corner, edge-edge 32, 16 or 8)
    __device__ __forceinline__ static void mass(const R x[10], R c, R F[10])
    {
        const R s = c * R(1.0 / 420.0);
        const R sc = (x[0] + x[1]) + (x[2] + x[3]);
        const R se = ((x[4] + x[5]) + (x[6] + x[7])) + (x[8] + x[9]);
        const R bc = sc - R(6) * se, be = R(16) * se - R(6) * sc;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const R e = (x[node(i, (i + 1) & 3)] + x[node(i, (i + 2) & 3)]) + x[node(i, (i + 3) & 3)];
            F[i] += s * (bc + R(5) * x[i] + R(2) * e);
        }
        const int opp[6] = {9, 7, 8, 5, 6, 4};  // edge opposite to edge node 4 + e
#pragma unroll
        for (int e = 0; e < 6; ++e)
            F[4 + e] += s * (be + R(2) * (x[t10_ea(e)] + x[t10_eb(e)]) + R(16) * x[4 + e] - R(8) * x[opp[e]]);
    }
};

// shared memory of one CTA
template <int ET, int NQ, int OP> struct PwSmem {
    using R = double;
    static constexpr int NF = op_in_fields(OP) / 3;  // fields with a gradient: u, udot, the direction
    static constexpr int NFO = OpFields<OP>::NFO;
    static constexpr size_t BASE = (size_t)NF * PW<ET, NQ>::NB * 32 * sizeof(R);
    static constexpr size_t OPER = (size_t)NQ * 9 * NFO * 32 * sizeof(R);
    static constexpr size_t SLOT = (size_t)3 * NFO * PW<ET, NQ>::NPE * 32 * sizeof(R);
    static constexpr size_t GPAR = OP == OP_VJP ? (size_t)NQ * 2 * 32 * sizeof(R) : 0;
    __host__ __device__ static constexpr size_t bytes(int umax, int meta_bytes)
    {
        return 128 + 2 * ((size_t)meta_bytes + AffRec<R>::BYTES) + up16((size_t)umax * Rec<OP, R>::REC * sizeof(R)) +
               BASE + OPER + SLOT + GPAR;
    }
};

// two CTAs per SM (168 registers): one CTA works while the other is at a
// barrier; one CTA at 255 registers, without the 340-390 bytes of spill, took
// 1210 us for the 60,000-element step instead of 963
template <int ET, int NQ, int OP> __global__ void __launch_bounds__(32 * NQ, 2) k_pw(const KParams<double> p)
{
    using R = double;
    using P = PW<ET, NQ>;
    using SM = PwSmem<ET, NQ, OP>;
    using RC = Rec<OP, R>;
    constexpr int NPE = P::NPE, REC = RC::REC, NT = 32 * NQ;
    constexpr bool HAS_V = OpFields<OP>::NFI == 3;
    constexpr int NF = SM::NF, NFO = SM::NFO, NB = P::NB;
    constexpr uint32_t AB = AffRec<R>::BYTES;
    extern __shared__ __align__(128) unsigned char smem[];
    const int tid = threadIdx.x, lane = tid & 31, q = tid >> 5;
    const int MB = p.meta_bytes;
    const size_t MRB = (size_t)MB + AB;
    uint64_t *mbar = reinterpret_cast<uint64_t *>(smem);
    unsigned char *mbuf = smem + 128;
    R *patch = reinterpret_cast<R *>(mbuf + 2 * MRB);
    R *sbase = reinterpret_cast<R *>(reinterpret_cast<unsigned char *>(patch) + up16((size_t)p.umax * REC * sizeof(R)));
    R *soper = sbase + SM::BASE / sizeof(R);
    R *slots = soper + SM::OPER / sizeof(R);
    R *gpar = slots + SM::SLOT / sizeof(R);

    const int n_tiles = p.tile_end - p.tile_begin;
    const int per = (n_tiles + (int)gridDim.x - 1) / (int)gridDim.x;
    const int t0 = p.tile_chunk ? p.tile_begin + (int)blockIdx.x * per : p.tile_begin + (int)blockIdx.x;
    const int tstep = p.tile_chunk ? 1 : (int)gridDim.x;
    const int n_my = p.tile_chunk ? max(0, min(per, n_tiles - (int)blockIdx.x * per))
                                  : (t0 < p.tile_end ? (p.tile_end - t0 + (int)gridDim.x - 1) / (int)gridDim.x : 0);
    const bool need_ud = p.visc != 0;
    const bool has_mass = (OP == OP_MATVEC || OP == OP_FM) && p.aM != R(0);
    const bool mass_only = OP == OP_MATVEC && p.mass_only != 0;

    if (tid == 0) {
        mbar_init(mbar, 1);
        mbar_init(mbar + 1, 1);
        fence_mbar_init();
    }
    __syncthreads();
    auto issue_meta = [&](int k) {  // metadata and affine record of the CTA's k-th tile into buffer k & 1
        const int t = t0 + k * tstep;
        unsigned char *dst = mbuf + (size_t)(k & 1) * MRB;
        mbar_arrive_expect_tx(mbar + (k & 1), (uint32_t)MRB);
        bulk_g2s(dst, p.meta + (size_t)t * MB, (uint32_t)MB, mbar + (k & 1));
        bulk_g2s(dst + MB, p.aff + (size_t)t * AFF_ROWS * 32, AB, mbar + (k & 1));
    };
    // the nodal inputs of the CTA's k-th tile into the patch, one record per
    // unique node, by asynchronous copies; false when its metadata never landed
    auto gather = [&](int k) -> bool {
        if (!mbar_wait_bounded(mbar + (k & 1), (uint32_t)((k >> 1) & 1))) return false;
        const unsigned char *M = mbuf + (size_t)(k & 1) * MRB;
        const int U = (int)bounds_clamp(*reinterpret_cast<const int32_t *>(M), (int64_t)p.umax + 1, p.status);
        const int32_t *nodes = reinterpret_cast<const int32_t *>(M + 16 + 128);
        for (int kk = tid; kk < U; kk += NT) {
            const int64_t n = bounds_clamp(nodes[kk], p.n_nodes, p.status);
            R *rec = patch + (size_t)kk * REC;
            const double *pu = p.u + 3 * n;
#pragma unroll
            for (int c = 0; c < 3; ++c) cp_async<8>(rec + c, pu + c);
            if (need_ud) {
                const R *pd = p.ud + 3 * n;
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    cp_async<8>(rec + RC::OFF_UD + c, pd + c);
            }
            if (HAS_V) {
                const R *pv = p.v + 3 * n;
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    cp_async<8>(rec + RC::OFF_V + c, pv + c);
            }
        }
        cp_async_commit();
        return true;
    };

    bool lost = false;  // a copy of metadata never landed
    int issued = 0;     // metadata records requested so far
    int bad = 0;
    if (n_my > 0) {
        if (tid == 0) issue_meta(0);
        issued = 1;
        lost = !gather(0);
    }
    for (int k = 0; k < n_my; ++k) {
        const int t = t0 + k * tstep;
        const unsigned char *M = mbuf + (size_t)(k & 1) * MRB;
        cp_async_wait<0>();
        if (__syncthreads_or(lost)) {
            lost = true;
            break;
        }
        if (k + 1 < n_my) {
            if (tid == 0) issue_meta(k + 1);
            issued = k + 2;
        }
        const int U = (int)bounds_clamp(*reinterpret_cast<const int32_t *>(M), (int64_t)p.umax + 1, p.status);
        const int e = reinterpret_cast<const int32_t *>(M + 16)[lane];
        const int32_t *nodes = reinterpret_cast<const int32_t *>(M + 16 + 128);
        const uint16_t *mlidx = reinterpret_cast<const uint16_t *>(M + 16 + 128 + 4 * p.umaxp);
        const uint16_t *spos = mlidx + NPE * 32;  // slot (i, lane) -> node-sorted position
        const uint16_t *soff = spos + NPE * 32;   // positions of unique node kk: [soff[kk], soff[kk + 1])
        const R *Aj = reinterpret_cast<const R *>(M + MB) + lane;
        const bool valid = e >= 0;
        auto rec_of = [&](int i) -> const R * {
            return patch + (int)bounds_clamp(mlidx[i * 32 + lane], U, p.status) * REC;
        };
        Mat<R> m = p.mat0;
        if (p.mats) m = p.mats[bounds_clamp(p.emat[(size_t)t * 32 + lane], p.n_mats, p.status)];
        if (p.elam) {
            m.mu = p.elam[((size_t)t * 2 + 0) * 32 + lane];
            m.lam = p.elam[((size_t)t * 2 + 1) * 32 + lane];
        }
        const bool visc = need_ud && (m.mu_v != R(0) || m.lam_v != R(0));
        const R detJ = Aj[9 * 32];

        if (!mass_only) {
            // ---- what the points share of each field's gradient
            if (q == 0) {
                V3 x[NPE];
#pragma unroll
                for (int i = 0; i < NPE; ++i) x[i] = pw_value<OP, 0>(rec_of(i));
#pragma unroll
                for (int i = 1; i < NPE; ++i) x[i] = x[i] - x[0];
                x[0] = {0.0, 0.0, 0.0};
                P::base(x, sbase + lane);
            }
            if (q == 1 && need_ud) {
                V3 x[NPE];
#pragma unroll
                for (int i = 0; i < NPE; ++i) x[i] = pw_value<OP, 1>(rec_of(i));
                P::base(x, sbase + NB * 32 + lane);
            }
            if constexpr (HAS_V)
                if (q == 2) {
                    V3 x[NPE];
#pragma unroll
                    for (int i = 0; i < NPE; ++i) x[i] = pw_value<OP, 2>(rec_of(i));
                    P::base(x, sbase + (NF - 1) * NB * 32 + lane);
                }
            __syncthreads();

            // ---- point q: gradients
            QP<R> s1;
            R D[9];
            {
                const int j = NQ == 5 ? q - 1 : q;  // the corner the point is close to; -1: the centroid
                V3 gu[3], gd[3], gv[3];
                auto ld_base = [&](int f, int o, V3 g[3]) {
                    const R *b = sbase + ((size_t)f * NB + o) * 32 + lane;
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        g[c] = {b[(c * 3) * 32], b[(c * 3 + 1) * 32], b[(c * 3 + 2) * 32]};
                    }
                };
                const int o = j < 0 ? 9 : 0;
                ld_base(0, o, gu);
                if (need_ud) ld_base(1, o, gd);
                if constexpr (HAS_V) ld_base(NF - 1, o, gv);
                if (j >= 0) {
                    constexpr R c4 = R(4.0 * (P::a - P::b));
                    const R *r0 = rec_of(P::node(0, j));
                    V3 d0, v0;
                    if (need_ud) d0 = pw_value<OP, 1>(r0);
                    if constexpr (HAS_V) v0 = pw_value<OP, 2>(r0);
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        const R *rk = rec_of(P::node(c + 1, j));
                        gu[c] = gu[c].fma(c4, pw_value<OP, 0>(rk) - pw_value<OP, 0>(r0));
                        if (need_ud) gd[c] = gd[c].fma(c4, pw_value<OP, 1>(rk) - d0);
                        if constexpr (HAS_V) gv[c] = gv[c].fma(c4, pw_value<OP, 2>(rk) - v0);
                    }
                }
                R J[9];
#pragma unroll
                for (int r = 0; r < 9; ++r) J[r] = Aj[r * 32];
                auto finish = [&](const V3 g[3], R *X) {  // X = (g_0 g_1 g_2) J^{-1}
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        const V3 col = (g[0] * J[c]).fma(J[3 + c], g[1]).fma(J[6 + c], g[2]);
                        X[c] = col.x;
                        X[3 + c] = col.y;
                        X[6 + c] = col.z;
                    }
                };
                finish(gu, s1.G);
#pragma unroll
                for (int c = 0; c < 9; ++c) s1.Fd[c] = D[c] = R(0);
                if (need_ud) finish(gd, s1.Fd);
                if constexpr (HAS_V) finish(gv, D);
            }

            // ---- point q: stress and operators
            R T[9];
            R *op = soper + (size_t)q * 9 * NFO * 32 + lane;
            stress_state<R>(m, s1, visc);
            bad += (valid && !s1.ok) ? 1 : 0;
            if constexpr (OP == OP_FORCE || OP == OP_FM) {
                first_piola<R>(s1, visc, T);
#pragma unroll
                for (int c = 0; c < 9; ++c) op[c * 32] = T[c];
            }
            if constexpr (OP == OP_MATVEC || OP == OP_FM) {
                dstress<R>(m, s1, visc, D, p.aK, p.aC, OP == OP_FM ? false : p.sym_only != 0, T);
#pragma unroll
                for (int c = 0; c < 9; ++c) op[((OP == OP_FM ? 9 : 0) + c) * 32] = T[c];
            }
            if constexpr (OP == OP_VJP) {
                R T1[9], gmu, glam;
                astress<R>(m, s1, visc, D, T, T1, gmu, glam);
                const R wq = quad_weight<ET, NQ, R>(q) * detJ;
                gpar[q * 64 + lane] = wq * gmu;
                gpar[q * 64 + 32 + lane] = wq * glam;
#pragma unroll
                for (int c = 0; c < 9; ++c) {
                    op[c * 32] = T[c];
                    op[(9 + c) * 32] = T1[c];
                }
            }
        }
        __syncthreads();

        // ---- the patch is dead now (but for the mass term, which reads the
        // direction from it): the next tile's nodes
        if (k + 1 < n_my && !has_mass) lost = !gather(k + 1);

        // ---- element vectors, one (output field, component) per warp and turn
        for (int task = q; task < 3 * NFO; task += NQ) {
            const int fo = task / 3, c = task - 3 * fo;
            R F[NPE];
            if (mass_only) {
#pragma unroll
                for (int i = 0; i < NPE; ++i) F[i] = R(0);
            } else {
                R J[9];
#pragma unroll
                for (int r = 0; r < 9; ++r) J[r] = Aj[r * 32];
                P::vectors(soper + (size_t)(fo * 9 + c * 3) * 32 + lane, 9 * NFO * 32, J, detJ, F);
            }
            if (has_mass && fo == NFO - 1) {
                R x[NPE];
                #pragma unroll
                for (int i = 0; i < NPE; ++i) x[i] = rec_of(i)[RC::OFF_V + c];
                P::mass(x, p.aM * m.rho * p.evol[(size_t)t * 32 + lane], F);
            }
            if (valid) {
                R *sl = slots + task * (NPE * 32);
#pragma unroll
                for (int i = 0; i < NPE; ++i) sl[(int)bounds_clamp(spos[i * 32 + lane], NPE * 32, p.status)] = F[i];
            }
        }
        if (OP == OP_VJP && q == NQ - 1 && valid && p.gth && bounds_ok(e, p.n_elem_total, p.status)) {
            R gmu = R(0), glam = R(0);
#pragma unroll
            for (int j = 0; j < NQ; ++j) {
                gmu += gpar[j * 64 + lane];
                glam += gpar[j * 64 + 32 + lane];
            }
            p.gth[(size_t)e * 2 + 0] = double(gmu);
            p.gth[(size_t)e * 2 + 1] = double(glam);
        }
        __syncthreads();
        if (k + 1 < n_my && has_mass) lost = !gather(k + 1);

        // ---- node sums: one thread per unique node and both output fields
        for (int kk = tid; kk < U; kk += NT) {
            const int s0 = (int)bounds_clamp(soff[kk], NPE * 32 + 1, p.status);
            const int s1e = (int)bounds_clamp(soff[kk + 1], NPE * 32 + 1, p.status);
            R s[NFO][3];
#pragma unroll
            for (int fo = 0; fo < NFO; ++fo) s[fo][0] = s[fo][1] = s[fo][2] = R(0);
            for (int sb = s0; sb < s1e; sb += 4) {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (sb + j < s1e)
#pragma unroll
                        for (int pl = 0; pl < 3 * NFO; ++pl) s[pl / 3][pl % 3] += slots[pl * (NPE * 32) + sb + j];
            }
            if (p.part0) {
                const int64_t P0 = reinterpret_cast<const int32_t *>(M)[1];
                if (!bounds_ok(P0 + kk, p.n_part, p.status)) continue;
#pragma unroll
                for (int fo = 0; fo < NFO; ++fo) {
                    R *dst = (fo == 0 ? p.part0 : p.part1) + (P0 + kk) * 3;
                    dst[0] = s[fo][0];
                    dst[1] = s[fo][1];
                    dst[2] = s[fo][2];
                }
            } else {
                const int64_t n = bounds_clamp(nodes[kk], p.n_nodes, p.status);
#pragma unroll
                for (int fo = 0; fo < NFO; ++fo) {
                    R *out = (fo == 0 ? p.out0 : p.out1) + 3 * n;
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        if (p.rmw_scatter) out[c] += s[fo][c];
                        else atomicAdd(out + c, s[fo][c]);
                    }
                }
            }
        }
    }
    if (lost) {
        // a copy never landed: record it, and wait (bounded) for whatever is
        // still in flight into shared memory before the CTA ends
        cp_async_wait<0>();
        if (tid == 0) {
            atomicAdd(p.status + ST_TIMEOUT, 1);
            if (issued > 0) mbar_wait_bounded(mbar + ((issued - 1) & 1), (uint32_t)(((issued - 1) >> 1) & 1));
        }
        __syncthreads();
    }
    const int nbad = __reduce_add_sync(0xffffffffu, bad);
    if (lane == 0 && nbad) atomicAdd(p.status + ST_INVERTED, nbad);
}

template <int OP, typename R> static void (*pw_kernel_for(int nq))(const KParams<R>)
{
    if constexpr (OP == OP_DIAG || sizeof(R) != 8) return nullptr;
    else return nq == 5 ? k_pw<ET_T10, 5, OP> : k_pw<ET_T10, 4, OP>;
}
// shared memory of a CTA
template <int OP> size_t pw_smem_for(int nq, int umax, int meta_bytes)
{
    return nq == 5 ? PwSmem<ET_T10, 5, OP>::bytes(umax, meta_bytes) : PwSmem<ET_T10, 4, OP>::bytes(umax, meta_bytes);
}

}  // namespace tlfe
