// Warp-per-element kernels for affine Q27 bricks (internal force, operator
// product, adjoint, Jacobi diagonal).
//
// A Q27 element vector holds 81 values: one thread per element cannot keep it
// (and the 78 nodal differences) in registers. Here one warp takes one element
// at a time; lane (i, j, k) = i + 3 j + 9 k < 27 owns both Gauss point and node
// (i, j, k) of the tensor grids:
//   A. the gradients of the fields at the points, by the tensor structure: the
//      three directions one after the other, each a 3-term sum along a line of
//      the grid with the 1D polynomials' values or derivatives at the Gauss
//      points (24 multiply-adds a component where the sum over the 27 nodes
//      takes 81), the intermediate values in shared rows; then J^{-1}, the
//      stress (or its derivative or adjoint), and the point's weighted operator
//      times J^{-T}, in a shared row;
//   B. the transposed sums, z then y then x, which leave node (i, j, k)'s
//      entry of the element vector in its lane; one atomic per component, or a
//      plain read-add-write in colour passes.
// The Jacobi diagonal, which is quadratic in the gradients, sums over the
// nodes with a per-CTA table of the 27 x 27 parent gradients instead.
// The element's nodal values come straight from global memory (one lane per
// node; the node arrays of a mesh this size stay in L2). The displacement
// differences d_n = u_n - u_13 (the brick's centre: the smallest differences,
// and with them the smallest rounding) are formed from the FP64 state as in the
// tile kernels (an FP32 (hi, lo) pair per value) and shared by all lanes
// through a small per-warp buffer. Warps take the block's element slots (the tile order
// of the mesh) interleaved or in contiguous runs, as the launch schedule says.
// No waits on other warps or on asynchronous copies: nothing to time out.
#pragma once

namespace tlfe {

// shared rows of a warp, four values each (three used): NF planes of nodal
// values, then two scratch areas of planes of 27 rows
template <typename R, int OP> struct Wpe {
    static constexpr bool DIAG = OP == OP_DIAG;
    static constexpr int NF = op_in_fields(OP) / 3, NFO = OpFields<OP>::NFO;
    static constexpr int ROW = 4, PLANE = 27 * ROW;
    static constexpr int R1 = DIAG ? 0 : (2 * NF > 3 * NFO ? 2 * NF : 3 * NFO);  // planes of the x / z-transposed sums
    static constexpr int R2 = DIAG ? 0 : 3 * (NF > NFO ? NF : NFO);              // planes of the y sums and operators
    static constexpr int TS = sizeof(R) == 4 ? 28 : 30;                          // diagonal: the 27 moduli of a point
    static constexpr int WARP = (NF + R1 + R2) * PLANE + (DIAG ? 27 * TS : 0);   // values per warp
    // diagonal: parent gradients [q][n][4]; else the 1D polynomials: values and
    // derivatives at Gauss point a [a][8], and their transposes [m][8]
    static constexpr int TAB = DIAG ? 27 * 27 * 4 : 48;
};

template <typename R, int OP> __host__ __device__ constexpr size_t wpe_smem_bytes(int wpb)
{
    return (size_t)(Wpe<R, OP>::TAB + wpb * Wpe<R, OP>::WARP) * sizeof(R);
}

// a shared row of three values
template <typename R> struct Row3 {
    R x, y, z;
    __device__ __forceinline__ Row3 fma(R s, const Row3 &v) const { return {x + s * v.x, y + s * v.y, z + s * v.z}; }
    __device__ __forceinline__ Row3 times(R s) const { return {x * s, y * s, z * s}; }
};
__device__ __forceinline__ Row3<float> ld_row(const float *p)
{
    const float4 v = lds4(p);
    return {v.x, v.y, v.z};
}
__device__ __forceinline__ Row3<double> ld_row(const double *p)
{
    const double2 v = *reinterpret_cast<const double2 *>(p);
    return {v.x, v.y, p[2]};
}
__device__ __forceinline__ void st_row(float *p, const Row3<float> &v)
{
    *reinterpret_cast<float4 *>(p) = make_float4(v.x, v.y, v.z, 0.f);
}
__device__ __forceinline__ void st_row(double *p, const Row3<double> &v)
{
    *reinterpret_cast<double2 *>(p) = make_double2(v.x, v.y);
    p[2] = v.z;
}
// sum of three rows `step` rows apart
template <typename R> __device__ __forceinline__ Row3<R> line_sum(const Row3<R> v[3], const R c[3])
{
    return v[0].times(c[0]).fma(c[1], v[1]).fma(c[2], v[2]);
}

// entry (i, j) of the 1D quadratic mass on [-1, 1] times 30/L: [[4, 2, -1], [2, 16, 2], [-1, 2, 4]]
__device__ __forceinline__ int q27_m1(int i, int j) { return i == j ? (i == 1 ? 16 : 4) : ((i == 1 || j == 1) ? 2 : -1); }

template <typename R, int OP, int MAT>
__global__ void __launch_bounds__(128, sizeof(R) == 4 ? 4 : 2) k_wpe_q27(const KParams<R> p)
{
    constexpr bool HAS_V = OpFields<OP>::NFI == 3;
    using WP = Wpe<R, OP>;
    constexpr bool DIAG = WP::DIAG;
    constexpr int NF = WP::NF, ROW = WP::ROW, PLANE = WP::PLANE, TS = WP::TS;
    extern __shared__ __align__(128) unsigned char smem[];
    R *tab = reinterpret_cast<R *>(smem);
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    R *nb = tab + WP::TAB + (size_t)wib * WP::WARP;  // [NF][27][ROW]
    R *r1 = nb + NF * PLANE;                         // [R1][27][ROW]
    R *r2 = r1 + WP::R1 * PLANE;                     // [R2][27][ROW]
    R *tb = r1;                                      // diagonal: [27][TS]

    if constexpr (DIAG) {  // parent gradients of the 3x3x3 Gauss points from the constant table
        for (int k = threadIdx.x; k < 27 * 27; k += blockDim.x) {
            const R *src;
            if constexpr (sizeof(R) == 4) src = kQ27F.g[k / 27] + (k % 27) * 3;
            else src = kQ27D.g[k / 27] + (k % 27) * 3;
            tab[k * 4 + 0] = src[0];
            tab[k * 4 + 1] = src[1];
            tab[k * 4 + 2] = src[2];
            tab[k * 4 + 3] = R(0);
        }
    } else {  // 1D values and derivatives: row a at a * 8, transposed row m at 24 + m * 8
        for (int k = threadIdx.x; k < 9; k += blockDim.x) {
            const int g = k / 3, m = k % 3;
            const double x = g == 0 ? -0.77459666924148337704 : (g == 1 ? 0.0 : 0.77459666924148337704);
            const R l = R(q27_l(m, x)), dl = R(q27_dl(m, x));
            tab[g * 8 + m] = l;
            tab[g * 8 + 3 + m] = dl;
            tab[24 + m * 8 + g] = l;
            tab[24 + m * 8 + 3 + g] = dl;
        }
    }
    __syncthreads();

    const int gw = blockIdx.x * (blockDim.x >> 5) + wib;
    const int W = gridDim.x * (blockDim.x >> 5);
    const int s_begin = p.tile_begin * TILE, s_end = p.tile_end * TILE;
    const int n_slots = s_end - s_begin;
    const int per = (n_slots + W - 1) / W;
    const int s0 = p.tile_chunk ? s_begin + gw * per : s_begin + gw;
    const int s1 = p.tile_chunk ? min(s_end, s0 + per) : s_end;
    const int sstep = p.tile_chunk ? 1 : W;
    const bool mass_only = OP == OP_MATVEC && p.mass_only != 0;
    const bool need_ud = p.visc != 0;
    const bool q_lane = lane < 27;  // phase A: point `lane`; phase B: node `lane`
    // tensor indices of the lane's point and node, and the first rows of its grid lines
    const int ln = q_lane ? lane : 0, ti = ln % 3, tj = (ln / 3) % 3, tk = ln / 9;
    const int lx = (ln - ti) * ROW, ly = (ln - 3 * tj) * ROW, lz = (ln - 9 * tk) * ROW;
    auto line = [&](const R *plane, int first, int step, Row3<R> v[3]) {
#pragma unroll
        for (int m = 0; m < 3; ++m) v[m] = ld_row(plane + first + m * step * ROW);
    };
    auto coeffs = [&](const R *t, R l[3], R dl[3]) {
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            l[m] = t[m];
            dl[m] = t[3 + m];
        }
    };
    int bad = 0;

    for (int s = s0; s < s1; s += sstep) {
        const int e = p.eid[s];
        if (e < 0) continue;  // warp-uniform
        const int t = s >> 5, l = s & 31;
        Mat<R> m = p.mat0;
        if (p.mats) m = p.mats[p.emat[s]];
        if (p.elam) {
            m.mu = p.elam[((size_t)t * 2 + 0) * 32 + l];
            m.lam = p.elam[((size_t)t * 2 + 1) * 32 + l];
        }
        if constexpr (MAT == MAT_NH || MAT == MAT_NH_KV) m.model = MODEL_NH;
        if constexpr (MAT == MAT_SVK || MAT == MAT_SVK_KV) m.model = MODEL_SVK;
        const bool visc = MAT == MAT_ANY ? (need_ud && (m.mu_v != R(0) || m.lam_v != R(0)))
                                         : (MAT == MAT_NH_KV || MAT == MAT_SVK_KV);
        R Ji[9];
#pragma unroll
        for (int r = 0; r < 9; ++r) Ji[r] = p.aff[((size_t)t * AFF_ROWS + r) * 32 + l];
        const R detJ = p.aff[((size_t)t * AFF_ROWS + 9) * 32 + l];

        // ---- nodal values of the element: lane n loads node n
        const int nl = q_lane ? lane : 0;
        const int64_t node = bounds_clamp(p.conn[bounds_clamp((int64_t)e - p.elem_base, p.n_elem_block, p.status) * 27 + nl],
                                          p.n_nodes, p.status);
        {
            double u3[3];
            R d[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) u3[a] = p.u[3 * node + a];
            if constexpr (sizeof(R) == 4) {
                float h[3], lo[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) split_f64(u3[a], h[a], lo[a]);
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const float h0 = __shfl_sync(0xffffffffu, h[a], 13), l0 = __shfl_sync(0xffffffffu, lo[a], 13);
                    d[a] = (h[a] - h0) + (lo[a] - l0);
                }
            } else {
#pragma unroll
                for (int a = 0; a < 3; ++a) d[a] = R(u3[a] - __shfl_sync(0xffffffffu, u3[a], 13));
            }
            if (q_lane) {
                R *row = nb + lane * ROW;
                st_row(row, Row3<R>{d[0], d[1], d[2]});
                if (visc) st_row(row + PLANE, Row3<R>{p.ud[3 * node], p.ud[3 * node + 1], p.ud[3 * node + 2]});
                if (HAS_V) st_row(row + 2 * PLANE, Row3<R>{p.v[3 * node], p.v[3 * node + 1], p.v[3 * node + 2]});
            }
        }
        __syncwarp();

        // ---- phase A: sums along x and y of every field (the point's own below)
        if constexpr (!DIAG) {
            if (!mass_only) {
                auto field = [&](int f) { return f == 0 || (f == 1 ? visc : HAS_V); };
                R l[3], dl[3];
                if (q_lane) {
                    coeffs(tab + ti * 8, l, dl);
#pragma unroll
                    for (int f = 0; f < NF; ++f) {
                        if (!field(f)) continue;
                        Row3<R> v[3];
                        line(nb + f * PLANE, lx, 1, v);
                        st_row(r1 + 2 * f * PLANE + ln * ROW, line_sum(v, l));
                        st_row(r1 + (2 * f + 1) * PLANE + ln * ROW, line_sum(v, dl));
                    }
                }
                __syncwarp();
                if (q_lane) {
                    coeffs(tab + tj * 8, l, dl);
#pragma unroll
                    for (int f = 0; f < NF; ++f) {
                        if (!field(f)) continue;
                        Row3<R> v[3];
                        line(r1 + 2 * f * PLANE, ly, 3, v);
                        st_row(r2 + 3 * f * PLANE + ln * ROW, line_sum(v, l));
                        st_row(r2 + (3 * f + 1) * PLANE + ln * ROW, line_sum(v, dl));
                        line(r1 + (2 * f + 1) * PLANE, ly, 3, v);
                        st_row(r2 + (3 * f + 2) * PLANE + ln * ROW, line_sum(v, l));
                    }
                }
                __syncwarp();
            }
        }
        // ---- point q = lane
        R gmu = R(0), glam = R(0);
        R T0[9], T1[9];
        if (q_lane && !mass_only) {
            const int q = lane;
            const R w = quad_weight<ET_Q27, 27, R>(q) * detJ;
            QP<R> s1;
            R D[9];
#pragma unroll
            for (int k2 = 0; k2 < 9; ++k2) {
                s1.G[k2] = R(0);
                s1.Fd[k2] = R(0);
                D[k2] = R(0);
            }
            if constexpr (DIAG) {
#pragma unroll
                for (int n = 0; n < 27; ++n) {
                    const R *g = tab + (q * 27 + n) * 4;
                    const R g0 = g[0], g1 = g[1], g2 = g[2];
                    auto add = [&](const R *row, R *X) {
#pragma unroll
                        for (int a = 0; a < 3; ++a) {
                            const R x = row[a];
                            X[a * 3 + 0] += x * g0;
                            X[a * 3 + 1] += x * g1;
                            X[a * 3 + 2] += x * g2;
                        }
                    };
                    if (n != 13) add(nb + n * ROW, s1.G);
                    if (visc) add(nb + PLANE + n * ROW, s1.Fd);
                }
            } else {
                R l[3], dl[3];
                coeffs(tab + tk * 8, l, dl);
                auto along_z = [&](int f, R *X) {
                    Row3<R> v[3];
                    line(r2 + (3 * f + 2) * PLANE, lz, 9, v);  // x derivative
                    const Row3<R> gx = line_sum(v, l);
                    line(r2 + (3 * f + 1) * PLANE, lz, 9, v);  // y derivative
                    const Row3<R> gy = line_sum(v, l);
                    line(r2 + 3 * f * PLANE, lz, 9, v);
                    const Row3<R> gz = line_sum(v, dl);
                    X[0] = gx.x, X[1] = gy.x, X[2] = gz.x;
                    X[3] = gx.y, X[4] = gy.y, X[5] = gz.y;
                    X[6] = gx.z, X[7] = gy.z, X[8] = gz.z;
                };
                along_z(0, s1.G);
                if (visc) along_z(1, s1.Fd);
                if constexpr (HAS_V) along_z(2, D);
            }
            {
                R T[9];
                mm3(s1.G, Ji, T);
#pragma unroll
                for (int k2 = 0; k2 < 9; ++k2) s1.G[k2] = T[k2];
                if (visc) {
                    mm3(s1.Fd, Ji, T);
#pragma unroll
                    for (int k2 = 0; k2 < 9; ++k2) s1.Fd[k2] = T[k2];
                }
                if (HAS_V) {
                    mm3(D, Ji, T);
#pragma unroll
                    for (int k2 = 0; k2 < 9; ++k2) D[k2] = T[k2];
                }
            }
            R P[9];
            stress<R>(m, s1, visc, P);
            bad += s1.ok ? 0 : 1;
            if constexpr (DIAG) {
                R *trow = tb + q * TS;
                // diagonal moduli A_d[c][b] = w dP_{d b} / dF_{d c}, d = 0..2
#pragma unroll
                for (int dd = 0; dd < 3; ++dd)
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        R E[9], dP[9];
#pragma unroll
                        for (int k2 = 0; k2 < 9; ++k2) E[k2] = (k2 == dd * 3 + c) ? R(1) : R(0);
                        dstress<R>(m, s1, visc, E, p.aK, p.aC, true, dP);
#pragma unroll
                        for (int b2 = 0; b2 < 3; ++b2) trow[dd * 9 + c * 3 + b2] = w * dP[dd * 3 + b2];
                    }
            } else {
                if (OP == OP_FORCE) {
#pragma unroll
                    for (int k2 = 0; k2 < 9; ++k2) T0[k2] = w * P[k2];
                } else if (OP == OP_MATVEC) {
                    dstress<R>(m, s1, visc, D, p.aK, p.aC, p.sym_only != 0, T0);
#pragma unroll
                    for (int k2 = 0; k2 < 9; ++k2) T0[k2] *= w;
                } else {
                    astress<R>(m, s1, visc, D, T0, T1, gmu, glam);
                    gmu *= w;
                    glam *= w;
#pragma unroll
                    for (int k2 = 0; k2 < 9; ++k2) {
                        T0[k2] *= w;
                        T1[k2] *= w;
                    }
                }
            }
        }
        __syncwarp();

        // ---- phase B: node n = lane
        R acc0[3] = {R(0), R(0), R(0)}, acc1[3] = {R(0), R(0), R(0)};
        const int n = lane;
        if constexpr (DIAG) {
            if (q_lane) {
#pragma unroll 3
                for (int q = 0; q < 27; ++q) {
                    const R *g = tab + (q * 27 + n) * 4;
                    const R g0 = g[0], g1 = g[1], g2 = g[2];
                    const R *trow = tb + q * TS;
                    R hh[3];
#pragma unroll
                    for (int c = 0; c < 3; ++c) hh[c] = g0 * Ji[c] + g1 * Ji[3 + c] + g2 * Ji[6 + c];
#pragma unroll
                    for (int dd = 0; dd < 3; ++dd) {
                        const R *A = trow + dd * 9;
                        acc0[dd] += hh[0] * (A[0] * hh[0] + A[1] * hh[1] + A[2] * hh[2]) +
                                    hh[1] * (A[3] * hh[0] + A[4] * hh[1] + A[5] * hh[2]) +
                                    hh[2] * (A[6] * hh[0] + A[7] * hh[1] + A[8] * hh[2]);
                    }
                }
            }
        } else if (!mass_only) {
            constexpr int NFO = WP::NFO;
            // the points' operators times J^{-T}, one row per parent direction
            if (q_lane) {
#pragma unroll
                for (int fo = 0; fo < NFO; ++fo) {
                    const R *T = fo == 0 ? T0 : T1;
#pragma unroll
                    for (int k2 = 0; k2 < 3; ++k2) {
                        auto dir = [&](int a) {
                            return T[a * 3] * Ji[k2 * 3] + T[a * 3 + 1] * Ji[k2 * 3 + 1] + T[a * 3 + 2] * Ji[k2 * 3 + 2];
                        };
                        st_row(r2 + (3 * fo + k2) * PLANE + ln * ROW, Row3<R>{dir(0), dir(1), dir(2)});
                    }
                }
            }
            __syncwarp();
            R l[3], dl[3];
            if (q_lane) {  // sums along z
                coeffs(tab + 24 + tk * 8, l, dl);
#pragma unroll
                for (int fo = 0; fo < NFO; ++fo) {
                    Row3<R> v[3];
#pragma unroll
                    for (int k2 = 0; k2 < 3; ++k2) {
                        line(r2 + (3 * fo + k2) * PLANE, lz, 9, v);
                        st_row(r1 + (3 * fo + k2) * PLANE + ln * ROW, line_sum(v, k2 == 2 ? dl : l));
                    }
                }
            }
            __syncwarp();
            if (q_lane) {  // along y: the x derivative's part, and the other two
                coeffs(tab + 24 + tj * 8, l, dl);
#pragma unroll
                for (int fo = 0; fo < NFO; ++fo) {
                    Row3<R> v[3];
                    line(r1 + 3 * fo * PLANE, ly, 3, v);
                    st_row(r2 + 2 * fo * PLANE + ln * ROW, line_sum(v, l));
                    line(r1 + (3 * fo + 1) * PLANE, ly, 3, v);
                    Row3<R> s = line_sum(v, dl);
                    line(r1 + (3 * fo + 2) * PLANE, ly, 3, v);
                    s = s.fma(l[0], v[0]).fma(l[1], v[1]).fma(l[2], v[2]);
                    st_row(r2 + (2 * fo + 1) * PLANE + ln * ROW, s);
                }
            }
            __syncwarp();
            if (q_lane) {  // along x
                coeffs(tab + 24 + ti * 8, l, dl);
#pragma unroll
                for (int fo = 0; fo < NFO; ++fo) {
                    Row3<R> v[3];
                    line(r2 + 2 * fo * PLANE, lx, 1, v);
                    Row3<R> s = line_sum(v, dl);
                    line(r2 + (2 * fo + 1) * PLANE, lx, 1, v);
                    s = s.fma(l[0], v[0]).fma(l[1], v[1]).fma(l[2], v[2]);
                    R *a3 = fo == 0 ? acc0 : acc1;
                    a3[0] = s.x, a3[1] = s.y, a3[2] = s.z;
                }
            }
        }
        if (q_lane) {
            // consistent mass of the parallelepiped: m_nj = rho V Mhat_nj with
            // Mhat the product of the normalised 1D quadratic masses
            if ((OP == OP_MATVEC || OP == OP_DIAG) && p.aM != R(0)) {
                const R c = p.aM * m.rho * p.evol[s] * R(1.0 / 27000.0);
                const int ni = n % 3, nj = (n / 3) % 3, nk = n / 9;
                if (OP == OP_MATVEC) {
#pragma unroll
                    for (int j = 0; j < 27; ++j) {
                        const R mh = c * R(q27_m1(ni, j % 3) * q27_m1(nj, (j / 3) % 3) * q27_m1(nk, j / 9));
                        const R *row = nb + 2 * PLANE + j * ROW;
                        acc0[0] += mh * row[0];
                        acc0[1] += mh * row[1];
                        acc0[2] += mh * row[2];
                    }
                } else {
                    const R mh = c * R(q27_m1(ni, ni) * q27_m1(nj, nj) * q27_m1(nk, nk));
                    acc0[0] += mh;
                    acc0[1] += mh;
                    acc0[2] += mh;
                }
            }
#pragma unroll
            for (int fo = 0; fo < OpFields<OP>::NFO; ++fo) {
                R *out = fo == 0 ? p.out0 : p.out1;
                R *part = fo == 0 ? p.part0 : p.part1;
                const R *a3 = fo == 0 ? acc0 : acc1;
                if (part) {  // sorted scatter: this element's partial for node n
                    const int64_t pos = (int64_t)((int)p.part_base + s * 27 + n);  // positions < 2^31
                    R *dst = part + bounds_clamp(pos, p.n_part, p.status) * 3;
                    dst[0] = a3[0];
                    dst[1] = a3[1];
                    dst[2] = a3[2];
                } else if (p.rmw_scatter) {
                    out[3 * node] += a3[0];
                    out[3 * node + 1] += a3[1];
                    out[3 * node + 2] += a3[2];
                } else {
                    atomicAdd(out + 3 * node, a3[0]);
                    atomicAdd(out + 3 * node + 1, a3[1]);
                    atomicAdd(out + 3 * node + 2, a3[2]);
                }
            }
        }
        if (OP == OP_VJP && p.gth && bounds_ok(e, p.n_elem_total, p.status)) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                gmu += __shfl_xor_sync(0xffffffffu, gmu, o);
                glam += __shfl_xor_sync(0xffffffffu, glam, o);
            }
            if (lane == 0) {
                p.gth[(size_t)e * 2 + 0] = double(gmu);
                p.gth[(size_t)e * 2 + 1] = double(glam);
            }
        }
        __syncwarp();  // nb and tb are rewritten by the next element
    }
    const int nbad = __reduce_add_sync(0xffffffffu, bad);
    if (lane == 0 && nbad) atomicAdd(p.status + ST_INVERTED, nbad);
}

template <int OP, typename R> static void (*wpe_kernel_for(int mat))(const KParams<R>)
{
    if constexpr (sizeof(R) == 4) {
        switch (mat) {
        case MAT_NH: return k_wpe_q27<R, OP, MAT_NH>;
        case MAT_NH_KV: return k_wpe_q27<R, OP, MAT_NH_KV>;
        case MAT_SVK: return k_wpe_q27<R, OP, MAT_SVK>;
        case MAT_SVK_KV: return k_wpe_q27<R, OP, MAT_SVK_KV>;
        default: break;
        }
    }
    return k_wpe_q27<R, OP, MAT_ANY>;
}

}  // namespace tlfe
