// Element kernels of the TL-FEA hot path (internal force, operator product,
// adjoint, Jacobi diagonal, and the force and operator product of one state
// in one pass), templated on element type, quadrature size, arithmetic type
// and operation.
//
// Work decomposition: one thread per element, one warp per tile of 32
// elements, warps independent of each other (persistent, grid-striding over
// tiles). Per warp:
//   - the tile's metadata (unique-node list, local indices, node-to-slot
//     lists) comes by cp.async.bulk one tile ahead into a double buffer, with
//     the per-element J^{-1} and det J record on the affine path;
//   - slab path only: the reference data of one quadrature point of one tile
//     (h_i rows and w_q J_p, a contiguous "slice" of the slab
//     [tile][q][3 npe + 1][32]) is streamed by cp.async.bulk into a ring of
//     NSLICE shared-memory slots, issued NSLICE slices ahead by lane 0 and
//     completed on one mbarrier per slot; the affine path instead forms
//     h_i = J^{-T} g_i from the parent gradients g_i at each point;
//   - the nodes of the next tile are prefetched into L2, after the first
//     quadrature point in the affine force, operator and diagonal kernels,
//     after the last one on the slab path (the affine adjoint runs faster
//     without);
//   - the nodal values of the tile's unique nodes (a list built at mesh
//     creation) are gathered into a shared-memory patch, one record per list
//     entry, with consecutive lanes on consecutive entries; each lane then
//     reads its element's nodes from the patch through precomputed local
//     indices. The list orders the nodes so that the 8 lanes of a quarter
//     warp, which read the same element-local node of their elements in one
//     16-byte load, hit distinct bank groups;
//   - each lane evaluates F = I + sum_i u_i h_i^T per quadrature point and the
//     stress, its directional derivative, its adjoint or the diagonal moduli,
//     accumulating its element vector sum_q w_q J_p (.) h_iq in registers. FP32
//     affine T10 and H8 blocks (column_path) instead form the gradients from
//     what their points share, keep them in the lane's own shared column and
//     evaluate two points at a time (k_t10.cuh, k_h8.cuh); they read the
//     per-lane tables of a tile straight from global memory;
//   - element vectors go to shared slots in node-sorted positions (a list
//     built at mesh creation); one lane per unique node sums that node's slots
//     and adds the sum to the global array with one atomic per component (a
//     plain read-add-write in colour passes, where no two elements of a launch
//     share a node).
// Every mbarrier wait is bounded; on timeout the kernel latches ST_TIMEOUT in
// the status word, waits (again bounded) for the copies it still has in
// flight, each by the parity of its barrier's one outstanding phase, and
// returns.
// Affine Q27 blocks do not come here: they run the warp-per-element kernels
// of k_wpe.cuh; nor do FP64 operations on affine T10 blocks (but the
// diagonal), which run one warp per quadrature point (k_pw.cuh). kernel_for /
// smem_for below dispatch on wpe_path and pw_path.
#pragma once

#include <string>
#include <type_traits>

#include "k_h8.cuh"
#include "k_t10.cuh"
#include "tlfe_elem.cuh"
#include "tlfe_internal.h"

namespace tlfe {

// ---------------------------------------------------------------------------
// PTX helpers: mbarrier, bulk async copy, cp.async
// ---------------------------------------------------------------------------

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// bulk copy global -> shared, completion counted in bytes on `bar`
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

template <int BYTES> __device__ __forceinline__ void cp_async(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_u32(dst)), "l"(src), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void prefetch_l2(const void *p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

constexpr long long MBAR_SPIN_LIMIT = 1ll << 20;  // try_wait rounds before giving up

// ---------------------------------------------------------------------------
// per-op sizes
// ---------------------------------------------------------------------------

template <int OP> struct OpFields {
    static constexpr int IN = op_in_fields(OP);   // input values per node (u, udot [, v])
    static constexpr int OUT = op_nf(OP) - IN;    // output values per node
    static constexpr int NFI = IN / 3;            // input vector fields per node
    static constexpr int NFO = OUT / 3;           // output vector fields per node
};

// Patch record of one node.
//   FP32 (12 floats, 48 B), laid out for paired arithmetic (FFMA2 on the x
//   and y components of a 3-vector, the z component alone):
//     [h0 h1 l0 l1 | h2 l2 ud2 v2 | ud0 ud1 v0 v1]
//   FP64: [u(3) | udot(3) | v(3)]  (6 or 10 doubles)
// The displacement arrives in FP64; FP32 kernels keep it as an unevaluated
// pair (h, l) with u = h + l to about 2^-46 |u|, so that element-relative
// differences u_i - u_0 are formed without the rounding of |u| (large rigid
// motions). The FP64 displacement is first copied into the record's bytes
// 0..23 (the h, l slots and the unused h2, l2 of slot 2's first half) and
// split there in place.
template <int OP, typename R> struct Rec {
    static constexpr bool PK = sizeof(R) == 4;
    // FP32 slots (float offsets)
    static constexpr int H01 = 0, L01 = 2, H2 = 4, L2 = 5, UD2 = 6, V2 = 7, UD01 = 8, V01 = 10;
    // FP64 offsets
    static constexpr int OFF_UD = 3;                            // udot
    static constexpr int OFF_V = 6;                             // direction / cotangent
    static constexpr int REC = PK ? 12 : (3 * OpFields<OP>::NFI + 1) / 2 * 2;
};

// packed FP32 pairs (sm_100 and later: one instruction for two lanes of work)
__device__ __forceinline__ float2 bc2(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float4 lds4(const float *r) { return *reinterpret_cast<const float4 *>(r); }
// shared-memory loads the compiler may not hoist out of the point loop and
// keep in registers (volatile): the force and adjoint kernels re-read each
// element's local node indices at every point, and the adjoint also its
// J^{-1} and node 0's displacement pair, instead of holding them across the
// loop, which frees registers for the point's arithmetic
__device__ __forceinline__ float lds_f32_volatile(const float *p)
{
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(smem_u32(p)));
    return v;
}
__device__ __forceinline__ float4 lds4_volatile(const float *p)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(smem_u32(p)));
    return v;
}
// loads of a tile's tables straight from global memory, issued where they stand
// (volatile): their latency overlaps what follows up to their first use
__device__ __forceinline__ int ldg_u16_volatile(const uint16_t *p)
{
    unsigned short v;
    asm volatile("ld.global.nc.u16 %0, [%1];" : "=h"(v) : "l"(p));
    return (int)v;
}
__device__ __forceinline__ float ldg_f32_volatile(const float *p)
{
    float v;
    asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ int lds_u16_volatile(const uint16_t *p)
{
    unsigned short v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(smem_u32(p)));
    return (int)v;
}

constexpr int NSLICE = 2;  // ring depth per warp (quadrature-point slices)

template <int ET, typename R> struct Slice {
    static constexpr int NPE = Elem<ET>::NPE;
    static constexpr int ROWS = NPE * 3 + 1;
    static constexpr uint32_t BYTES = ROWS * 32 * sizeof(R);  // multiple of 128
};

// per-element affine record of a tile: J^{-1} (row-major, 9 rows) and det J, [10][32]
template <typename R> struct AffRec {
    static constexpr int ROWS = AFF_ROWS;
    static constexpr uint32_t BYTES = ROWS * 32 * sizeof(R);  // multiple of 16
};

// element-vector slots of a tile. Wide slots (FP32, but for the diagonal and
// for T4 with one output field) hold the vectors of all output fields, one
// 16-byte slot (x, y, z of the first field, x of the second) and for two
// fields one 8-byte slot (y, z of the second) per position; the others one
// field at a time, [position][3]. The T4 force alone is slower with wide slots
// (34.2 against 32.8 us on 849k elements): its four positions a lane leave no
// instructions to save against the larger slots' bank conflicts.
template <int ET, typename R, int OP> __host__ __device__ constexpr bool wide_slots()
{
    return sizeof(R) == 4 && OP != OP_DIAG && (ET != ET_T4 || OpFields<OP>::NFO == 2);
}
template <int ET, typename R, int OP> __host__ __device__ constexpr size_t slot_bytes()
{
    const size_t n = (size_t)Elem<ET>::NPE * 32;
    if (wide_slots<ET, R, OP>()) return n * (OpFields<OP>::NFO == 2 ? 24 : 16);
    return n * 3 * sizeof(R);
}

// FP32 affine T10 blocks run the point records of k_t10.cuh (all but the
// diagonal): per lane the gradients of the fields at four points, u, udot
// where the material mode is damped (or not known) and the direction
template <typename R> __host__ __device__ constexpr bool t10_path(int et, int op, bool aff)
{
    return sizeof(R) == 4 && et == ET_T10 && aff && op != OP_DIAG;
}
__host__ __device__ constexpr bool mat_damped(int mat) { return mat == MAT_ANY || mat == MAT_NH_KV || mat == MAT_SVK_KV; }
__host__ __device__ constexpr int t10_fields(int op, int mat) { return op_in_fields(op) / 3 - (mat_damped(mat) ? 0 : 1); }

// FP32 affine H8 blocks run on the coefficients of the trilinear fields
// (k_h8.cuh), all but the diagonal: per lane 7 x 3 values a field, and the sum
// of the direction's nodal values for the mass term
template <typename R> __host__ __device__ constexpr bool h8_path(int et, int op, bool aff)
{
    return sizeof(R) == 4 && et == ET_H8 && aff && op != OP_DIAG;
}
// whether its points are evaluated two at a time: where the state of two
// points and the accumulators fit the registers
__host__ __device__ constexpr bool h8_pairs(int op, int mat) { return mat != MAT_ANY && (op == OP_FORCE || (op == OP_MATVEC && mat == MAT_SVK)); }

// T10 and H8 blocks on those paths read the per-lane tables of a tile (local
// indices, slot positions, affine record) once each, straight from global
// memory: of the metadata record only the head (unique-node count, element
// ids, node list) and the node offsets at its end go through shared memory
template <typename R> __host__ __device__ constexpr bool column_path(int et, int op, bool aff)
{
    return t10_path<R>(et, op, aff) || h8_path<R>(et, op, aff);
}
__host__ __device__ constexpr int meta_head_bytes(int umaxp) { return 16 + 128 + 4 * umaxp; }
__host__ __device__ constexpr int meta_lane_bytes(int npe) { return 2 * npe * 32 * 2; }  // local indices, positions

// shared memory of one warp: slice ring (isoparametric path only), two
// metadata buffers (each followed, on the affine path, by the tile's affine
// record), and a work area holding first the node patch [umax][REC] and later
// the element-vector slots; rounded up to 128 bytes so that every bulk-copy
// destination stays 16-byte aligned. On the T10 path the work area also holds,
// between the two, the lanes' J^{-1} [9][32], their point records [2][9 fields][32] float2 and, with
// a mass term (`mass`), behind them the lanes' mass vectors [30][32]; on the
// H8 path the lanes' J^{-1} and coefficients.
template <int ET, typename R, int OP, bool AFF>
__host__ __device__ constexpr size_t warp_region_bytes(int umax, int meta_bytes, int mat, bool mass)
{
    const size_t patch = (size_t)umax * Rec<OP, R>::REC * sizeof(R);
    const size_t slots = slot_bytes<ET, R, OP>();
    const size_t ring = AFF ? 0 : (size_t)NSLICE * Slice<ET, R>::BYTES;
    const size_t mrec = column_path<R>(ET, OP, AFF) ? (size_t)meta_bytes - meta_lane_bytes(Elem<ET>::NPE)
                                                    : (size_t)meta_bytes + (AFF ? AffRec<R>::BYTES : 0);
    size_t work = patch > slots ? patch : slots;
    if (t10_path<R>(ET, OP, AFF)) {
        const size_t rec = ((size_t)9 + 4 * 9 * t10_fields(OP, mat) + (mass ? 30 : 0)) * 32 * sizeof(R);
        work = work > rec ? work : rec;
    }
    if (h8_path<R>(ET, OP, AFF)) {
        const size_t c = ((size_t)9 + 21 * t10_fields(OP, mat) + 3) * 32 * sizeof(R);
        work = work > c ? work : c;
    }
    return (ring + 2 * mrec + work + 127) / 128 * 128;
}

// dynamic shared memory of one CTA with `wpb` warps (mbarriers, then the warp regions)
constexpr size_t cta_smem_bytes(size_t region, int wpb) { return 128 + (size_t)wpb * region; }

// 3-vectors at compile-time offsets of a 16-byte-aligned shared record, with
// the widest aligned vector accesses the offset allows
template <int OFF> __device__ __forceinline__ void ld3c(const float *r, float &x, float &y, float &z)
{
    if constexpr (OFF % 4 == 0) {
        const float4 v = *reinterpret_cast<const float4 *>(r + OFF);
        x = v.x, y = v.y, z = v.z;
    } else if constexpr (OFF % 4 == 2) {
        const float2 v = *reinterpret_cast<const float2 *>(r + OFF);
        x = v.x, y = v.y, z = r[OFF + 2];
    } else {
        const float2 v = *reinterpret_cast<const float2 *>(r + OFF + 1);
        x = r[OFF], y = v.x, z = v.y;
    }
}
template <int OFF> __device__ __forceinline__ void ld3c(const double *r, double &x, double &y, double &z)
{
    if constexpr (OFF % 2 == 0) {
        const double2 v = *reinterpret_cast<const double2 *>(r + OFF);
        x = v.x, y = v.y, z = r[OFF + 2];
    } else {
        const double2 v = *reinterpret_cast<const double2 *>(r + OFF + 1);
        x = r[OFF], y = v.x, z = v.y;
    }
}
template <int OFF> __device__ __forceinline__ void st3c(float *r, float x, float y, float z)
{
    if constexpr (OFF % 4 == 0) {
        *reinterpret_cast<float4 *>(r + OFF) = make_float4(x, y, z, 0.f);
    } else if constexpr (OFF % 4 == 2) {
        *reinterpret_cast<float2 *>(r + OFF) = make_float2(x, y);
        r[OFF + 2] = z;
    } else {
        r[OFF] = x;
        *reinterpret_cast<float2 *>(r + OFF + 1) = make_float2(y, z);
    }
}
template <int OFF> __device__ __forceinline__ void st3c(double *r, double x, double y, double z)
{
    if constexpr (OFF % 2 == 0) {
        *reinterpret_cast<double2 *>(r + OFF) = make_double2(x, y);
        r[OFF + 2] = z;
    } else {
        r[OFF] = x;
        *reinterpret_cast<double2 *>(r + OFF + 1) = make_double2(y, z);
    }
}
// FP64 displacement of a record (the FP32 kernels read their (h, l) pairs
// from the paired slots directly)
__device__ __forceinline__ void ld_u(const double *r, double h[3], double l[3])
{
    ld3c<0>(r, h[0], h[1], h[2]);
    l[0] = l[1] = l[2] = 0.0;
}

// x = hi + lo to about 2^-46 |x| with hi, lo in FP32, by integer and FP32
// operations only (the FP64 pipe of this GPU runs at a small fraction of the
// FP32 rate): hi keeps the leading 24 significant bits of x (exact in FP32),
// lo the next 23 bits scaled by 2^(e - 46). |x| < 2^-126 gives (+-0, +-0);
// |x| >= 2^128, inf and NaN fall back to the plain FP32 rounding with lo = 0.
__device__ __forceinline__ void split_f64(double x, float &hi, float &lo)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const unsigned hw = (unsigned)(b >> 32), lw = (unsigned)b;
    const unsigned sign = hw & 0x80000000u;
    const int e = (int)((hw >> 20) & 0x7FFu) - 1023;  // unbiased binary exponent
    if (e < -126) {
        hi = __uint_as_float(sign);
        lo = __uint_as_float(sign);
    } else if (e <= 127) {
        const unsigned mhi = ((hw & 0xFFFFFu) << 3) | (lw >> 29);  // significand bits 51..29
        hi = __uint_as_float(sign | ((unsigned)(e + 127) << 23) | mhi);
        const unsigned r = (lw >> 6) & 0x7FFFFFu;                   // significand bits 28..6
        const float rf = __uint_as_float(0x4B000000u | r) - 8388608.0f;  // = r exactly
        const float sc = e >= -80 ? __uint_as_float((unsigned)(e + 81) << 23) : 0.0f;  // 2^(e - 46)
        lo = __uint_as_float(sign | __float_as_uint(rf * sc));
    } else {
        hi = (float)x;
        lo = 0.0f;
    }
}

// bounded wait on an mbarrier phase; returns false when the limit ran out
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, uint32_t parity)
{
    long long spins = 0;
    while (!mbar_try_wait(bar, parity))
        if (++spins > MBAR_SPIN_LIMIT) return false;
    return true;
}

// Resident CTAs (of 4 warps) per SM the register allocation aims at, by
// measurement. Column paths (affine T10 and H8): 12 warps in 168 registers
// with at most a few spilled values, the force 16 warps in 128; the generic
// law keeps 8 warps and all its registers. Slab T10 adjoint and force +
// operator product: 8 warps at 255 registers; at 12 warps they spill 150-210
// bytes and the curved T10 step (194k elements) takes 158 us instead of 137.
// So too with damped Saint Venant-Kirchhoff (323k: 208 -> 195 us) and the
// undamped neo-Hookean law (323k: 201 -> 195); undamped Saint Venant-Kirchhoff
// spills little and keeps 12 warps (99k: 64.3 us at 8, 58.6 at 12; 960k: 435
// and 425).
// The damped neo-Hookean law alone also gains by that in the H8 adjoint and
// one pass (step of 140k bricks 111.0 -> 106.8 us; 86.7 -> 92.4 without
// damping). Not so the slab T10 operator product, which spills less: at 8
// warps 62 us instead of 64.5 on 194k elements, but 267 instead of 254 on 960k.
// T4, and H8 on the slab: 12 warps where the law's state fits 168 registers.
// FP64 kernels take all 255 registers, and so do Q27 kernels (81-entry element
// vectors; their shared-memory footprint limits the resident warps anyway).
template <int ET, typename R, int OP, bool AFF, int MAT> constexpr int min_ctas()
{
    if (sizeof(R) != 4 || ET == ET_Q27) return 1;
    if (h8_path<R>(ET, OP, AFF) && (OP == OP_FM || OP == OP_VJP) && MAT == MAT_NH_KV) return 2;
    if (t10_path<R>(ET, OP, AFF) || h8_path<R>(ET, OP, AFF)) return OP == OP_FORCE ? 4 : (MAT == MAT_ANY ? 2 : 3);
    if (OP == OP_VJP || OP == OP_FM) {
        if (ET == ET_T10) return MAT == MAT_SVK ? 3 : 2;
        return ET == ET_T4 || MAT != MAT_ANY ? 3 : 2;
    }
    return (OP == OP_FORCE && AFF) ? 4 : 3;
}

__device__ __forceinline__ void mbar_inval(uint64_t *bar)
{
    asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// The work of one warp on the tiles t0, t0 + tstep, ... (n_my of them) of
// the pass described by p: wbase is the warp's shared-memory region (laid out
// by warp_region_bytes) and bar its NSLICE + 2 mbarriers, freshly initialised
// by the caller (every phase count starts at 0). Returns false when a bounded
// wait ran out (the status word has the timeout, and every copy the warp had
// in flight has been waited for).
template <int ET, int NQ, typename R, int OP, bool AFF, int MAT>
__device__ __forceinline__ bool elem_tiles(const KParams<R> &p, unsigned char *wbase, uint64_t *bar, int t0,
                                           int tstep, int n_my)
{
    constexpr int NPE = Elem<ET>::NPE;
    using RC = Rec<OP, R>;
    constexpr int REC = RC::REC;
    constexpr int OFF_UD = RC::OFF_UD;
    constexpr int OFF_V = RC::OFF_V;
    constexpr bool PK = RC::PK;                        // FP32: paired (x, y) arithmetic
    constexpr bool PKA = PK && OP != OP_DIAG;          // ... and paired element-vector accumulators
    constexpr int NFO = OpFields<OP>::NFO;
    constexpr bool HAS_V = OpFields<OP>::NFI == 3;
    constexpr bool DD_REG = OP == OP_FORCE || OP == OP_DIAG;
    using SL = Slice<ET, R>;
    constexpr int ROWS = SL::ROWS;
    using PG = ParentGrad<ET, NQ, R>;
    constexpr uint32_t AB = AFF ? AffRec<R>::BYTES : 0;
    constexpr bool T10R = t10_path<R>(ET, OP, AFF);    // point records (k_t10.cuh)
    constexpr bool H8C = h8_path<R>(ET, OP, AFF);      // trilinear coefficients (k_h8.cuh)
    constexpr bool LANECOL = T10R || H8C;  // the lane keeps its fields in its own shared column
    constexpr bool PF_EARLY = AFF && OP != OP_VJP;  // where the next tile's L2 prefetch goes (see prefetch_next)
    constexpr bool PF_NONE = AFF && OP == OP_VJP;
    constexpr bool LI_REREAD = OP == OP_FORCE || OP == OP_VJP || OP == OP_FM;
    // two element vectors per element: the adjoint's (g_u, g_udot) and the
    // fused force + operator product's (f, y)
    constexpr bool TWO = OP == OP_VJP || OP == OP_FM;
    // the adjoint (and the fused force + operator product, which holds as
    // many accumulators) also re-reads J^{-1} (affine record) and node 0's
    // pair at every point: 168 registers without spill (12 warps per SM)
    constexpr bool DIET = OP == OP_VJP || OP == OP_FM;

    const int lane = threadIdx.x & 31;
    const int MB = p.meta_bytes;
    uint64_t *mbar = bar + NSLICE;
    const int HB = meta_head_bytes(p.umaxp), TB = MB - HB - meta_lane_bytes(NPE);  // head, node offsets
    const size_t MRB = LANECOL ? (size_t)(HB + TB) : (size_t)MB + AB;  // bytes of a metadata buffer
    unsigned char *ring = wbase;
    unsigned char *mbuf = wbase + (AFF ? 0 : NSLICE * SL::BYTES);  // [2][MB + AB]
    R *work = reinterpret_cast<R *>(mbuf + 2 * MRB);           // patch [umax][REC], later slots

    const bool mass_only = OP == OP_MATVEC && p.mass_only != 0;
    const int n_slices = (mass_only || AFF) ? 0 : n_my * NQ;
    const bool need_ud = p.visc != 0;

    auto issue = [&](int j) {  // slab slice j of this warp into ring slot j % NSLICE
        const int t = t0 + (j / NQ) * tstep;
        const int q = j % NQ;
        const int b = j % NSLICE;
        mbar_arrive_expect_tx(bar + b, SL::BYTES);
        bulk_g2s(ring + (size_t)b * SL::BYTES, p.slab + ((size_t)t * NQ + q) * ROWS * 32, SL::BYTES, bar + b);
    };
    auto issue_meta = [&](int k) {  // metadata (+ affine record) of the warp's k-th tile into buffer k & 1
        const int t = t0 + k * tstep;
        unsigned char *dst = mbuf + (size_t)(k & 1) * MRB;
        mbar_arrive_expect_tx(mbar + (k & 1), (uint32_t)MRB);
        const unsigned char *src = p.meta + (size_t)t * MB;
        if constexpr (LANECOL) {
            bulk_g2s(dst, src, (uint32_t)HB, mbar + (k & 1));
            bulk_g2s(dst + HB, src + (MB - TB), (uint32_t)TB, mbar + (k & 1));
        } else {
            bulk_g2s(dst, src, (uint32_t)MB, mbar + (k & 1));
        }
        if constexpr (AFF && !LANECOL) bulk_g2s(dst + MB, p.aff + (size_t)t * AffRec<R>::ROWS * 32, AB, mbar + (k & 1));
    };
    if (lane == 0) {
        if (n_my > 0) issue_meta(0);
        for (int j = 0; j < NSLICE && j < n_slices; ++j) issue(j);
    }
    // copies issued and waited for, counted alike in every lane (the issue
    // decisions are warp-uniform): slices j < sl_issued and metadata records
    // k < mt_issued were requested, those below sl_done / mt_done have landed.
    // A barrier never holds more than one outstanding phase (slot b is
    // re-armed only after its previous slice was consumed; record k + 1 is
    // requested only after record k - 1, the previous user of its barrier,
    // was waited for), so the timeout drain below can wait on each
    // outstanding phase by its parity without ambiguity.
    int sl_issued = n_slices < NSLICE ? n_slices : NSLICE, sl_done = 0;
    int mt_issued = n_my > 0 ? 1 : 0, mt_done = 0;

    bool timed_out = false;
    for (int k = 0; k < n_my; ++k) {
        const int t = t0 + k * tstep;
        // ---- metadata of this tile (prefetched one tile ahead)
        if (!mbar_wait_bounded(mbar + (k & 1), (uint32_t)((k >> 1) & 1))) timed_out = true;
        if (__any_sync(0xffffffffu, timed_out)) {
            timed_out = true;
            break;
        }
        mt_done = k + 1;
        if (k + 1 < n_my) {
            if (lane == 0) issue_meta(k + 1);
            mt_issued = k + 2;
        }
        const unsigned char *M = mbuf + (size_t)(k & 1) * MRB;
        const int U = (int)bounds_clamp(*reinterpret_cast<const int32_t *>(M), (int64_t)p.umax + 1, p.status);
        const int e = reinterpret_cast<const int32_t *>(M + 16)[lane];
        const int32_t *nodes = reinterpret_cast<const int32_t *>(M + 16 + 128);
        // in shared memory, or in global memory on the column paths
        const uint16_t *mlidx = reinterpret_cast<const uint16_t *>((LANECOL ? p.meta + (size_t)t * MB : M) + HB);
        const uint16_t *spos = mlidx + NPE * 32;  // slot (i, lane) -> node-sorted position
        // positions of unique node kk: [soff[kk], soff[kk + 1])
        const uint16_t *soff = LANECOL ? reinterpret_cast<const uint16_t *>(M + HB) : spos + NPE * 32;

        // ---- gather the tile's nodal inputs into the patch, one record per
        // unique node: every lane issues asynchronous copies (cp.async) for all
        // of its nodes before waiting once, so that the load latencies of the
        // whole tile overlap without holding registers; FP32 kernels then
        // split the FP64 displacement in place into its (hi, lo) pair (both
        // take the same 24 bytes of the record)
        for (int kk = lane; kk < U; kk += 32) {
            const int64_t n = bounds_clamp(nodes[kk], p.n_nodes, p.status);
            R *rec = work + (size_t)kk * REC;
#pragma unroll
            for (int a = 0; a < 3; ++a) cp_async<8>(reinterpret_cast<double *>(rec) + a, p.u + 3 * n + a);
            if constexpr (PK) {
                if (need_ud) {
                    cp_async<4>(rec + RC::UD01, p.ud + 3 * n);
                    cp_async<4>(rec + RC::UD01 + 1, p.ud + 3 * n + 1);
                    cp_async<4>(rec + RC::UD2, p.ud + 3 * n + 2);
                }
                if (HAS_V) {
                    cp_async<4>(rec + RC::V01, p.v + 3 * n);
                    cp_async<4>(rec + RC::V01 + 1, p.v + 3 * n + 1);
                    cp_async<4>(rec + RC::V2, p.v + 3 * n + 2);
                }
            } else {
                if (need_ud)
#pragma unroll
                    for (int a = 0; a < 3; ++a) cp_async<sizeof(R)>(rec + OFF_UD + a, p.ud + 3 * n + a);
                if (HAS_V)
#pragma unroll
                    for (int a = 0; a < 3; ++a) cp_async<sizeof(R)>(rec + OFF_V + a, p.v + 3 * n + a);
            }
        }
        cp_async_commit();
        int li[NPE];
        R Ji[9], detJ = R(0);  // affine path: J^{-1} and det J of this lane's element (Sec. 6, affine case)
        if constexpr (LANECOL) {  // in flight together with the gather
#pragma unroll
            for (int i = 0; i < NPE; ++i) li[i] = ldg_u16_volatile(mlidx + i * 32 + lane);
            const R *A = p.aff + (size_t)t * AFF_ROWS * 32 + lane;
#pragma unroll
            for (int r = 0; r < 9; ++r) Ji[r] = ldg_f32_volatile(A + r * 32);
            detJ = ldg_f32_volatile(A + 9 * 32);
        }
        cp_async_wait<0>();
        if constexpr (PK) {
            for (int kk = lane; kk < U; kk += 32) {
                R *rec = work + (size_t)kk * REC;
                const double2 u01 = *reinterpret_cast<const double2 *>(rec);
                const double u2 = reinterpret_cast<const double *>(rec)[2];
                float h[3], l[3];
                split_f64(u01.x, h[0], l[0]);
                split_f64(u01.y, h[1], l[1]);
                split_f64(u2, h[2], l[2]);
                *reinterpret_cast<float4 *>(rec) = make_float4(h[0], h[1], l[0], l[1]);
                *reinterpret_cast<float2 *>(rec + RC::H2) = make_float2(h[2], l[2]);
            }
        }
#pragma unroll
        for (int i = 0; i < NPE; ++i) li[i] = (int)bounds_clamp(LANECOL ? li[i] : mlidx[i * 32 + lane], U, p.status);
        const bool valid = e >= 0;
        Mat<R> m = p.mat0;
        if (p.mats) m = p.mats[bounds_clamp(p.emat[(size_t)t * 32 + lane], p.n_mats, p.status)];
        if (p.elam) {
            m.mu = p.elam[((size_t)t * 2 + 0) * 32 + lane];
            m.lam = p.elam[((size_t)t * 2 + 1) * 32 + lane];
        }
        // material: the law and the presence of the viscous term are
        // compile-time constants when the block allows (MAT != MAT_ANY)
        if constexpr (MAT == MAT_NH || MAT == MAT_NH_KV) m.model = MODEL_NH;
        if constexpr (MAT == MAT_SVK || MAT == MAT_SVK_KV) m.model = MODEL_SVK;
        const bool visc = MAT == MAT_ANY ? (need_ud && (m.mu_v != R(0) || m.lam_v != R(0)))
                                         : (MAT == MAT_NH_KV || MAT == MAT_SVK_KV);
        if constexpr (AFF && !LANECOL) {
            const R *A = reinterpret_cast<const R *>(M + MB) + lane;
#pragma unroll
            for (int r = 0; r < 9; ++r) Ji[r] = A[r * 32];
            detJ = A[9 * 32];
        }
        __syncwarp();

        // element-relative displacements d_i = u_i - u_0 (sum_i h_i = 0, so
        // G = sum_i u_i h_i^T = sum_{i>0} d_i h_i^T, with rigid translation
        // removed exactly). Kept in registers by the force and diagonal
        // kernels; the operator and adjoint kernels, which hold more
        // accumulators, re-form them from the patch at every point.
        R h0v[3], l0v[3];
        R dd[NPE][3];
        // FP32: node 0's pair, negated, with x and y paired; d_i = (h_i - h_0)
        // + (l_i - l_0) as (h_i + (-h_0)) + (l_i + (-l_0)), the same roundings
        float2 nh01 = make_float2(0.f, 0.f), nl01 = make_float2(0.f, 0.f), dp[NPE];
        float nh2 = 0.f, nl2 = 0.f;
        if constexpr (LANECOL) {
            // formed where the nodes are read, below
        } else if constexpr (PK) {
            const float4 A = lds4(work + li[0] * REC), B = lds4(work + li[0] * REC + 4);
            nh01 = make_float2(-A.x, -A.y);
            nl01 = make_float2(-A.z, -A.w);
            nh2 = -B.x;
            nl2 = -B.y;
        } else {
            ld_u(work + li[0] * REC, h0v, l0v);
        }
        if constexpr (DD_REG && !LANECOL) {
#pragma unroll
            for (int i = 1; i < NPE; ++i) {
                if constexpr (PK) {
                    const float4 A = lds4(work + li[i] * REC), B = lds4(work + li[i] * REC + 4);
                    dp[i] = add2(add2(make_float2(A.x, A.y), nh01), add2(make_float2(A.z, A.w), nl01));
                    dd[i][2] = (B.x + nh2) + (B.y + nl2);
                } else {
                    R hv[3], lv[3];
                    ld_u(work + li[i] * REC, hv, lv);
#pragma unroll
                    for (int a = 0; a < 3; ++a) dd[i][a] = (hv[a] - h0v[a]) + (lv[a] - l0v[a]);
                }
            }
        }
        // element vectors: FP32 keeps (x, y) of each node as a pair and z alone
        R acc0[NPE][3], acc1[NPE][3];
        float2 ap0[NPE], ap1[NPE];
#pragma unroll
        for (int i = 0; i < NPE; ++i) {
            if constexpr (PKA) {
                ap0[i] = make_float2(0.f, 0.f);
                acc0[i][2] = R(0);
                if (TWO) {
                    ap1[i] = make_float2(0.f, 0.f);
                    acc1[i][2] = R(0);
                }
            } else {
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    acc0[i][d] = R(0);
                    if (TWO) acc1[i][d] = R(0);
                }
            }
        }
        R gmu_acc = R(0), glam_acc = R(0);
        int bad = 0;
        int sp[NPE];  // column paths: slot positions, loaded ahead of their use
        auto load_positions = [&]() {
#pragma unroll
            for (int i = 0; i < NPE; ++i) sp[i] = ldg_u16_volatile(spos + i * 32 + lane);
        };

        // ---- the next tile's nodal inputs towards L2 (its metadata was
        // requested at the start of this tile); false when that metadata never
        // landed. Issued after this tile's first point on the affine path
        // (force, operator, diagonal), after the last on the slab path, and
        // not at all by the affine adjoint: measured on the beam, the early
        // prefetch cut the affine K v kernel by 18 % and the force by 12 %,
        // and slowed the slab path; the affine adjoint runs 4-5 % faster
        // without it than with it early or late, also with the L2 flushed
        // before the launch. (The tile-start wait on the metadata barrier
        // stands without it.)
        // the next tile's per-lane tables towards L2 (column paths): the
        // 128-byte lines of its local indices and positions, and of its affine record
        auto prefetch_tables = [&]() {
            if constexpr (LANECOL) {
                if (k + 1 >= n_my) return;
                constexpr int NL = (meta_lane_bytes(NPE) + 127) / 128 + 1, NA = (int)(AffRec<R>::BYTES / 128);
                const size_t tn = (size_t)(t + tstep);
                if (lane < NL) prefetch_l2(p.meta + tn * MB + HB + min(lane * 128, meta_lane_bytes(NPE) - 1));
                else if (lane < NL + NA) prefetch_l2(reinterpret_cast<const unsigned char *>(p.aff + tn * AFF_ROWS * 32) + (lane - NL) * 128);
            }
        };
        auto prefetch_next = [&]() -> bool {
            if (k + 1 >= n_my) return true;
            const bool ok = mbar_wait_bounded(mbar + ((k + 1) & 1), (uint32_t)(((k + 1) >> 1) & 1));
            if (__any_sync(0xffffffffu, !ok)) return false;
            const unsigned char *Mn = mbuf + (size_t)((k + 1) & 1) * MRB;
            const int Un = *reinterpret_cast<const int32_t *>(Mn);
            const int32_t *nodes_n = reinterpret_cast<const int32_t *>(Mn + 16 + 128);
            for (int kk = lane; kk < Un; kk += 32) {
                const int64_t n = nodes_n[kk];
                prefetch_l2(p.u + 3 * n);
                if (need_ud) prefetch_l2(p.ud + 3 * n);
                if (HAS_V) prefetch_l2(p.v + 3 * n);
            }
            prefetch_tables();
            return true;
        };

        // ---- FP32 affine T10 and H8: the fields of the lane's element in its
        // own shared column, the points two at a time (and the centroid of the
        // T10 rule alone), the element vectors from the points' operators
        // (k_t10.cuh, k_h8.cuh)
        if constexpr (LANECOL) {
            constexpr int NF = t10_fields(OP, MAT);  // fields held: u, [udot,] [the direction]
            constexpr int FV = NF - 1;
            constexpr bool DAMPED = mat_damped(MAT);
            float *Aj = work + lane;          // the lane's J^{-1}, read again where it is used
            float *const cols = Aj + 9 * 32;  // the lane's columns
            // nodal values: displacements relative to node 0 (pair by pair),
            // velocities, the direction. The columns go over the patch: every
            // lane reads all of its nodes first
            auto nodal = [&](V3f(*x)[NPE]) {
                float4 A0 = make_float4(0.f, 0.f, 0.f, 0.f), B0 = A0;
#pragma unroll
                for (int i = 0; i < NPE; ++i) {
                    const float *rc = work + li[i] * REC;
                    const float4 A = lds4(rc), B = lds4(rc + 4);
                    if (i == 0) {
                        A0 = A;
                        B0 = B;
                        x[0][0] = {make_float2(0.f, 0.f), 0.f};
                    } else {
                        x[0][i] = {add2(add2(make_float2(A.x, A.y), make_float2(-A0.x, -A0.y)),
                                        add2(make_float2(A.z, A.w), make_float2(-A0.z, -A0.w))),
                                   (B.x - B0.x) + (B.y - B0.y)};
                    }
                    if constexpr (NF > 1) {
                        const float4 C4 = lds4(rc + 8);
                        if constexpr (DAMPED) x[1][i] = {make_float2(C4.x, C4.y), B.z};
                        if constexpr (HAS_V) x[FV][i] = {make_float2(C4.z, C4.w), B.w};
                    }
                }
                if constexpr (DAMPED)
                    if (!need_ud)  // the generic law without a velocity: its slots hold nothing
#pragma unroll
                        for (int i = 0; i < NPE; ++i) x[1][i] = {make_float2(0.f, 0.f), 0.f};
                __syncwarp();
#pragma unroll
                for (int r = 0; r < 9; ++r) Aj[r * 32] = Ji[r];
            };
            // state and operators of one point or two (V), from the gradients g
            // of the fields (9 each)
            auto point = [&](auto *g, auto *T0, auto *T1, R w) {
                using V = typename std::remove_pointer<decltype(g)>::type;
                QP<V> s1;
                V D[9];
#pragma unroll
                for (int k2 = 0; k2 < 9; ++k2) {
                    s1.G[k2] = g[k2];
                    s1.Fd[k2] = DAMPED ? g[9 + k2] : V(0.f);
                    D[k2] = HAS_V ? g[FV * 9 + k2] : V(0.f);
                }
                stress_state<R>(m, s1, visc);
                if constexpr (OP == OP_FORCE || OP == OP_FM) first_piola(s1, visc, T0);
                if constexpr (OP == OP_MATVEC) dstress<R>(m, s1, visc, D, p.aK, p.aC, p.sym_only != 0, T0);
                if constexpr (OP == OP_FM) dstress<R>(m, s1, visc, D, p.aK, p.aC, false, T1);
                if constexpr (OP == OP_VJP) {
                    V gmu, glam;
                    astress<R>(m, s1, visc, D, T0, T1, gmu, glam);
                    gmu_acc += w * sum_of(gmu);
                    glam_acc += w * sum_of(glam);
                }
                bad += valid ? count_not(s1.ok) : 0;
            };
            auto store = [&](int fo, const V3f *F) {
#pragma unroll
                for (int i = 0; i < NPE; ++i) {
                    (fo == 0 ? ap0 : ap1)[i] = F[i].xy;
                    (fo == 0 ? acc0 : acc1)[i][2] = F[i].z;
                }
            };
            if constexpr (T10R) {
            constexpr int NV = 9 * NF;
            float2 *rec = reinterpret_cast<float2 *>(work + 9 * 32) + lane;
            float *stash = cols + 4 * NV * 32;  // the lane's mass vector
            if (!mass_only) {
                float g0[NV];
                {
                    V3f x[NF][NPE];
                    nodal(x);
#pragma unroll
                    for (int f = 0; f < NF; ++f) t10_gradients<NQ, NV>(x[f], Ji, rec + f * 9 * 32, g0 + f * 9);
                    if constexpr (HAS_V)
                        if (p.aM != R(0)) {
                            V3f y[NPE];
                            t10_mass(x[FV], p.aM * m.rho * p.evol[(size_t)t * 32 + lane], y);
#pragma unroll
                            for (int i = 0; i < NPE; ++i) {
                                stash[(i * 3) * 32] = y[i].xy.x;
                                stash[(i * 3 + 1) * 32] = y[i].xy.y;
                                stash[(i * 3 + 2) * 32] = y[i].z;
                            }
                        }
                }
                if constexpr (PF_NONE) prefetch_tables();
                if (PF_EARLY && !prefetch_next()) {
                    timed_out = true;
                    break;
                }
                constexpr float w1 = float(T10Rule<NQ>::w), w0 = float(T10Rule<NQ>::w0);
                float c0[TWO ? 18 : 9];  // the centroid's operators in units of the other points' weight
#pragma unroll
                for (int k2 = 0; k2 < (TWO ? 18 : 9); ++k2) c0[k2] = 0.f;
                if constexpr (NQ == 5) {
                    float T0[9], T1[9];
                    point(g0, T0, T1, w0 * detJ);
                    constexpr float c = float(T10Rule<NQ>::w0 / (4.0 * T10Rule<NQ>::w));
#pragma unroll
                    for (int k2 = 0; k2 < 9; ++k2) {
                        c0[k2] = c * T0[k2];
                        if constexpr (TWO) c0[9 + k2] = c * T1[k2];
                    }
                }
#pragma unroll 1
                for (int h = 0; h < 2; ++h) {
                    float2 *rh = rec + h * NV * 32;
                    F2 g[NV], T0[9], T1[9];
#pragma unroll
                    for (int k2 = 0; k2 < NV; ++k2) g[k2] = rh[k2 * 32];
                    point(g, T0, T1, w1 * detJ);
#pragma unroll
                    for (int k2 = 0; k2 < 9; ++k2) {
                        rh[k2 * 32] = NQ == 5 ? add2(T0[k2].v, bc2(c0[k2])) : T0[k2].v;
                        if constexpr (TWO) rh[(9 + k2) * 32] = NQ == 5 ? add2(T1[k2].v, bc2(c0[9 + k2])) : T1[k2].v;
                    }
                }
                load_positions();
                float Jw[9];
#pragma unroll
                for (int r = 0; r < 9; ++r) Jw[r] = (w1 * detJ) * Aj[r * 32];
#pragma unroll
                for (int fo = 0; fo < NFO; ++fo) {
                    V3f F[NPE];
                    t10_vectors<NQ, NV>(rec + fo * 9 * 32, Jw, F);
                    store(fo, F);
                }
            }
            // the mass vector of the lane's element into the operator product
            // (the second element vector of OP_FM): stashed before the points,
            // or formed here from the patch where there are none
            if constexpr (OP == OP_MATVEC || OP == OP_FM)
                if (p.aM != R(0)) {
                    float2 *apy = OP == OP_FM ? ap1 : ap0;
                    R(*accy)[3] = OP == OP_FM ? acc1 : acc0;
                    if (mass_only) {
                        load_positions();
                        V3f xv[NPE], y[NPE];
#pragma unroll
                        for (int i = 0; i < NPE; ++i) {
                            const float *rc = work + li[i] * REC;
                            xv[i] = {*reinterpret_cast<const float2 *>(rc + RC::V01), rc[RC::V2]};
                        }
                        t10_mass(xv, p.aM * m.rho * p.evol[(size_t)t * 32 + lane], y);
#pragma unroll
                        for (int i = 0; i < NPE; ++i) {
                            apy[i] = y[i].xy;
                            accy[i][2] = y[i].z;
                        }
                    } else {
#pragma unroll
                        for (int i = 0; i < NPE; ++i) {
                            apy[i] = add2(apy[i], make_float2(stash[(i * 3) * 32], stash[(i * 3 + 1) * 32]));
                            accy[i][2] += stash[(i * 3 + 2) * 32];
                        }
                    }
                }
            }
            if constexpr (H8C) {
                float *col = cols;  // [NF][7][3] coefficients, then the direction's sum
                float *vsum = col + 21 * NF * 32;
                {
                    V3f x[NF][NPE];
                    nodal(x);
#pragma unroll
                    for (int f = 0; f < NF; ++f) {
                        h8_transform(x[f]);
#pragma unroll
                        for (int c = 1; c < 8; ++c) {
                            const V3f v = x[f][c] * h8_scale(c);
                            float *o = col + (f * 21 + (c - 1) * 3) * 32;
                            o[0] = v.xy.x;
                            o[32] = v.xy.y;
                            o[64] = v.z;
                        }
                    }
                    if constexpr (HAS_V) {
                        vsum[0] = x[FV][0].xy.x;
                        vsum[32] = x[FV][0].xy.y;
                        vsum[64] = x[FV][0].z;
                    }
                }
                if constexpr (PF_NONE) prefetch_tables();
                if (PF_EARLY && !mass_only && !prefetch_next()) {
                    timed_out = true;
                    break;
                }
                V3f C[NFO][8];
#pragma unroll
                for (int fo = 0; fo < NFO; ++fo)
#pragma unroll
                    for (int c = 0; c < 8; ++c) C[fo][c] = {make_float2(0.f, 0.f), 0.f};
                constexpr bool PAIR = h8_pairs(OP, MAT);
                using V = typename std::conditional<PAIR, F2, float>::type;
#pragma unroll 1
                for (int q = 0; q < (mass_only ? 0 : (PAIR ? 4 : 8)); ++q) {
                    const float sy = (q & 1) ? 1.f : -1.f, sz = (q & 2) ? 1.f : -1.f;
                    V sx, g[9 * NF], T0[9], T1[9];
                    if constexpr (PAIR) sx = F2(make_float2(-1.f, 1.f));
                    else sx = (q & 4) ? 1.f : -1.f;
                    {
                        float J[9];
#pragma unroll
                        for (int r = 0; r < 9; ++r) J[r] = Aj[r * 32];
#pragma unroll
                        for (int f = 0; f < NF; ++f) h8_gradients<V>(col + f * 21 * 32, sx, sy, sz, J, g + f * 9);
                    }
                    point(g, T0, T1, detJ);
                    h8_accumulate<V>(T0, sx, sy, sz, Aj, detJ, C[0]);
                    if constexpr (TWO) h8_accumulate<V>(T1, sx, sy, sz, Aj, detJ, C[1]);
                }
                load_positions();
#pragma unroll
                for (int fo = 0; fo < NFO; ++fo) {
#pragma unroll
                    for (int c = 1; c < 8; ++c) C[fo][c] = C[fo][c] * h8_scale(c);
                    if constexpr (OP == OP_MATVEC || OP == OP_FM)
                        if (fo == NFO - 1 && p.aM != R(0)) {
                            const float r = p.aM * m.rho * p.evol[(size_t)t * 32 + lane];
#pragma unroll
                            for (int c = 0; c < 8; ++c) {
                                const float *o = c == 0 ? vsum : col + (FV * 21 + (c - 1) * 3) * 32;
                                const float s = r * float(c == 0 ? h8_mass(0) : h8_mass(c) / h8_scale(c));
                                C[fo][c] = C[fo][c].fma(s, V3f{make_float2(o[0], o[32]), o[64]});
                            }
                        }
                    h8_transform_t(C[fo]);
                    store(fo, C[fo]);
                }
            }
        }

#pragma unroll 1
        for (int q = 0; q < (LANECOL || mass_only ? 0 : NQ); ++q) {
            // reference gradients of this point: the slab slice (isoparametric
            // path), or the parent gradients g_i with h_i = J^{-T} g_i (affine path)
            const R *sl = nullptr;
            PG pg;
            R w;
            if constexpr (AFF) {
                pg.at(q);
                w = quad_weight<ET, NQ, R>(q) * detJ;
            } else {
                const int j = k * NQ + q;
                const int b = j % NSLICE;
                if (!mbar_wait_bounded(bar + b, (uint32_t)((j / NSLICE) & 1))) timed_out = true;
                if (__any_sync(0xffffffffu, timed_out)) {
                    timed_out = true;
                    break;
                }
                sl_done = j + 1;
                sl = reinterpret_cast<const R *>(ring + (size_t)b * SL::BYTES) + lane;
                w = sl[NPE * 3 * 32];
            }
            // gradient entry k of node i; nz(i, k) = false where it vanishes identically
            auto grad = [&](int i, int k2) -> R { return AFF ? pg.g(i, k2) : sl[(i * 3 + k2) * 32]; };
            auto nz = [&](int i, int k2) -> bool { return !AFF || PG::nz(i, k2); };

            // kinematics: G = sum d_i h_i^T, Fd = sum udot_i h_i^T, D = sum v_i h_i^T
            // (affine path: the same sums against g_i, then times J^{-1})
            QP<R> s1;
            R D[9];
            if constexpr (PK) {
                // rows 0 and 1 of G', Fd', D' paired per column k, row 2 alone
                if constexpr (DIET && !DD_REG) {  // node 0's negated pair, read again for this point
                    const int l0 = (int)bounds_clamp(lds_u16_volatile(mlidx + lane), U, p.status);
                    const float4 A0 = lds4_volatile(work + l0 * REC), B0 = lds4_volatile(work + l0 * REC + 4);
                    nh01 = make_float2(-A0.x, -A0.y);
                    nl01 = make_float2(-A0.z, -A0.w);
                    nh2 = -B0.x;
                    nl2 = -B0.y;
                }
                float2 Gp[3], Fp[3], Dp[3];
                float Gs[3], Fs[3], Ds[3];
#pragma unroll
                for (int k2 = 0; k2 < 3; ++k2) {
                    Gp[k2] = Fp[k2] = Dp[k2] = make_float2(0.f, 0.f);
                    Gs[k2] = Fs[k2] = Ds[k2] = 0.f;
                }
#pragma unroll
                for (int i = 0; i < NPE; ++i) {
                    R hk[3];
#pragma unroll
                    for (int k2 = 0; k2 < 3; ++k2) hk[k2] = nz(i, k2) ? grad(i, k2) : R(0);
                    const int lii = LI_REREAD ? (int)bounds_clamp(lds_u16_volatile(mlidx + i * 32 + lane), U, p.status)
                                              : li[i];
                    const float *rec = work + lii * REC;
                    float4 B = make_float4(0.f, 0.f, 0.f, 0.f);
                    if ((i > 0 && !DD_REG) || visc || HAS_V) B = lds4(rec + 4);
                    if (i > 0) {
                        float2 d01;
                        float d2;
                        if constexpr (DD_REG) {
                            d01 = dp[i];
                            d2 = dd[i][2];
                        } else {
                            const float4 A = lds4(rec);
                            d01 = add2(add2(make_float2(A.x, A.y), nh01), add2(make_float2(A.z, A.w), nl01));
                            d2 = (B.x + nh2) + (B.y + nl2);
                        }
#pragma unroll
                        for (int k2 = 0; k2 < 3; ++k2)
                            if (nz(i, k2)) {
                                Gp[k2] = fma2(d01, bc2(hk[k2]), Gp[k2]);
                                Gs[k2] = fmaf(d2, hk[k2], Gs[k2]);
                            }
                    }
                    if (visc || HAS_V) {
                        const float4 C4 = lds4(rec + 8);
                        if (visc)
#pragma unroll
                            for (int k2 = 0; k2 < 3; ++k2)
                                if (nz(i, k2)) {
                                    Fp[k2] = fma2(make_float2(C4.x, C4.y), bc2(hk[k2]), Fp[k2]);
                                    Fs[k2] = fmaf(B.z, hk[k2], Fs[k2]);
                                }
                        if (HAS_V)
#pragma unroll
                            for (int k2 = 0; k2 < 3; ++k2)
                                if (nz(i, k2)) {
                                    Dp[k2] = fma2(make_float2(C4.z, C4.w), bc2(hk[k2]), Dp[k2]);
                                    Ds[k2] = fmaf(B.w, hk[k2], Ds[k2]);
                                }
                    }
                }
                // affine path: X = X' J^{-1}, rows 0 and 1 paired
                auto finish = [&](const float2 Xp[3], const float Xs[3], float *X) {
#pragma unroll
                    for (int b2 = 0; b2 < 3; ++b2) {
                        if constexpr (AFF) {
                            const float *Ajl = reinterpret_cast<const float *>(M + MB) + lane;
                            const float j0 = DIET ? lds_f32_volatile(Ajl + b2 * 32) : Ji[b2];
                            const float j3 = DIET ? lds_f32_volatile(Ajl + (3 + b2) * 32) : Ji[3 + b2];
                            const float j6 = DIET ? lds_f32_volatile(Ajl + (6 + b2) * 32) : Ji[6 + b2];
                            float2 q2 = mul2(Xp[0], bc2(j0));
                            q2 = fma2(Xp[1], bc2(j3), q2);
                            q2 = fma2(Xp[2], bc2(j6), q2);
                            X[b2] = q2.x;
                            X[3 + b2] = q2.y;
                            X[6 + b2] = fmaf(Xs[2], j6, fmaf(Xs[1], j3, Xs[0] * j0));
                        } else {
                            X[b2] = Xp[b2].x;
                            X[3 + b2] = Xp[b2].y;
                            X[6 + b2] = Xs[b2];
                        }
                    }
                };
                finish(Gp, Gs, s1.G);
                if (visc) finish(Fp, Fs, s1.Fd);
                else
#pragma unroll
                    for (int k2 = 0; k2 < 9; ++k2) s1.Fd[k2] = 0.f;
                if (HAS_V) finish(Dp, Ds, D);
                else
#pragma unroll
                    for (int k2 = 0; k2 < 9; ++k2) D[k2] = 0.f;
            } else {
#pragma unroll
            for (int k2 = 0; k2 < 9; ++k2) {
                s1.G[k2] = R(0);
                s1.Fd[k2] = R(0);
                D[k2] = R(0);
            }
#pragma unroll
            for (int i = 0; i < NPE; ++i) {
                R hk[3];
#pragma unroll
                for (int k2 = 0; k2 < 3; ++k2) hk[k2] = nz(i, k2) ? grad(i, k2) : R(0);
                const R *rec = work + li[i] * REC;
                R x[3];
                if (i > 0) {
                    if constexpr (!DD_REG) {
                        R hv[3], lv[3];
                        ld_u(rec, hv, lv);
#pragma unroll
                        for (int a = 0; a < 3; ++a) dd[i][a] = (hv[a] - h0v[a]) + (lv[a] - l0v[a]);
                    }
#pragma unroll
                    for (int a = 0; a < 3; ++a)
#pragma unroll
                        for (int k2 = 0; k2 < 3; ++k2)
                            if (nz(i, k2)) s1.G[a * 3 + k2] += dd[i][a] * hk[k2];
                }
                if (visc) {
                    ld3c<OFF_UD>(rec, x[0], x[1], x[2]);
#pragma unroll
                    for (int a = 0; a < 3; ++a)
#pragma unroll
                        for (int k2 = 0; k2 < 3; ++k2)
                            if (nz(i, k2)) s1.Fd[a * 3 + k2] += x[a] * hk[k2];
                }
                if (HAS_V) {
                    ld3c<OFF_V>(rec, x[0], x[1], x[2]);
#pragma unroll
                    for (int a = 0; a < 3; ++a)
#pragma unroll
                        for (int k2 = 0; k2 < 3; ++k2)
                            if (nz(i, k2)) D[a * 3 + k2] += x[a] * hk[k2];
                }
            }
            if constexpr (AFF) {
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
            }
            R P[9];
            stress<R>(m, s1, visc, P);
            bad += (valid && !s1.ok) ? 1 : 0;

            if (OP == OP_DIAG) {
                // diagonal of a_K K^e + a_C C: A_d[c][b] = dP_{d b} / dF_{d c}
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    R A[9];
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        R E[9], dP[9];
#pragma unroll
                        for (int k2 = 0; k2 < 9; ++k2) E[k2] = (k2 == d * 3 + c) ? R(1) : R(0);
                        dstress<R>(m, s1, visc, E, p.aK, p.aC, true, dP);
#pragma unroll
                        for (int b2 = 0; b2 < 3; ++b2) A[c * 3 + b2] = w * dP[d * 3 + b2];
                    }
#pragma unroll
                    for (int i = 0; i < NPE; ++i) {
                        R hh[3];
#pragma unroll
                        for (int c = 0; c < 3; ++c) {
                            if constexpr (AFF) {  // h_i = J^{-T} g_i
                                hh[c] = R(0);
#pragma unroll
                                for (int k2 = 0; k2 < 3; ++k2)
                                    if (nz(i, k2)) hh[c] += grad(i, k2) * Ji[k2 * 3 + c];
                            } else {
                                hh[c] = grad(i, c);
                            }
                        }
                        const R h0 = hh[0], h1 = hh[1], h2 = hh[2];
                        acc0[i][d] += h0 * (A[0] * h0 + A[1] * h1 + A[2] * h2) +
                                      h1 * (A[3] * h0 + A[4] * h1 + A[5] * h2) +
                                      h2 * (A[6] * h0 + A[7] * h1 + A[8] * h2);
                    }
                }
            } else {
                R T0[9], T1[9];  // element-vector operators of this point (scaled by w below)
                if (OP == OP_FORCE) {
#pragma unroll
                    for (int k2 = 0; k2 < 9; ++k2) T0[k2] = P[k2];
                } else if (OP == OP_MATVEC) {
                    dstress<R>(m, s1, visc, D, p.aK, p.aC, p.sym_only != 0, T0);
                } else if (OP == OP_FM) {
                    // FP32 only: the force's and the operator product's
                    // element vectors are accumulated one after the other below
                } else {
                    R gmu, glam;
                    astress<R>(m, s1, visc, D, T0, T1, gmu, glam);
                    gmu_acc += w * gmu;
                    glam_acc += w * glam;
                }
                if constexpr (PKA) {
                    // w T h_i = w (T J^{-T}) g_i: rows 0 and 1 of the point's
                    // operator paired per column, then accumulated into the
                    // paired element vectors
                    auto pack = [&](const float *T, float2 Tp[3], float Ts[3]) {
#pragma unroll
                        for (int k2 = 0; k2 < 3; ++k2) {
                            if constexpr (AFF) {
                                const float *Ajl = reinterpret_cast<const float *>(M + MB) + lane;
                                const float j0 = DIET ? lds_f32_volatile(Ajl + (k2 * 3) * 32) : Ji[k2 * 3];
                                const float j1 = DIET ? lds_f32_volatile(Ajl + (k2 * 3 + 1) * 32) : Ji[k2 * 3 + 1];
                                const float j2 = DIET ? lds_f32_volatile(Ajl + (k2 * 3 + 2) * 32) : Ji[k2 * 3 + 2];
                                float2 q2 = mul2(make_float2(T[0], T[3]), bc2(j0));
                                q2 = fma2(make_float2(T[1], T[4]), bc2(j1), q2);
                                q2 = fma2(make_float2(T[2], T[5]), bc2(j2), q2);
                                Tp[k2] = mul2(q2, bc2(w));
                                Ts[k2] = w * fmaf(T[8], j2, fmaf(T[7], j1, T[6] * j0));
                            } else {
                                Tp[k2] = mul2(make_float2(T[k2], T[3 + k2]), bc2(w));
                                Ts[k2] = w * T[6 + k2];
                            }
                        }
                    };
                    if constexpr (OP == OP_FM) {
                        // force first (P packed and accumulated, then dead),
                        // then the stress derivative along the direction, so
                        // that the two point operators are never live together
                        float2 Tp[3];
                        float Ts[3];
                        pack(P, Tp, Ts);
#pragma unroll
                        for (int i = 0; i < NPE; ++i)
#pragma unroll
                            for (int k2 = 0; k2 < 3; ++k2)
                                if (nz(i, k2)) {
                                    const float hk = grad(i, k2);
                                    ap0[i] = fma2(Tp[k2], bc2(hk), ap0[i]);
                                    acc0[i][2] = fmaf(Ts[k2], hk, acc0[i][2]);
                                }
                        dstress<R>(m, s1, visc, D, p.aK, p.aC, p.sym_only != 0, T1);
                        pack(T1, Tp, Ts);
#pragma unroll
                        for (int i = 0; i < NPE; ++i)
#pragma unroll
                            for (int k2 = 0; k2 < 3; ++k2)
                                if (nz(i, k2)) {
                                    const float hk = grad(i, k2);
                                    ap1[i] = fma2(Tp[k2], bc2(hk), ap1[i]);
                                    acc1[i][2] = fmaf(Ts[k2], hk, acc1[i][2]);
                                }
                    } else {
                    float2 Tp0[3], Tp1[3];
                    float Ts0[3], Ts1[3];
                    pack(T0, Tp0, Ts0);
                    if (TWO) pack(T1, Tp1, Ts1);
#pragma unroll
                    for (int i = 0; i < NPE; ++i) {
#pragma unroll
                        for (int k2 = 0; k2 < 3; ++k2)
                            if (nz(i, k2)) {
                                const float hk = grad(i, k2);
                                ap0[i] = fma2(Tp0[k2], bc2(hk), ap0[i]);
                                acc0[i][2] = fmaf(Ts0[k2], hk, acc0[i][2]);
                                if (TWO) {
                                    ap1[i] = fma2(Tp1[k2], bc2(hk), ap1[i]);
                                    acc1[i][2] = fmaf(Ts1[k2], hk, acc1[i][2]);
                                }
                            }
                    }
                    }
                } else {
#pragma unroll
                for (int k2 = 0; k2 < 9; ++k2) {
                    T0[k2] *= w;
                    if (TWO) T1[k2] *= w;
                }
                if constexpr (AFF) {
                    // T h_i = (T J^{-T}) g_i
                    R T[9];
#pragma unroll
                    for (int a = 0; a < 3; ++a)
#pragma unroll
                        for (int k2 = 0; k2 < 3; ++k2)
                            T[a * 3 + k2] = T0[a * 3] * Ji[k2 * 3] + T0[a * 3 + 1] * Ji[k2 * 3 + 1] +
                                            T0[a * 3 + 2] * Ji[k2 * 3 + 2];
#pragma unroll
                    for (int k2 = 0; k2 < 9; ++k2) T0[k2] = T[k2];
                    if (TWO) {
#pragma unroll
                        for (int a = 0; a < 3; ++a)
#pragma unroll
                            for (int k2 = 0; k2 < 3; ++k2)
                                T[a * 3 + k2] = T1[a * 3] * Ji[k2 * 3] + T1[a * 3 + 1] * Ji[k2 * 3 + 1] +
                                                T1[a * 3 + 2] * Ji[k2 * 3 + 2];
#pragma unroll
                        for (int k2 = 0; k2 < 9; ++k2) T1[k2] = T[k2];
                    }
                }
#pragma unroll
                for (int i = 0; i < NPE; ++i) {
                    R hk[3];
#pragma unroll
                    for (int k2 = 0; k2 < 3; ++k2) hk[k2] = nz(i, k2) ? grad(i, k2) : R(0);
#pragma unroll
                    for (int a = 0; a < 3; ++a)
#pragma unroll
                        for (int k2 = 0; k2 < 3; ++k2)
                            if (nz(i, k2)) {
                                acc0[i][a] += T0[a * 3 + k2] * hk[k2];
                                if (TWO) acc1[i][a] += T1[a * 3 + k2] * hk[k2];
                            }
                }
                }
            }
            if (PF_EARLY && q == 0 && !prefetch_next()) {
                timed_out = true;
                break;
            }
            if constexpr (!AFF) {
                // slot b is no longer read: hand it to the slice NSLICE ahead
                const int j = k * NQ + q;
                __syncwarp();
                if (j + NSLICE < n_slices) {
                    if (lane == 0) {
                        fence_proxy_async();
                        issue(j + NSLICE);
                    }
                    sl_issued = j + NSLICE + 1;
                }
            }
        }
        if (timed_out) break;

        if (!PF_NONE && !(PF_EARLY && !mass_only) && !prefetch_next()) {
            timed_out = true;
            break;
        }

        // consistent mass of affine elements: m_ij = rho V Mhat_ij (Sec. 4.1),
        // into the operator product (the second element vector of OP_FM)
        if (!LANECOL && (OP == OP_MATVEC || OP == OP_DIAG || OP == OP_FM) && p.aM != R(0)) {
            const R c = p.aM * m.rho * p.evol[(size_t)t * 32 + lane];
            if (OP == OP_MATVEC || OP == OP_FM) {
                float2 *apy = OP == OP_FM ? ap1 : ap0;
                R(*accy)[3] = OP == OP_FM ? acc1 : acc0;
#pragma unroll
                for (int jn = 0; jn < NPE; ++jn) {
                    const int lj = LI_REREAD ? (int)bounds_clamp(lds_u16_volatile(mlidx + jn * 32 + lane), U, p.status)
                                             : li[jn];
                    if constexpr (PKA) {
                        const float *rec = work + lj * REC;
                        const float2 v01 = *reinterpret_cast<const float2 *>(rec + RC::V01);
                        const float v2 = rec[RC::V2];
#pragma unroll
                        for (int i = 0; i < NPE; ++i) {
                            const float mh = c * float(mass_hat(ET, i, jn));
                            apy[i] = fma2(v01, bc2(mh), apy[i]);
                            accy[i][2] += mh * v2;
                        }
                    } else {
                        R x[3];
                        ld3c<OFF_V>(work + lj * REC, x[0], x[1], x[2]);
#pragma unroll
                        for (int i = 0; i < NPE; ++i) {
                            const R mh = c * R(mass_hat(ET, i, jn));
                            accy[i][0] += mh * x[0];
                            accy[i][1] += mh * x[1];
                            accy[i][2] += mh * x[2];
                        }
                    }
                }
            } else {
#pragma unroll
                for (int i = 0; i < NPE; ++i) {
                    const R mh = c * R(mass_hat(ET, i, i));
                    acc0[i][0] += mh;
                    acc0[i][1] += mh;
                    acc0[i][2] += mh;
                }
            }
        }
        if (OP == OP_VJP && valid && p.gth && bounds_ok(e, p.n_elem_total, p.status)) {
            p.gth[(size_t)e * 2 + 0] = double(gmu_acc);
            p.gth[(size_t)e * 2 + 1] = double(glam_acc);
        }
        const int nbad = __reduce_add_sync(0xffffffffu, bad);
        if (lane == 0 && nbad) atomicAdd(p.status + ST_INVERTED, nbad);

        // ---- each lane writes its element vector into the node-sorted position
        // array (the patch is dead now), then one lane per unique node sums that
        // node's contiguous positions and adds the sum to the global array. The
        // sorted scatter stores the sum as the tile's partial instead (word 1 of
        // the record: the tile's first partial position); it runs as its own copy
        // of the loop, so that the adding path compiles as it does without it.
        // Wide slots: one walk over the positions sums every field, 2 shared
        // loads and 3 packed additions a position of two fields where one walk
        // per field over [position][3] took 6 and 6 and twice the loop around
        // them, and 2 stores instead of 6 (beam step of 480k T10 273.6 -> 262.7
        // us, 40-body batch 339 -> 317).
        if constexpr (wide_slots<ET, R, OP>()) {
            float4 *sA = reinterpret_cast<float4 *>(work);
            float2 *sB = reinterpret_cast<float2 *>(sA + NPE * 32);
            __syncwarp();
            if (valid) {
#pragma unroll
                for (int i = 0; i < NPE; ++i) {
                    const int ps = (int)bounds_clamp(LANECOL ? sp[i] : spos[i * 32 + lane], NPE * 32, p.status);
                    sA[ps] = make_float4(ap0[i].x, ap0[i].y, acc0[i][2], TWO ? ap1[i].x : 0.f);
                    if constexpr (TWO) sB[ps] = make_float2(ap1[i].y, acc1[i][2]);
                }
            }
            __syncwarp();
            auto node_sums = [&](int kk, float4 &a, float2 &b) {
                const int s0 = (int)bounds_clamp(soff[kk], NPE * 32 + 1, p.status);
                const int s1e = (int)bounds_clamp(soff[kk + 1], NPE * 32 + 1, p.status);
                float2 xy = make_float2(0.f, 0.f), zx = xy;
                b = xy;
                for (int sb = s0; sb < s1e; sb += 4) {
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (sb + j < s1e) {
                            const float4 v = sA[sb + j];
                            xy = add2(xy, make_float2(v.x, v.y));
                            if constexpr (TWO) {
                                zx = add2(zx, make_float2(v.z, v.w));
                                b = add2(b, sB[sb + j]);
                            } else {
                                zx.x += v.z;
                            }
                        }
                }
                a = make_float4(xy.x, xy.y, zx.x, zx.y);
            };
            if (p.part0) {
                const int64_t P0 = reinterpret_cast<const int32_t *>(M)[1];
                for (int kk = lane; kk < U; kk += 32) {
                    if (!bounds_ok(P0 + kk, p.n_part, p.status)) continue;
                    float4 a;
                    float2 b;
                    node_sums(kk, a, b);
                    R *d0 = p.part0 + (P0 + kk) * 3;
                    d0[0] = a.x;
                    d0[1] = a.y;
                    d0[2] = a.z;
                    if constexpr (TWO) {
                        R *d1 = p.part1 + (P0 + kk) * 3;
                        d1[0] = a.w;
                        d1[1] = b.x;
                        d1[2] = b.y;
                    }
                }
            } else {
                for (int kk = lane; kk < U; kk += 32) {
                    const int64_t n = bounds_clamp(nodes[kk], p.n_nodes, p.status);
                    float4 a;
                    float2 b;
                    node_sums(kk, a, b);
                    R *o0 = p.out0 + 3 * n, *o1 = TWO ? p.out1 + 3 * n : nullptr;
                    if (p.rmw_scatter) {
                        o0[0] += a.x;
                        o0[1] += a.y;
                        o0[2] += a.z;
                        if constexpr (TWO) {
                            o1[0] += a.w;
                            o1[1] += b.x;
                            o1[2] += b.y;
                        }
                    } else {
                        atomicAdd(o0, a.x);
                        atomicAdd(o0 + 1, a.y);
                        atomicAdd(o0 + 2, a.z);
                        if constexpr (TWO) {
                            atomicAdd(o1, a.w);
                            atomicAdd(o1 + 1, b.x);
                            atomicAdd(o1 + 2, b.y);
                        }
                    }
                }
            }
        } else {
        auto slots_in = [&](int fo) {
            __syncwarp();
            if (valid) {
#pragma unroll
                for (int i = 0; i < NPE; ++i) {
                    const int ps = (int)bounds_clamp(spos[i * 32 + lane], NPE * 32, p.status);
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        if constexpr (PKA) work[ps * 3 + d] = d == 0 ? ap0[i].x : (d == 1 ? ap0[i].y : acc0[i][2]);
                        else work[ps * 3 + d] = fo == 0 ? acc0[i][d] : acc1[i][d];
                    }
                }
            }
            __syncwarp();
        };
        auto node_sum = [&](int kk, R &a0, R &a1, R &a2) {
            const int s0 = (int)bounds_clamp(soff[kk], NPE * 32 + 1, p.status);
            const int s1e = (int)bounds_clamp(soff[kk + 1], NPE * 32 + 1, p.status);
            a0 = a1 = a2 = R(0);
            for (int sb = s0; sb < s1e; sb += 4) {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (sb + j < s1e) {
                        a0 += work[(sb + j) * 3 + 0];
                        a1 += work[(sb + j) * 3 + 1];
                        a2 += work[(sb + j) * 3 + 2];
                    }
            }
        };
        if (p.part0) {
#pragma unroll
            for (int fo = 0; fo < NFO; ++fo) {
                slots_in(fo);
                const int64_t P0 = reinterpret_cast<const int32_t *>(M)[1];
                R *dst = (fo == 0 ? p.part0 : p.part1) + P0 * 3;
                for (int kk = lane; kk < U; kk += 32) {
                    if (!bounds_ok(P0 + kk, p.n_part, p.status)) continue;
                    R a0, a1, a2;
                    node_sum(kk, a0, a1, a2);
                    dst[kk * 3] = a0;
                    dst[kk * 3 + 1] = a1;
                    dst[kk * 3 + 2] = a2;
                }
            }
        } else {
#pragma unroll
            for (int fo = 0; fo < NFO; ++fo) {
                R *out = fo == 0 ? p.out0 : p.out1;
                slots_in(fo);
                for (int kk = lane; kk < U; kk += 32) {
                    const int64_t n = bounds_clamp(nodes[kk], p.n_nodes, p.status);
                    R a0, a1, a2;
                    node_sum(kk, a0, a1, a2);
                    if (p.rmw_scatter) {
                        out[3 * n] += a0;
                        out[3 * n + 1] += a1;
                        out[3 * n + 2] += a2;
                    } else {
                        atomicAdd(out + 3 * n, a0);
                        atomicAdd(out + 3 * n + 1, a1);
                        atomicAdd(out + 3 * n + 2, a2);
                    }
                }
            }
        }
        }
        __syncwarp();
    }
    if (timed_out) {
        // a copy never landed: record it, then wait (bounded) for every copy
        // this warp still has in flight, by the parity of the one phase its
        // barrier has outstanding, so that no bulk copy is still writing into
        // shared memory when the CTA exits
        if (lane == 0) atomicAdd(p.status + ST_TIMEOUT, 1);
        for (int j = sl_done; j < sl_issued; ++j) mbar_wait_bounded(bar + j % NSLICE, (uint32_t)((j / NSLICE) & 1));
        for (int k = mt_done; k < mt_issued; ++k) mbar_wait_bounded(mbar + (k & 1), (uint32_t)((k >> 1) & 1));
        return false;
    }
    return true;
}

// One element kernel per (type, quadrature, precision, op, path, material
// mode): one launch per pass, warps persistent over the pass's tiles.
template <int ET, int NQ, typename R, int OP, bool AFF, int MAT>
__global__ void __launch_bounds__(128, min_ctas<ET, R, OP, AFF, MAT>()) k_elem(const KParams<R> p)
{
    extern __shared__ __align__(128) unsigned char smem[];
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    const int wpb = blockDim.x >> 5;
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem) + wib * (NSLICE + 2);  // [wpb][NSLICE + 2] (<= 128 B)
    unsigned char *wbase = smem + 128 + (size_t)wib * p.wreg;

    const int gw = blockIdx.x * wpb + wib;
    const int W = gridDim.x * wpb;
    // tiles of this warp: interleaved (t0 + k W) or, with tile_chunk, one
    // contiguous run of neighbouring tiles (which share nodes through L2)
    const int n_tiles = p.tile_end - p.tile_begin;
    const int per = (n_tiles + W - 1) / W;
    const int t0 = p.tile_chunk ? p.tile_begin + gw * per : p.tile_begin + gw;
    const int tstep = p.tile_chunk ? 1 : W;
    const int n_my = p.tile_chunk ? max(0, min(per, n_tiles - gw * per))
                                  : (t0 < p.tile_end ? (p.tile_end - t0 + W - 1) / W : 0);
    if (lane == 0) {
        for (int b = 0; b < NSLICE + 2; ++b) mbar_init(bar + b, 1);
        fence_mbar_init();
    }
    __syncwarp();
    elem_tiles<ET, NQ, R, OP, AFF, MAT>(p, wbase, bar, t0, tstep, n_my);
}

}  // namespace tlfe

#include "k_pw.cuh"
#include "k_wpe.cuh"

namespace tlfe {

template <int OP, typename R, bool AFF, int MAT> static void (*kernel_for_(int et, int nq))(const KParams<R>)
{
    if constexpr (OP == OP_FM) {  // the fused force + operator product: FP32 T4, T10 and H8 blocks
        if (sizeof(R) != 4 || et == ET_Q27) return nullptr;
    }
    if (et == ET_T4 && nq == 1) return k_elem<ET_T4, 1, R, OP, AFF, MAT>;
    if constexpr (!pw_path(ET_T10, AFF, OP, sizeof(R) == 4)) {
        if (et == ET_T10 && nq == 4) return k_elem<ET_T10, 4, R, OP, AFF, MAT>;
        if (et == ET_T10 && nq == 5) return k_elem<ET_T10, 5, R, OP, AFF, MAT>;
    }
    if (et == ET_H8 && nq == 8) return k_elem<ET_H8, 8, R, OP, AFF, MAT>;
    if constexpr (OP != OP_FM)
        if (et == ET_Q27 && nq == 27) return k_elem<ET_Q27, 27, R, OP, AFF, MAT>;
    return nullptr;
}
// FP32 kernels are specialised on the material mode; FP64 kernels (the plain
// reference path, FP64-pipe bound) use the generic mode only
template <int OP, typename R, bool AFF> static void (*kernel_for_m(int et, int nq, int mat))(const KParams<R>)
{
    if constexpr (sizeof(R) == 4) {
        switch (mat) {
        case MAT_NH: return kernel_for_<OP, R, AFF, MAT_NH>(et, nq);
        case MAT_NH_KV: return kernel_for_<OP, R, AFF, MAT_NH_KV>(et, nq);
        case MAT_SVK: return kernel_for_<OP, R, AFF, MAT_SVK>(et, nq);
        case MAT_SVK_KV: return kernel_for_<OP, R, AFF, MAT_SVK_KV>(et, nq);
        default: break;
        }
    }
    return kernel_for_<OP, R, AFF, MAT_ANY>(et, nq);
}
template <int OP, typename R> static void (*kernel_for(int et, int nq, bool aff, int mat))(const KParams<R>)
{
    if constexpr (OP == OP_FM) {
        if (wpe_path(et, aff)) return nullptr;
    } else {
        if (wpe_path(et, aff)) return wpe_kernel_for<OP, R>(mat);
    }
    if (pw_path(et, aff, OP, sizeof(R) == 4)) return pw_kernel_for<OP, R>(nq);
    if constexpr (OP == OP_FM && sizeof(R) != 4) return nullptr;
    else return aff ? kernel_for_m<OP, R, true>(et, nq, mat) : kernel_for_m<OP, R, false>(et, nq, mat);
}

// bytes of one warp's shared-memory region in the tile kernels (0: no such kernel)
template <int OP, typename R, bool AFF> size_t region_for_(int et, int umax, int meta_bytes, int mat, bool mass)
{
    if (et == ET_T4) return warp_region_bytes<ET_T4, R, OP, AFF>(umax, meta_bytes, mat, mass);
    if (et == ET_T10) return warp_region_bytes<ET_T10, R, OP, AFF>(umax, meta_bytes, mat, mass);
    if (et == ET_H8) return warp_region_bytes<ET_H8, R, OP, AFF>(umax, meta_bytes, mat, mass);
    if (et == ET_Q27 && OP != OP_FM) return warp_region_bytes<ET_Q27, R, OP, AFF>(umax, meta_bytes, mat, mass);
    return 0;
}
template <int OP, typename R> size_t region_for(int et, int umax, int meta_bytes, bool aff, int mat, bool mass)
{
    return aff ? region_for_<OP, R, true>(et, umax, meta_bytes, mat, mass)
               : region_for_<OP, R, false>(et, umax, meta_bytes, mat, mass);
}
template <int OP, typename R>
size_t smem_for(int et, int nq, int umax, int meta_bytes, int wpb, bool aff, int mat, bool mass)
{
    if constexpr (OP == OP_FM) {
        if (wpe_path(et, aff)) return 0;
    } else {
        if (wpe_path(et, aff)) return wpe_smem_bytes<R, OP>(wpb);
    }
    if (pw_path(et, aff, OP, sizeof(R) == 4)) return pw_smem_for<OP>(nq, umax, meta_bytes);
    const size_t w = region_for<OP, R>(et, umax, meta_bytes, aff, mat, mass);
    return w ? cta_smem_bytes(w, wpb) : 0;
}

// resident warps per SM for the best CTA size among 4, 2 and 1 warps, or for
// the CTA size *wpb_io when it is positive on entry. The point-per-warp
// kernels have one CTA size, nq warps, which answers for 4.
template <int OP, typename R>
int occupancy_op(int et, int nq, bool aff, int mat, bool mass, int umax, int meta_bytes, int *wpb_io, std::string *why)
{
    void (*kern)(const KParams<R>) = kernel_for<OP, R>(et, nq, aff, mat);
    const int only = *wpb_io;
    *wpb_io = 0;
    if (!kern) {
        *why = "no kernel for this element type and quadrature size";
        return 0;
    }
    const bool pw = pw_path(et, aff, OP, sizeof(R) == 4);
    int best = 0;
    for (int size : {4, 2, 1}) {
        if (only > 0 && size != only && !(pw && only == nq)) continue;
        if (pw && size != 4) continue;
        const int wpb = pw ? nq : size;
        const size_t smem = smem_for<OP, R>(et, nq, umax, meta_bytes, wpb, aff, mat, mass);
        if (smem > 227 * 1024) continue;
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        int nb = 0;
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, 32 * wpb, smem);
        if (e != cudaSuccess) {
            *why = std::string("occupancy query failed: ") + cudaGetErrorString(e);
            return 0;
        }
        if (nb * wpb > best) {
            best = nb * wpb;
            *wpb_io = wpb;
        }
    }
    if (best == 0)
        *why = "shared memory per warp too large (patch of " + std::to_string(umax) + " nodes, metadata " +
               std::to_string(meta_bytes) + " B)";
    return best;
}

// launch on the affine path when p.aff is set, else on the isoparametric
// (slab) path; material mode p.mat_mode
template <int OP, typename R>
cudaError_t launch_op(int et, int nq, const KParams<R> &p0, int grid, int wpb, cudaStream_t s)
{
    KParams<R> p = p0;
    const bool aff = p.aff != nullptr;
    void (*kern)(const KParams<R>) = kernel_for<OP, R>(et, nq, aff, p.mat_mode);
    if (!kern) return cudaErrorInvalidValue;
    const bool mass = p.aM != R(0);
    const size_t smem = smem_for<OP, R>(et, nq, p.umax, p.meta_bytes, wpb, aff, p.mat_mode, mass);
    p.wreg = (int)region_for<OP, R>(et, p.umax, p.meta_bytes, aff, p.mat_mode, mass);
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return err;
    kern<<<grid, 32 * wpb, smem, s>>>(p);
    return cudaGetLastError();
}

}  // namespace tlfe
