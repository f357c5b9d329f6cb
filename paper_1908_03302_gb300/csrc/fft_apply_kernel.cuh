// J m and J^T d with every entry of J recomputed inside each product instead of stored
// (Sec. II-C), tile-centric on sm_103a.
//
// Work decomposition
//   * The voxel grid is cut into 16 x 16 x 8 tiles. Each tile has a list of candidate rows
//     (built once per geometry by a conservative cull). A work item is a tile and a range of
//     its rows; a unit is one region of one item: an 8 x 8 x 8 region (four 8 x 4 x 4
//     sub-bricks, four regions per tile) for the single-column modes, an 8 x 8 x 4 region
//     (two sub-bricks, eight per tile) for the four- and eight-column ones. Every warp of the persistent
//     grid pulls units from a counter, heaviest items first, on its own (the only CTA barrier
//     follows the table load). The launch shape (warps per CTA, CTAs per SM) is picked per
//     variant from its register budget and the shared memory the band tables take.
//   * Lane l owns 4 consecutive x voxels of each sub-brick of its warp's region. Per chunk of
//     32 rows, lane l loads row l, moves its geometry into the tile's pair frame and tests it
//     against the region's sub-bricks (tangent-plane bounds of the convex detour); the rows
//     that reach one are staged in shared memory and broadcast, and each is evaluated on the
//     sub-bricks it reaches.
//   * Per (row, voxel): pair-frame coordinates by FFMA from per-lane offsets, normalised
//     detour (cancellation-free form), Phi from the band table in shared memory (one 64-bit
//     load, linear interpolation), geometric factor 1 / (R_xs R_xr). A lane's voxels are
//     evaluated as packed pairs (eval_deep, eval4).
//   * J^T accumulates per voxel in registers over the item's rows (gather, no atomics).
//     J folds each row's lane partials to 8 with two shuffles, parks them in the row's
//     consumed staging record, and the row's own lane sums them after the chunk: one partial
//     per (entry, region); a second kernel sums each row's partials in a fixed order. Both are
//     deterministic.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "fft_common.cuh"
#include "fft_device.cuh"

namespace fftgb {

// MODE_COV: sensitivity coverage sum_p |J[p, v] w_p| (J^T of |J|, same gather as MODE_JT).
// MODE_JT4 / MODE_J4, MODE_JT8 / MODE_J8: J^T and J for up to four or eight right-hand sides at once
// (every evaluated entry is applied to all; blocks are column-major: column r at r * V or r * M).
// MODE_JTC / MODE_JC: J^T and J with compensated FP32 sums, for the solver (fft_cg.cu says why): an
// entry's product goes into a pair of floats (fma2_comp), rows' weights are pairs as well, J folds the
// pairs, and the partials are stored as pairs (J^T) or in FP64 (J).
enum { MODE_JT = 0, MODE_J = 1, MODE_COUNT = 2, MODE_FROB = 3, MODE_COV = 4, MODE_JT4 = 5, MODE_J4 = 6, MODE_JT8 = 7,
       MODE_J8 = 8, MODE_JTC = 9, MODE_JC = 10 };
constexpr int STG_PER_WARP = 128;    // staged float4 per warp: 32 rows x (3 or 4)
constexpr int STG_PER_WARP8 = 160;   // the eight-column J^T: 32 rows x 5
// CTA of the eight-column kernels: one per SM, of 16 warps at 128 registers (64 of them hold a lane's
// accumulators or model values: 8 voxels x 8 columns), the sharp-band ones of 12 at 168, which
// would spill 600 bytes at 128. With 12 warps the plain ones were bound by latency (issue slots 59 %
// active): ring256, block of 8 columns, J and J^T 6.91 -> 6.13 ms, slices3d J^T 100.9 -> 96.4 ms.
template <bool SHARP>
constexpr int col8_warps() {
    return SHARP ? 12 : 16;
}

template <int MODE>
constexpr int apply_ncol() {
    return (MODE == MODE_JT8 || MODE == MODE_J8) ? 8 : ((MODE == MODE_JT4 || MODE == MODE_J4) ? 4 : 1);
}
template <int MODE>
constexpr int apply_stage() {
    return MODE == MODE_JT8 ? STG_PER_WARP8 : STG_PER_WARP;
}

struct ApplyParams {
    const RowRec* rec;
    const RowRec64* rec64;
    const int32_t* row_band;
    const float2* tab;
    int n_bands;
    int n_tab;
    const BandConst* bc;     // device [n_bands]
    const int32_t* tile_rows;
    const float4* ebase;     // [E] (p + hl, p - hl, c1, c2) of each entry's tile origin (pair frame)
    const float* ebase3;     // [E] c3 of each entry's tile origin
    const Item* items;
    int n_items;
    int32_t* counter;
    int tiles_x, tiles_y;
    int nx, ny, nz;
    int z_lo, z_end, mirror;   // layers to evaluate, mirror plane (fft_geom_s)
    const uint8_t* zw;         // COUNT, FROB: weight of each layer (null: 1)
    double org[3];
    double h;
    const float* vin;        // J: m [V]; J^T: d [M]
    float* vout;             // J: jpart [E * 4]; J^T: g [V]
    float* gpart;            // J^T partials of multi-item tiles
    float* vlow;             // JTC: what a voxel's value lacks after rounding (written beside vout)
    float* gpart_low;        // JTC: the same of the J^T partials
    double* vpart;           // JC: jpart in FP64 [E * 4]
    double* dsum;            // FROB: one per unit [n_items * 4]
    unsigned long long* icount;   // COUNT
    int trig_nq;             // PHI_TRIG: coefficient groups of 4 per band
    int seg_n;               // PHI_SEG: segments per band
    int64_t nvox, nrow;      // column lengths of the batch modes' blocks (V, M)
    int ncol;                // columns of the block (at most the mode's; the others count as zero)
};

// Where the kernels find Phi: `tab` the shared address of the bands' tables or segments, `seg2` that
// of the segments' c2, scale and nq as in phi_lookup_at, phi_seg and phi_trig.
struct PhiAt {
    uint32_t tab, seg2;
    float scale;
    int nq;
};

// Phi of the normalised detour v (fft_device.cuh); row_m is the magic number of the row's band
// (PHI_TRIG: the bits of the shared address of the band's block).
template <int PHI>
__device__ __forceinline__ float phi_eval(float v, float row_m, const PhiAt& at) {
    if (PHI == PHI_TRIG) return phi_trig(v, __float_as_uint(row_m), at.nq);
    if (PHI == PHI_SEG) return phi_seg(v, row_m, at.scale, at.tab, at.seg2);
    return phi_lookup_at(v, row_m, at.scale, at.tab);
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// FP64 detour for the precision-study mode: voxel (ix, iy, iz), row record in metres.
__device__ __forceinline__ float detour_v64(const RowRec64& r, double ox, double oy, double oz, double h,
                                            int ix, int iy, int iz, double U, float& w_band) {
    double x = ox + ix * h, y = oy + iy * h, z = oz + iz * h;
    double ex = r.xr[0] - r.xs[0], ey = r.xr[1] - r.xs[1], ez = r.xr[2] - r.xs[2];
    double L = sqrt(ex * ex + ey * ey + ez * ez);
    ex /= L; ey /= L; ez /= L;
    double dx = x - 0.5 * (r.xs[0] + r.xr[0]), dy = y - 0.5 * (r.xs[1] + r.xr[1]),
           dz = z - 0.5 * (r.xs[2] + r.xr[2]);
    double p = dx * ex + dy * ey + dz * ez;
    double c1 = dy * ez - dz * ey, c2 = dz * ex - dx * ez, c3 = dx * ey - dy * ex;
    double q2 = c1 * c1 + c2 * c2 + c3 * c3;
    double hl = 0.5 * L, ps = p + hl, pr = p - hl;
    double Rs = sqrt(ps * ps + q2), Rr = sqrt(pr * pr + q2);
    if (Rs == 0.0 || Rr == 0.0) {
        w_band = 0.0f;
        return 0.0f;
    }
    double A = Rs + fabs(ps), B = Rr + fabs(pr);
    double R = q2 * (A + B) / (A * B) + ((fabs(ps) - ps) + (fabs(pr) + pr));
    w_band = (float)(U * U / (Rs * Rr));
    double v = R / U;
    return (float)(v < 0.0 ? 0.0 : (v > 1.0 ? 1.0 : v));
}

// Resident 8-warp CTAs per SM the register budget is sized for: 4 (64 registers) for the
// stable-detour table kernels, 3 (80) for the others, 2 (128) for the four-column ones and the
// other sharp-band ones. The single-column stable-detour table variants are sized separately
// (apply_sharp_wide and apply_plain_wide below).
template <int MODE, int DT, bool SHARP, int PHI>
constexpr int apply_min_blocks() {
    return (SHARP || apply_ncol<MODE>() == 4) ? 2
                                                          : ((DT == FFT_DT_STABLE && PHI != PHI_TRIG) ? 4 : 3);
}

// Sub-bricks per unit and units (regions) per item of each mode: see sub_dy below.
template <int MODE>
constexpr int apply_nsub() {
    return apply_ncol<MODE>() > 1 ? 2 : 4;
}
template <int MODE>
constexpr int apply_regions() {
    return 16 / apply_nsub<MODE>();   // 16 sub-bricks of 8 x 4 x 4 per 16 x 16 x 8 tile
}

// Sub-bricks of a unit. The single-column modes take an 8 x 8 x 8 region (NSUB = 4) and the
// batch modes, whose per-voxel state is four or eight times larger, an 8 x 8 x 4 region (NSUB =
// 2). Sub-brick s of a lane sits at y offset sub_dy(s) and z offset sub_dz(s) from sub-brick 0;
// for NSUB = 4 the order (0,0), (4,0), (4,4), (0,4) lets every step between consecutive
// sub-bricks move along one axis only.
template <int NSUB>
__device__ __forceinline__ constexpr int sub_dy(int s) {
    return NSUB == 2 ? 4 * s : ((s == 1 || s == 2) ? 4 : 0);
}
template <int NSUB>
__device__ __forceinline__ constexpr int sub_dz(int s) {
    return NSUB == 2 ? 0 : (s >= 2 ? 4 : 0);
}

// Pair-frame values of a lane's first voxel moved from sub-brick s - 1 to sub-brick s (s >= 1):
// +4 voxels in y (s = 1), +4 in z (s = 2), -4 in y (s = 3). A step d along an axis changes
// p by d . e and c = (x - o) x e by d x e. The main loop and the FP64 re-decision both reach
// sub-brick s through these same operations, so their FP32 values agree bit for bit.
template <int NSUB, bool PL>
__device__ __forceinline__ void sub_step(int s, float hx, float hy, float hz, float& ps, float& pr, float& c1,
                                         float& c2, float& c3) {
    if (s == 1 || s == 3) {
        const float f = (s == 1) ? 4.0f : -4.0f;
        ps = fmaf(f, hy, ps);
        pr = fmaf(f, hy, pr);
        if (!PL) c1 = fmaf(f, hz, c1);
        c3 = fmaf(-f, hx, c3);
    } else if (s == 2) {
        if (!PL) {
            ps = fmaf(4.0f, hz, ps);
            pr = fmaf(4.0f, hz, pr);
        }
        c1 = fmaf(-4.0f, hy, c1);
        c2 = fmaf(4.0f, hx, c2);
    }
}

// Detour form of a sub-brick (staged per row): general, between the pair's transducer planes
// (no absolute values), deep inside the pair's sphere (fft_device.cuh).
enum { FORM_GENERAL = 0, FORM_INNER = 1, FORM_DEEP = 2 };

// Staged flag word: band (bits 0-7), sharp band (8), planar pair (9), and per sub-brick s of the
// unit: the row may reach it (12 + s), it is inner (16 + s), it is deep (20 + s); and per z layer h
// of the unit (sub-bricks 2 h and 2 h + 1): both are reached and deep (24 + h). In the support count also:
// the support holds the sub-brick whole (28 + s).
__device__ __forceinline__ int form_of(uint32_t cw, int s) {
    return ((cw >> (20 + s)) & 1u) ? FORM_DEEP : (((cw >> (16 + s)) & 1u) ? FORM_INNER : FORM_GENERAL);
}

// Per-row values of the deep form at a lane: X = ps pr + q2 is a quadratic in the voxel index t
// along the lane's run, X(t) = X(0) + t (b + t h^2) with b = 2 h (x - o)_x the same in every
// sub-brick, so that the run needs no stepped axial offsets.
struct DeepRow {
    float b, hh;              // 2 h (x - o)_x and h^2
    float lam, l2;            // L / U and its square
    float k2, k3, k4, k5;     // lam DEEP_C2 .. lam DEEP_C5
};

__device__ __forceinline__ void deep_init(DeepRow& d, float lam) {
    d.lam = lam;
    d.l2 = __fmul_rn(lam, lam);
    d.k2 = __fmul_rn(lam, DEEP_C2);
    d.k3 = __fmul_rn(lam, DEEP_C3);
    d.k4 = __fmul_rn(lam, DEEP_C4);
    d.k5 = __fmul_rn(lam, DEEP_C5);
}

template <bool PL>
__device__ __forceinline__ void deep_row(DeepRow& d, float ps, float pr, float c2, float c3, float hx, float hy,
                                         float hz) {
    float g = __fmul_rn(c3, hy);
    d.hh = fmaf(hx, hx, __fmul_rn(hy, hy));
    if (!PL) {
        g = fmaf(-c2, hz, g);
        d.hh = fmaf(hz, hz, d.hh);
    }
    d.b = fmaf(2.0f, g, __fmul_rn(hx, __fadd_rn(ps, pr)));
}

// Saturates the detour v = m0 m1 of each voxel pair to [0, 1]. SH: near becomes the smallest |v - 1|
// seen before saturation.
template <bool SH>
__device__ __forceinline__ f2 settle(f2 m0, f2 m1, float& near) {
    if (SH) {
        const float2 d = up(add2(mul2(m0, m1), pk1(-1.0f)));
        near = fminf(fminf(near, fabsf(d.x)), fabsf(d.y));
    }
    const float2 a = up(m0), b = up(m1);
    return pk(__saturatef(a.x * b.x), __saturatef(a.y * b.y));
}

// q2 of a lane's four voxels t = 0 .. 3 of one sub-brick from the pair-frame values at t = 0, as
// pairs (0, 1), (2, 3). c12 is c1^2 + c2^2 for a planar pair (constant along the run), c1^2
// otherwise.
template <bool PL>
__device__ __forceinline__ void line_q2(float c2, float c3, float c12, float hy, float hz, f2 (&q2)[2]) {
    const f2 T[2] = {pk(0.0f, 1.0f), pk(2.0f, 3.0f)};
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const f2 c3t = fma2(T[j], pk1(hy), pk1(c3));
        q2[j] = fma2(c3t, c3t, pk1(c12));
        if (!PL) {
            const f2 c2t = fma2(T[j], pk1(-hz), pk1(c2));
            q2[j] = fma2(c2t, c2t, q2[j]);
        }
    }
}

// Detours v (saturated) and w = 1 / (R_xs R_xr) of the lane's four voxels in each of NS deep
// sub-bricks, stage by stage over all of them: 2 NS independent chains hide the latency of the
// special-function unit better than one sub-brick's two.
template <int NS, bool SH, bool PL>
__device__ __forceinline__ void eval_deep(const float (&ps)[NS], const float (&pr)[NS], const float (&c2)[NS],
                                          const float (&c3)[NS], const float (&c12)[NS], float hy, float hz,
                                          const DeepRow& k, f2 (&v)[NS][2], f2 (&w)[NS][2], float& near) {
    const f2 T[2] = {pk(0.0f, 1.0f), pk(2.0f, 3.0f)};
    f2 q2[NS][2], X[NS][2], y[NS][2], Q[NS][2];
#pragma unroll
    for (int s = 0; s < NS; ++s) line_q2<PL>(c2[s], c3[s], c12[s], hy, hz, q2[s]);
#define FFT_EACH _Pragma("unroll") for (int s = 0; s < NS; ++s) _Pragma("unroll") for (int j = 0; j < 2; ++j)
    FFT_EACH X[s][j] = fma2(T[j], fma2(T[j], pk1(k.hh), pk1(k.b)), pk1(fmaf(ps[s], pr[s], up(q2[s][0]).x)));
    FFT_EACH Q[s][j] = fma2(X[s][j], X[s][j], mul2(pk1(k.l2), q2[s][j]));   // D
    FFT_EACH w[s][j] = rsqrt2(Q[s][j]);
    FFT_EACH y[s][j] = rcp2(fma2(Q[s][j], w[s][j], neg2(X[s][j])));
    FFT_EACH y[s][j] = mul2(q2[s][j], y[s][j]);
    FFT_EACH Q[s][j] = fma2(pk1(k.k5), y[s][j], pk1(k.k4));
    FFT_EACH Q[s][j] = fma2(Q[s][j], y[s][j], pk1(k.k3));
    FFT_EACH Q[s][j] = fma2(Q[s][j], y[s][j], pk1(k.k2));
    FFT_EACH Q[s][j] = fma2(Q[s][j], y[s][j], pk1(k.lam));
    FFT_EACH v[s][j] = settle<SH>(y[s][j], Q[s][j], near);
#undef FFT_EACH
}

// The same for one sub-brick in the other forms (general, inner).
template <int DT, bool GUARD, bool SH, int FORM, bool PL>
__device__ __forceinline__ void eval4(float ps, float pr, float c2, float c3, float c12, float hx, float hy, float hz,
                                      float hl, f2 (&v)[2], f2 (&w)[2], float& near) {
    const f2 T[2] = {pk(0.0f, 1.0f), pk(2.0f, 3.0f)};
    f2 q2[2];
    line_q2<PL>(c2, c3, c12, hy, hz, q2);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const f2 pst = fma2(T[j], pk1(hx), pk1(ps)), prt = fma2(T[j], pk1(hx), pk1(pr));
        f2 m0, m1;   // v is the product m0 m1
        if (DT == FFT_DT_STABLE && !GUARD && FORM == FORM_INNER) {
            const f2 ss = fma2(pst, pst, q2[j]), rr = fma2(prt, prt, q2[j]);
            const f2 is = rsqrt2(ss), ir = rsqrt2(rr);
            const f2 A = fma2(ss, is, pst), B = fma2(rr, ir, neg2(prt));
            w[j] = mul2(is, ir);
            m0 = mul2(q2[j], add2(A, B));
            m1 = rcp2(mul2(A, B));
        } else {
            const float2 a = up(pst), b = up(prt), q = up(q2[j]);
            float is0, ir0, is1, ir1;
            const float v0 = detour_v<DT, GUARD, FORM == FORM_INNER, true>(a.x, b.x, q.x, hl, is0, ir0);
            const float v1 = detour_v<DT, GUARD, FORM == FORM_INNER, true>(a.y, b.y, q.y, hl, is1, ir1);
            w[j] = pk(is0 * ir0, is1 * ir1);
            m0 = pk(v0, v1);
            m1 = pk1(1.0f);
        }
        v[j] = settle<SH>(m0, m1, near);
    }
}

// One voxel's detour before saturation, by the operations that eval_deep and eval4 pack (the same bits): t the
// voxel of the run, the other arguments as there.
template <int DT, bool GUARD>
__device__ __forceinline__ float eval1_raw(int form, bool planar, int t, float ps, float pr, float c2, float c3,
                                           float c12, float hx, float hy, float hz, float hl, const DeepRow& k,
                                           float& w) {
    const float ft = (float)t;
    auto q2_at = [&](float f) {
        const float c3t = fmaf(f, hy, c3);
        float q = fmaf(c3t, c3t, c12);
        if (!planar) {
            const float c2t = fmaf(f, -hz, c2);
            q = fmaf(c2t, c2t, q);
        }
        return q;
    };
    const float q2 = q2_at(ft);
    if (form == FORM_DEEP) {
        const float x0 = fmaf(ps, pr, q2_at(0.0f));
        const float X = fmaf(ft, fmaf(ft, k.hh, k.b), x0);
        const float D = fmaf(X, X, __fmul_rn(k.l2, q2));
        w = rsqrt_approx(D);
        const float y = __fmul_rn(q2, rcp_approx(fmaf(D, w, -X)));
        float Q = fmaf(k.k5, y, k.k4);
        Q = fmaf(Q, y, k.k3);
        Q = fmaf(Q, y, k.k2);
        return __fmul_rn(y, fmaf(Q, y, k.lam));
    }
    const float pst = fmaf(ft, hx, ps), prt = fmaf(ft, hx, pr);
    float is, ir;
    const float v = form == FORM_INNER ? detour_v<DT, GUARD, true, true>(pst, prt, q2, hl, is, ir)
                                       : detour_v<DT, GUARD, false, true>(pst, prt, q2, hl, is, ir);
    w = is * ir;
    return v;
}

// The FP64 re-decision of the sharp-band kernels, out of line (called only for an entry where
// some lane's FP32 detour lies within CUT_BAND of the cut), so that its FP64 temporaries do not
// weigh on the register allocation of the main loop. For each of the lane's 4 NSUB voxels
// (k = 4 s + t) it recomputes the FP32 detour by the operations of the main pass, and for the
// voxels near the cut re-decides dt < dt_max in FP64. It returns in d[k] what the main pass's
// term has to change by: val2 - val1 (J, J^T, four-column modes), |val2| - |val1| (coverage),
// val2^2 - val1^2 (Frobenius), +1 / -1 (support count), 0 where nothing changes. p is the row.
template <int MODE, int DT, bool GUARD, int PHI, int NSUB>
__device__ __noinline__ void sharp_fix(const ApplyParams& P, float4 A, float4 B, float4 C, int p, float Xl, float Yl,
                                       float Zl, const PhiAt& at, int ix0, int iy0, int iz0, float* d) {
    const float hx = B.x, hy = B.y, hz = B.z;
    const float hl = 0.5f * (A.x - A.y);
    const uint32_t cw = (uint32_t)__float_as_int(C.w);
    const bool planar = (cw >> 9) & 1u;
    const double U = P.bc[cw & 0xffu].U;
    DeepRow dr;
    deep_init(dr, C.z);
    // one voxel per iteration, each recomputed from the lane base (few values live across
    // iterations, which keeps the caller's register saves around this call small)
#pragma unroll 1
    for (int k = 0; k < 4 * NSUB; ++k) {
        const int s = k >> 2, t = k & 3;
        d[k] = 0.0f;
        if (!((cw >> (12 + s)) & 1u)) continue;   // the main pass skipped the sub-brick
        const float offs = planar ? fmaf(Xl, hx, Yl * hy) : fmaf(Xl, hx, fmaf(Yl, hy, Zl * hz));
        float pss = A.x + offs, prs = A.y + offs;
        float c1s = planar ? fmaf(-Zl, hy, A.z) : fmaf(Yl, hz, fmaf(-Zl, hy, A.z));
        float c2s = planar ? fmaf(Zl, hx, A.w) : fmaf(Zl, hx, fmaf(-Xl, hz, A.w));
        float c3s = fmaf(Xl, hy, fmaf(-Yl, hx, B.w));
        if (planar)
            deep_row<true>(dr, pss, prs, c2s, c3s, hx, hy, hz);
        else
            deep_row<false>(dr, pss, prs, c2s, c3s, hx, hy, hz);
#pragma unroll 1
        for (int q = 1; q <= s; ++q) {
            if (planar)
                sub_step<NSUB, true>(q, hx, hy, hz, pss, prs, c1s, c2s, c3s);
            else
                sub_step<NSUB, false>(q, hx, hy, hz, pss, prs, c1s, c2s, c3s);
        }
        const float c1sq = __fmul_rn(c1s, c1s);
        const float c12 = planar ? fmaf(c2s, c2s, c1sq) : c1sq;
        float w;
        const float vr = eval1_raw<DT, GUARD>(DT == FFT_DT_STABLE ? form_of(cw, s) : FORM_GENERAL, planar, t, pss, prs,
                                              c2s, c3s, c12, hx, hy, hz, hl, dr, w);
        if (!(fabsf(vr - 1.0f) < CUT_BAND)) continue;
        const float v = __saturatef(vr);
        const bool in = in_support64(P.rec64[p], P.org[0], P.org[1], P.org[2], P.h, ix0 + t, iy0 + sub_dy<NSUB>(s),
                                     iz0 + sub_dz<NSUB>(s), U);
        const float v2 = settle_cut(v, in);
        if (v2 == v) continue;
        if (MODE == MODE_COUNT) {
            d[k] = (v2 < 1.0f) ? 1.0f : -1.0f;
            continue;
        }
        const float val1 = phi_eval<PHI>(v, C.y, at) * w;
        const float val2 = phi_eval<PHI>(v2, C.y, at) * w;
        if (MODE == MODE_COV) d[k] = fabsf(val2) - fabsf(val1);
        else if (MODE == MODE_FROB) d[k] = val2 * val2 - val1 * val1;
        else d[k] = val2 - val1;
    }
}

// The sharp-band stable-detour table variants (single column) are built for CTAs of up to 20
// warps at one per SM (96 registers used): one CTA of 20 warps shares one copy of the band
// tables, and keeps more warps resident than 8-warp CTAs do (two per SM at this register
// count, fewer where large tables fill shared memory). Measured against 24 warps at 80
// registers and 16 warps at 128: the spills of the first and the lower occupancy of the
// second cost more.
template <int MODE, int DT, bool SHARP, int PHI>
constexpr bool apply_sharp_wide() {
    return SHARP && DT == FFT_DT_STABLE && PHI != PHI_TRIG && apply_ncol<MODE>() == 1;
}
constexpr int SHARP_MAX_WARPS = 20;
// (the compensated J^T, 16 more registers a lane, for 16 warps at 128: it would spill 336 bytes at 96)
template <int MODE>
constexpr int sharp_bound_warps() {
    return MODE == MODE_JTC ? 16 : SHARP_MAX_WARPS;
}

// The plain stable-detour table variants (single column) are built for blocks of up to 24
// warps at one per SM, i.e. 80 registers: their 16 per-lane voxels (8 x 8 x 8 units) want more
// than 64, and one wide CTA shares one copy of the band tables. Measured against 32 warps at
// 64 registers: slices3d J^T 408.0 -> 407.6 ms, J 412.6 -> 411.4 ms, ring256 J^T 3.75 -> 3.72 ms.
template <int MODE, int DT, bool SHARP, int PHI>
constexpr bool apply_plain_wide() {
    return !SHARP && DT == FFT_DT_STABLE && PHI != PHI_TRIG && apply_ncol<MODE>() == 1;
}
constexpr int PLAIN_MAX_WARPS = 24;

template <int MODE, int DT, bool SHARP, int PHI>
constexpr int apply_block_bound() {
    return apply_ncol<MODE>() == 8                    ? 32 * col8_warps<SHARP>()
           : apply_sharp_wide<MODE, DT, SHARP, PHI>() ? 32 * sharp_bound_warps<MODE>()
           : apply_plain_wide<MODE, DT, SHARP, PHI>() ? 32 * PLAIN_MAX_WARPS
                                                      : APPLY_THREADS;
}

template <int MODE, int DT, bool GUARD, bool SHARP, int PHI>
__global__ void __launch_bounds__(apply_block_bound<MODE, DT, SHARP, PHI>(),
                                  apply_block_bound<MODE, DT, SHARP, PHI>() == APPLY_THREADS
                                      ? apply_min_blocks<MODE, DT, SHARP, PHI>()
                                      : 1)
    apply_kernel(const __grid_constant__ ApplyParams P) {
    extern __shared__ __align__(16) unsigned char smem[];
    float2* s_tab = reinterpret_cast<float2*>(smem);
    const int tab_len = P.n_bands * P.n_tab;
    float4* s_stage = reinterpret_cast<float4*>(smem + (((size_t)tab_len * sizeof(float2) + 15) & ~(size_t)15));

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int i = tid; i < tab_len; i += blockDim.x) s_tab[i] = P.tab[i];
    __syncthreads();   // the only CTA-wide barrier: from here on every warp runs on its own

    const uint32_t tab_addr = smem_addr(s_tab);
    PhiAt at;
    at.tab = tab_addr;
    at.seg2 = tab_addr + (uint32_t)(P.n_bands * (P.seg_n + SEG_PAD)) * 8u;
    at.scale = (float)(PHI == PHI_SEG ? P.seg_n : P.n_tab - 1) * MAGIC2_ULP;
    at.nq = P.trig_nq;
    const int lx = lane & 1, ly = (lane >> 1) & 3, lz = lane >> 3;
    constexpr int NC = apply_ncol<MODE>();
    constexpr bool JTN = (MODE == MODE_JT4 || MODE == MODE_JT8), JN = (MODE == MODE_J4 || MODE == MODE_J8);
    constexpr bool BATCH = NC > 1;
    constexpr bool JT1 = (MODE == MODE_JT || MODE == MODE_JTC), J1 = (MODE == MODE_J || MODE == MODE_JC);
    constexpr int SR = JTN ? 3 + NC / 4 : (MODE == MODE_JTC ? 4 : 3);   // staged float4 per row
    constexpr int NSUB = apply_nsub<MODE>();
    constexpr int NREG = apply_regions<MODE>();
    float4* stg = s_stage + warp * apply_stage<MODE>();
    const int n_units = P.n_items * NREG;

    for (;;) {
        // A unit is one region of one item (unit = item * NREG + region): 8 x 8 x 8 voxels for
        // the single-column modes (regions 2 x 2 x 1 per tile), 8 x 8 x 4 for the four-column
        // ones (2 x 2 x 2 per tile).
        int unit = 0;
        if (lane == 0) unit = atomicAdd(P.counter, 1);
        unit = __shfl_sync(0xffffffffu, unit, 0);
        if (unit >= n_units) break;
        const int it = unit / NREG, region = unit % NREG;
        const Item item = P.items[it];
        const int tx = item.tile % P.tiles_x;
        const int ty = (item.tile / P.tiles_x) % P.tiles_y;
        const int tz = item.tile / (P.tiles_x * P.tiles_y);
        const int TX = TILE_X * tx, TY = TILE_Y * ty, TZ = TILE_Z * tz;
        const int wx = region & 1, wy = (region >> 1) & 1, wz = (NSUB == 2) ? (region >> 2) : 0;
        // lane voxel offsets in the tile (sub-brick 0, first of its 4 x voxels)
        const int oxi = 8 * wx + 4 * lx, oyi = 8 * wy + ly, ozi = 4 * wz + lz;
        const float Xl = (float)oxi, Yl = (float)oyi, Zl = (float)ozi;

        // validity of this lane's voxels (bit 4 s + t) and of the region's sub-bricks (bit s)
        auto lane_vmask = [&]() {
            uint32_t vm = 0;
#pragma unroll
            for (int s = 0; s < NSUB; ++s) {
                const int z = TZ + ozi + sub_dz<NSUB>(s);
                if (z >= P.z_lo && z < P.z_end && TY + oyi + sub_dy<NSUB>(s) < P.ny) {
#pragma unroll
                    for (int t = 0; t < NX_LANE; ++t)
                        if (TX + oxi + t < P.nx) vm |= 1u << (4 * s + t);
                }
            }
            return vm;
        };
        uint32_t sub_ok = 0;
#pragma unroll
        for (int s = 0; s < NSUB; ++s)
            if (TX + 8 * wx < P.nx && TY + 8 * wy + sub_dy<NSUB>(s) < P.ny && TZ + 4 * wz + sub_dz<NSUB>(s) < P.z_end &&
                TZ + 4 * wz + sub_dz<NSUB>(s) + 3 >= P.z_lo)
                sub_ok |= 1u << s;
        // the gather modes need the mask only for their stores: recomputed there
        constexpr bool VM_LIVE = !(JT1 || MODE == MODE_COV || JTN);
        const uint32_t vmask = VM_LIVE ? lane_vmask() : 0u;
        const int64_t vbase = ((int64_t)(TZ + ozi) * P.ny + TY + oyi) * P.nx + TX + oxi;
        // voxels from this lane's run in sub-brick s to its mirror image (0: none)
        auto mirror_off = [&](int s) {
            return (int64_t)mirror_step(P.mirror, TZ + ozi + sub_dz<NSUB>(s), P.nz) * P.ny * P.nx;
        };
        // the count and the Frobenius norm weigh a run with its layer and its image (8 bits per
        // sub-brick; at most 2 STACK_MAX_SLICES)
        uint32_t mult = 0;
        if (MODE == MODE_COUNT || MODE == MODE_FROB) {
#pragma unroll
            for (int s = 0; s < NSUB; ++s) {
                const int z = TZ + ozi + sub_dz<NSUB>(s);
                if (z >= P.nz) continue;
                const int zs = mirror_step(P.mirror, z, P.nz);
                uint32_t w = P.zw ? P.zw[z] : 1u;
                if (zs != 0) w += P.zw ? P.zw[z + zs] : 1u;
                mult |= w << (8 * s);
            }
        }

        // accumulators (J^T) or model values (J) of the lane's voxels, as pairs (0, 1), (2, 3) of
        // each run
        f2 acc[NSUB][2], accl[NSUB][2], mv[NSUB][2];   // (accl: low parts, JTC only)
        f2 accn[2][2][NC], mvn[2][2][NC];   // batch modes only (NSUB = 2)
        double dacc = 0.0;
        unsigned long long cnt = 0, cnt_eval = 0;
#pragma unroll
        for (int s = 0; s < NSUB; ++s)
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int64_t vo = vbase + ((int64_t)sub_dz<NSUB>(s) * P.ny + sub_dy<NSUB>(s)) * P.nx + 2 * j;
                const bool ok0 = (vmask >> (4 * s + 2 * j)) & 1u, ok1 = (vmask >> (4 * s + 2 * j + 1)) & 1u;
                acc[s][j] = accl[s][j] = mv[s][j] = 0ull;
                if (J1) {
                    mv[s][j] = pk(ok0 ? __ldg(P.vin + vo) : 0.0f, ok1 ? __ldg(P.vin + vo + 1) : 0.0f);
                    if (const int64_t mo = mirror_off(s))
                        mv[s][j] = add2(mv[s][j], pk(ok0 ? __ldg(P.vin + vo + mo) : 0.0f,
                                                     ok1 ? __ldg(P.vin + vo + mo + 1) : 0.0f));
                }
                if (BATCH && s < 2) {
#pragma unroll
                    for (int r = 0; r < NC; ++r) {
                        accn[s & 1][j][r] = mvn[s & 1][j][r] = 0ull;
                        if (JN && r < P.ncol) {
                            const float* mr = P.vin + (int64_t)r * P.nvox + vo;
                            mvn[s & 1][j][r] = pk(ok0 ? __ldg(mr) : 0.0f, ok1 ? __ldg(mr + 1) : 0.0f);
                            if (const int64_t mo = mirror_off(s))
                                mvn[s & 1][j][r] = add2(mvn[s & 1][j][r], pk(ok0 ? __ldg(mr + mo) : 0.0f,
                                                                             ok1 ? __ldg(mr + mo + 1) : 0.0f));
                        }
                    }
                }
            }

        for (int64_t e0 = item.e0; e0 < item.e1; e0 += 32) {
            // ---- stage: lane l prepares row e0 + l
            const int64_t e = e0 + lane;
            const bool have = e < item.e1;
            uint32_t okb = 0;   // sub-bricks the row may reach
            if (have) {
                const int p = P.tile_rows[e];
                const float4 base = P.ebase[e];
                const float base3 = P.ebase3[e];
                const RowRec r = P.rec[p];
                const int b = P.row_band[p];
                const BandConst bc = P.bc[b];
                const float hb = bc.h;
                float W = r.b.w;
                float Wlow = 0.0f;   // what W lacks after rounding
                if (JT1) {
                    const float x = __ldg(P.vin + p), C = W;
                    W *= x;
                    if (MODE == MODE_JTC) Wlow = fmaf(C, x, -W);
                }
                if (MODE == MODE_COV) W = fabsf(W) * (P.vin ? fabsf(__ldg(P.vin + p)) : 1.0f);
                float Wn[NC];
                bool any_w = false;
                if (JTN) {
#pragma unroll
                    for (int r = 0; r < NC; ++r) {
                        Wn[r] = r < P.ncol ? W * __ldg(P.vin + (int64_t)r * P.nrow + p) : 0.0f;
                        any_w = any_w || Wn[r] != 0.0f;
                    }
                }
                const float ex = r.b.x, ey = r.b.y, ez = r.b.z, hl = r.a.w;
                // sub-brick centres relative to the pair midpoint (FP32; used by the bound only)
                const float dx = fmaf((float)TX, hb, bc.org[0]) - r.a.x;
                const float dy = fmaf((float)TY, hb, bc.org[1]) - r.a.y;
                const float dz = fmaf((float)TZ, hb, bc.org[2]) - r.a.z;
                const float cx = fmaf(8.0f * wx + 3.5f, hb, dx);
                const float hxx = 3.5f * hb, hyy = 1.5f * hb;
                // rows with zero weight add exactly nothing to J^T: skip them
                const bool live = JTN ? any_w : ((!JT1 && MODE != MODE_COV) || (W != 0.0f));
                const float pext = hxx * fabsf(ex) + hyy * (fabsf(ey) + fabsf(ez)) + 1e-3f;
                // deep sub-bricks: their voxel centres (half diagonal sqrt(3.5^2 + 2 1.5^2) = 4.1 steps)
                // keep DEEP_MARGIN steps off the pair's sphere
                const float lam = 2.0f * hl;
                const float rim = hl - (4.1f + DEEP_MARGIN) * hb;
                const float rim2 = (DT == FFT_DT_STABLE && lam >= DEEP_MIN_L && rim > 0.0f) ? rim * rim : -1.0f;
                uint32_t inb = 0, dpb = 0, full = 0;
#pragma unroll
                for (int s = 0; s < NSUB; ++s) {
                    const float cy = fmaf(8.0f * wy + (float)sub_dy<NSUB>(s) + 1.5f, hb, dy);
                    const float cz = fmaf(4.0f * wz + (float)sub_dz<NSUB>(s) + 1.5f, hb, dz);
                    if (live && ((sub_ok >> s) & 1u) && box_may_touch(cx, cy, cz, ex, ey, ez, hl, hxx, hyy, hyy))
                        okb |= 1u << s;
                    // the support count takes sub-bricks that the support holds whole as they are
                    // (a ring of 256 calibrated elements: 3.41 -> 2.63 ms)
                    if (MODE == MODE_COUNT && DT != FFT_DT_FP64 && ((okb >> s) & 1u) &&
                        box_inside(cx, cy, cz, ex, ey, ez, hl, hxx, hyy, hyy))
                        full |= 1u << s;
                    // sub-bricks whose voxels all satisfy |p| <= hl (between the transducer planes)
                    if (fabsf(fmaf(cx, ex, fmaf(cy, ey, cz * ez))) + pext <= hl) inb |= 1u << s;
                    if (fmaf(cx, cx, fmaf(cy, cy, cz * cz)) <= rim2) dpb |= 1u << s;
                }
                const uint32_t od = okb & dpb & ~full;
                const uint32_t both = ((od & 3u) == 3u ? 1u : 0u) | ((od & 12u) == 12u ? 2u : 0u);
                const uint32_t fl = (okb << 12) | (inb << 16) | (dpb << 20) | (both << 24) | (full << 28);
                stg[lane * SR + 0] = base;
                stg[lane * SR + 1] = make_float4(r.c.x, r.c.y, r.c.z, base3);
                // planar pair (both transducers at one z): stepping along x changes only c3
                const int planar = (ez == 0.0f) ? 1 : 0;
                // third word: the band's place (the magic number of its lookups; PHI_TRIG: the
                // shared address of its block), the pair's length; fourth: see form_of
                const float row_m =
                    PHI == PHI_TRIG ? __uint_as_float(tab_addr + (uint32_t)(b * P.n_tab) * 8u)
                                    : fmaf((float)(b * (PHI == PHI_SEG ? P.seg_n + SEG_PAD : P.n_tab)), MAGIC2_ULP, MAGIC2);
                stg[lane * SR + 2] = make_float4(W, row_m, DT == FFT_DT_FP64 ? __int_as_float(p) : lam,
                                                 __int_as_float(b | (bc.sharp << 8) | (planar << 9) | (int)fl));
                if (MODE == MODE_JTC) stg[lane * SR + 3].x = Wlow;
                if (JTN) {
#pragma unroll
                    for (int k = 0; k < NC / 4; ++k)
                        stg[lane * SR + 3 + k] = make_float4(Wn[4 * k], Wn[4 * k + 1], Wn[4 * k + 2], Wn[4 * k + 3]);
                }
            }
            uint32_t mm = __ballot_sync(0xffffffffu, okb != 0u);
            __syncwarp();
            float mypart = 0.0f;
            double mypart64 = 0.0;   // JC
            while (mm) {
                const int bit = __ffs(mm) - 1;
                mm &= mm - 1;
                const float4 A = stg[bit * SR + 0];
                const float4 B = stg[bit * SR + 1];
                const float4 C = stg[bit * SR + 2];
                float Wr[NC];
                if (JTN) {
#pragma unroll
                    for (int k = 0; k < NC / 4; ++k) {
                        const float4 x = stg[bit * SR + 3 + k];
                        Wr[4 * k] = x.x;
                        Wr[4 * k + 1] = x.y;
                        Wr[4 * k + 2] = x.z;
                        Wr[4 * k + 3] = x.w;
                    }
                }
                const float hx = B.x, hy = B.y, hz = B.z, W = C.x, row_m = C.y;
                const float Wlow = MODE == MODE_JTC ? stg[bit * SR + 3].x : 0.0f;
                const float hl = 0.5f * (A.x - A.y);   // used by the textbook (NAIVE) detour only
                const uint32_t cw = (uint32_t)__float_as_int(C.w);
                const bool planar = (DT != FFT_DT_FP64) && ((cw >> 9) & 1u);
                DeepRow dr;
                deep_init(dr, C.z);
                float near = 2.0f;   // smallest |v - 1| of this lane's voxels (sharp bands)
                f2 part = 0ull, partl = 0ull;   // (partl: low part, JC only)
                f2 partn[NC];
#pragma unroll
                for (int r = 0; r < NC; ++r) partn[r] = 0ull;
                uint32_t n_in = 0;
                float fsum = 0.0f;
                // Phi and the mode's sum over one sub-brick's four voxels.
                auto accumulate = [&](int s, const f2 (&v)[2], const f2 (&w)[2]) {
                    const float2 va = up(v[0]), vb = up(v[1]);
                    if (MODE == MODE_COUNT) {
                        const uint32_t vm = (vmask >> (4 * s)) & 15u;
                        const uint32_t in = (va.x < 1.0f ? 1u : 0u) | (va.y < 1.0f ? 2u : 0u) | (vb.x < 1.0f ? 4u : 0u) |
                                            (vb.y < 1.0f ? 8u : 0u);
                        n_in += (__popc(in & vm) | (__popc(vm) << 16)) * ((mult >> (8 * s)) & 255u);
                        return;
                    }
                    float ph[NX_LANE];
                    if (PHI == PHI_TRIG) {
                        const float vv[NX_LANE] = {va.x, va.y, vb.x, vb.y};
                        phi_trig_n<NX_LANE>(vv, __float_as_uint(row_m), at.nq, ph);
                    } else if (PHI == PHI_SEG) {
                        ph[0] = phi_eval<PHI>(va.x, row_m, at);
                        ph[1] = phi_eval<PHI>(va.y, row_m, at);
                        ph[2] = phi_eval<PHI>(vb.x, row_m, at);
                        ph[3] = phi_eval<PHI>(vb.y, row_m, at);
                    } else {
                        const float2 ta = up(fma2_rd(v[0], pk1(at.scale), pk1(row_m)));
                        const float2 tb = up(fma2_rd(v[1], pk1(at.scale), pk1(row_m)));
                        const float2 T0 = lds_f2_table(tab_addr, ta.x), T1 = lds_f2_table(tab_addr, ta.y);
                        const float2 T2 = lds_f2_table(tab_addr, tb.x), T3 = lds_f2_table(tab_addr, tb.y);
                        ph[0] = fmaf(va.x, T0.y, T0.x);
                        ph[1] = fmaf(va.y, T1.y, T1.x);
                        ph[2] = fmaf(vb.x, T2.y, T2.x);
                        ph[3] = fmaf(vb.y, T3.y, T3.x);
                    }
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const f2 val = mul2(pk(ph[2 * j], ph[2 * j + 1]), w[j]);
                        if (MODE == MODE_JT) acc[s][j] = fma2(val, pk1(W), acc[s][j]);
                        if (MODE == MODE_JTC) {
                            fma2_comp(val, pk1(W), acc[s][j], accl[s][j]);
                            accl[s][j] = fma2(val, pk1(Wlow), accl[s][j]);
                        }
                        if (MODE == MODE_COV) {
                            const float2 x = up(val);
                            acc[s][j] = fma2(pk(fabsf(x.x), fabsf(x.y)), pk1(W), acc[s][j]);
                        }
                        if (MODE == MODE_J) part = fma2(val, mv[s][j], part);
                        if (MODE == MODE_JC) fma2_comp(val, mv[s][j], part, partl);
                        if (JTN) {
#pragma unroll
                            for (int r = 0; r < NC; ++r) accn[s & 1][j][r] = fma2(val, pk1(Wr[r]), accn[s & 1][j][r]);
                        }
                        if (JN) {
#pragma unroll
                            for (int r = 0; r < NC; ++r) partn[r] = fma2(val, mvn[s & 1][j][r], partn[r]);
                        }
                        if (MODE == MODE_FROB) {
                            const float2 x = up(val);
                            const float f = (float)((mult >> (8 * s)) & 255u);
                            if ((vmask >> (4 * s + 2 * j)) & 1u) fsum = fmaf(f * x.x, x.x, fsum);
                            if ((vmask >> (4 * s + 2 * j + 1)) & 1u) fsum = fmaf(f * x.y, x.y, fsum);
                        }
                    }
                };
                // The entry's evaluation, specialised for planar pairs (both transducers at one
                // z: the axis has no z component, so h_z = 0 exactly, c1 and c2 do not change
                // along the lane's voxels or between sub-bricks at one z, and p does not change
                // in z). The lane base (sub-brick 0, t = 0) is a small offset added to the tile
                // origin's FP64-derived values.
                // SH: the near-cut checks, for rows of a band whose Phi does not vanish at the cut.
                auto entry_body = [&](auto planar_tag, auto sharp_tag) {
                    constexpr bool PL = decltype(planar_tag)::value;
                    constexpr bool SH = decltype(sharp_tag)::value;
                    const float off = PL ? fmaf(Xl, hx, Yl * hy) : fmaf(Xl, hx, fmaf(Yl, hy, Zl * hz));
                    float psb = A.x + off, prb = A.y + off;
                    float c1 = PL ? fmaf(-Zl, hy, A.z) : fmaf(Yl, hz, fmaf(-Zl, hy, A.z));
                    float c2 = PL ? fmaf(Zl, hx, A.w) : fmaf(Zl, hx, fmaf(-Xl, hz, A.w));
                    float c3 = fmaf(Xl, hy, fmaf(-Yl, hx, B.w));
                    float c12_planar = PL ? fmaf(c2, c2, __fmul_rn(c1, c1)) : 0.0f;
                    if (DT == FFT_DT_STABLE) deep_row<PL>(dr, psb, prb, c2, c3, hx, hy, hz);
                    // two sub-bricks at a time (one z layer of the unit)
#pragma unroll
                    for (int h = 0; h < NSUB / 2; ++h) {
                        if (h > 0) {   // from sub-brick 1 to 2: +4 in z
                            sub_step<NSUB, PL>(2, hx, hy, hz, psb, prb, c1, c2, c3);
                            if (PL) c12_planar = fmaf(c2, c2, __fmul_rn(c1, c1));
                        }
                        float psv[2], prv[2], c2v[2], c3v[2], c12v[2];
                        psv[0] = psb;
                        prv[0] = prb;
                        c2v[0] = c2;
                        c3v[0] = c3;
                        c12v[0] = PL ? c12_planar : __fmul_rn(c1, c1);
                        sub_step<NSUB, PL>(2 * h + 1, hx, hy, hz, psb, prb, c1, c2, c3);
                        psv[1] = psb;
                        prv[1] = prb;
                        c2v[1] = c2;
                        c3v[1] = c3;
                        c12v[1] = PL ? c12_planar : __fmul_rn(c1, c1);
                        // (the recurrence, inlined at each use, is one use fewer per layer without it: five series cut
                        // after six periods, 96 elements, J 9.4 ms with and 6.1 ms without, 7.1 ms by the general form)
                        if (DT == FFT_DT_STABLE && PHI != PHI_TRIG && ((cw >> (24 + h)) & 1u)) {
                            f2 v[2][2], w[2][2];
                            eval_deep<2, SH, PL>(psv, prv, c2v, c3v, c12v, hy, hz, dr, v, w, near);
                            accumulate(2 * h, v[0], w[0]);
                            accumulate(2 * h + 1, v[1], w[1]);
                            continue;
                        }
#pragma unroll
                        for (int q = 0; q < 2; ++q) {
                            const int s = 2 * h + q;
                            if (!((cw >> (12 + s)) & 1u)) continue;
                            if (MODE == MODE_COUNT && ((cw >> (28 + s)) & 1u)) {
                                n_in += (uint32_t)__popc((vmask >> (4 * s)) & 15u) * 0x10001u * ((mult >> (8 * s)) & 255u);
                                continue;
                            }
                            f2 v[2], w[2];
                            if (DT == FFT_DT_FP64) {
                                const RowRec64 r64 = P.rec64[__float_as_int(C.z)];
                                const double U = P.bc[cw & 0xffu].U;
                                float vv[NX_LANE], ww[NX_LANE];
#pragma unroll
                                for (int t = 0; t < NX_LANE; ++t)
                                    vv[t] = detour_v64(r64, P.org[0], P.org[1], P.org[2], P.h, TX + oxi + t,
                                                       TY + oyi + sub_dy<NSUB>(s), TZ + ozi + sub_dz<NSUB>(s), U, ww[t]);
                                v[0] = pk(vv[0], vv[1]);
                                v[1] = pk(vv[2], vv[3]);
                                w[0] = pk(ww[0], ww[1]);
                                w[1] = pk(ww[2], ww[3]);
                            } else if (DT == FFT_DT_STABLE && form_of(cw, s) == FORM_DEEP) {
                                f2 v1[1][2], w1[1][2];
                                const float a[1] = {psv[q]}, b[1] = {prv[q]}, c[1] = {c2v[q]}, d[1] = {c3v[q]},
                                            f[1] = {c12v[q]};
                                eval_deep<1, SH, PL>(a, b, c, d, f, hy, hz, dr, v1, w1, near);
                                v[0] = v1[0][0];
                                v[1] = v1[0][1];
                                w[0] = w1[0][0];
                                w[1] = w1[0][1];
                            } else if (DT == FFT_DT_STABLE && form_of(cw, s) == FORM_INNER) {
                                eval4<DT, GUARD, SH, FORM_INNER, PL>(psv[q], prv[q], c2v[q], c3v[q], c12v[q], hx, hy, hz, hl,
                                                                     v, w, near);
                            } else {
                                eval4<DT, GUARD, SH, FORM_GENERAL, PL>(psv[q], prv[q], c2v[q], c3v[q], c12v[q], hx, hy, hz,
                                                                       hl, v, w, near);
                            }
                            accumulate(s, v, w);
                        }
                    }
                };
                // (a launch's rows are all of one kind: launch_split)
                if (planar)
                    entry_body(std::true_type{}, std::integral_constant<bool, SHARP>{});
                else
                    entry_body(std::false_type{}, std::integral_constant<bool, SHARP>{});
                if (SHARP && DT != FFT_DT_FP64 && __any_sync(0xffffffffu, near < CUT_BAND)) {
                    // FP64 re-decision of the voxels whose FP32 detour lies within CUT_BAND of
                    // the cut; d[k] is the change of this entry's term for voxel k = 4 s + t
                    float d[4 * NSUB];
                    if (near < CUT_BAND)
                        sharp_fix<MODE, DT, GUARD, PHI, NSUB>(P, A, B, C, P.tile_rows[e0 + bit], Xl, Yl, Zl, at,
                                                              TX + oxi, TY + oyi, TZ + ozi, d);
#pragma unroll
                    for (int s = 0; s < NSUB; ++s) {
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            const float d0 = near < CUT_BAND ? d[4 * s + 2 * j] : 0.0f;
                            const float d1 = near < CUT_BAND ? d[4 * s + 2 * j + 1] : 0.0f;
                            if (d0 == 0.0f && d1 == 0.0f) continue;
                            const f2 dk = pk(d0, d1);
                            const bool ok0 = (vmask >> (4 * s + 2 * j)) & 1u, ok1 = (vmask >> (4 * s + 2 * j + 1)) & 1u;
                            const int f = (int)((mult >> (8 * s)) & 255u);   // count, Frobenius
                            if (MODE == MODE_COUNT) n_in += f * ((ok0 ? (int)d0 : 0) + (ok1 ? (int)d1 : 0));
                            if (JT1 || MODE == MODE_COV) acc[s][j] = fma2(dk, pk1(W), acc[s][j]);
                            if (J1) part = fma2(dk, mv[s][j], part);
                            if (JTN) {
#pragma unroll
                                for (int r = 0; r < NC; ++r) accn[s & 1][j][r] = fma2(dk, pk1(Wr[r]), accn[s & 1][j][r]);
                            }
                            if (JN) {
#pragma unroll
                                for (int r = 0; r < NC; ++r) partn[r] = fma2(dk, mvn[s & 1][j][r], partn[r]);
                            }
                            if (MODE == MODE_FROB) fsum += (float)f * ((ok0 ? d0 : 0.0f) + (ok1 ? d1 : 0.0f));
                        }
                    }
                }
                if (MODE == MODE_COUNT) {
                    cnt += n_in & 0xffffu;
                    cnt_eval += n_in >> 16;
                }
                if (MODE == MODE_J) {
                    // Fold the row's 32 lane partials to 8 (lanes 0-7 then hold distinct sums)
                    // and park them in the row's own staged record, which every lane has read
                    // by now; the row's lane adds the 8 in a fixed order after the chunk.
                    const float2 p2 = up(part);
                    float ps = p2.x + p2.y;
                    ps += __shfl_xor_sync(0xffffffffu, ps, 16);
                    ps += __shfl_xor_sync(0xffffffffu, ps, 8);
                    __syncwarp();
                    if (lane < 8) reinterpret_cast<float*>(stg + bit * SR)[lane] = ps;
                }
                if (MODE == MODE_JC) {
                    // the same with (sum, low part) pairs, to 4 lanes; the row's lane adds those in FP64
                    const float2 p2 = up(part), l2 = up(partl);
                    float ps, pl = two_sum(p2.x, p2.y, ps) + (l2.x + l2.y);
#pragma unroll
                    for (int o = 16; o >= 4; o >>= 1) {
                        const float qs = __shfl_xor_sync(0xffffffffu, ps, o), ql = __shfl_xor_sync(0xffffffffu, pl, o);
                        const float low = two_sum(ps, qs, ps);
                        pl = low + (pl + ql);
                    }
                    __syncwarp();
                    if (lane < 4) reinterpret_cast<float2*>(stg + bit * SR)[lane] = make_float2(ps, pl);
                }
                if (JN) {
                    // Transposing fold: each exchange halves the columns a lane carries (NC / 2 + .. + 1
                    // shuffles), the others add the lanes that hold one column; the first of them
                    // parks the column in the row's consumed record: 6 shuffles (four columns) instead of
                    // the 20 of four butterflies (ring256, a block of 8 columns: J and J^T 10.93 -> 10.54 ms).
                    float q[NC];
#pragma unroll
                    for (int r = 0; r < NC; ++r) {
                        const float2 p2 = up(partn[r]);
                        q[r] = p2.x + p2.y;
                    }
                    constexpr int LANES = 32 / NC;   // lanes of a column
#pragma unroll
                    for (int o = 16, n = NC / 2; o >= LANES; o >>= 1, n >>= 1) {
                        const bool hi = lane & o;
#pragma unroll
                        for (int r = 0; r < n; ++r)
                            q[r] = (hi ? q[r + n] : q[r]) + __shfl_xor_sync(0xffffffffu, hi ? q[r] : q[r + n], o);
                    }
#pragma unroll
                    for (int o = LANES / 2; o > 0; o >>= 1) q[0] += __shfl_xor_sync(0xffffffffu, q[0], o);
                    __syncwarp();
                    if (lane % LANES == 0) reinterpret_cast<float*>(stg + bit * SR)[lane / LANES] = q[0];
                }
                if (MODE == MODE_FROB) dacc += (double)fsum * (double)W * (double)W;
            }
            if (J1) {
                __syncwarp();
                if (have) {
                    if (okb) {
                        const float4 r0 = stg[lane * SR + 0];
                        const float4 r1 = stg[lane * SR + 1];
                        const float Wl = stg[lane * SR + 2].x;
                        if (MODE == MODE_JC)
                            mypart64 = (((double)r0.x + (double)r0.z) + ((double)r1.x + (double)r1.z) +
                                        (double)((r0.y + r0.w) + (r1.y + r1.w))) * (double)Wl;
                        else
                            mypart = (r0.x + r0.y + r0.z + r0.w + r1.x + r1.y + r1.z + r1.w) * Wl;
                    }
                    if (MODE == MODE_JC)
                        P.vpart[e * NREG + region] = mypart64;
                    else
                        P.vout[e * NREG + region] = mypart;
                }
            }
            if (JN) {
                __syncwarp();
                if (have) {
#pragma unroll
                    for (int k = 0; k < NC / 4; ++k) {
                        float4 r0 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                        if (okb) {
                            r0 = stg[lane * SR + k];
                            const float Wl = stg[lane * SR + 2].x;
                            r0 = make_float4(r0.x * Wl, r0.y * Wl, r0.z * Wl, r0.w * Wl);
                        }
                        *reinterpret_cast<float4*>(P.vout + (e * NREG + region) * NC + 4 * k) = r0;
                    }
                }
            }
            __syncwarp();
        }

        if (JT1 || MODE == MODE_COV) {
            const uint32_t vm = lane_vmask();
#pragma unroll
            for (int s = 0; s < NSUB; ++s) {
                const int dy = sub_dy<NSUB>(s), dz = sub_dz<NSUB>(s);
                const float2 a0 = up(acc[s][0]), a1 = up(acc[s][1]);
                float av[NX_LANE] = {a0.x, a0.y, a1.x, a1.y}, lv[NX_LANE];
                if (MODE == MODE_JTC) {
                    const float2 l0 = up(accl[s][0]), l1 = up(accl[s][1]);
                    const float low[NX_LANE] = {l0.x, l0.y, l1.x, l1.y};
#pragma unroll
                    for (int t = 0; t < NX_LANE; ++t) lv[t] = two_sum(av[t], low[t], av[t]);
                }
                if (item.slot < 0) {
                    const int64_t mo = mirror_off(s);
#pragma unroll
                    for (int t = 0; t < NX_LANE; ++t)
                        if ((vm >> (4 * s + t)) & 1u) {
                            const int64_t at_v = vbase + ((int64_t)dz * P.ny + dy) * P.nx + t;
                            P.vout[at_v] = av[t];
                            if (mo != 0) P.vout[at_v + mo] = av[t];
                            if (MODE == MODE_JTC) {
                                P.vlow[at_v] = lv[t];
                                if (mo != 0) P.vlow[at_v + mo] = lv[t];
                            }
                        }
                } else {
                    // local index inside the tile: (z * 16 + y) * 16 + x
                    const int loc = (((ozi + dz) * TILE_Y) + oyi + dy) * TILE_X + oxi;
                    *reinterpret_cast<float4*>(P.gpart + (int64_t)item.slot * TILE_VOX + loc) =
                        make_float4(av[0], av[1], av[2], av[3]);
                    if (MODE == MODE_JTC)
                        *reinterpret_cast<float4*>(P.gpart_low + (int64_t)item.slot * TILE_VOX + loc) =
                            make_float4(lv[0], lv[1], lv[2], lv[3]);
                }
            }
        }
        if (JTN) {
            static_assert(!BATCH || NSUB == 2, "the batch modes take 8 x 8 x 4 regions");
            const uint32_t vm = lane_vmask();
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const int loc = ((ozi * TILE_Y) + oyi + 4 * s) * TILE_X + oxi;
#pragma unroll
                for (int r = 0; r < NC; ++r) {
                    const float2 a0 = up(accn[s][0][r]), a1 = up(accn[s][1][r]);
                    const float av[NX_LANE] = {a0.x, a0.y, a1.x, a1.y};
                    if (r >= P.ncol) continue;
                    if (item.slot < 0) {
                        const int64_t mo = mirror_off(s);
#pragma unroll
                        for (int t = 0; t < NX_LANE; ++t)
                            if ((vm >> (4 * s + t)) & 1u) {
                                float* o = P.vout + (int64_t)r * P.nvox + vbase + (int64_t)(4 * s) * P.nx + t;
                                o[0] = av[t];
                                if (mo != 0) o[mo] = av[t];
                            }
                    } else {
                        *reinterpret_cast<float4*>(P.gpart + ((int64_t)item.slot * NC + r) * TILE_VOX + loc) =
                            make_float4(av[0], av[1], av[2], av[3]);
                    }
                }
            }
        }
        if (MODE == MODE_FROB) {
            dacc = warp_sum_d(dacc);
            if (lane == 0) P.dsum[unit] = dacc;
        }
        if (MODE == MODE_COUNT) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
                cnt_eval += __shfl_xor_sync(0xffffffffu, cnt_eval, o);
            }
            if (lane == 0) {
                if (cnt) atomicAdd(P.icount, cnt);
                if (cnt_eval) atomicAdd(P.icount + 1, cnt_eval);
            }
        }
    }
}

template <int MODE, int DT, bool G, bool S, int PHI>
inline fft_status set_attr_one(size_t smem) {
    FFT_CUDA(cudaFuncSetAttribute(apply_kernel<MODE, DT, G, S, PHI>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)smem));
    return FFT_OK;
}

template <int MODE, int DT, int PHI>
inline fft_status set_attr_dt(size_t smem) {
    fft_status rc;
    if ((rc = set_attr_one<MODE, DT, false, false, PHI>(smem)) != FFT_OK) return rc;
    if ((rc = set_attr_one<MODE, DT, true, false, PHI>(smem)) != FFT_OK) return rc;
    if ((rc = set_attr_one<MODE, DT, false, true, PHI>(smem)) != FFT_OK) return rc;
    return set_attr_one<MODE, DT, true, true, PHI>(smem);
}

template <int MODE>
inline fft_status set_attr_mode_impl(size_t smem) {
    fft_status rc;
    if ((rc = set_attr_dt<MODE, FFT_DT_STABLE, PHI_TABLE>(smem)) != FFT_OK) return rc;
    if ((rc = set_attr_dt<MODE, FFT_DT_NAIVE, PHI_TABLE>(smem)) != FFT_OK) return rc;
    if (MODE != MODE_COUNT && (rc = set_attr_dt<MODE, FFT_DT_STABLE, PHI_TRIG>(smem)) != FFT_OK) return rc;
    if (MODE != MODE_COUNT && (rc = set_attr_dt<MODE, FFT_DT_STABLE, PHI_SEG>(smem)) != FFT_OK) return rc;
    return set_attr_one<MODE, FFT_DT_FP64, false, false, PHI_TABLE>(smem);
}

size_t apply_smem(fft_geom g, int warps);
size_t apply_smem8(fft_geom g, int warps);
// Resident CTAs per SM of the J^T kernel (stable detour, tables; plain or sharp).
int apply_blocks_per_sm(bool sharp, int threads, size_t smem);

// One apply launch over P's items: sharp single-column variants in the geometry's sharp CTA
// shape, plain stable-detour table variants in the plain shape, the others in 8-warp CTAs on
// the persistent grid.
template <int MODE, int DT, bool G, bool S, int PHI>
inline void launch_apply(fft_geom g, const ApplyParams& P, cudaStream_t st) {
    if (apply_ncol<MODE>() == 8) {
        apply_kernel<MODE, DT, G, S, PHI><<<g->sms, 32 * col8_warps<S>(), apply_smem8(g, col8_warps<S>()), st>>>(P);
    } else if (apply_sharp_wide<MODE, DT, S, PHI>()) {
        const int w = std::min(g->sharp_warps, sharp_bound_warps<MODE>());
        apply_kernel<MODE, DT, G, S, PHI><<<g->sharp_ctas, 32 * w, apply_smem(g, w), st>>>(P);
    } else if (apply_plain_wide<MODE, DT, S, PHI>() && g->plain_warps > APPLY_WARPS) {
        apply_kernel<MODE, DT, G, S, PHI><<<g->plain_ctas, 32 * g->plain_warps, apply_smem(g, g->plain_warps), st>>>(P);
    } else {
        apply_kernel<MODE, DT, G, S, PHI><<<g->apply_ctas, APPLY_THREADS, apply_smem(g), st>>>(P);
    }
}

// A sharp geometry's plain items (rows of bands whose Phi vanishes at the cut) run in the plain
// variant, its sharp-band items in the sharp one: two launches, each pulling units from its own
// counter. Other geometries run all items in one launch.
template <int MODE, int DT, bool G, int PHI>
inline void launch_split(fft_geom g, const ApplyParams& P, cudaStream_t st) {
    if (!g->sharp) {
        launch_apply<MODE, DT, G, false, PHI>(g, P, st);
        return;
    }
    const int np = g->n_items_plain, ns = g->n_items - g->n_items_plain;
    if (np > 0) {
        ApplyParams Q = P;
        Q.n_items = np;
        launch_apply<MODE, DT, G, false, PHI>(g, Q, st);
    }
    if (ns > 0) {
        ApplyParams Q = P;
        Q.items = P.items + np;
        Q.n_items = ns;
        Q.counter = P.counter + 1;
        // (per-unit partials follow the plain launch's)
        if (Q.dsum) Q.dsum = P.dsum + (size_t)np * apply_regions<MODE>();
        launch_apply<MODE, DT, G, true, PHI>(g, Q, st);
    }
}

template <int MODE>
inline fft_status launch_mode_impl(fft_geom g, const ApplyParams& P, cudaStream_t st) {
    if (g->unusable) return check_usable(g);
    FFT_CUDA(cudaMemsetAsync(g->counter, 0, 2 * sizeof(int32_t), st));
    if (g->n_items == 0) return FFT_OK;
    // MODE_COUNT evaluates no Phi: the table variant serves every representation
    constexpr int PHI_T = MODE == MODE_COUNT ? PHI_TABLE : PHI_TRIG, PHI_S = MODE == MODE_COUNT ? PHI_TABLE : PHI_SEG;
#define FFT_LAUNCH_GS(DTV, PV)                                      \
    do {                                                            \
        if (g->guard) launch_split<MODE, DTV, true, PV>(g, P, st);  \
        else launch_split<MODE, DTV, false, PV>(g, P, st);          \
    } while (0)
    if (g->phi_eval == PHI_TRIG) {   // geometry creation guarantees dt_mode STABLE for series
        FFT_LAUNCH_GS(FFT_DT_STABLE, PHI_T);
    } else if (g->phi_eval == PHI_SEG) {
        FFT_LAUNCH_GS(FFT_DT_STABLE, PHI_S);
    } else if (g->dt_mode == FFT_DT_STABLE) {
        FFT_LAUNCH_GS(FFT_DT_STABLE, PHI_TABLE);
    } else if (g->dt_mode == FFT_DT_NAIVE) {
        FFT_LAUNCH_GS(FFT_DT_NAIVE, PHI_TABLE);
    } else {   // FP64 detour: the cut is decided in FP64 everywhere, one plain launch
        launch_apply<MODE, FFT_DT_FP64, false, false, PHI_TABLE>(g, P, st);
    }
#undef FFT_LAUNCH_GS
    FFT_CUDA(cudaGetLastError());
    return FFT_OK;
}

// The modes that exist for the stable detour only: batches, compensated sums.
template <int MODE>
inline fft_status launch_batch_impl(fft_geom g, const ApplyParams& P, cudaStream_t st) {
    if (g->unusable) return check_usable(g);
    FFT_CUDA(cudaMemsetAsync(g->counter, 0, 2 * sizeof(int32_t), st));
    if (g->n_items == 0) return FFT_OK;
#define FFT_LAUNCH_G(PV)                                                          \
    do {                                                                          \
        if (g->guard) launch_split<MODE, FFT_DT_STABLE, true, PV>(g, P, st);      \
        else launch_split<MODE, FFT_DT_STABLE, false, PV>(g, P, st);              \
    } while (0)
    if (g->phi_eval == PHI_TRIG)
        FFT_LAUNCH_G(PHI_TRIG);
    else if (g->phi_eval == PHI_SEG)
        FFT_LAUNCH_G(PHI_SEG);
    else
        FFT_LAUNCH_G(PHI_TABLE);
#undef FFT_LAUNCH_G
    FFT_CUDA(cudaGetLastError());
    return FFT_OK;
}

// Entry points of the modes' translation units (fft_apply_*.cu): each instantiates its own
// kernels, so that they compile in parallel.
template <int MODE>
fft_status launch_mode(fft_geom g, const ApplyParams& P, cudaStream_t st);
template <int MODE>
fft_status launch_batch(fft_geom g, const ApplyParams& P, cudaStream_t st);
template <int MODE>
fft_status set_attr_mode(size_t smem);
template <> fft_status launch_mode<MODE_JT>(fft_geom g, const ApplyParams& P, cudaStream_t st);
template <> fft_status launch_mode<MODE_J>(fft_geom g, const ApplyParams& P, cudaStream_t st);
template <> fft_status launch_mode<MODE_JTC>(fft_geom g, const ApplyParams& P, cudaStream_t st);
template <> fft_status launch_mode<MODE_JC>(fft_geom g, const ApplyParams& P, cudaStream_t st);
template <> fft_status launch_mode<MODE_COUNT>(fft_geom g, const ApplyParams& P, cudaStream_t st);
template <> fft_status launch_mode<MODE_FROB>(fft_geom g, const ApplyParams& P, cudaStream_t st);
template <> fft_status launch_mode<MODE_COV>(fft_geom g, const ApplyParams& P, cudaStream_t st);
template <> fft_status launch_batch<MODE_JT4>(fft_geom g, const ApplyParams& P, cudaStream_t st);
template <> fft_status launch_batch<MODE_JT8>(fft_geom g, const ApplyParams& P, cudaStream_t st);
template <> fft_status launch_batch<MODE_J4>(fft_geom g, const ApplyParams& P, cudaStream_t st);
template <> fft_status launch_batch<MODE_J8>(fft_geom g, const ApplyParams& P, cudaStream_t st);
template <> fft_status set_attr_mode<MODE_JT>(size_t smem);
template <> fft_status set_attr_mode<MODE_J>(size_t smem);
template <> fft_status set_attr_mode<MODE_JTC>(size_t smem);
template <> fft_status set_attr_mode<MODE_JC>(size_t smem);
template <> fft_status set_attr_mode<MODE_COUNT>(size_t smem);
template <> fft_status set_attr_mode<MODE_FROB>(size_t smem);
template <> fft_status set_attr_mode<MODE_COV>(size_t smem);
template <> fft_status set_attr_mode<MODE_JT4>(size_t smem);
template <> fft_status set_attr_mode<MODE_JT8>(size_t smem);
template <> fft_status set_attr_mode<MODE_J4>(size_t smem);
template <> fft_status set_attr_mode<MODE_J8>(size_t smem);

}  // namespace fftgb
