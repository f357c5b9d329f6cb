// J m and J^T d with every entry of J recomputed inside each product instead of stored
// (Sec. II-C), tile-centric on sm_103a.
//
// Work decomposition
//   * The voxel grid is cut into 16 x 16 x 8 tiles. Each tile has a list of candidate rows
//     (built once per geometry by a conservative cull). A work item is a tile and a range of
//     its rows; a unit is one region of one item: an 8 x 8 x 8 region (four 8 x 4 x 4
//     sub-bricks, four regions per tile) for the single-column modes, an 8 x 8 x 4 region
//     (two sub-bricks, eight per tile) for the four-column ones. Every warp of the persistent
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
//     load, linear interpolation), geometric factor 1 / (R_xs R_xr).
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
// MODE_JT4 / MODE_J4: J^T and J for four right-hand sides at once (every evaluated entry is
// applied to all four; blocks are column-major: column r at r * V or r * M).
enum { MODE_JT = 0, MODE_J = 1, MODE_COUNT = 2, MODE_FROB = 3, MODE_COV = 4, MODE_JT4 = 5, MODE_J4 = 6 };
constexpr int STG_PER_WARP = 128;   // staged float4 per warp: 32 rows x (3 or 4)

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
    double org[3];
    double h;
    const float* vin;        // J: m [V]; J^T: d [M]
    float* vout;             // J: jpart [E * 4]; J^T: g [V]
    float* gpart;            // J^T partials of multi-item tiles
    double* dsum;            // FROB: one per unit [n_items * 4]
    unsigned long long* icount;   // COUNT
    int trig_nq;             // PHI_TRIG: coefficient groups of 4 per band
    int seg_n;               // PHI_SEG: segments per band
    int64_t nvox, nrow;      // column lengths of the batch modes' blocks (V, M)
};

// Phi of the normalised detour v (table lookup, sine series or its piecewise quadratics, see
// fft_device.cuh): tb is the band data's shared address (PHI_SEG: the bits of the band's magic
// number, `tab` the shared address of all bands' segments and `seg2` that of their c2).
template <int PHI>
__device__ __forceinline__ float phi_eval(float v, uint32_t tb, float nm1, int nq, uint32_t tab, uint32_t seg2) {
    if (PHI == PHI_TRIG) return phi_trig(v, tb, nq);
    if (PHI == PHI_SEG) return phi_seg(v, __uint_as_float(tb), nm1, tab, seg2);
    return phi_lookup(v, tb, nm1);
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
    return (SHARP || MODE == MODE_JT4 || MODE == MODE_J4) ? 2
                                                          : ((DT == FFT_DT_STABLE && PHI != PHI_TRIG) ? 4 : 3);
}

// Sub-bricks per unit and units (regions) per item of each mode: see sub_dy below.
template <int MODE>
constexpr int apply_nsub() {
    return (MODE == MODE_JT4 || MODE == MODE_J4) ? 2 : 4;
}
template <int MODE>
constexpr int apply_regions() {
    return 16 / apply_nsub<MODE>();   // 16 sub-bricks of 8 x 4 x 4 per 16 x 16 x 8 tile
}

// Sub-bricks of a unit. The single-column modes take an 8 x 8 x 8 region (NSUB = 4) and the
// four-column modes, whose per-voxel state is four times larger, an 8 x 8 x 4 region (NSUB =
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

// The FP64 re-decision of the sharp-band kernels, out of line (called only for an entry where
// some lane's FP32 detour lies within CUT_BAND of the cut), so that its FP64 temporaries do not
// weigh on the register allocation of the main loop. For each of the lane's 4 NSUB voxels
// (k = 4 s + t) it recomputes the FP32 detour by the operations of the main pass, and for the
// voxels near the cut re-decides dt < dt_max in FP64. It returns in d[k] what the main pass's
// term has to change by: val2 - val1 (J, J^T, four-column modes), |val2| - |val1| (coverage),
// val2^2 - val1^2 (Frobenius), +1 / -1 (support count), 0 where nothing changes. `inner` holds
// the sub-bricks lying between the transducer planes (bit s).
template <int MODE, int DT, bool GUARD, int PHI, int NSUB>
__device__ __noinline__ void sharp_fix(const ApplyParams& P, float4 A, float4 B, float4 C, float Xl, float Yl,
                                       float Zl, bool planar, uint32_t inner_bits, float cutb, uint32_t tb,
                                       float nm1, int nq, uint32_t tab, uint32_t seg2, int ix0, int iy0, int iz0,
                                       float* d) {
    const float hx = B.x, hy = B.y, hz = B.z;
    const float hl = 0.5f * (A.x - A.y);
    const int b = __float_as_int(C.w) & 0xff;
    const double U = P.bc[b].U;
    // one voxel per iteration, each recomputed from the lane base (few values live across
    // iterations, which keeps the caller's register saves around this call small)
#pragma unroll 1
    for (int k = 0; k < 4 * NSUB; ++k) {
        const int s = k >> 2, t = k & 3;
        d[k] = 0.0f;
        const float offs = planar ? fmaf(Xl, hx, Yl * hy) : fmaf(Xl, hx, fmaf(Yl, hy, Zl * hz));
        float pss = A.x + offs, prs = A.y + offs;
        float c1s = planar ? fmaf(-Zl, hy, A.z) : fmaf(Yl, hz, fmaf(-Zl, hy, A.z));
        float c2s = planar ? fmaf(Zl, hx, A.w) : fmaf(Zl, hx, fmaf(-Xl, hz, A.w));
        float c3s = fmaf(Xl, hy, fmaf(-Yl, hx, B.w));
#pragma unroll 1
        for (int q = 1; q <= s; ++q) {
            if (planar)
                sub_step<NSUB, true>(q, hx, hy, hz, pss, prs, c1s, c2s, c3s);
            else
                sub_step<NSUB, false>(q, hx, hy, hz, pss, prs, c1s, c2s, c3s);
        }
        const float ft = (float)t;
        const float c1sq = c1s * c1s;
        const float pst = (t == 0 ? pss : fmaf(ft, hx, pss));
        const float prt = (t == 0 ? prs : fmaf(ft, hx, prs));
        const float c3t = (t == 0 ? c3s : fmaf(ft, hy, c3s));
        float q2;
        if (planar) {
            q2 = fmaf(c3t, c3t, fmaf(c2s, c2s, c1sq));
        } else {
            const float c2t = (t == 0 ? c2s : fmaf(-ft, hz, c2s));
            q2 = fmaf(c2t, c2t, fmaf(c3t, c3t, c1sq));
        }
        const bool inner = (DT == FFT_DT_STABLE) && ((inner_bits >> s) & 1u);
        float is, ir;
        const float vr = inner ? detour_v<DT, GUARD, true, true>(pst, prt, q2, hl, is, ir)
                               : detour_v<DT, GUARD, false, true>(pst, prt, q2, hl, is, ir);
        if (!(fabsf(vr - 1.0f) < cutb)) continue;
        const float v = __saturatef(vr);
        const bool in = in_support64(P.rec64[__float_as_int(C.z)], P.org[0], P.org[1], P.org[2], P.h, ix0 + t,
                                     iy0 + sub_dy<NSUB>(s), iz0 + sub_dz<NSUB>(s), U);
        const float v2 = settle_cut(v, in);
        if (v2 == v) continue;
        if (MODE == MODE_COUNT) {
            d[k] = (v2 < 1.0f) ? 1.0f : -1.0f;
            continue;
        }
        const float w = is * ir;
        const float val1 = phi_eval<PHI>(v, tb, nm1, nq, tab, seg2) * w;
        const float val2 = phi_eval<PHI>(v2, tb, nm1, nq, tab, seg2) * w;
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
    return SHARP && DT == FFT_DT_STABLE && PHI != PHI_TRIG && MODE != MODE_JT4 && MODE != MODE_J4;
}
constexpr int SHARP_MAX_WARPS = 20;

// The plain stable-detour table variants (single column) are built for blocks of up to 24
// warps at one per SM, i.e. 80 registers: their 16 per-lane voxels (8 x 8 x 8 units) want more
// than 64, and one wide CTA shares one copy of the band tables. Measured against 32 warps at
// 64 registers: slices3d J^T 408.0 -> 407.6 ms, J 412.6 -> 411.4 ms, ring256 J^T 3.75 -> 3.72 ms.
template <int MODE, int DT, bool SHARP, int PHI>
constexpr bool apply_plain_wide() {
    return !SHARP && DT == FFT_DT_STABLE && PHI != PHI_TRIG && MODE != MODE_JT4 && MODE != MODE_J4;
}
constexpr int PLAIN_MAX_WARPS = 24;

template <int MODE, int DT, bool SHARP, int PHI>
constexpr int apply_block_bound() {
    return apply_sharp_wide<MODE, DT, SHARP, PHI>()   ? 32 * SHARP_MAX_WARPS
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
    // table lookups scale v by n_tab - 1, segment lookups by seg_n 2^-22
    const float nm1 = PHI == PHI_SEG ? (float)P.seg_n * MAGIC2_ULP : (float)(P.n_tab - 1);
    const uint32_t seg2_addr = tab_addr + (uint32_t)(P.n_bands * (P.seg_n + SEG_PAD)) * 8u;
    const int nq = P.trig_nq;
    const int lx = lane & 1, ly = (lane >> 1) & 3, lz = lane >> 3;
    constexpr bool BATCH = (MODE == MODE_JT4 || MODE == MODE_J4);
    constexpr int SR = BATCH ? 4 : 3;   // staged float4 per row
    constexpr int NSUB = apply_nsub<MODE>();
    constexpr int NREG = apply_regions<MODE>();
    constexpr bool FLAGW = (NSUB == 4);
    float4* stg = s_stage + warp * STG_PER_WARP;
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
                if (TZ + ozi + sub_dz<NSUB>(s) < P.nz && TY + oyi + sub_dy<NSUB>(s) < P.ny) {
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
            if (TX + 8 * wx < P.nx && TY + 8 * wy + sub_dy<NSUB>(s) < P.ny && TZ + 4 * wz + sub_dz<NSUB>(s) < P.nz)
                sub_ok |= 1u << s;
        // the gather modes need the mask only for their stores: recomputed there
        constexpr bool VM_LIVE = !(MODE == MODE_JT || MODE == MODE_COV || MODE == MODE_JT4);
        const uint32_t vmask = VM_LIVE ? lane_vmask() : 0u;
        const int64_t vbase = ((int64_t)(TZ + ozi) * P.ny + TY + oyi) * P.nx + TX + oxi;

        float acc[NSUB][NX_LANE];
        float mv[NSUB][NX_LANE];
        float acc4[2][NX_LANE][4];   // four-column modes only (NSUB = 2)
        float mv4[2][NX_LANE][4];
        double dacc = 0.0;
        unsigned long long cnt = 0, cnt_eval = 0;
#pragma unroll
        for (int s = 0; s < NSUB; ++s)
#pragma unroll
            for (int t = 0; t < NX_LANE; ++t) {
                const int64_t vo = vbase + ((int64_t)sub_dz<NSUB>(s) * P.ny + sub_dy<NSUB>(s)) * P.nx + t;
                acc[s][t] = 0.0f;
                mv[s][t] = 0.0f;
                if (MODE == MODE_J && ((vmask >> (4 * s + t)) & 1u)) mv[s][t] = __ldg(P.vin + vo);
                if (BATCH && s < 2) {
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        acc4[s & 1][t][r] = 0.0f;
                        mv4[s & 1][t][r] = 0.0f;
                        if (MODE == MODE_J4 && ((vmask >> (4 * s + t)) & 1u))
                            mv4[s & 1][t][r] = __ldg(P.vin + (int64_t)r * P.nvox + vo);
                    }
                }
            }

        for (int64_t e0 = item.e0; e0 < item.e1; e0 += 32) {
            // ---- stage: lane l prepares row e0 + l
            const int64_t e = e0 + lane;
            const bool have = e < item.e1;
            uint32_t okb = 0, inb = 0;   // sub-bricks the row may reach / lying between its transducer planes
            if (have) {
                const int p = P.tile_rows[e];
                const float4 base = P.ebase[e];
                const float base3 = P.ebase3[e];
                const RowRec r = P.rec[p];
                const int b = P.row_band[p];
                const BandConst bc = P.bc[b];
                const float hb = bc.h;
                float W = r.b.w;
                if (MODE == MODE_JT) W *= __ldg(P.vin + p);
                if (MODE == MODE_COV) W = fabsf(W) * (P.vin ? fabsf(__ldg(P.vin + p)) : 1.0f);
                float4 W4 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (MODE == MODE_JT4)
                    W4 = make_float4(W * __ldg(P.vin + p), W * __ldg(P.vin + P.nrow + p),
                                     W * __ldg(P.vin + 2 * P.nrow + p), W * __ldg(P.vin + 3 * P.nrow + p));
                const float ex = r.b.x, ey = r.b.y, ez = r.b.z, hl = r.a.w;
                // sub-brick centres relative to the pair midpoint (FP32; used by the bound only)
                const float dx = fmaf((float)TX, hb, bc.org[0]) - r.a.x;
                const float dy = fmaf((float)TY, hb, bc.org[1]) - r.a.y;
                const float dz = fmaf((float)TZ, hb, bc.org[2]) - r.a.z;
                const float cx = fmaf(8.0f * wx + 3.5f, hb, dx);
                const float hxx = 3.5f * hb, hyy = 1.5f * hb;
                // rows with zero weight add exactly nothing to J^T: skip them
                const bool live = (MODE == MODE_JT4) ? (W4.x != 0.0f || W4.y != 0.0f || W4.z != 0.0f || W4.w != 0.0f)
                                                     : ((MODE != MODE_JT && MODE != MODE_COV) || (W != 0.0f));
                const float pext = hxx * fabsf(ex) + hyy * (fabsf(ey) + fabsf(ez)) + 1e-3f;
#pragma unroll
                for (int s = 0; s < NSUB; ++s) {
                    const float cy = fmaf(8.0f * wy + (float)sub_dy<NSUB>(s) + 1.5f, hb, dy);
                    const float cz = fmaf(4.0f * wz + (float)sub_dz<NSUB>(s) + 1.5f, hb, dz);
                    if (live && ((sub_ok >> s) & 1u) && box_may_touch(cx, cy, cz, ex, ey, ez, hl, hxx, hyy, hyy))
                        okb |= 1u << s;
                    // sub-bricks whose voxels all satisfy |p| <= hl (between the transducer planes)
                    if (fabsf(fmaf(cx, ex, fmaf(cy, ey, cz * ez))) + pext <= hl) inb |= 1u << s;
                }
                const uint32_t tb =
                    PHI == PHI_SEG ? __float_as_uint(fmaf((float)(b * (P.seg_n + SEG_PAD)), MAGIC2_ULP, MAGIC2))
                                   : tab_addr + (uint32_t)(b * P.n_tab) * 8u - (PHI == PHI_TABLE ? MAGIC_BITS_X8 : 0u);
                stg[lane * SR + 0] = base;
                stg[lane * SR + 1] = make_float4(hb * ex, hb * ey, hb * ez, base3);
                if (MODE == MODE_JT4) stg[lane * SR + 3] = W4;
                // planar pair (both transducers at one z): stepping along x changes only c3
                const int planar = (ez == 0.0f) ? 1 : 0;
                // flags word: band (bits 0-7), sharp band (8), planar pair (9); with four
                // sub-bricks also the sub-bricks the row may reach (12 + s) and the inner ones
                // (16 + s)
                const uint32_t fl = FLAGW ? ((okb << 12) | (inb << 16)) : 0u;
                stg[lane * SR + 2] = make_float4(W, __uint_as_float(tb), __int_as_float(p),
                                                __int_as_float(b | (bc.sharp << 8) | (planar << 9) | (int)fl));
            }
            // With two sub-bricks the per-row tests read warp-uniform ballots (uniform branches);
            // with four, the row's staged flag word (eight ballots per chunk cost more there).
            uint32_t mk[NSUB], ik[NSUB];
#pragma unroll
            for (int s = 0; s < NSUB; ++s) {
                mk[s] = FLAGW ? 0u : __ballot_sync(0xffffffffu, (okb >> s) & 1u);
                ik[s] = FLAGW ? 0u : __ballot_sync(0xffffffffu, (inb >> s) & 1u);
            }
            uint32_t mm = __ballot_sync(0xffffffffu, okb != 0u);
            __syncwarp();
            float mypart = 0.0f;
            float mypart4[4] = {0.0f, 0.0f, 0.0f, 0.0f};
            while (mm) {
                const int bit = __ffs(mm) - 1;
                mm &= mm - 1;
                const float4 A = stg[bit * SR + 0];
                const float4 B = stg[bit * SR + 1];
                const float4 C = stg[bit * SR + 2];
                const float4 W4 = (MODE == MODE_JT4) ? stg[bit * SR + 3] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                const float Wr[4] = {W4.x, W4.y, W4.z, W4.w};
                const float hx = B.x, hy = B.y, hz = B.z, W = C.x;
                const float hl = 0.5f * (A.x - A.y);   // used by the textbook (NAIVE) detour only
                const uint32_t tb = __float_as_uint(C.y);
                const uint32_t cw = (uint32_t)__float_as_int(C.w);
                // voxels whose FP32 detour falls within CUT_BAND of a sharp band's cut-off
                const float cutb = (SHARP && ((cw >> 8) & 1u)) ? CUT_BAND : -1.0f;
                const bool planar = (DT != FFT_DT_FP64) && ((cw >> 9) & 1u);
                bool near = false;   // a voxel of this lane has its FP32 detour within CUT_BAND of the cut
                // lane base (sub-brick 0, t = 0) in the pair frame: small offsets added to the
                // tile origin's FP64-derived values
                float part = 0.0f;
                float part4[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                // The entry's evaluation, specialised for planar pairs (both transducers at one
                // z: the axis has no z component, so h_z = 0 exactly, c1 and c2 do not change
                // along the lane's voxels or between sub-bricks at one z, and p does not change
                // in z).
                // SH: the near-cut checks, only for rows of a band whose Phi does not vanish at
                // the cut (the other rows of a sharp geometry take the plain evaluation; both
                // give the same values there).
                auto entry_body = [&](auto planar_tag, auto sharp_tag) {
                    constexpr bool PL = decltype(planar_tag)::value;
                    constexpr bool SH = decltype(sharp_tag)::value;
                const float off = PL ? fmaf(Xl, hx, Yl * hy) : fmaf(Xl, hx, fmaf(Yl, hy, Zl * hz));
                float psb = A.x + off, prb = A.y + off;
                float c1 = PL ? fmaf(-Zl, hy, A.z) : fmaf(Yl, hz, fmaf(-Zl, hy, A.z));
                float c2 = PL ? fmaf(Zl, hx, A.w) : fmaf(Zl, hx, fmaf(-Xl, hz, A.w));
                float c3 = fmaf(Xl, hy, fmaf(-Yl, hx, B.w));
                float c12_planar = PL ? fmaf(c2, c2, c1 * c1) : 0.0f;
#pragma unroll
                for (int s = 0; s < NSUB; ++s) {
                    if (s > 0) {
                        sub_step<NSUB, PL>(s, hx, hy, hz, psb, prb, c1, c2, c3);
                        if (PL && s == 2) c12_planar = fmaf(c2, c2, c1 * c1);
                    }
                    if (!(FLAGW ? ((cw >> (12 + s)) & 1u) : ((mk[s] >> bit) & 1u))) continue;
                    const float c1sq = PL ? 0.0f : c1 * c1;
                    const bool inner = (DT == FFT_DT_STABLE) &&
                                       (FLAGW ? ((cw >> (16 + s)) & 1u) : ((ik[s] >> bit) & 1u));
#define FFT_EVAL_SUB(INNER_V, PLANAR_V)                                                              \
    float vv[NX_LANE], ww[NX_LANE];                                                                \
    _Pragma("unroll") for (int t = 0; t < NX_LANE; ++t) {                                          \
        const float ft = (float)t;                                                                 \
        float is, ir, v, w;                                                                        \
        if (DT == FFT_DT_FP64) {                                                                   \
            const RowRec64 r64 = P.rec64[__float_as_int(C.z)];                                     \
            const int b = (int)(cw & 0xffu);                                                       \
            v = detour_v64(r64, P.org[0], P.org[1], P.org[2], P.h, TX + oxi + t,                   \
                           TY + oyi + sub_dy<NSUB>(s), TZ + ozi + sub_dz<NSUB>(s), P.bc[b].U, w);  \
            is = 1.0f;                                                                             \
            ir = w;                                                                                \
        } else {                                                                                   \
            const float pst = (t == 0 ? psb : fmaf(ft, hx, psb));                                  \
            const float prt = (t == 0 ? prb : fmaf(ft, hx, prb));                                  \
            const float c3t = (t == 0 ? c3 : fmaf(ft, hy, c3));                                    \
            float q2;                                                                              \
            if (PLANAR_V) {                                                                        \
                q2 = fmaf(c3t, c3t, c12sq);                                                        \
            } else {                                                                               \
                const float c2t = (t == 0 ? c2 : fmaf(-ft, hz, c2));                               \
                q2 = fmaf(c2t, c2t, fmaf(c3t, c3t, c1sq));                                         \
            }                                                                                      \
            if (SH) {                                                                              \
                v = detour_v<DT, GUARD, INNER_V, true>(pst, prt, q2, hl, is, ir);                  \
                near |= (fabsf(v - 1.0f) < cutb);                                                  \
                v = __saturatef(v);                                                                \
            } else {                                                                               \
                v = detour_v<DT, GUARD, INNER_V>(pst, prt, q2, hl, is, ir);                        \
            }                                                                                      \
        }                                                                                          \
        if (MODE == MODE_COUNT) {                                                                  \
            if ((vmask >> (4 * s + t)) & 1u) {                                                     \
                ++cnt_eval;                                                                        \
                if (v < 1.0f) ++cnt;                                                               \
            }                                                                                      \
            continue;                                                                              \
        }                                                                                          \
        if constexpr (PHI == PHI_TRIG) {                                                           \
            vv[t] = v;                                                                             \
            ww[t] = is * ir;                                                                       \
            continue;                                                                              \
        }                                                                                          \
        const float val = phi_eval<PHI>(v, tb, nm1, nq, tab_addr, seg2_addr) * (is * ir);          \
        if (MODE == MODE_JT) acc[s][t] = fmaf(val, W, acc[s][t]);                                  \
        if (MODE == MODE_COV) acc[s][t] = fmaf(fabsf(val), W, acc[s][t]);                          \
        if (MODE == MODE_JT4) {                                                                    \
            _Pragma("unroll") for (int r = 0; r < 4; ++r) acc4[s & 1][t][r] = fmaf(val, Wr[r], acc4[s & 1][t][r]); \
        }                                                                                          \
        if (MODE == MODE_J4) {                                                                     \
            _Pragma("unroll") for (int r = 0; r < 4; ++r) part4[r] = fmaf(val, mv4[s & 1][t][r], part4[r]); \
        }                                                                                          \
        if (MODE == MODE_J) part = fmaf(val, mv[s][t], part);                                      \
        if (MODE == MODE_FROB) {                                                                   \
            if ((vmask >> (4 * s + t)) & 1u) part = fmaf(val, val, part);                          \
        }                                                                                          \
    }                                                                                              \
    if constexpr (PHI == PHI_TRIG && MODE != MODE_COUNT) {                                         \
        float ph[NX_LANE];                                                                         \
        phi_trig_n<NX_LANE>(vv, tb, nq, ph);                                                       \
        _Pragma("unroll") for (int t = 0; t < NX_LANE; ++t) {                                      \
            const float val = ph[t] * ww[t];                                                       \
            if (MODE == MODE_JT) acc[s][t] = fmaf(val, W, acc[s][t]);                              \
            if (MODE == MODE_COV) acc[s][t] = fmaf(fabsf(val), W, acc[s][t]);                      \
            if (MODE == MODE_JT4) {                                                                \
                _Pragma("unroll") for (int r = 0; r < 4; ++r) acc4[s & 1][t][r] = fmaf(val, Wr[r], acc4[s & 1][t][r]); \
            }                                                                                      \
            if (MODE == MODE_J4) {                                                                 \
                _Pragma("unroll") for (int r = 0; r < 4; ++r) part4[r] = fmaf(val, mv4[s & 1][t][r], part4[r]); \
            }                                                                                      \
            if (MODE == MODE_J) part = fmaf(val, mv[s][t], part);                                  \
            if (MODE == MODE_FROB) {                                                               \
                if ((vmask >> (4 * s + t)) & 1u) part = fmaf(val, val, part);                      \
            }                                                                                      \
        }                                                                                          \
    }
                    const float c12sq = PL ? c12_planar : fmaf(c2, c2, c1sq);
                    if (inner) {
                        FFT_EVAL_SUB(true, PL)
                    } else {
                        FFT_EVAL_SUB(false, PL)
                    }
                }
                };
                if (SHARP && cutb > 0.0f) {
                    if (planar)
                        entry_body(std::true_type{}, std::integral_constant<bool, SHARP>{});
                    else
                        entry_body(std::false_type{}, std::integral_constant<bool, SHARP>{});
                } else {
                    if (planar)
                        entry_body(std::true_type{}, std::false_type{});
                    else
                        entry_body(std::false_type{}, std::false_type{});
                }
#undef FFT_EVAL_SUB
                if (SHARP && DT != FFT_DT_FP64 && __any_sync(0xffffffffu, near)) {
                    // FP64 re-decision of the voxels whose FP32 detour lies within CUT_BAND of
                    // the cut; d[k] is the change of this entry's term for voxel k = 4 s + t
                    float d[4 * NSUB];
                    uint32_t inner_bits = (cw >> 16) & 15u;
                    if (!FLAGW) {
                        inner_bits = 0u;
#pragma unroll
                        for (int s = 0; s < NSUB; ++s) inner_bits |= ((ik[s] >> bit) & 1u) << s;
                    }
                    if (near)
                        sharp_fix<MODE, DT, GUARD, PHI, NSUB>(P, A, B, C, Xl, Yl, Zl, planar, inner_bits, cutb, tb, nm1,
                                                              nq, tab_addr, seg2_addr, TX + oxi, TY + oyi, TZ + ozi, d);
#pragma unroll
                    for (int s = 0; s < NSUB; ++s) {
#pragma unroll
                        for (int t = 0; t < NX_LANE; ++t) {
                            const float dk = near ? d[4 * s + t] : 0.0f;
                            if (dk == 0.0f) continue;
                            const bool valid = (vmask >> (4 * s + t)) & 1u;
                            if (MODE == MODE_COUNT && valid) cnt += (dk > 0.0f) ? 1ull : ~0ull;
                            if (MODE == MODE_JT || MODE == MODE_COV) acc[s][t] = fmaf(dk, W, acc[s][t]);
                            if (MODE == MODE_J) part = fmaf(dk, mv[s][t], part);
                            if (MODE == MODE_JT4) {
#pragma unroll
                                for (int r = 0; r < 4; ++r) acc4[s & 1][t][r] = fmaf(dk, Wr[r], acc4[s & 1][t][r]);
                            }
                            if (MODE == MODE_J4) {
#pragma unroll
                                for (int r = 0; r < 4; ++r) part4[r] = fmaf(dk, mv4[s & 1][t][r], part4[r]);
                            }
                            if (MODE == MODE_FROB && valid) part += dk;
                        }
                    }
                }
                if (MODE == MODE_J) {
                    // Fold the row's 32 lane partials to 8 (lanes 0-7 then hold distinct sums)
                    // and park them in the row's own staged record, which every lane has read
                    // by now; the row's lane adds the 8 in a fixed order after the chunk.
                    part += __shfl_xor_sync(0xffffffffu, part, 16);
                    part += __shfl_xor_sync(0xffffffffu, part, 8);
                    __syncwarp();
                    if (lane < 8) reinterpret_cast<float*>(stg + bit * SR)[lane] = part;
                }
                if (MODE == MODE_J4) {
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const float pr4 = warp_sum(part4[r]);
                        if (lane == bit) mypart4[r] = pr4 * W;
                    }
                }
                if (MODE == MODE_FROB) dacc += (double)part * (double)W * (double)W;
            }
            if (MODE == MODE_J) {
                __syncwarp();
                if (have) {
                    if (okb) {
                        const float4 r0 = stg[lane * SR + 0];
                        const float4 r1 = stg[lane * SR + 1];
                        const float Wl = stg[lane * SR + 2].x;
                        mypart = (r0.x + r0.y + r0.z + r0.w + r1.x + r1.y + r1.z + r1.w) * Wl;
                    }
                    P.vout[e * NREG + region] = mypart;
                }
            }
            if (MODE == MODE_J4 && have)
                *reinterpret_cast<float4*>(P.vout + (e * NREG + region) * 4) =
                    make_float4(mypart4[0], mypart4[1], mypart4[2], mypart4[3]);
            __syncwarp();
        }

        if (MODE == MODE_JT || MODE == MODE_COV) {
            const uint32_t vm = lane_vmask();
#pragma unroll
            for (int s = 0; s < NSUB; ++s) {
                const int dy = sub_dy<NSUB>(s), dz = sub_dz<NSUB>(s);
                if (item.slot < 0) {
#pragma unroll
                    for (int t = 0; t < NX_LANE; ++t)
                        if ((vm >> (4 * s + t)) & 1u)
                            P.vout[vbase + ((int64_t)dz * P.ny + dy) * P.nx + t] = acc[s][t];
                } else {
                    // local index inside the tile: (z * 16 + y) * 16 + x
                    const int loc = (((ozi + dz) * TILE_Y) + oyi + dy) * TILE_X + oxi;
                    float4 v4 = make_float4(acc[s][0], acc[s][1], acc[s][2], acc[s][3]);
                    *reinterpret_cast<float4*>(P.gpart + (int64_t)item.slot * TILE_VOX + loc) = v4;
                }
            }
        }
        if (MODE == MODE_JT4) {
            static_assert(!BATCH || NSUB == 2, "the four-column modes take 8 x 8 x 4 regions");
            const uint32_t vm = lane_vmask();
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const int loc = ((ozi * TILE_Y) + oyi + 4 * s) * TILE_X + oxi;
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    if (item.slot < 0) {
#pragma unroll
                        for (int t = 0; t < NX_LANE; ++t)
                            if ((vm >> (4 * s + t)) & 1u)
                                P.vout[(int64_t)r * P.nvox + vbase + (int64_t)(4 * s) * P.nx + t] = acc4[s][t][r];
                    } else {
                        float4 v4 = make_float4(acc4[s][0][r], acc4[s][1][r], acc4[s][2][r], acc4[s][3][r]);
                        *reinterpret_cast<float4*>(P.gpart + ((int64_t)item.slot * 4 + r) * TILE_VOX + loc) = v4;
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
// Resident CTAs per SM of the J^T kernel (stable detour, tables; plain or sharp).
int apply_blocks_per_sm(bool sharp, int threads, size_t smem);

// One apply launch over P's items: sharp single-column variants in the geometry's sharp CTA
// shape, plain stable-detour table variants in the plain shape, the others in 8-warp CTAs on
// the persistent grid.
template <int MODE, int DT, bool G, bool S, int PHI>
inline void launch_apply(fft_geom g, const ApplyParams& P, cudaStream_t st) {
    if (apply_sharp_wide<MODE, DT, S, PHI>()) {
        apply_kernel<MODE, DT, G, S, PHI><<<g->sharp_ctas, 32 * g->sharp_warps, apply_smem(g, g->sharp_warps), st>>>(P);
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
        if (Q.dsum) Q.dsum = P.dsum + (size_t)np * apply_regions<MODE>();   // per-unit partials follow the plain launch's
        launch_apply<MODE, DT, G, true, PHI>(g, Q, st);
    }
}

template <int MODE>
inline fft_status launch_mode_impl(fft_geom g, const ApplyParams& P, cudaStream_t st) {
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

// The four-column modes (stable detour only).
template <int MODE>
inline fft_status launch_batch_impl(fft_geom g, const ApplyParams& P, cudaStream_t st) {
    const size_t smem = apply_smem(g);
    const int ctas = g->apply_ctas;
    FFT_CUDA(cudaMemsetAsync(g->counter, 0, sizeof(int32_t), st));
    if (g->n_items == 0) return FFT_OK;
#define FFT_LAUNCH(GV, SV, PV) apply_kernel<MODE, FFT_DT_STABLE, GV, SV, PV><<<ctas, APPLY_THREADS, smem, st>>>(P)
#define FFT_LAUNCH_GS(PV)                                           \
    do {                                                            \
        if (g->guard) {                                             \
            if (g->sharp) FFT_LAUNCH(true, true, PV);               \
            else FFT_LAUNCH(true, false, PV);                       \
        } else {                                                    \
            if (g->sharp) FFT_LAUNCH(false, true, PV);              \
            else FFT_LAUNCH(false, false, PV);                      \
        }                                                           \
    } while (0)
    if (g->phi_eval == PHI_TRIG)
        FFT_LAUNCH_GS(PHI_TRIG);
    else if (g->phi_eval == PHI_SEG)
        FFT_LAUNCH_GS(PHI_SEG);
    else
        FFT_LAUNCH_GS(PHI_TABLE);
#undef FFT_LAUNCH_GS
#undef FFT_LAUNCH
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
template <> fft_status launch_mode<MODE_COUNT>(fft_geom g, const ApplyParams& P, cudaStream_t st);
template <> fft_status launch_mode<MODE_FROB>(fft_geom g, const ApplyParams& P, cudaStream_t st);
template <> fft_status launch_mode<MODE_COV>(fft_geom g, const ApplyParams& P, cudaStream_t st);
template <> fft_status launch_batch<MODE_JT4>(fft_geom g, const ApplyParams& P, cudaStream_t st);
template <> fft_status launch_batch<MODE_J4>(fft_geom g, const ApplyParams& P, cudaStream_t st);
template <> fft_status set_attr_mode<MODE_JT>(size_t smem);
template <> fft_status set_attr_mode<MODE_J>(size_t smem);
template <> fft_status set_attr_mode<MODE_COUNT>(size_t smem);
template <> fft_status set_attr_mode<MODE_FROB>(size_t smem);
template <> fft_status set_attr_mode<MODE_COV>(size_t smem);
template <> fft_status set_attr_mode<MODE_JT4>(size_t smem);
template <> fft_status set_attr_mode<MODE_J4>(size_t smem);

}  // namespace fftgb
