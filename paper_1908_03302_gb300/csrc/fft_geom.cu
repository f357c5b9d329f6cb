// Geometry set-up: per-row records, band tables in the device layout, and the culled
// (tile, row) lists that make the truncated operator sparse (Sec. II-C: truncating the
// maximum detour controls the sparsity of F).
//
// A (tile, row) entry is kept unless a lower bound of the detour over the tile's voxel
// centres is >= the band's cut-off: R is convex, so its tangent plane at the tile centre
// bounds it from below over the tile. The tile-major lists are built by one CTA per tile
// scanning all rows (rows ascending, so the order is deterministic); the row-major view
// used by the J reduction is the same set, grouped by row with entries in ascending order.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <cstring>
#include <numeric>
#include <vector>

#include "fft_common.cuh"
#include "fft_device.cuh"

namespace fftgb {

namespace {

constexpr int CULL_THREADS = 256;

struct CullParams {
    const RowRec* rec;
    const int32_t* row_band;
    const BandConst* bc;
    int64_t M;
    int tiles_x, tiles_y;
    int nx, ny, nz;
};

__device__ __forceinline__ bool tile_keeps_row(const CullParams& C, int T, int64_t p) {
    const int tx = T % C.tiles_x, ty = (T / C.tiles_x) % C.tiles_y, tz = T / (C.tiles_x * C.tiles_y);
    const RowRec r = C.rec[p];
    const BandConst bc = C.bc[C.row_band[p]];
    const float hb = bc.h;
    const float cx = fmaf((float)(TILE_X * tx) + 0.5f * (TILE_X - 1), hb, bc.org[0]) - r.a.x;
    const float cy = fmaf((float)(TILE_Y * ty) + 0.5f * (TILE_Y - 1), hb, bc.org[1]) - r.a.y;
    const float cz = fmaf((float)(TILE_Z * tz) + 0.5f * (TILE_Z - 1), hb, bc.org[2]) - r.a.z;
    if (!box_may_touch(cx, cy, cz, r.b.x, r.b.y, r.b.z, r.a.w, 0.5f * (TILE_X - 1) * hb,
                       0.5f * (TILE_Y - 1) * hb, 0.5f * (TILE_Z - 1) * hb))
        return false;
    // keep the row only if one of the tile's 16 sub-bricks (8 x 4 x 4, the apply kernels'
    // culling unit) inside the grid may reach the support: rows that reach none of them
    // would be staged by every region for nothing
    const float x0 = cx - 0.5f * (TILE_X - 1) * hb, y0 = cy - 0.5f * (TILE_Y - 1) * hb,
                z0 = cz - 0.5f * (TILE_Z - 1) * hb;
    for (int sb = 0; sb < 16; ++sb) {
        const int sx = 8 * (sb & 1), sy = 4 * ((sb >> 1) & 3), sz = 4 * (sb >> 3);
        if (TILE_X * tx + sx >= C.nx || TILE_Y * ty + sy >= C.ny || TILE_Z * tz + sz >= C.nz) continue;
        if (box_may_touch(fmaf((float)sx + 3.5f, hb, x0), fmaf((float)sy + 1.5f, hb, y0),
                          fmaf((float)sz + 1.5f, hb, z0), r.b.x, r.b.y, r.b.z, r.a.w, 3.5f * hb, 1.5f * hb,
                          1.5f * hb))
            return true;
    }
    return false;
}

// Kept rows of tile T (cnt), and of those the rows of bands that are not sharp (cnt_plain,
// nullable; counted only when `split`).
__global__ void tile_count_kernel(const CullParams C, int split, int64_t* __restrict__ cnt,
                                  int64_t* __restrict__ cnt_plain) {
    __shared__ int64_t sh[2][CULL_THREADS / 32];
    const int T = blockIdx.x;
    int64_t c = 0, cp = 0;
    for (int64_t p = threadIdx.x; p < C.M; p += CULL_THREADS) {
        if (tile_keeps_row(C, T, p)) {
            ++c;
            if (split && !C.bc[C.row_band[p]].sharp) ++cp;
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        c += __shfl_xor_sync(0xffffffffu, c, o);
        cp += __shfl_xor_sync(0xffffffffu, cp, o);
    }
    if ((threadIdx.x & 31) == 0) {
        sh[0][threadIdx.x >> 5] = c;
        sh[1][threadIdx.x >> 5] = cp;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int64_t s = 0, sp = 0;
        for (int w = 0; w < CULL_THREADS / 32; ++w) {
            s += sh[0][w];
            sp += sh[1][w];
        }
        cnt[T] = s;
        if (cnt_plain) cnt_plain[T] = sp;
    }
}

// Writes the kept rows of tile T in ascending row order; with `split` (nplain given) the rows of
// bands that are not sharp first (from off[T]) and the rows of sharp bands after them (from
// off[T] + nplain[T]), each part in ascending row order.
__global__ void tile_fill_kernel(const CullParams C, const int64_t* __restrict__ off,
                                 const int64_t* __restrict__ nplain, int32_t* __restrict__ rows) {
    __shared__ int wsum[2][CULL_THREADS / 32];
    const int T = blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t base0 = off[T], base1 = nplain ? off[T] + nplain[T] : off[T + 1];
    for (int64_t p0 = 0; p0 < C.M; p0 += CULL_THREADS) {
        const int64_t p = p0 + threadIdx.x;
        const bool keep = p < C.M && tile_keeps_row(C, T, p);
        const bool sharp = keep && nplain && C.bc[C.row_band[p]].sharp;
        const uint32_t bal0 = __ballot_sync(0xffffffffu, keep && !sharp);
        const uint32_t bal1 = __ballot_sync(0xffffffffu, sharp);
        if (lane == 0) {
            wsum[0][warp] = __popc(bal0);
            wsum[1][warp] = __popc(bal1);
        }
        __syncthreads();
        int before0 = 0, total0 = 0, before1 = 0, total1 = 0;
        for (int w = 0; w < CULL_THREADS / 32; ++w) {
            if (w < warp) {
                before0 += wsum[0][w];
                before1 += wsum[1][w];
            }
            total0 += wsum[0][w];
            total1 += wsum[1][w];
        }
        const uint32_t below = (1u << lane) - 1u;
        if (keep) {
            const int64_t pos = sharp ? base1 + before1 + __popc(bal1 & below) : base0 + before0 + __popc(bal0 & below);
            if (pos < off[T + 1]) rows[pos] = (int32_t)p;
        }
        base0 += total0;
        base1 += total1;
        __syncthreads();
    }
}

// FP64 pair-frame coordinates of each entry's tile origin (voxel (TX, TY, TZ) centre) in band
// units: p = (x_T - o).e and c = (x_T - o) x e. Computing them here in double precision keeps
// the large (~L/2) coordinates out of FP32 arithmetic; the kernels add only small offsets.
// The rows' frames come from a pass of their own: the square root and the divisions, an entry's most
// expensive FP64 operations, once per row instead of once per entry (ring256: 0.75 -> 0.20 ms).
struct RowFrame {
    double o[3], e[3];   // pair midpoint (m), unit axis
    double hl, inv_u;    // half pair length (band units), 1 / U
};
__global__ void row_frame_kernel(const double* __restrict__ tx, const int32_t* __restrict__ pairs,
                                 const int32_t* __restrict__ row_band, const BandConst* __restrict__ bc, int64_t M,
                                 RowFrame* __restrict__ frame) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= M) return;
    const double* xs = tx + 3 * (int64_t)pairs[2 * p];
    const double* xr = tx + 3 * (int64_t)pairs[2 * p + 1];
    const double U = bc[row_band[p]].U;
    const double ax = xr[0] - xs[0], ay = xr[1] - xs[1], az = xr[2] - xs[2];
    const double L = sqrt(ax * ax + ay * ay + az * az);
    RowFrame f;
    for (int a = 0; a < 3; ++a) f.o[a] = 0.5 * (xs[a] + xr[a]);
    f.e[0] = ax / L;
    f.e[1] = ay / L;
    f.e[2] = az / L;
    f.hl = 0.5 * L / U;
    f.inv_u = 1.0 / U;
    frame[p] = f;
}

__global__ void entry_base_kernel(const int64_t* __restrict__ off, const int32_t* __restrict__ rows_of_entry,
                                  const RowFrame* __restrict__ frame, double ox, double oy, double oz, double h,
                                  int tiles_x, int tiles_y, float4* __restrict__ ebase, float* __restrict__ ebase3) {
    const int T = blockIdx.x;
    const int tx_ = T % tiles_x, ty_ = (T / tiles_x) % tiles_y, tz_ = T / (tiles_x * tiles_y);
    const double xT = ox + (double)(TILE_X * tx_) * h;
    const double yT = oy + (double)(TILE_Y * ty_) * h;
    const double zT = oz + (double)(TILE_Z * tz_) * h;
    for (int64_t e = off[T] + threadIdx.x; e < off[T + 1]; e += blockDim.x) {
        const RowFrame f = frame[rows_of_entry[e]];
        const double ax = f.e[0], ay = f.e[1], az = f.e[2];
        const double dx = (xT - f.o[0]) * f.inv_u, dy = (yT - f.o[1]) * f.inv_u, dz = (zT - f.o[2]) * f.inv_u;
        const double pp = dx * ax + dy * ay + dz * az, hl = f.hl;
        // p + hl and p - hl are the axial offsets from the emitter and the receiver; forming
        // them here keeps them exact when small (voxels near a transducer)
        ebase[e] = make_float4((float)(pp + hl), (float)(pp - hl), (float)(dy * az - dz * ay),
                               (float)(dz * ax - dx * az));
        ebase3[e] = (float)(dx * ay - dy * ax);
    }
}

// Row-major view of the entries [e0, e1).
__global__ void row_count_kernel(const int32_t* __restrict__ tile_rows, int64_t e0, int64_t e1,
                                 int32_t* __restrict__ cnt) {
    int64_t e = e0 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < e1) atomicAdd(&cnt[tile_rows[e]], 1);
}

__global__ void row_fill_kernel(const int32_t* __restrict__ tile_rows, int64_t e0, int64_t e1,
                                const int64_t* __restrict__ row_off, int32_t* __restrict__ cursor,
                                int64_t* __restrict__ row_ent) {
    int64_t e = e0 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= e1) return;
    int p = tile_rows[e];
    int k = atomicAdd(&cursor[p], 1);
    row_ent[row_off[p] + k] = e;
}

// Insertion sort of each row's (short) entry list, so that its order does not depend on
// the order in which the fill kernel's atomics were served.
__global__ void row_sort_kernel(const int64_t* __restrict__ row_off, int64_t M, int64_t* __restrict__ row_ent) {
    int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= M) return;
    int64_t a = row_off[p], b = row_off[p + 1];
    for (int64_t i = a + 1; i < b; ++i) {
        int64_t x = row_ent[i], j = i - 1;
        while (j >= a && row_ent[j] > x) {
            row_ent[j + 1] = row_ent[j];
            --j;
        }
        row_ent[j + 1] = x;
    }
}

__global__ void pack_table_kernel(const double* __restrict__ phi, int n, float2* __restrict__ out) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    // Entry k holds (Phi_k - k dPhi_k, (n - 1) dPhi_k), dPhi_k = Phi_{k+1} - Phi_k, formed in FP64:
    // the interpolant on [k, k + 1) is then one FFMA in the normalised detour. The last entry
    // is the cut-off: Phi = 0 at and beyond dt_max (hard truncation), so it holds (0, 0).
    if (k == n - 1) {
        out[k] = make_float2(0.0f, 0.0f);
    } else {
        const double d = phi[k + 1] - phi[k];
        out[k] = make_float2((float)(phi[k] - (double)k * d), (float)(d * (double)(n - 1)));
    }
}

// Phi of a sine series at x = theta v (0 at and outside [0, 1)): Clenshaw's recurrence in FP64.
double series_phi(const fft_table t, double v) {
    if (!(v > 0.0) || v >= 1.0) return 0.0;
    const double x = t->dw * t->dt_max * v, c2 = 2.0 * cos(x);
    double b1 = 0.0, b2 = 0.0;
    for (int j = t->n; j >= 1; --j) {
        const double b0 = t->coef[j - 1] + c2 * b1 - b2;
        b2 = b1;
        b1 = b0;
    }
    return b1 * sin(x);
}

// Piecewise quadratics of the bands' series (device layout of PHI_SEG, see phi_seg): (c0, c1) of all
// bands' entries, then their c2. The fewest segments (a power of two) whose quadratics stay
// within 5e-8 of each band's max |Phi| (a third of a segment off its ends and middle, where the
// cubic remainder peaks), i.e. inside the FP32 rounding of the values: 2048 for spectra of the usual
// width cut after three periods. Returns 0 if they do not fit `max_bytes` of shared memory: such series
// (many bands, or cut after tens of periods) keep the recurrence.
int build_segments(const fft_table* tables, int n_bands, size_t max_bytes, std::vector<float2>& packed) {
    for (int n = 512; (size_t)n_bands * (n + SEG_PAD) * 12 <= max_bytes; n *= 2) {
        const int ne = n + SEG_PAD;
        packed.assign((size_t)n_bands * ne * 3 / 2, make_float2(0.0f, 0.0f));
        float* c2 = reinterpret_cast<float*>(packed.data() + (size_t)n_bands * ne);
        bool good = true;
        for (int b = 0; b < n_bands && good; ++b) {
            const fft_table t = tables[b];
            // the series just below the cut-off, not the truncated 0 there, ends the last segment
            const double end = 1.0 - 1e-12;
            double mx = 0.0, err = 0.0, f2 = series_phi(t, 0.0);
            for (int k = 0; k < n; ++k) {
                const double f0 = f2, f1 = series_phi(t, (k + 0.5) / n);
                f2 = series_phi(t, k + 1 < n ? (k + 1.0) / n : end);
                const double a1 = -3.0 * f0 + 4.0 * f1 - f2, a2 = 2.0 * f0 - 4.0 * f1 + 2.0 * f2;
                mx = fmax(mx, fmax(fabs(f0), fabs(f1)));
                for (double u : {0.21, 0.79})
                    err = fmax(err, fabs(f0 + u * (a1 + u * a2) - series_phi(t, (k + u) / n)));
                const double s = 4194304.0;   // u is kept times 2^-22
                packed[(size_t)b * ne + k] = make_float2((float)f0, (float)(a1 * s));
                c2[(size_t)b * ne + k] = (float)(a2 * s * s);
            }
            good = err <= 5e-8 * mx;
        }
        if (good) return n;
    }
    return 0;
}

// Sets z_lo, z_end and mirror. K0 depends on a voxel's distances to the two transducers alone, so
// with all of them in one plane z = z0 the layers k and K - k, K = 2 (z0 - origin_z) / h, have equal
// entries if K is a whole number (to 1e-9 voxel: the layers then mirror each other to FP64
// rounding): a single ring or plane array on a lattice with the plane on or half way between its
// layers. Items then cover the layers up to the plane where every layer above it has its image below, else
// those from the plane up. It halves the evaluations (ring256 J 3.56 -> 1.93 ms, J^T 3.52 -> 1.86 ms,
// three bands J 11.98 -> 6.58 ms; error against 64 bits of J 0.9e-7 -> 1.2e-7, of J^T unchanged).
// Below MIRROR_MIN_ENTRIES a product is bound by launches and latency, not by evaluations (the
// 32-element ring: 8 k entries), and one evaluation per voxel keeps independent roundings.
constexpr int64_t MIRROR_MIN_ENTRIES = 65536;
void find_mirror(fft_geom g, const double* tx, const int32_t* rows) {
    const fft_grid& gr = g->grid;
    g->z_lo = 0;
    g->z_end = gr.nz;
    g->mirror = -1;
    if (g->E < MIRROR_MIN_ENTRIES) return;
    const double z0 = tx[3 * rows[0] + 2];
    for (int64_t p = 0; p < 2 * g->M; ++p)
        if (tx[3 * rows[p] + 2] != z0) return;
    const double k = 2.0 * (z0 - gr.origin[2]) / gr.h;
    if (!(k >= 1.0 && k <= 2.0 * gr.nz - 3.0) || fabs(k - nearbyint(k)) > 1e-9) return;
    g->mirror = (int32_t)nearbyint(k);
    if (g->mirror >= gr.nz - 1)
        g->z_end = g->mirror / 2 + 1;
    else
        g->z_lo = (g->mirror + 1) / 2;
}

template <typename T>
fft_status dmalloc(fft_geom g, T** p, size_t count) {
    *p = nullptr;
    if (count == 0) count = 1;
    cudaError_t e = device_malloc(reinterpret_cast<void**>(p), count * sizeof(T));
    if (e != cudaSuccess) {
        cudaGetLastError();
        set_error("fft_geom_create: cudaMalloc of " + std::to_string(count * sizeof(T)) + " bytes failed");
        return FFT_ERR_OOM;
    }
    g->scratch_bytes += (int64_t)(count * sizeof(T));
    return FFT_OK;
}

void free_geom(fft_geom g) {
    if (!g) return;
    for (StackClass& c : g->stk) free_geom(c.sub);
    if (g->nested) g->jpart = g->jpart4 = g->gpart = g->gpart4 = nullptr;   // the parent's
    void* ptrs[] = {g->d_band, g->rec, g->rec64, g->row_band, g->tab, g->tile_off, g->tile_rows, g->ebase, g->ebase3,
                    g->row_off, g->row_ent, g->items, g->tile_slot0, g->tile_nslot, g->jpart,
                    g->gpart, g->counter, g->cg_r, g->cg_q, g->cg_s, g->cg_ql, g->cg_sl, g->cg_jpart,
                    g->cg_gpart, g->cg_p, g->cg_d, g->cg_m,
                    g->cg_scal, g->cg_dots, g->cg_status, g->cg_hist, g->vol, g->jpart4, g->gpart4,
                    g->jpart4_kept, g->gpart4_kept,
                    g->psf_crec, g->stk_rows, g->stk_x, g->stk_d, g->stk_jpart, g->stk_gpart, g->zw};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    if (g->cg_graph) cudaGraphExecDestroy((cudaGraphExec_t)g->cg_graph);
    if (g->cg_graph_cont) cudaGraphExecDestroy((cudaGraphExec_t)g->cg_graph_cont);
    if (g->cg_stream) cudaStreamDestroy((cudaStream_t)g->cg_stream);
    delete g;
}

}  // namespace

int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }

// Rows per work item of a launch over E entries when no tuning has chosen it. Small items cost J^T
// a partial slot each (8 KB written and read back, ~3 ns), large ones leave warps idle while the
// last are finished (about 0.2 us per row: a unit's rows run one after another in one warp). The
// sum of the two, 3 ns E / n + 0.2 us n, is least at n = sqrt(0.015 E): 230 rows on ring256 (3.5 M
// entries; the autotuner picks 242 there), 11 on the 32-element ring (8 k entries), where it also
// makes about one unit per resident warp. Against eight items per CTA of at least 64 rows: ring256 J
// 3.79 -> 3.56 ms, its three-band J 14.05 -> 11.98 ms, a 20-iteration solve of four 32-element
// slices 8.1 -> 5.2 ms.
int64_t default_item_rows(int64_t E) {
    const int64_t n = std::max<int64_t>(8, (int64_t)sqrt(0.015 * (double)E));
    return n < 32 ? n : ceil_div(n, 32) * 32;
}

// Rows per work item for about items_per_cta items per persistent CTA.
int64_t item_rows(int64_t E, int items_per_cta, int ctas) {
    const int64_t target = (int64_t)items_per_cta * ctas;
    const int64_t ch = std::max<int64_t>(64, ceil_div(std::max<int64_t>(E, 1), std::max<int64_t>(target, 1)));
    return ceil_div(ch, 32) * 32;
}

// Does tile T hold layers the products evaluate?
static bool tile_used(fft_geom g, int64_t T) {
    const int64_t tz = T / ((int64_t)g->tiles[0] * g->tiles[1]);
    return TILE_Z * tz < g->z_end && TILE_Z * (tz + 1) > g->z_lo;
}

// Work items: a tile's candidate rows in ranges of at most ch rows, ch chosen so that each
// persistent CTA sees about items_per_cta items (at least 64 rows, a multiple of 32), or by
// default_item_rows when items_per_cta is 0; tiles split over several items write J^T partial
// slots. Heaviest items first. Replaces the geometry's previous items, slots and partial buffers
// (the J partials do not depend on them); those go first, so that tuning needs no more memory than the
// larger of the two takes. If the new ones can't be had the operator is unusable until a later call succeeds.
fft_status build_items(fft_geom g, const std::vector<int64_t>& toff, int items_per_cta) {
    // plain rows [toff, toff + nplain) and sharp-band rows [toff + nplain, toff1) of a split
    // geometry go to different items and launches; the tile's slots number its plain items first
    const bool split = !g->tile_nplain.empty();
    int64_t chp, chs;   // rows per plain and per sharp item
    if (items_per_cta > 0) {
        chp = chs = item_rows(g->E, items_per_cta, g->apply_ctas);
    } else {
        int64_t Ep = 0, Es = 0;   // entries of the two launches
        for (int64_t T = 0; T < g->n_tiles; ++T) {
            if (!tile_used(g, T)) continue;
            const int64_t n = toff[T + 1] - toff[T], np = split ? g->tile_nplain[T] : n;
            Ep += np;
            Es += n - np;
        }
        chp = default_item_rows(Ep);
        chs = default_item_rows(Es);
    }
    std::vector<Item> items, items_sharp;
    std::vector<int32_t> slot0(g->n_tiles, -2), nslot(g->n_tiles, 0);
    int32_t slots = 0;
    for (int64_t T = 0; T < g->n_tiles; ++T) {
        const int64_t n = toff[T + 1] - toff[T];
        if (n == 0 || !tile_used(g, T)) continue;
        const int64_t np = split ? g->tile_nplain[T] : n;
        const int64_t kp = ceil_div(np, chp), ks = ceil_div(n - np, chs), k = kp + ks;
        if (k == 1) {
            (kp == 1 ? items : items_sharp).push_back(Item{(int32_t)T, -1, toff[T], toff[T + 1]});
            slot0[T] = -1;
        } else {
            slot0[T] = slots;
            nslot[T] = (int32_t)k;
            for (int64_t q = 0; q < k; ++q) {
                const int64_t lo = q < kp ? toff[T] : toff[T] + np, hi = q < kp ? toff[T] + np : toff[T + 1];
                const int64_t a = lo + (q < kp ? q * chp : (q - kp) * chs), b = std::min(hi, a + (q < kp ? chp : chs));
                (q < kp ? items : items_sharp).push_back(Item{(int32_t)T, slots + (int32_t)q, a, b});
            }
            slots += (int32_t)k;
        }
    }
    auto heavier = [](const Item& x, const Item& y) { return (x.e1 - x.e0) > (y.e1 - y.e0); };
    std::stable_sort(items.begin(), items.end(), heavier);
    std::stable_sort(items_sharp.begin(), items_sharp.end(), heavier);
    g->n_items_plain = (int32_t)items.size();
    items.insert(items.end(), items_sharp.begin(), items_sharp.end());
    // a captured CG loop holds the old item list: capture again on the next solve
    if (g->cg_graph) {
        cudaGraphExecDestroy((cudaGraphExec_t)g->cg_graph);
        g->cg_graph = nullptr;
        g->cg_graph_iters = -1;
    }
    if (g->cg_graph_cont) {
        cudaGraphExecDestroy((cudaGraphExec_t)g->cg_graph_cont);
        g->cg_graph_cont = nullptr;
        g->cg_graph_cont_iters = -1;
    }
    if (g->nested) g->jpart4 = g->gpart = g->gpart4 = nullptr;   // the parent's (stack_scratch sets them again)
    free_batch_scratch(g);   // rebuilt with the new slot count on first use
    if (g->items) {          // the buffers below are replaced: take them out of the scratch count
        g->scratch_bytes -= (int64_t)(sizeof(Item) * g->n_items + 2 * sizeof(int32_t) * g->n_tiles);
        if (!g->nested) g->scratch_bytes -= (int64_t)(sizeof(float) * (size_t)g->n_slots * TILE_VOX);
    }
    void* old[] = {g->items, g->tile_slot0, g->tile_nslot, g->gpart, g->cg_gpart};   // (cg_gpart: at the next solve)
    for (void* q : old)
        if (q) cudaFree(q);
    g->items = nullptr;
    g->tile_slot0 = g->tile_nslot = nullptr;
    g->gpart = g->cg_gpart = nullptr;
    g->n_items = (int32_t)items.size();
    g->n_slots = slots;
    g->items_per_cta = items_per_cta;
    g->unusable = true;
    const int64_t before = g->scratch_bytes;
    fft_status rc = dmalloc(g, &g->items, items.size());
    if (rc == FFT_OK) rc = dmalloc(g, &g->tile_slot0, g->n_tiles);
    if (rc == FFT_OK) rc = dmalloc(g, &g->tile_nslot, g->n_tiles);
    if (rc == FFT_OK && !g->nested) rc = dmalloc(g, &g->gpart, (size_t)slots * TILE_VOX);
    cudaError_t e = cudaSuccess;
    if (rc == FFT_OK && !items.empty())
        e = cudaMemcpy(g->items, items.data(), sizeof(Item) * items.size(), cudaMemcpyHostToDevice);
    if (rc == FFT_OK && e == cudaSuccess)
        e = cudaMemcpy(g->tile_slot0, slot0.data(), sizeof(int32_t) * g->n_tiles, cudaMemcpyHostToDevice);
    if (rc == FFT_OK && e == cudaSuccess)
        e = cudaMemcpy(g->tile_nslot, nslot.data(), sizeof(int32_t) * g->n_tiles, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) rc = cuda_fail(e, "work items");
    if (rc != FFT_OK) {
        void* got[] = {g->items, g->tile_slot0, g->tile_nslot, g->gpart};
        for (void* q : got)
            if (q) cudaFree(q);
        g->items = nullptr;
        g->tile_slot0 = g->tile_nslot = nullptr;
        g->gpart = nullptr;
        g->n_items = g->n_items_plain = g->n_slots = 0;
        g->scratch_bytes = before;
        return rc;
    }
    g->unusable = false;
    return FFT_OK;
}

// The partial buffers that a stack's operators share: their passes follow each other on one stream.
// (J^T partials grow with the items; the J partials do not.)
fft_status stack_scratch(fft_geom g) {
    int64_t need = 0;
    for (StackClass& c : g->stk) need = std::max(need, (int64_t)c.sub->n_slots * c.sub->batch_cols * TILE_VOX);
    if (need > g->stk_gpart_cap || !g->stk_gpart) {
        cudaFree(g->stk_gpart);
        g->scratch_bytes -= (int64_t)sizeof(float) * g->stk_gpart_cap;
        g->stk_gpart = nullptr;
        g->stk_gpart_cap = 0;
        const fft_status rc = dmalloc(g, &g->stk_gpart, (size_t)std::max<int64_t>(need, 1));
        if (rc != FFT_OK) return rc;
        g->stk_gpart_cap = std::max<int64_t>(need, 1);
    }
    for (StackClass& c : g->stk) {
        c.sub->jpart = c.sub->jpart4 = g->stk_jpart;
        c.sub->gpart = c.sub->gpart4 = g->stk_gpart;
    }
    return FFT_OK;
}

// Work items of the operators of a stack (the autotuner's candidates).
fft_status stack_build_items(fft_geom g, int items_per_cta) {
    g->unusable = true;   // the classes' operators lose their buffers here, until stack_scratch succeeds
    for (StackClass& c : g->stk) {
        std::vector<int64_t> toff(c.sub->n_tiles + 1);
        FFT_CUDA(cudaMemcpy(toff.data(), c.sub->tile_off, sizeof(int64_t) * toff.size(), cudaMemcpyDeviceToHost));
        c.sub->apply_ctas = g->apply_ctas;
        const fft_status rc = build_items(c.sub, toff, items_per_cta);
        if (rc != FFT_OK) return rc;
    }
    const fft_status rc = stack_scratch(g);
    g->unusable = rc != FFT_OK;
    return rc;
}

namespace {

fft_status create_geom(const double* tx_xyz, int32_t n_tx, const int32_t* rows, int64_t n_rows,
                       const int32_t* band_of_row, const fft_grid* grid, double c0, const fft_table* tables,
                       int32_t n_tables, int32_t dt_mode, bool nested, fft_geom* out);

void drop_stack(fft_geom g) {
    for (StackClass& c : g->stk) free_geom(c.sub);
    g->stk.clear();
    void* ptrs[] = {g->stk_rows, g->stk_x, g->stk_d, g->stk_jpart, g->stk_gpart};
    for (void* q : ptrs)
        if (q) cudaFree(q);
    g->stk_rows = nullptr;
    g->stk_x = g->stk_d = g->stk_jpart = g->stk_gpart = nullptr;
    g->stk_gpart_cap = 0;
}

// Do J^T of sparse columns, the PSFs, go through the classes? Few rows have a weight, so that the general path
// does little, while a class's pass costs what its slices' extended volumes take to write, reduce and add,
// and five launches. Measured by the entries per voxel of those volumes (fill), six PSFs, general path against
// classes, one column at a time and four: 64 elements in 11 slices (fill 0.11) 1.89 against 2.27 and 1.71
// against 2.92 ms, 100 in 5 (0.23) 2.28 / 1.67 and 2.14 / 2.28, 128 in 7 (0.26) 3.27 / 2.71 and 3.15 / 3.06,
// 128 in 2 (0.6) 2.49 / 1.71 and 2.29 / 1.74, 200 in 11 (0.7) 41.3 / 15.6 and 32.3 / 18.1; three classes of
// 96 in 9 (1.3e6 entries) 1.89 / 2.21 and 1.71 / 1.72.
void sparse_pays(fft_geom g) {
    double vox = 0.0;
    for (const StackClass& c : g->stk) vox += (double)c.off.size() * (double)c.sub->V;
    const double fill = (double)g->E_used / vox;
    const bool enough = g->E_used >= STACK_MIN_ENTRIES / 2 * (int64_t)g->stk.size();
    g->stk_psf1 = enough && fill >= 0.2;
    g->stk_psf4 = enough && fill >= 0.3;
}

// Operators of an elevation stack's classes where they pay: from STACK_MIN_ENTRIES entries (below, a
// product is bound by launches and the classes add more of them: a PSF of ten 57-element slices, about
// 6e5 entries of which few have a weight, 0.35 -> 0.41 ms with them), with at most 0.8 of the entries of a
// pass over all rows left to evaluate, and with memory to spare. g stays as it is otherwise.
void build_stack(fft_geom g, const double* tx, const int32_t* rows, const int32_t* band, const fft_table* tables) {
    std::vector<StackPlan> plan;
    if (g->nested || g->dt_mode != FFT_DT_STABLE || g->E_used < STACK_MIN_ENTRIES) return;
    if (!find_stack(tx, rows, g->M, band, g->grid, plan) || stack_cost(plan, g->M, g->grid) > 0.8) return;
    size_t mem_free = 0, mem_total = 0;
    if (cudaMemGetInfo(&mem_free, &mem_total) != cudaSuccess) {
        cudaGetLastError();
        return;
    }
    const int64_t plane = (int64_t)g->grid.nx * g->grid.ny;
    // (an operator's entries: 32 bytes of lists and 256 of partials each, about a slice's share of E)
    double need = 0.0;
    for (const StackPlan& c : plan)
        need = std::max(need, 288.0 * (double)g->E * (double)c.rows[0].size() / (double)g->M +
                                  32.0 * (double)plane * (g->grid.nz + c.shift.back()));
    if (2.0 * need > 0.5 * (double)mem_free) return;
    const int64_t before = g->scratch_bytes;
    std::vector<int32_t> ids;
    ids.reserve((size_t)g->M);
    int64_t v_max = 0, m_max = 0, e_max = 0;
    int cols = 4;
    bool ok = true;
    for (const StackPlan& c : plan) {
        const int32_t top = c.shift.back();
        fft_grid eg = g->grid;
        eg.nz += top;
        eg.origin[2] -= top * eg.h;
        // the transducers of the lowest slice alone, in the order of its rows
        std::vector<double> stx;
        std::vector<int32_t> srows, sband, at;
        const std::vector<int32_t>& base = c.rows[0];
        at.assign((size_t)g->n_tx, -1);
        for (int32_t p : base) {
            for (int e = 0; e < 2; ++e) {
                const int32_t t = rows[2 * (int64_t)p + e];
                if (at[t] < 0) {
                    at[t] = (int32_t)(stx.size() / 3);
                    stx.insert(stx.end(), tx + 3 * (int64_t)t, tx + 3 * (int64_t)t + 3);
                }
                srows.push_back(at[t]);
            }
            sband.push_back(band ? band[p] : 0);
        }
        StackClass k;
        if (create_geom(stx.data(), (int32_t)(stx.size() / 3), srows.data(), (int64_t)base.size(), sband.data(), &eg, g->c0,
                        tables, g->n_bands, g->dt_mode, true, &k.sub) != FFT_OK) {
            ok = false;
            break;
        }
        k.row0 = (int64_t)ids.size();
        std::vector<uint8_t> zw((size_t)eg.nz, 0);
        for (size_t s = 0; s < c.rows.size(); ++s) {
            k.off.push_back(top - c.shift[s]);
            ids.insert(ids.end(), c.rows[s].begin(), c.rows[s].end());
            for (int z = 0; z < g->grid.nz; ++z) ++zw[z + k.off[s]];
        }
        k.sub->batch_cols = (c.rows.size() > 4 && k.sub->col8) ? 8 : 4;
        cols = std::max(cols, k.sub->batch_cols);
        g->stk.push_back(k);
        ok = dmalloc(k.sub, &k.sub->zw, zw.size()) == FFT_OK &&
             cudaMemcpy(k.sub->zw, zw.data(), zw.size(), cudaMemcpyHostToDevice) == cudaSuccess;
        if (!ok) break;
        g->scratch_bytes += k.sub->scratch_bytes;
        v_max = std::max(v_max, k.sub->V);
        m_max = std::max(m_max, k.sub->M);
        e_max = std::max(e_max, k.sub->E * k.sub->batch_cols);
    }
    ok = ok && stack_entries(g, 1) <= 0.8 * (double)g->E_used;
    ok = ok && dmalloc(g, &g->stk_rows, ids.size()) == FFT_OK &&
         cudaMemcpy(g->stk_rows, ids.data(), sizeof(int32_t) * ids.size(), cudaMemcpyHostToDevice) == cudaSuccess &&
         dmalloc(g, &g->stk_x, cols * (size_t)v_max) == FFT_OK && dmalloc(g, &g->stk_d, cols * (size_t)m_max) == FFT_OK &&
         dmalloc(g, &g->stk_jpart, 8 * (size_t)e_max) == FFT_OK && stack_scratch(g) == FFT_OK;
    if (!ok) {
        cudaGetLastError();
        drop_stack(g);
        g->scratch_bytes = before;
        return;
    }
    // several columns at once: against passes of the same width over all rows
    g->stk_batch = stack_entries(g, 8) <= pass_cost(8, g->col8) * (double)g->E_used;
    sparse_pays(g);
}

}  // namespace

}  // namespace fftgb

using namespace fftgb;

namespace fftgb {

namespace {

// nested: an operator of a stack's class (fft_geom_s): no partial buffers of its own, no support count.
fft_status create_geom(const double* tx_xyz, int32_t n_tx, const int32_t* rows, int64_t n_rows,
                       const int32_t* band_of_row, const fft_grid* grid, double c0, const fft_table* tables,
                       int32_t n_tables, int32_t dt_mode, bool nested, fft_geom* out) {
    FFT_ARG(out, "fft_geom_create: null out");
    *out = nullptr;
    FFT_ARG(tx_xyz && n_tx >= 2, "fft_geom_create: need at least two transducers");
    FFT_ARG(rows && n_rows >= 1 && n_rows < (int64_t)INT32_MAX, "fft_geom_create: need 1 .. 2^31-2 rows");
    FFT_ARG(grid && grid->nx >= 1 && grid->ny >= 1 && grid->nz >= 1 && grid->h > 0,
            "fft_geom_create: invalid grid");
    FFT_ARG(c0 > 0 && isfinite(c0), "fft_geom_create: c0 must be > 0");
    FFT_ARG(tables && n_tables >= 1 && n_tables <= MAX_BANDS, "fft_geom_create: need 1 .. 8 tables");
    FFT_ARG(dt_mode == FFT_DT_STABLE || dt_mode == FFT_DT_NAIVE || dt_mode == FFT_DT_FP64,
            "fft_geom_create: unknown dt_mode");
    int dev = 0;
    FFT_CUDA(cudaGetDevice(&dev));
    for (int b = 0; b < n_tables; ++b) {
        FFT_ARG(tables[b], "fft_geom_create: null table");
        FFT_ARG(tables[b]->kind == tables[0]->kind,
                "fft_geom_create: tables must be all sampled tables or all sine series");
        if (tables[0]->kind == PHI_TABLE)
            FFT_ARG(tables[b]->n == tables[0]->n, "fft_geom_create: all tables must have the same sample count");
        if (tables[b]->dev != dev) {
            set_error("fft_geom_create: table was built on another device");
            return FFT_ERR_STATE;
        }
    }
    const int32_t phi_kind = tables[0]->kind;
    FFT_ARG(phi_kind == PHI_TABLE || dt_mode == FFT_DT_STABLE,
            "fft_geom_create: sine-series tables need dt_mode FFT_DT_STABLE");
    // device layout of one band's Phi: n_tab float2 entries. Series: a 16-byte header (theta =
    // dw dt_max, the series argument at the cut-off) and the coefficients in groups of 4.
    int32_t trig_terms = 0;
    for (int b = 0; b < n_tables; ++b) trig_terms = std::max(trig_terms, tables[b]->n);
    const int32_t trig_nq = (trig_terms + 3) / 4;
    int32_t n_tab = phi_kind == PHI_TABLE ? tables[0]->n : 2 + 2 * trig_nq;
    const int64_t V = (int64_t)grid->nx * grid->ny * grid->nz;
    FFT_ARG(V < ((int64_t)1 << 40), "fft_geom_create: grid too large");
    for (int64_t p = 0; p < n_rows; ++p) {
        int32_t s = rows[2 * p], r = rows[2 * p + 1];
        FFT_ARG(s >= 0 && s < n_tx && r >= 0 && r < n_tx, "fft_geom_create: row transducer index out of range");
        FFT_ARG(s != r, "fft_geom_create: a row has the same emitter and receiver");
        if (band_of_row)
            FFT_ARG(band_of_row[p] >= 0 && band_of_row[p] < n_tables, "fft_geom_create: band index out of range");
    }
    int32_t phi_eval = phi_kind, seg_n = 0;
    std::vector<float2> segments;
    {
        int optin = 0;
        FFT_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
        if (phi_kind == PHI_TRIG) {   // piecewise quadratics where they leave room for 16 warps' staging
            const size_t stage = (size_t)2 * APPLY_WARPS * 128 * sizeof(float4);
            if ((size_t)optin > stage) seg_n = build_segments(tables, n_tables, (size_t)optin - stage, segments);
            if (seg_n > 0) {
                phi_eval = PHI_SEG;
                n_tab = (seg_n + SEG_PAD) / 2 * 3;   // float2 words per band
            }
        }
        size_t need = (((size_t)n_tables * n_tab * sizeof(float2) + 15) & ~(size_t)15) +
                      (size_t)APPLY_WARPS * 128 * sizeof(float4);
        if (need > (size_t)optin) {
            set_error("fft_geom_create: the tables (n_tables x n_samples x 8 bytes) do not fit in shared memory");
            return FFT_ERR_ARG;
        }
    }
    fft_geom g = new fft_geom_s();
    g->nested = nested;
    g->dev = dev;
    g->M = n_rows;
    g->V = V;
    g->n_tx = n_tx;
    g->grid = *grid;
    g->c0 = c0;
    g->n_bands = n_tables;
    g->n_tab = n_tab;
    g->dt_mode = dt_mode;
    g->phi_kind = phi_kind;
    g->phi_eval = phi_eval;
    g->seg_n = seg_n;
    g->trig_nq = phi_eval == PHI_TRIG ? trig_nq : 0;
    g->trig_terms = phi_kind == PHI_TRIG ? trig_terms : 0;
    g->guard = false;
    fft_status rc = FFT_OK;
#define GEOM_TRY(x)              \
    do {                         \
        rc = (x);                \
        if (rc != FFT_OK) {      \
            free_geom(g);        \
            return rc;           \
        }                        \
    } while (0)
#define GEOM_CUDA(x)                                 \
    do {                                             \
        cudaError_t _e = (x);                        \
        if (_e != cudaSuccess) {                     \
            rc = cuda_fail(_e, #x);                  \
            free_geom(g);                            \
            return rc;                               \
        }                                            \
    } while (0)

    // ---- bands
    std::vector<BandConst> hb(n_tables);
    for (int b = 0; b < n_tables; ++b) {
        double U = c0 * tables[b]->dt_max;
        g->dt_max[b] = tables[b]->dt_max;
        hb[b].U = U;
        hb[b].h = (float)(grid->h / U);
        for (int a = 0; a < 3; ++a) hb[b].org[a] = (float)(grid->origin[a] / U);
        // Is Phi just below the cut-off non-negligible? (table: its sample at dt_max)
        std::vector<double> phi;
        if (phi_kind == PHI_TABLE) {
            phi.resize(tables[b]->n);
            cudaError_t ce = cudaMemcpy(phi.data(), tables[b]->d_phi, sizeof(double) * phi.size(), cudaMemcpyDeviceToHost);
            if (ce != cudaSuccess) {
                rc = cuda_fail(ce, "fft_geom_create: table copy");
                free_geom(g);
                return rc;
            }
        } else {   // the series on 4096 points of [0, dt_max]
            phi.resize(4096);
            for (size_t k = 0; k + 1 < phi.size(); ++k) phi[k] = series_phi(tables[b], (double)k / (double)(phi.size() - 1));
            phi.back() = series_phi(tables[b], 1.0 - 1e-12);
        }
        double mx = 0.0;
        for (double v : phi) mx = fmax(mx, fabs(v));
        hb[b].sharp = (fabs(phi[phi.size() - 1]) > 1e-7 * mx) ? 1 : 0;
        hb[b].pad = 0;
        g->band[b] = hb[b];
    }
    bool any_sharp = false;
    for (int b = 0; b < n_tables; ++b) any_sharp = any_sharp || hb[b].sharp;
    g->sharp = any_sharp && dt_mode != FFT_DT_FP64;
    const bool need64 = (dt_mode == FFT_DT_FP64) || any_sharp;
    GEOM_TRY(dmalloc(g, &g->d_band, n_tables));
    GEOM_CUDA(cudaMemcpy(g->d_band, hb.data(), sizeof(BandConst) * n_tables, cudaMemcpyHostToDevice));

    // ---- tables in the device layout
    GEOM_TRY(dmalloc(g, &g->tab, (size_t)n_tables * g->n_tab));
    if (phi_kind == PHI_TABLE) {
        for (int b = 0; b < n_tables; ++b) {
            pack_table_kernel<<<(unsigned)ceil_div(g->n_tab, 256), 256>>>(tables[b]->d_phi, g->n_tab,
                                                                            g->tab + (size_t)b * g->n_tab);
            GEOM_CUDA(cudaGetLastError());
        }
    } else if (phi_eval == PHI_SEG) {
        GEOM_CUDA(cudaMemcpy(g->tab, segments.data(), sizeof(float2) * segments.size(), cudaMemcpyHostToDevice));
    } else {
        // per band: (theta, 0), (0, 0), then a_1 .. a_{4 nq} as float pairs (zeros past n)
        std::vector<float2> packed((size_t)n_tables * n_tab, make_float2(0.0f, 0.0f));
        for (int b = 0; b < n_tables; ++b) {
            float2* blk = packed.data() + (size_t)b * n_tab;
            blk[0].x = (float)(tables[b]->dw * tables[b]->dt_max);
            float* a = reinterpret_cast<float*>(blk + 2);
            for (int j = 0; j < tables[b]->n; ++j) a[j] = (float)tables[b]->coef[j];
        }
        GEOM_CUDA(cudaMemcpy(g->tab, packed.data(), sizeof(float2) * packed.size(), cudaMemcpyHostToDevice));
    }

    // ---- row records
    {
        std::vector<RowRec> rec(n_rows);
        std::vector<RowRec64> rec64(need64 ? n_rows : 0);
        std::vector<int32_t> rb(n_rows);
        const double h3 = grid->h * grid->h * grid->h;
        for (int64_t p = 0; p < n_rows; ++p) {
            const double* xs = tx_xyz + 3 * rows[2 * p];
            const double* xr = tx_xyz + 3 * rows[2 * p + 1];
            int b = band_of_row ? band_of_row[p] : 0;
            rb[p] = b;
            double U = hb[b].U;
            double ax = xr[0] - xs[0], ay = xr[1] - xs[1], az = xr[2] - xs[2];
            double L = sqrt(ax * ax + ay * ay + az * az);
            if (!(L > 0)) {
                free_geom(g);
                set_error("fft_geom_create: a row has coincident emitter and receiver positions");
                return FFT_ERR_ARG;
            }
            RowRec& R = rec[p];
            R.a = make_float4((float)(0.5 * (xs[0] + xr[0]) / U), (float)(0.5 * (xs[1] + xr[1]) / U),
                              (float)(0.5 * (xs[2] + xr[2]) / U), (float)(0.5 * L / U));
            // K0 dV = -L h^3 / (2 pi c0^3 R_xs R_xr) Phi = C Phi / (Rs_band Rr_band)
            double C = -L * h3 / (2.0 * M_PI * c0 * c0 * c0 * U * U);
            R.b = make_float4((float)(ax / L), (float)(ay / L), (float)(az / L), (float)C);
            const double hU = grid->h / U;
            R.c = make_float4((float)(hU * (ax / L)), (float)(hU * (ay / L)), (float)(hU * (az / L)), 0.0f);
            if (need64) {
                for (int a = 0; a < 3; ++a) {
                    rec64[p].xs[a] = xs[a];
                    rec64[p].xr[a] = xr[a];
                }
            }
        }
        GEOM_TRY(dmalloc(g, &g->rec, n_rows));
        GEOM_TRY(dmalloc(g, &g->row_band, n_rows));
        GEOM_CUDA(cudaMemcpy(g->rec, rec.data(), sizeof(RowRec) * n_rows, cudaMemcpyHostToDevice));
        GEOM_CUDA(cudaMemcpy(g->row_band, rb.data(), sizeof(int32_t) * n_rows, cudaMemcpyHostToDevice));
        if (need64) {
            GEOM_TRY(dmalloc(g, &g->rec64, n_rows));
            GEOM_CUDA(cudaMemcpy(g->rec64, rec64.data(), sizeof(RowRec64) * n_rows, cudaMemcpyHostToDevice));
        }
    }

    // ---- tiles
    g->tiles[0] = (int32_t)ceil_div(grid->nx, TILE_X);
    g->tiles[1] = (int32_t)ceil_div(grid->ny, TILE_Y);
    g->tiles[2] = (int32_t)ceil_div(grid->nz, TILE_Z);
    g->n_tiles = (int64_t)g->tiles[0] * g->tiles[1] * g->tiles[2];
    if (g->n_tiles >= (int64_t)INT32_MAX) {
        free_geom(g);
        set_error("fft_geom_create: grid too large");
        return FFT_ERR_ARG;
    }

    // Guarded kernels are needed only if a voxel centre of the tile-padded lattice coincides
    // (to within 1e-3 h) with a transducer: there R_xs = 0 and the plain form divides 0 by 0.
    for (int t = 0; t < n_tx && !g->guard; ++t) {
        bool on = true;
        for (int a = 0; a < 3; ++a) {
            double u = (tx_xyz[3 * t + a] - grid->origin[a]) / grid->h;
            double ru = nearbyint(u);
            int lim = g->tiles[a] * (a == 0 ? TILE_X : (a == 1 ? TILE_Y : TILE_Z));
            if (fabs(u - ru) > 1e-3 || ru < 0 || ru >= lim) on = false;
        }
        if (on) g->guard = true;
    }

    CullParams C;
    C.rec = g->rec;
    C.row_band = g->row_band;
    C.bc = g->d_band;
    C.M = n_rows;
    C.tiles_x = g->tiles[0];
    C.nx = grid->nx;
    C.ny = grid->ny;
    C.nz = grid->nz;
    C.tiles_y = g->tiles[1];

    std::vector<int64_t> tcnt(g->n_tiles), toff(g->n_tiles + 1, 0);
    // sharp geometries keep each tile's plain rows ahead of its sharp-band rows, so that the
    // two kinds run in separate launches (the plain kernels need fewer registers)
    const bool split = g->sharp;
    int64_t* d_nplain = nullptr;
    {
        int64_t* d_cnt = nullptr;
        GEOM_TRY(dmalloc(g, &g->tile_off, g->n_tiles + 1));
        d_cnt = g->tile_off;   // counts first, offsets after
        if (split) GEOM_CUDA(cudaMalloc(&d_nplain, sizeof(int64_t) * g->n_tiles));
        tile_count_kernel<<<(unsigned)g->n_tiles, CULL_THREADS>>>(C, split ? 1 : 0, d_cnt, d_nplain);
        cudaError_t e = cudaGetLastError();
        if (e == cudaSuccess)
            e = cudaMemcpy(tcnt.data(), d_cnt, sizeof(int64_t) * g->n_tiles, cudaMemcpyDeviceToHost);
        if (e == cudaSuccess && split) {
            g->tile_nplain.resize(g->n_tiles);
            e = cudaMemcpy(g->tile_nplain.data(), d_nplain, sizeof(int64_t) * g->n_tiles, cudaMemcpyDeviceToHost);
        }
        for (int64_t T = 0; T < g->n_tiles; ++T) toff[T + 1] = toff[T] + tcnt[T];
        g->E = toff[g->n_tiles];
        if (e == cudaSuccess)
            e = cudaMemcpy(g->tile_off, toff.data(), sizeof(int64_t) * (g->n_tiles + 1), cudaMemcpyHostToDevice);
        if (e != cudaSuccess) cudaFree(d_nplain);
        GEOM_CUDA(e);
    }
    {
        fft_status r2 = dmalloc(g, &g->tile_rows, g->E);
        if (r2 == FFT_OK && g->E > 0) {
            tile_fill_kernel<<<(unsigned)g->n_tiles, CULL_THREADS>>>(C, g->tile_off, d_nplain, g->tile_rows);
            cudaError_t e = cudaGetLastError();
            if (e == cudaSuccess) e = cudaDeviceSynchronize();
            if (e != cudaSuccess) r2 = cuda_fail(e, "tile lists");
        }
        cudaFree(d_nplain);
        GEOM_TRY(r2);
    }

    // ---- FP64 pair-frame bases of the entries
    GEOM_TRY(dmalloc(g, &g->ebase, g->E));
    GEOM_TRY(dmalloc(g, &g->ebase3, g->E));
    if (g->E > 0) {
        double* d_tx = nullptr;
        int32_t* d_pairs = nullptr;
        cudaError_t e = cudaMalloc(&d_tx, sizeof(double) * 3 * n_tx);
        if (e == cudaSuccess) e = cudaMalloc(&d_pairs, sizeof(int32_t) * 2 * n_rows);
        if (e == cudaSuccess) e = cudaMemcpy(d_tx, tx_xyz, sizeof(double) * 3 * n_tx, cudaMemcpyHostToDevice);
        if (e == cudaSuccess) e = cudaMemcpy(d_pairs, rows, sizeof(int32_t) * 2 * n_rows, cudaMemcpyHostToDevice);
        RowFrame* d_frame = nullptr;
        if (e == cudaSuccess) e = cudaMalloc(&d_frame, sizeof(RowFrame) * n_rows);
        if (e == cudaSuccess) {
            row_frame_kernel<<<(unsigned)ceil_div(n_rows, 128), 128>>>(d_tx, d_pairs, g->row_band, g->d_band, n_rows, d_frame);
            entry_base_kernel<<<(unsigned)g->n_tiles, 256>>>(g->tile_off, g->tile_rows, d_frame, grid->origin[0],
                                                             grid->origin[1], grid->origin[2], grid->h, g->tiles[0],
                                                             g->tiles[1], g->ebase, g->ebase3);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = cudaDeviceSynchronize();
        cudaFree(d_frame);
        cudaFree(d_tx);
        cudaFree(d_pairs);
        GEOM_CUDA(e);
    }

    // ---- row-major view of the entries that the products evaluate (the tiles of the layers
    // [z_lo, z_end), one range of tiles as z is their slowest index)
    find_mirror(g, tx_xyz, rows);
    {
        const int64_t per_z = (int64_t)g->tiles[0] * g->tiles[1];
        const int64_t e_lo = toff[per_z * (g->z_lo / TILE_Z)], e_hi = toff[per_z * ceil_div(g->z_end, TILE_Z)];
        const int64_t Ek = e_hi - e_lo;
        g->E_used = Ek;
        int32_t* d_rc = nullptr;
        int32_t* d_cur = nullptr;
        cudaError_t ea = cudaMalloc(&d_rc, sizeof(int32_t) * n_rows);
        if (ea == cudaSuccess) ea = cudaMalloc(&d_cur, sizeof(int32_t) * n_rows);
        if (ea == cudaSuccess) ea = cudaMemset(d_rc, 0, sizeof(int32_t) * n_rows);
        if (ea == cudaSuccess) ea = cudaMemset(d_cur, 0, sizeof(int32_t) * n_rows);
        if (ea != cudaSuccess) {
            cudaFree(d_rc);
            cudaFree(d_cur);
        }
        GEOM_CUDA(ea);
        if (Ek > 0) row_count_kernel<<<(unsigned)ceil_div(Ek, 256), 256>>>(g->tile_rows, e_lo, e_hi, d_rc);
        std::vector<int32_t> rc32(n_rows);
        cudaError_t e = cudaMemcpy(rc32.data(), d_rc, sizeof(int32_t) * n_rows, cudaMemcpyDeviceToHost);
        std::vector<int64_t> roff(n_rows + 1, 0);
        for (int64_t p = 0; p < n_rows; ++p) roff[p + 1] = roff[p] + rc32[p];
        fft_status r2 = (e == cudaSuccess) ? dmalloc(g, &g->row_off, n_rows + 1) : cuda_fail(e, "row counts");
        if (r2 == FFT_OK) r2 = dmalloc(g, &g->row_ent, Ek);
        if (r2 == FFT_OK) {
            e = cudaMemcpy(g->row_off, roff.data(), sizeof(int64_t) * (n_rows + 1), cudaMemcpyHostToDevice);
            if (e == cudaSuccess && Ek > 0) {
                row_fill_kernel<<<(unsigned)ceil_div(Ek, 256), 256>>>(g->tile_rows, e_lo, e_hi, g->row_off, d_cur,
                                                                      g->row_ent);
                row_sort_kernel<<<(unsigned)ceil_div(n_rows, 128), 128>>>(g->row_off, n_rows, g->row_ent);
                e = cudaGetLastError();
            }
            if (e != cudaSuccess) r2 = cuda_fail(e, "row lists");
        }
        cudaFree(d_rc);
        cudaFree(d_cur);
        GEOM_TRY(r2);
    }

    // ---- work items
    GEOM_TRY(set_apply_attributes(g));
    // commit the no-allocation PSF's static scratch on this device now, so that
    // fft_psf_noalloc itself never loads a module or allocates
    GEOM_TRY(noalloc_prepare(g->dev));
    g->apply_ctas = apply_occupancy(g);
    sharp_launch_shape(g);
    plain_launch_shape(g);
    build_stack(g, tx_xyz, rows, band_of_row, tables);
    // one J partial per (entry, 8 x 8 x 8 region); a stack's products use its classes' buffer
    if (!nested && g->stk.empty()) GEOM_TRY(dmalloc(g, &g->jpart, (size_t)g->E * 4));
    GEOM_TRY(dmalloc(g, &g->counter, 4));
    GEOM_TRY(build_items(g, toff, DEFAULT_ITEMS_PER_CTA));
    GEOM_CUDA(cudaDeviceSynchronize());
    if (!nested) GEOM_TRY(count_support(g, &g->support, &g->evaluated));
    GEOM_CUDA(cudaDeviceSynchronize());
#undef GEOM_TRY
#undef GEOM_CUDA
    *out = g;
    return FFT_OK;
}

}  // namespace

}  // namespace fftgb

extern "C" fft_status fft_geom_create(const double* tx_xyz, int32_t n_tx, const int32_t* rows,
                                      int64_t n_rows, const int32_t* band_of_row, const fft_grid* grid,
                                      double c0, const fft_table* tables, int32_t n_tables,
                                      int32_t dt_mode, fft_geom* out) {
    FFT_API_RANGE("fft_geom_create");
    return create_geom(tx_xyz, n_tx, rows, n_rows, band_of_row, grid, c0, tables, n_tables, dt_mode, false, out);
}

extern "C" void fft_geom_destroy(fft_geom g) {
    if (!g) return;
    int cur = 0;
    cudaGetDevice(&cur);
    if (cur != g->dev) cudaSetDevice(g->dev);
    cudaDeviceSynchronize();
    int dev = g->dev;
    free_geom(g);
    if (cur != dev) cudaSetDevice(cur);
}

// Kernels of one J or J^T of one column: an item kernel per kind of rows and a reduction, per pass of a class of
// a stack two more.
static int product_launches(fft_geom g) {
    int n = 0;
    for (const StackClass& c : g->stk)
        for (int64_t left = (int64_t)c.off.size(); left > 0;) {
            n += product_launches(c.sub) + 2;
            left -= pass_columns(c.sub, left);
        }
    if (!g->stk.empty()) return n;
    const bool split = g->sharp && g->dt_mode != FFT_DT_FP64;
    return 1 + (split ? (g->n_items_plain > 0 ? 1 : 0) + (g->n_items > g->n_items_plain ? 1 : 0) : 1);
}

extern "C" fft_status fft_geom_route(fft_geom g, fft_route_t* route) {
    FFT_ARG(g && route, "fft_geom_route: null argument");
    route->mirror = g->mirror;
    route->stack_classes = (int32_t)g->stk.size();
    route->stack_batch = g->stk_batch ? 1 : 0;
    route->stack_psf = (g->stk_psf1 ? 1 : 0) + (g->stk_psf4 ? 2 : 0);
    route->batch_cols = g->batch_cols;
    route->segments = g->seg_n;
    route->solver_comp = has_compensated(g) ? 1 : 0;
    route->launches = product_launches(g);
    return FFT_OK;
}

extern "C" fft_status fft_geom_info(fft_geom g, fft_geom_info_t* info) {
    FFT_ARG(g && info, "fft_geom_info: null argument");
    info->n_rows = g->M;
    info->n_vox = g->V;
    info->n_entries = g->E;
    info->n_items = g->n_items;
    info->support_evals = g->support;
    info->evaluated_evals = g->evaluated;
    info->scratch_bytes = g->scratch_bytes;
    info->dt_mode = g->dt_mode;
    info->phi_terms = g->trig_terms;
    info->psf_tc_mma_flops = g->psf_tc_mma_flops;
    info->psf_tc_entries = g->psf_tc_entries;
    return FFT_OK;
}
