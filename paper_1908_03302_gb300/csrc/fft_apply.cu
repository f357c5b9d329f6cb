// J m and J^T d: the host side of the apply kernels (fft_apply_kernel.cuh) - launch shapes,
// scratch, the row and tile reductions - and the C entry points.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <vector>

#include "fft_apply_kernel.cuh"

namespace fftgb {

// d_p = sum over the row's entries (ascending tile order) and the 4 regions of the partials.
// LOW (the compensated form): the partials are FP64 and summed in it, and what d_p lacks after rounding goes to low.
template <bool LOW>
__global__ void __launch_bounds__(256) j_reduce_kernel(const int64_t* __restrict__ row_off,
                                                       const int64_t* __restrict__ row_ent,
                                                       const void* __restrict__ jpart, int64_t M,
                                                       float* __restrict__ d, float* __restrict__ low) {
    // one warp per row: lane l takes the row's entries l, l + 32, ... in order (the 4 region
    // partials of an entry pairwise in FP32, entries accumulated in FP64), then a fixed
    // butterfly over the lanes; the order never depends on scheduling
    const int lane = threadIdx.x & 31;
    const int64_t p = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (p >= M) return;
    auto four = [&](int64_t j) {
        if (LOW) {
            const double2* a = reinterpret_cast<const double2*>(jpart) + row_ent[j] * 2;
            const double2 a0 = __ldg(a), a1 = __ldg(a + 1);
            return (a0.x + a0.y) + (a1.x + a1.y);
        }
        const float4 a = __ldg(reinterpret_cast<const float4*>(jpart) + row_ent[j]);
        return (double)((a.x + a.y) + (a.z + a.w));
    };
    double s = 0.0;
    const int64_t j1 = row_off[p + 1];
    int64_t j = row_off[p] + lane;
    for (; j + 32 < j1; j += 64) {   // two entries in flight, added in the same order
        const double a0 = four(j), a1 = four(j + 32);
        s += a0;
        s += a1;
    }
    if (j < j1) s += four(j);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane != 0) return;
    d[p] = (float)s;
    if (LOW) low[p] = (float)(s - (double)(float)s);
}

// The batch form of j_reduce_kernel: jpart[(entry * 8 + region) * NC + r]; the same lane order,
// pairing and butterfly per column, d[r * M + p], columns r < ncol.
template <int NC>
__global__ void __launch_bounds__(256) j_reduce_n_kernel(const int64_t* __restrict__ row_off,
                                                         const int64_t* __restrict__ row_ent,
                                                         const float* __restrict__ jpart, int64_t M, int ncol,
                                                         float* __restrict__ d) {
    const int lane = threadIdx.x & 31;
    const int64_t p = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (p >= M) return;
    double s[NC];
#pragma unroll
    for (int r = 0; r < NC; ++r) s[r] = 0.0;
    const int64_t j1 = row_off[p + 1];
    for (int64_t j = row_off[p] + lane; j < j1; j += 32) {
#pragma unroll
        for (int h = 0; h < NC / 4; ++h) {
            const float4* q = reinterpret_cast<const float4*>(jpart + row_ent[j] * (8 * NC)) + h;
            float4 g[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) g[k] = __ldg(q + k * (NC / 4));
            s[4 * h] += (double)(((g[0].x + g[1].x) + (g[2].x + g[3].x)) + ((g[4].x + g[5].x) + (g[6].x + g[7].x)));
            s[4 * h + 1] += (double)(((g[0].y + g[1].y) + (g[2].y + g[3].y)) + ((g[4].y + g[5].y) + (g[6].y + g[7].y)));
            s[4 * h + 2] += (double)(((g[0].z + g[1].z) + (g[2].z + g[3].z)) + ((g[4].z + g[5].z) + (g[6].z + g[7].z)));
            s[4 * h + 3] += (double)(((g[0].w + g[1].w) + (g[2].w + g[3].w)) + ((g[4].w + g[5].w) + (g[6].w + g[7].w)));
        }
    }
#pragma unroll
    for (int r = 0; r < NC; ++r) {
        double v = s[r];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0 && r < ncol) d[(int64_t)r * M + p] = (float)v;
    }
}

// g for voxels of tiles with several items (the sum of their slots) or with none (0); tiles with
// one item were written by the apply kernel. A CTA takes 32 runs of 4 x voxels of a tile, a lane
// each; warp w adds slots w, w + 8, .. in that order (compensated, so that the sum does not lose
// to the number of slots), the eight partial sums are added as two floats: a fixed order, and eight times
// as many loads in flight as with one thread per run, which a tile cut into many small items
// needs (32-element ring: about 45 slots per tile). (In FP64 those eight took half of the kernel.)
// NCOL = 4, 8: the batch forms, slot q of column r at gpart[((s0 + q) * NCOL + r) * TILE_VOX],
// g[r * V + v], columns r < ncol. LOW (the compensated form, one column): the partials have low
// parts (gpart_low), and what g lacks after rounding goes to g_low.
constexpr int RED_WARPS = 8;
template <int NCOL, bool LOW>
__global__ void __launch_bounds__(32 * RED_WARPS) jt_reduce_kernel(const int32_t* __restrict__ slot0,
                                                                   const int32_t* __restrict__ nslot,
                                                                   const float* __restrict__ gpart, int nx, int ny,
                                                                   int nz, int z_lo, int z_end, int mirror,
                                                                   int tiles_x, int tiles_y, int ncol,
                                                                   float* __restrict__ g,
                                                                   const float* __restrict__ gpart_low,
                                                                   float* __restrict__ g_low) {
    __shared__ float4 sh[RED_WARPS][32], sh_low[LOW ? RED_WARPS : 1][32];
    constexpr int PER_TILE = TILE_VOX / (4 * 32);   // CTAs per tile
    const int T = blockIdx.x / PER_TILE, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int s0 = slot0[T];
    if (s0 == -1) return;
    const int loc = 4 * (32 * (int)(blockIdx.x % PER_TILE) + lane);
    const int ix = TILE_X * (T % tiles_x) + loc % TILE_X;
    const int iy = TILE_Y * ((T / tiles_x) % tiles_y) + (loc / TILE_X) % TILE_Y;
    const int iz = TILE_Z * (T / (tiles_x * tiles_y)) + loc / (TILE_X * TILE_Y);
    const int64_t V = (int64_t)nx * ny * nz;
    const int64_t v = ((int64_t)iz * ny + iy) * nx + ix;
    const bool inside = iy < ny && iz >= z_lo && iz < z_end && ix < nx;
    const int64_t mo = (int64_t)mirror_step(mirror, iz, nz) * ny * nx;   // to the mirrored layer (0: none)
    const int ns = (s0 == -2 || !inside) ? 0 : nslot[T];
    for (int r = 0; r < ncol; ++r) {
        float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f}, low[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        const float* base = ns > 0 ? gpart + ((int64_t)s0 * NCOL + r) * TILE_VOX + loc : nullptr;
        auto add = [&](const float4& x) {
            const float xv[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {   // Kahan's sum (an infinite one, of infinite data, has nothing to add)
                const float y = xv[k] - low[k], t = acc[k] + y;
                low[k] = isinf(t) ? 0.0f : (t - acc[k]) - y;
                acc[k] = t;
            }
        };
        const float* lbase = LOW && ns > 0 ? gpart_low + (int64_t)s0 * TILE_VOX + loc : nullptr;
        float lows[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        auto add_low = [&](const float4& x) {
            lows[0] += x.x;
            lows[1] += x.y;
            lows[2] += x.z;
            lows[3] += x.w;
        };
        int q = w;
        for (; q + 3 * RED_WARPS < ns; q += 4 * RED_WARPS) {   // four slots in flight
            float4 x[4], y[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int64_t slot = q + k * RED_WARPS;
                x[k] = __ldcs(reinterpret_cast<const float4*>(base + slot * NCOL * TILE_VOX));
                if (LOW) y[k] = __ldcs(reinterpret_cast<const float4*>(lbase + slot * TILE_VOX));
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                add(x[k]);
                if (LOW) add_low(y[k]);
            }
        }
        for (; q < ns; q += RED_WARPS) {
            add(__ldcs(reinterpret_cast<const float4*>(base + (int64_t)q * NCOL * TILE_VOX)));
            if (LOW) add_low(__ldcs(reinterpret_cast<const float4*>(lbase + (int64_t)q * TILE_VOX)));
        }
        sh[w][lane] = make_float4(acc[0], acc[1], acc[2], acc[3]);
        if (LOW)   // (low is what acc has too much)
            sh_low[w][lane] = make_float4(lows[0] - low[0], lows[1] - low[1], lows[2] - low[2], lows[3] - low[3]);
        __syncthreads();
        if (w < 4) {   // warp w: component w of the 32 runs
            float s = 0.0f, l = 0.0f;   // the sum and what it lacks
#pragma unroll
            for (int k = 0; k < RED_WARPS; ++k) {
                l += two_sum(s, reinterpret_cast<const float*>(&sh[k][lane])[w], s);
                if (LOW) l += reinterpret_cast<const float*>(&sh_low[k][lane])[w];
            }
            if (!isinf(s)) l = two_sum(s, l, s);
            if (inside && ix + w < nx) {
                g[(int64_t)r * V + v + w] = s;
                if (mo != 0) g[(int64_t)r * V + v + mo + w] = s;
                if (LOW) {
                    g_low[v + w] = l;
                    if (mo != 0) g_low[v + mo + w] = l;
                }
            }
        }
        if (NCOL > 1) __syncthreads();
    }
}

fft_status check_usable(fft_geom g) {
    if (!g->unusable) return FFT_OK;
    set_error("the operator has no work items: fft_geom_autotune ran out of memory (tune again or make a new one)");
    return FFT_ERR_STATE;
}

static ApplyParams make_params(fft_geom g) {
    ApplyParams P;
    P.rec = g->rec;
    P.rec64 = g->rec64;
    P.row_band = g->row_band;
    P.tab = g->tab;
    P.n_bands = g->n_bands;
    P.n_tab = g->n_tab;
    P.bc = g->d_band;
    P.tile_rows = g->tile_rows;
    P.ebase = g->ebase;
    P.ebase3 = g->ebase3;
    P.items = g->items;
    P.n_items = g->n_items;
    P.counter = g->counter;
    P.tiles_x = g->tiles[0];
    P.tiles_y = g->tiles[1];
    P.nx = g->grid.nx;
    P.ny = g->grid.ny;
    P.nz = g->grid.nz;
    P.z_lo = g->z_lo;
    P.z_end = g->z_end;
    P.mirror = g->mirror;
    P.zw = g->zw;
    for (int a = 0; a < 3; ++a) P.org[a] = g->grid.origin[a];
    P.h = g->grid.h;
    P.vin = nullptr;
    P.vout = nullptr;
    P.gpart = g->gpart;
    P.vlow = P.gpart_low = nullptr;
    P.vpart = nullptr;
    P.dsum = nullptr;
    P.icount = nullptr;
    P.trig_nq = g->trig_nq;
    P.seg_n = g->seg_n;
    P.nvox = g->V;
    P.nrow = g->M;
    P.ncol = 1;
    return P;
}

size_t apply_smem(fft_geom g, int warps) {
    size_t tab = ((size_t)g->n_bands * g->n_tab * sizeof(float2) + 15) & ~(size_t)15;
    return tab + (size_t)warps * STG_PER_WARP * sizeof(float4);
}

size_t apply_smem(fft_geom g) { return apply_smem(g, APPLY_WARPS); }

size_t apply_smem8(fft_geom g, int warps) { return apply_smem(g, 0) + (size_t)warps * STG_PER_WARP8 * sizeof(float4); }

// Most warps (a multiple of 8, at most 24) one sharp-variant CTA can stage for.
static int sharp_max_warps(fft_geom g) {
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    int w = SHARP_MAX_WARPS;
    while (w > APPLY_WARPS && apply_smem(g, w) > (size_t)optin) w -= 4;
    return w;
}

// Most warps (at most 32) one plain wide CTA can stage for.
static int plain_max_warps(fft_geom g) {
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    int w = PLAIN_MAX_WARPS;
    while (w > APPLY_WARPS && apply_smem(g, w) > (size_t)optin) w -= 8;
    return w;
}

// Raise the dynamic shared-memory limit of every kernel instantiation once per geometry
// (outside any stream capture), so launches need no attribute calls. The limit belongs to the
// kernel, not to the handle: always the device's largest, so that a handle with small tables does not
// lower it under a live one with large tables. (Occupancy and launches go by the size that they use.)
fft_status set_apply_attributes(fft_geom g) {
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    const size_t smem = (size_t)optin;
    fft_status rc;
    if ((rc = set_attr_mode<MODE_JT>(smem)) != FFT_OK) return rc;
    if ((rc = set_attr_mode<MODE_J>(smem)) != FFT_OK) return rc;
    if ((rc = set_attr_mode<MODE_JTC>(smem)) != FFT_OK) return rc;
    if ((rc = set_attr_mode<MODE_JC>(smem)) != FFT_OK) return rc;
    if ((rc = set_attr_mode<MODE_COUNT>(smem)) != FFT_OK) return rc;
    if ((rc = set_attr_mode<MODE_COV>(smem)) != FFT_OK) return rc;
    // batch modes: stable detour only (other geometries apply the columns one by one)
    if ((rc = set_attr_mode<MODE_JT4>(smem)) != FFT_OK) return rc;
    if ((rc = set_attr_mode<MODE_J4>(smem)) != FFT_OK) return rc;
    cudaDeviceGetAttribute(&g->sms, cudaDevAttrMultiProcessorCount, dev);
    g->sms = std::max(g->sms, 1);
    g->col8 = g->dt_mode == FFT_DT_STABLE && apply_smem8(g, col8_warps<false>()) <= smem;
    if (g->col8) {
        if ((rc = set_attr_mode<MODE_JT8>(smem)) != FFT_OK) return rc;
        if ((rc = set_attr_mode<MODE_J8>(smem)) != FFT_OK) return rc;
    }
    return set_attr_mode<MODE_FROB>(smem);
}

// Persistent grid size: resident CTAs per SM of the J^T kernel times the SM count.
int apply_occupancy(fft_geom g) {
    int sms = 0, dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int per_sm = apply_blocks_per_sm(false, APPLY_THREADS, apply_smem(g));
    if (per_sm < 1) per_sm = 1;
    if (sms < 1) sms = 1;
    return per_sm * sms;
}

// CTA shape of the sharp variants: the block of 8, 12, 16 or 20 warps with the most resident
// warps per SM (the smaller block on a tie), and the persistent grid that fills the GPU.
void sharp_launch_shape(fft_geom g) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms < 1) sms = 1;
    int best_w = APPLY_WARPS, best_b = 1, best_res = 0;
    for (int w = APPLY_WARPS; w <= sharp_max_warps(g); w += 4) {
        const int b = apply_blocks_per_sm(true, 32 * w, apply_smem(g, w));
        if (b * w > best_res) {
            best_res = b * w;
            best_w = w;
            best_b = b;
        }
    }
    cudaGetLastError();
    g->sharp_warps = best_w;
    g->sharp_ctas = std::max(best_b, 1) * sms;
}

// CTA shape of the plain stable-detour table variants: 8-warp CTAs on the (autotuned)
// persistent grid, unless one wide CTA of 16, 24 or 32 warps keeps more warps resident per SM
// (large multi-band tables), then one such CTA per SM.
void plain_launch_shape(fft_geom g) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms < 1) sms = 1;
    const int b8 = apply_blocks_per_sm(false, APPLY_THREADS, apply_smem(g));
    int best_w = APPLY_WARPS, best_b = std::max(b8, 1), best_res = b8 * APPLY_WARPS;
    for (int w = 2 * APPLY_WARPS; w <= plain_max_warps(g); w += APPLY_WARPS) {
        const int b = apply_blocks_per_sm(false, 32 * w, apply_smem(g, w));
        if (b * w > best_res) {
            best_res = b * w;
            best_w = w;
            best_b = b;
        }
    }
    cudaGetLastError();
    g->plain_warps = best_w;
    g->plain_ctas = std::max(best_b, 1) * sms;
}

static int64_t batch_bytes(fft_geom g, int cols) {
    return (int64_t)sizeof(float) * cols * (g->E * 8 + (int64_t)g->n_slots * TILE_VOX);
}

static cudaError_t alloc_batch(fft_geom g, int cols, float** jp, float** gp) {
    *jp = *gp = nullptr;
    cudaError_t e = device_malloc((void**)jp, sizeof(float) * (size_t)(g->E > 0 ? g->E : 1) * 8 * cols);
    if (e == cudaSuccess && g->n_slots > 0)
        e = device_malloc((void**)gp, sizeof(float) * (size_t)g->n_slots * cols * TILE_VOX);
    if (e == cudaSuccess) return e;
    cudaGetLastError();
    cudaFree(*jp);
    *jp = *gp = nullptr;
    return e;
}

// Partials of a batch of n columns: for eight columns at once where n is more than four, the kernels
// fit and memory allows it (asked once), else for four. A caller may have captured a call that uses the
// four-column buffers, so they stay beside the eight-column ones, until new work items replace both.
static fft_status batch_scratch(fft_geom g, int n, cudaStream_t st) {
    if (g->nested) return FFT_OK;   // the parent's (stack_scratch)
    const bool wide = n > 4 && g->col8 && !g->batch8_refused;
    if (g->batch_cols == 8 || (g->batch_cols == 4 && !wide)) return FFT_OK;
    if (wide) {
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        FFT_CUDA(cudaStreamIsCapturing(st, &cap));
        if (cap == cudaStreamCaptureStatusNone) {
            // (relaxed: growing must not break a capture that another stream is in the middle of)
            cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
            FFT_CUDA(cudaThreadExchangeStreamCaptureMode(&mode));
            size_t mem_free = 0, mem_total = 0;
            float *jp = nullptr, *gp = nullptr;
            const bool grown = cudaMemGetInfo(&mem_free, &mem_total) == cudaSuccess &&
                               2.0 * (double)batch_bytes(g, 8) <= (double)mem_free &&
                               alloc_batch(g, 8, &jp, &gp) == cudaSuccess;
            cudaThreadExchangeStreamCaptureMode(&mode);
            if (grown) {
                g->jpart4_kept = g->jpart4;
                g->gpart4_kept = g->gpart4;
                g->jpart4 = jp;
                g->gpart4 = gp;
                g->batch_cols = 8;
                g->scratch_bytes += batch_bytes(g, 8);
                return FFT_OK;
            }
            g->batch8_refused = true;
        }
        if (g->batch_cols == 4) return FFT_OK;
    }
    if (alloc_batch(g, 4, &g->jpart4, &g->gpart4) != cudaSuccess) {
        set_error("batch apply: cudaMalloc of the partial buffers failed");
        return FFT_ERR_OOM;
    }
    g->batch_cols = 4;
    g->scratch_bytes += batch_bytes(g, 4);
    return FFT_OK;
}

void free_batch_scratch(fft_geom g) {
    if (g->nested || g->batch_cols == 0) return;
    g->scratch_bytes -= batch_bytes(g, g->batch_cols) + (g->jpart4_kept ? batch_bytes(g, 4) : 0);
    for (float* p : {g->jpart4, g->gpart4, g->jpart4_kept, g->gpart4_kept}) cudaFree(p);
    g->jpart4 = g->gpart4 = g->jpart4_kept = g->gpart4_kept = nullptr;
    g->batch_cols = 0;
    g->batch8_refused = false;
}

// Columns of the next pass of rem columns: one alone, two to four in a four-column pass, five to eight
// in an eight-column one. Over the same rows of slices3d J^T the three take 25.6, 32.5 and 38.9 ms, so
// that two columns already pay for the wider kernel (ring256, block of 8, J and J^T: 10.54 ms in two
// four-column passes, 6.91 ms in one).
int pass_columns(fft_geom g, int64_t rem) {
    if (rem > 4 && g->batch_cols == 8) return (int)std::min<int64_t>(rem, 8);
    return (int)std::min<int64_t>(rem, 4);
}

template <int NC, int MODE>
static fft_status j_pass(fft_geom g, const float* m, int nc, float* d, cudaStream_t st) {
    ApplyParams P = make_params(g);
    P.vin = m;
    P.vout = g->jpart4;
    P.ncol = nc;
    fft_status rc = launch_batch<MODE>(g, P, st);
    if (rc != FFT_OK || g->M == 0) return rc;
    j_reduce_n_kernel<NC><<<(unsigned)ceil_div(g->M, 8), 256, 0, st>>>(g->row_off, g->row_ent, g->jpart4, g->M, nc, d);
    FFT_CUDA(cudaGetLastError());
    return FFT_OK;
}

template <int NCOL, bool LOW = false>
static fft_status launch_jt_reduce(fft_geom g, const float* gpart, int ncol, float* gout, cudaStream_t st,
                                   const float* gpart_low = nullptr, float* g_low = nullptr) {
    if (g->n_tiles == 0) return FFT_OK;
    jt_reduce_kernel<NCOL, LOW><<<(unsigned)(g->n_tiles * (TILE_VOX / 128)), 32 * RED_WARPS, 0, st>>>(
        g->tile_slot0, g->tile_nslot, gpart, g->grid.nx, g->grid.ny, g->grid.nz, g->z_lo, g->z_end, g->mirror,
        g->tiles[0], g->tiles[1], ncol, gout, gpart_low, g_low);
    FFT_CUDA(cudaGetLastError());
    return FFT_OK;
}

template <int NC, int MODE>
static fft_status jt_pass(fft_geom g, const float* d, int nc, float* gout, cudaStream_t st) {
    ApplyParams P = make_params(g);
    P.vin = d;
    P.vout = gout;
    P.gpart = g->gpart4;
    P.ncol = nc;
    fft_status rc = launch_batch<MODE>(g, P, st);
    if (rc != FFT_OK) return rc;
    return launch_jt_reduce<NC>(g, g->gpart4, nc, gout, st);
}

// Columns of the next pass of n from column c on, and whether it goes through the single-column kernels:
// fewer than four columns (they need no batch scratch; a stack's operator has it), those of other detour modes,
// and a last column alone in its group of eight (of four where the tables leave no room for the kernels of
// eight). Passes of four and eight give a column the same bits, so the result does not depend on which of
// the two there was memory for.
static int next_pass(fft_geom g, int n, int c, bool batch, bool& single) {
    const int nc = batch ? pass_columns(g, n - c) : 1;
    single = !batch || (nc == 1 && c % (g->col8 ? 8 : 4) == 0);
    return nc;
}

// d[:, c] = J m[:, c] for n columns.
fft_status launch_J_batch(fft_geom g, const float* m, int n, float* d, cudaStream_t st) {
    if (!g->stk.empty() && (n < 4 || g->stk_batch)) return stack_J(g, m, n, d, st);
    const bool batch = g->dt_mode == FFT_DT_STABLE && (n >= 4 || g->nested);
    fft_status rc = batch ? batch_scratch(g, n, st) : FFT_OK;
    for (int c = 0; c < n && rc == FFT_OK;) {
        bool single;
        const int nc = next_pass(g, n, c, batch, single);
        const float* mc = m + (int64_t)c * g->V;
        float* dc = d + (int64_t)c * g->M;
        if (single)
            rc = launch_J(g, mc, dc, st);
        else
            rc = nc > 4 ? j_pass<8, MODE_J8>(g, mc, nc, dc, st) : j_pass<4, MODE_J4>(g, mc, nc, dc, st);
        c += nc;
    }
    return rc;
}

// g[:, c] = J^T d[:, c] for n columns.
fft_status launch_JT_batch(fft_geom g, const float* din, int n, float* gout, cudaStream_t st, bool sparse) {
    if (!g->stk.empty() && (n < 4 || g->stk_batch) && (!sparse || g->stk_psf4)) return stack_JT(g, din, n, gout, st);
    const bool batch = g->dt_mode == FFT_DT_STABLE && (n >= 4 || g->nested);
    fft_status rc = batch ? batch_scratch(g, n, st) : FFT_OK;
    for (int c = 0; c < n && rc == FFT_OK;) {
        bool single;
        const int nc = next_pass(g, n, c, batch, single);
        const float* dc = din + (int64_t)c * g->M;
        float* gc = gout + (int64_t)c * g->V;
        if (single)
            rc = launch_JT(g, dc, gc, st);
        else
            rc = nc > 4 ? jt_pass<8, MODE_JT8>(g, dc, nc, gc, st) : jt_pass<4, MODE_JT4>(g, dc, nc, gc, st);
        c += nc;
    }
    return rc;
}

fft_status launch_J(fft_geom g, const float* m, float* d, cudaStream_t st) {
    if (!g->stk.empty()) return stack_J(g, m, 1, d, st);
    ApplyParams P = make_params(g);
    P.vin = m;
    P.vout = g->jpart;
    fft_status rc = launch_mode<MODE_J>(g, P, st);
    if (rc != FFT_OK) return rc;
    if (g->M > 0) {
        int64_t blocks = ceil_div(g->M, 8);   // 8 rows (warps) per block
        j_reduce_kernel<false><<<(unsigned)blocks, 256, 0, st>>>(g->row_off, g->row_ent, g->jpart, g->M, d, nullptr);
        FFT_CUDA(cudaGetLastError());
    }
    return FFT_OK;
}

fft_status launch_JT(fft_geom g, const float* din, float* gout, cudaStream_t st, bool sparse) {
    if (!g->stk.empty() && (!sparse || g->stk_psf1)) return stack_JT(g, din, 1, gout, st);
    ApplyParams P = make_params(g);
    P.vin = din;
    P.vout = gout;
    fft_status rc = launch_mode<MODE_JT>(g, P, st);
    if (rc != FFT_OK) return rc;
    return launch_jt_reduce<1>(g, g->gpart, 1, gout, st);
}

// J and J^T with compensated sums (MODE_JC, MODE_JTC), the result as the sum of two floats: d + d_low, g + g_low.
// The caller's scratch: jpart64 [E * 4], gpart_low [n_slots * TILE_VOX].
bool has_compensated(fft_geom g) {
    return g->dt_mode == FFT_DT_STABLE && g->stk.empty() && g->E_used <= COMP_MAX_ENTRIES;
}

fft_status launch_J_comp(fft_geom g, const float* m, float* d, float* d_low, double* jpart64, cudaStream_t st) {
    ApplyParams P = make_params(g);
    P.vin = m;
    P.vpart = jpart64;
    const fft_status rc = launch_mode<MODE_JC>(g, P, st);
    if (rc != FFT_OK || g->M == 0) return rc;
    j_reduce_kernel<true><<<(unsigned)ceil_div(g->M, 8), 256, 0, st>>>(g->row_off, g->row_ent, jpart64, g->M, d, d_low);
    FFT_CUDA(cudaGetLastError());
    return FFT_OK;
}

fft_status launch_JT_comp(fft_geom g, const float* din, float* gout, float* g_low, float* gpart_low,
                          cudaStream_t st) {
    ApplyParams P = make_params(g);
    P.vin = din;
    P.vout = gout;
    P.vlow = g_low;
    P.gpart_low = gpart_low;
    const fft_status rc = launch_mode<MODE_JTC>(g, P, st);
    if (rc != FFT_OK) return rc;
    return launch_jt_reduce<1, true>(g, g->gpart, 1, gout, st, gpart_low, g_low);
}

// cov_v = sum_p |J[p, v] w_p| (w null: all ones), gathered like J^T.
fft_status launch_cov(fft_geom g, const float* w, float* cov, cudaStream_t st) {
    ApplyParams P = make_params(g);
    P.vin = w;
    P.vout = cov;
    fft_status rc = launch_mode<MODE_COV>(g, P, st);
    if (rc != FFT_OK) return rc;
    return launch_jt_reduce<1>(g, g->gpart, 1, cov, st);
}

// In-support evaluations (dt < dt_max) of one apply and evaluations actually performed.
fft_status count_support(fft_geom g, int64_t* support, int64_t* evaluated) {
    if (!g->stk.empty()) {   // each class's operator counts its slices through zw
        *support = *evaluated = 0;
        for (StackClass& c : g->stk) {
            int64_t s = 0, e = 0;
            const fft_status rc = count_support(c.sub, &s, &e);
            if (rc != FFT_OK) return rc;
            *support += s;
            *evaluated += e;
        }
        return FFT_OK;
    }
    ApplyParams P = make_params(g);
    unsigned long long* d_cnt = nullptr;
    FFT_CUDA(cudaMalloc(&d_cnt, 2 * sizeof(unsigned long long)));
    cudaError_t e0 = cudaMemset(d_cnt, 0, 2 * sizeof(unsigned long long));
    if (e0 != cudaSuccess) {
        cudaFree(d_cnt);
        return cuda_fail(e0, "count_support: cudaMemset");
    }
    P.icount = d_cnt;
    fft_status rc = launch_mode<MODE_COUNT>(g, P, 0);
    unsigned long long h[2] = {0, 0};
    if (rc == FFT_OK) {
        cudaError_t e = cudaMemcpy(h, d_cnt, sizeof(h), cudaMemcpyDeviceToHost);
        if (e != cudaSuccess) rc = cuda_fail(e, "count_support");
    }
    cudaFree(d_cnt);
    *support = (int64_t)h[0];
    *evaluated = (int64_t)h[1];
    return rc;
}

fft_status compute_frob2(fft_geom g, double* out) {
    if (!g->stk.empty()) {
        *out = 0.0;
        for (StackClass& c : g->stk) {
            double s = 0.0;
            const fft_status rc = compute_frob2(c.sub, &s);
            if (rc != FFT_OK) return rc;
            *out += s;
        }
        return FFT_OK;
    }
    ApplyParams P = make_params(g);
    double* d_sum = nullptr;
    size_t n = (size_t)(g->n_items > 0 ? g->n_items : 1) * APPLY_WARPS;   // one per unit
    FFT_CUDA(cudaMalloc(&d_sum, n * sizeof(double)));
    cudaError_t e0 = cudaMemset(d_sum, 0, n * sizeof(double));
    if (e0 != cudaSuccess) {
        cudaFree(d_sum);
        return cuda_fail(e0, "frob2: cudaMemset");
    }
    P.dsum = d_sum;
    fft_status rc = launch_mode<MODE_FROB>(g, P, 0);
    std::vector<double> h(n, 0.0);
    if (rc == FFT_OK) {
        cudaError_t e = cudaMemcpy(h.data(), d_sum, n * sizeof(double), cudaMemcpyDeviceToHost);
        if (e != cudaSuccess) rc = cuda_fail(e, "frob2");
    }
    cudaFree(d_sum);
    double s = 0.0;
    for (size_t i = 0; i < n; ++i) s += h[i];
    *out = s;
    return rc;
}

}  // namespace fftgb

using namespace fftgb;

extern "C" fft_status fft_J_apply(fft_geom g, const float* m_dev, float* d_dev, void* stream) {
    FFT_API_RANGE("fft_J_apply");
    FFT_ARG(g && m_dev && d_dev, "fft_J_apply: null argument");
    fft_status rc = check_device(g->dev);
    if (rc != FFT_OK) return rc;
    return launch_J(g, m_dev, d_dev, (cudaStream_t)stream);
}

extern "C" fft_status fft_JT_apply(fft_geom g, const float* d_dev, float* g_dev, void* stream) {
    FFT_API_RANGE("fft_JT_apply");
    FFT_ARG(g && d_dev && g_dev, "fft_JT_apply: null argument");
    fft_status rc = check_device(g->dev);
    if (rc != FFT_OK) return rc;
    return launch_JT(g, d_dev, g_dev, (cudaStream_t)stream);
}

extern "C" fft_status fft_J_apply_batch(fft_geom g, const float* m_dev, int32_t n, float* d_dev, void* stream) {
    FFT_API_RANGE("fft_J_apply_batch");
    FFT_ARG(g && m_dev && d_dev, "fft_J_apply_batch: null argument");
    FFT_ARG(n >= 1, "fft_J_apply_batch: need n >= 1 columns");
    fft_status rc = check_device(g->dev);
    if (rc != FFT_OK) return rc;
    return launch_J_batch(g, m_dev, n, d_dev, (cudaStream_t)stream);
}

extern "C" fft_status fft_JT_apply_batch(fft_geom g, const float* d_dev, int32_t n, float* g_dev, void* stream) {
    FFT_API_RANGE("fft_JT_apply_batch");
    FFT_ARG(g && d_dev && g_dev, "fft_JT_apply_batch: null argument");
    FFT_ARG(n >= 1, "fft_JT_apply_batch: need n >= 1 columns");
    fft_status rc = check_device(g->dev);
    if (rc != FFT_OK) return rc;
    return launch_JT_batch(g, d_dev, n, g_dev, (cudaStream_t)stream);
}

extern "C" fft_status fft_coverage(fft_geom g, const float* w_dev, float* cov_dev, void* stream) {
    FFT_API_RANGE("fft_coverage");
    FFT_ARG(g && cov_dev, "fft_coverage: null argument");
    fft_status rc = check_device(g->dev);
    if (rc != FFT_OK) return rc;
    return launch_cov(g, w_dev, cov_dev, (cudaStream_t)stream);
}

extern "C" fft_status fft_frob2(fft_geom g, double* out) {
    FFT_API_RANGE("fft_frob2");
    FFT_ARG(g && out, "fft_frob2: null argument");
    fft_status rc = check_device(g->dev);
    if (rc != FFT_OK) return rc;
    if (g->frob2 < 0.0) {
        double v = 0.0;
        rc = compute_frob2(g, &v);
        if (rc != FFT_OK) return rc;
        g->frob2 = v;
    }
    *out = g->frob2;
    return FFT_OK;
}
