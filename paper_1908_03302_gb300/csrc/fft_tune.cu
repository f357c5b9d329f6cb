// Autotuning of the J / J^T work decomposition. The tile (16 x 16 x 8 voxels) is cut into
// work items of a tile and a range of its candidate rows; how many rows an item takes (set
// through the number of items per persistent CTA) trades load balance at the end of a launch
// against per-item overhead and J^T partial slots, and the persistent grid may hold fewer
// CTAs per SM than fit. Both depend on the acquisition, so they are chosen by timing J and
// J^T on the device for each candidate and keeping the fastest.
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "fft_common.cuh"

namespace fftgb {

namespace {

__global__ void tune_fill_kernel(float* x, int64_t n, float scale) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) x[i] = scale * (float)((i * 2654435761u) % 1000u - 500) * 1e-3f;
}

}  // namespace

}  // namespace fftgb

using namespace fftgb;

extern "C" fft_status fft_geom_autotune(fft_geom g, void* stream, fft_tune_info_t* info) {
    FFT_API_RANGE("fft_geom_autotune");
    FFT_ARG(g, "fft_geom_autotune: null geometry");
    fft_status rc = check_device(g->dev);
    if (rc != FFT_OK) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    int dev = 0, sms = 1;
    FFT_CUDA(cudaGetDevice(&dev));
    FFT_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int occ = std::max(1, apply_occupancy(g) / std::max(sms, 1));
    std::vector<int64_t> toff(g->n_tiles + 1);
    FFT_CUDA(cudaMemcpy(toff.data(), g->tile_off, sizeof(int64_t) * (g->n_tiles + 1), cudaMemcpyDeviceToHost));

    float *m = nullptr, *d = nullptr, *out_v = nullptr, *out_m = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr, e2 = nullptr;
    cudaError_t e = cudaMalloc(&m, sizeof(float) * (size_t)g->V);
    if (e == cudaSuccess) e = cudaMalloc(&d, sizeof(float) * (size_t)g->M);
    if (e == cudaSuccess) e = cudaMalloc(&out_v, sizeof(float) * (size_t)g->V);
    if (e == cudaSuccess) e = cudaMalloc(&out_m, sizeof(float) * (size_t)g->M);
    if (e == cudaSuccess) e = cudaEventCreate(&e0);
    if (e == cudaSuccess) e = cudaEventCreate(&e1);
    if (e == cudaSuccess) e = cudaEventCreate(&e2);
    if (e == cudaSuccess) {
        tune_fill_kernel<<<(unsigned)ceil_div(g->V, 256), 256, 0, st>>>(m, g->V, 1.0f);
        tune_fill_kernel<<<(unsigned)ceil_div(g->M, 256), 256, 0, st>>>(d, g->M, 1e-8f);
        e = cudaGetLastError();
    }
    // Search: the sizes that the rule gives an untuned operator (0: default_item_rows), then all item sizes
    // at the occupancy limit (stopping once two sizes in a row are slower than the best of them by more
    // than 2 %), then one CTA per SM fewer around the best size, nine candidates at most. The rule's sizes are
    // given up only for ones more than 2 % faster: at least 64 rows an item cost small arrays half their
    // speed (a 20-iteration solve of four 32-element slices: 8.1 ms against 5.2 ms by the rule).
    // A candidate gets an untimed pass first unless the last application took over 20 ms (then
    // first-launch effects are lost in the measurement and the pass would double the cost of tuning a large
    // acquisition), and the least of three timed ones unless they take that long.
    const int cand_items[] = {0, 4, 8, 16, 32, 64, 128};
    const int n_cand = 7, max_tried = 9;
    double best = 1e300, best_j = 0.0, best_jt = 0.0, last = 0.0;
    int best_items = g->items_per_cta, best_ctas = g->apply_ctas / std::max(sms, 1), tried = 0, best_ii = 0,
        best_n_items = g->n_items;
    // Items of the operator and, for an elevation stack, of its classes' operators.
    auto set_items = [&](int n_ctas, int items_per_cta) {
        g->apply_ctas = n_ctas;
        const fft_status r = build_items(g, toff, items_per_cta);
        return r == FFT_OK && !g->stk.empty() ? stack_build_items(g, items_per_cta) : r;
    };
    // The listed sizes of small operators come to the same rows an item: one of them is timed.
    const bool wide = g->plain_warps > APPLY_WARPS && g->phi_eval != PHI_TRIG && g->dt_mode == FFT_DT_STABLE;
    std::vector<std::vector<int64_t>> seen;
    auto timed_before = [&](int ctas, int ii) {
        std::vector<int64_t> key = {wide ? 0 : ctas, item_rows(g->E, cand_items[ii], ctas * sms)};
        for (const StackClass& k : g->stk) key.push_back(item_rows(k.sub->E, cand_items[ii], ctas * sms));
        if (std::find(seen.begin(), seen.end(), key) != seen.end()) return true;
        seen.push_back(key);
        return false;
    };
    const int old_ctas = g->apply_ctas, old_items = g->items_per_cta;
    auto try_one = [&](int ctas, int ii) -> bool {
        if ((rc = set_items(ctas * sms, cand_items[ii])) != FFT_OK) return false;
        if (tried == 0 || last < 20.0) {
            if ((rc = launch_JT(g, d, out_v, st)) != FFT_OK) return false;
            if ((rc = launch_J(g, m, out_m, st)) != FFT_OK) return false;
        }
        double ms_j = 1e300, ms_jt = 1e300;
        for (int rep = 0; rep < 3 && (rep == 0 || ms_j + ms_jt < 20.0); ++rep) {
            e = cudaEventRecord(e0, st);
            if (e == cudaSuccess && (rc = launch_JT(g, d, out_v, st)) != FFT_OK) return false;
            if (e == cudaSuccess) e = cudaEventRecord(e1, st);
            if (e == cudaSuccess && (rc = launch_J(g, m, out_m, st)) != FFT_OK) return false;
            if (e == cudaSuccess) e = cudaEventRecord(e2, st);
            if (e == cudaSuccess) e = cudaEventSynchronize(e2);
            float t_jt = 0.0f, t_j = 0.0f;
            if (e == cudaSuccess) e = cudaEventElapsedTime(&t_jt, e0, e1);
            if (e == cudaSuccess) e = cudaEventElapsedTime(&t_j, e1, e2);
            if (e != cudaSuccess) return false;
            ms_jt = std::min(ms_jt, (double)t_jt);
            ms_j = std::min(ms_j, (double)t_j);
        }
        ++tried;
        last = ms_j + ms_jt;
        if (last < (best_ii == 0 ? 0.98 : 1.0) * best) {
            best = last;
            best_j = ms_j;
            best_jt = ms_jt;
            best_items = cand_items[ii];
            best_ii = ii;
            best_ctas = ctas;
            best_n_items = g->n_items;
        }
        return true;
    };
    if (e == cudaSuccess && try_one(occ, 0)) {
        int worse = 0, centre = 1;
        double swept = 1e300;   // the best of the listed sizes
        for (int ii = 1; ii < n_cand && !timed_before(occ, ii); ++ii) {   // (then the larger ones are alike too)
            if (!try_one(occ, ii)) break;
            worse = (last > 1.02 * swept) ? worse + 1 : 0;
            if (worse == 2) break;
            if (last < swept) {
                swept = last;
                centre = ii;
            }
        }
        if (e == cudaSuccess && rc == FFT_OK && occ > 1) {
            for (int ii = std::max(1, centre - 1); ii <= std::min(n_cand - 1, centre + 1) && tried < max_tried; ++ii)
                if (!timed_before(occ - 1, ii) && !try_one(occ - 1, ii)) break;
        }
    }
    if (e == cudaSuccess && rc == FFT_OK) rc = set_items(best_ctas * sms, best_items);
    // an operator that lost its items to a failed allocation gets the ones back that it came with
    if (g->unusable) set_items(old_ctas, old_items);
    if (e == cudaSuccess && rc == FFT_OK) e = cudaStreamSynchronize(st);
    cudaFree(m);
    cudaFree(d);
    cudaFree(out_v);
    cudaFree(out_m);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (e2) cudaEventDestroy(e2);
    if (rc != FFT_OK) return rc;
    if (e != cudaSuccess) return cuda_fail(e, "fft_geom_autotune");
    if (info) {
        info->items_per_cta = best_items;
        if (best_items == 0) {   // the listed size nearest to the rule's
            info->items_per_cta = 4;
            while (info->items_per_cta < 128 && best_n_items > 1.41 * info->items_per_cta * best_ctas * sms)
                info->items_per_cta *= 2;
        }
        info->ctas_per_sm = best_ctas;
        info->ms_J = best_j;
        info->ms_JT = best_jt;
        info->n_tried = tried;
    }
    return FFT_OK;
}
