// Elevation stacks: one ring stepped in z, the acquisition of Sec. IV. A row of one slice and the same
// pair of another slice a whole number of layers away have the same entries of J, shifted by those
// layers, since an entry depends on a voxel's distances to the two transducers alone. The slices are
// grouped into classes whose members lie whole numbers of layers apart. Each class has one operator (a
// geometry of its own, `sub`) for the rows of its lowest slice on a grid extended in z so that it
// holds the layers of every member as that slice sees them, and J and J^T apply it to the members as
// columns: an entry is evaluated once for up to eight slices by the batch kernels, and half as often
// again where the slice's plane mirrors the extended lattice (find_mirror).
//
//   J m on slice s     = sub J (m moved down by the slice's layers)
//   J^T d              = sum over slices of (sub J^T d_s) moved up by the slice's layers
//
// Bound by the evaluations as the plain products are; the moves are one pass over the volume (~0.1 ms
// of slices3d's 93 ms, which was 371 with each slice's entries evaluated by themselves).
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <map>
#include <utility>
#include <vector>

#include "fft_common.cuh"

namespace fftgb {

namespace {

// Up to eight (column, slice) jobs that one pass of a class's operator serves.
constexpr int MAX_JOBS = 8;
struct StackJobs {
    int n;
    int32_t col[MAX_JOBS];           // column of the call
    int32_t off[MAX_JOBS];           // grid layer z of the slice is layer z + off of the extended grid
    const int32_t* rows[MAX_JOBS];   // the slice's rows in the order of the operator's rows
    int32_t first[MAX_JOBS];         // the first contribution to its column: J^T overwrites
};

// X[c][e] = m[col][e - off layers], 0 outside the grid.
__global__ void __launch_bounds__(256) stack_models_kernel(const StackJobs J, const float* __restrict__ m, int64_t V,
                                                           int64_t plane, int64_t V_ext, float* __restrict__ X) {
    const int c = blockIdx.y;
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= V_ext) return;
    const int64_t k = e - J.off[c] * plane;
    X[(int64_t)c * V_ext + e] = (k >= 0 && k < V) ? __ldg(m + (int64_t)J.col[c] * V + k) : 0.0f;
}

// D[c][p] = d[col][rows[p]].
__global__ void __launch_bounds__(256) stack_gather_kernel(const StackJobs J, const float* __restrict__ d, int64_t M,
                                                           int64_t M_sub, float* __restrict__ D) {
    const int c = blockIdx.y;
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p < M_sub) D[(int64_t)c * M_sub + p] = __ldg(d + (int64_t)J.col[c] * M + J.rows[c][p]);
}

// d[col][rows[p]] = D[c][p].
__global__ void __launch_bounds__(256) stack_scatter_kernel(const StackJobs J, const float* __restrict__ D,
                                                            int64_t M_sub, int64_t M, float* __restrict__ d) {
    const int c = blockIdx.y;
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p < M_sub) d[(int64_t)J.col[c] * M + J.rows[c][p]] = D[(int64_t)c * M_sub + p];
}

// g[col][v] (+)= sum over the jobs of the column of Y[c][v + off layers]; a pass's jobs in FP64.
__global__ void __launch_bounds__(256) stack_sum_kernel(const StackJobs J, const float* __restrict__ Y, int64_t V_ext,
                                                        int64_t V, int64_t plane, float* __restrict__ g) {
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= V) return;
    double s = 0.0;
    bool over = false;
#pragma unroll
    for (int c = 0; c < MAX_JOBS; ++c) {
        if (c >= J.n) break;
        s += (double)__ldg(Y + (int64_t)c * V_ext + v + J.off[c] * plane);
        over = over || J.first[c];
        if (c + 1 == J.n || J.col[c + 1] != J.col[c]) {
            float* o = g + (int64_t)J.col[c] * V + v;
            *o = (float)(over ? s : s + (double)*o);
            s = 0.0;
            over = false;
        }
    }
}

template <class F>
fft_status for_each_pass(fft_geom g, int n, F&& pass) {
    for (size_t k = 0; k < g->stk.size(); ++k) {
        StackClass& C = g->stk[k];
        const int ns = (int)C.off.size();
        const int64_t jobs = (int64_t)n * ns;
        for (int64_t j0 = 0; j0 < jobs;) {
            StackJobs J;
            J.n = pass_columns(C.sub, jobs - j0);
            for (int c = 0; c < J.n; ++c) {
                const int s = (int)((j0 + c) % ns);
                J.col[c] = (int32_t)((j0 + c) / ns);
                J.off[c] = C.off[s];
                J.rows[c] = g->stk_rows + C.row0 + (int64_t)s * C.sub->M;
                J.first[c] = k == 0 && s == 0;
            }
            fft_status rc = pass(C.sub, J);
            if (rc != FFT_OK) return rc;
            j0 += J.n;
        }
    }
    return FFT_OK;
}

}  // namespace

// Cost of a pass over jobs columns in single-column passes (slices3d, J^T: the single-, four- and
// eight-column kernels take 25.6, 32.5 and 38.9 ms over the same rows; a 96-element ring, J and J^T, 0.147, 0.182,
// 0.217 and 0.141, 0.160, 0.196 ms, with three bands off one plane 0.57, 0.83, 1.00 and 0.56, 0.71, 0.86 ms).
double pass_cost(int64_t jobs, bool col8) {
    double cost = 0.0;
    for (; jobs > 0;) {
        const int64_t n = (jobs > 4 && col8) ? std::min<int64_t>(jobs, 8) : std::min<int64_t>(jobs, 4);
        cost += n > 4 ? 1.52 : (n > 1 ? 1.27 : 1.0);
        jobs -= n;
    }
    return cost;
}

// Groups the slices of an acquisition into classes (host only). Every row has to lie in one plane z
// and every slice of a class to hold the same pairs (equal x and y of both transducers) and bands in the
// same order. Returns no class where that does not hold, or where it would not pay.
bool find_stack(const double* tx, const int32_t* rows, int64_t M, const int32_t* band, const fft_grid& gr,
                std::vector<StackPlan>& plan) {
    plan.clear();
    std::map<double, int> slice_of_z;
    std::vector<std::vector<int32_t>> slice;   // rows of each slice, ascending
    double last_z = 0.0;
    int last = -1;
    for (int64_t p = 0; p < M; ++p) {
        const double z = tx[3 * (int64_t)rows[2 * p] + 2];
        if (!(z == tx[3 * (int64_t)rows[2 * p + 1] + 2])) return false;
        if (last < 0 || z != last_z) {
            const auto at = slice_of_z.emplace(z, (int)slice.size());
            if (at.second) {
                if (slice.size() == STACK_MAX_SLICES) return false;
                slice.emplace_back();
            }
            last = at.first->second;
            last_z = z;
        }
        slice[last].push_back((int32_t)p);
    }
    if (slice.size() < 2) return false;
    auto same_rows = [&](const std::vector<int32_t>& a, const std::vector<int32_t>& b) {
        if (a.size() != b.size()) return false;
        for (size_t i = 0; i < a.size(); ++i) {
            if (band && band[a[i]] != band[b[i]]) return false;
            for (int e = 0; e < 2; ++e) {
                const double* u = tx + 3 * (int64_t)rows[2 * (int64_t)a[i] + e];
                const double* v = tx + 3 * (int64_t)rows[2 * (int64_t)b[i] + e];
                if (u[0] != v[0] || u[1] != v[1]) return false;
            }
        }
        return true;
    };
    for (const auto& zs : slice_of_z) {   // ascending z: a class's first slice is its lowest
        bool placed = false;
        for (StackPlan& c : plan) {
            const double k = (zs.first - c.z) / gr.h, kr = nearbyint(k);
            if (!(fabs(k - kr) <= 1e-9) || kr > 3.0 * gr.nz || !same_rows(c.rows[0], slice[zs.second])) continue;
            c.shift.push_back((int32_t)kr);
            c.rows.push_back(slice[zs.second]);
            placed = true;
            break;
        }
        if (placed) continue;
        if (2 * (plan.size() + 1) > slice.size() || plan.size() == STACK_MAX_CLASSES) {
            plan.clear();
            return false;
        }
        StackPlan c;
        c.z = zs.first;
        c.shift.push_back(0);
        c.rows.push_back(slice[zs.second]);
        plan.push_back(std::move(c));
    }
    return true;
}

// Expected cost of the classes' passes against one pass over all rows (1.0), before anything is
// built: a class's pass costs its share of the rows, half where its plane mirrors the lattice, and a
// sixth more for the layers of an extended grid that a slice at the edge does not need.
double stack_cost(const std::vector<StackPlan>& plan, int64_t M, const fft_grid& gr) {
    double cost = 0.0;
    for (const StackPlan& c : plan) {
        const double k = 2.0 * (c.z - gr.origin[2]) / gr.h;
        const bool mirrors = fabs(k - nearbyint(k)) <= 1e-9;
        const double share = (double)c.rows[0].size() / (double)M;
        cost += pass_cost((int64_t)c.rows.size(), true) * share * (mirrors ? 0.5 : 1.0) * (7.0 / 6.0);
    }
    return cost;
}

// One J or J^T of n columns in entries evaluated (the measure that decides between the two ways).
double stack_entries(fft_geom g, int64_t n) {
    double c = 0.0;
    for (const StackClass& k : g->stk)
        c += pass_cost(n * (int64_t)k.off.size(), k.sub->batch_cols == 8) * (double)k.sub->E_used;
    return c;
}

fft_status stack_J(fft_geom g, const float* m, int n, float* d, cudaStream_t st) {
    if (g->unusable) return check_usable(g);
    const int64_t plane = (int64_t)g->grid.nx * g->grid.ny;
    return for_each_pass(g, n, [&](fft_geom sub, const StackJobs& J) -> fft_status {
        stack_models_kernel<<<dim3((unsigned)ceil_div(sub->V, 256), J.n), 256, 0, st>>>(J, m, g->V, plane, sub->V,
                                                                                         g->stk_x);
        FFT_CUDA(cudaGetLastError());
        const fft_status rc = launch_J_batch(sub, g->stk_x, J.n, g->stk_d, st);
        if (rc != FFT_OK) return rc;
        stack_scatter_kernel<<<dim3((unsigned)ceil_div(sub->M, 256), J.n), 256, 0, st>>>(J, g->stk_d, sub->M, g->M, d);
        FFT_CUDA(cudaGetLastError());
        return FFT_OK;
    });
}

fft_status stack_JT(fft_geom g, const float* d, int n, float* gout, cudaStream_t st) {
    if (g->unusable) return check_usable(g);
    const int64_t plane = (int64_t)g->grid.nx * g->grid.ny;
    return for_each_pass(g, n, [&](fft_geom sub, const StackJobs& J) -> fft_status {
        stack_gather_kernel<<<dim3((unsigned)ceil_div(sub->M, 256), J.n), 256, 0, st>>>(J, d, g->M, sub->M, g->stk_d);
        FFT_CUDA(cudaGetLastError());
        const fft_status rc = launch_JT_batch(sub, g->stk_d, J.n, g->stk_x, st);
        if (rc != FFT_OK) return rc;
        stack_sum_kernel<<<(unsigned)ceil_div(g->V, 256), 256, 0, st>>>(J, g->stk_x, sub->V, g->V, plane, gout);
        FFT_CUDA(cudaGetLastError());
        return FFT_OK;
    });
}

}  // namespace fftgb
