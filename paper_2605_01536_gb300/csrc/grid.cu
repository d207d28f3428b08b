// Queries on a rectilinear grid with ray reuse (Supp. S3): every cell of one
// (x, y) column shares the +z ray direction and the projected position, so the
// perturbed 2-D edge tests of a triangle do not depend on z, and the crossing test of
// cell k reduces to "the plane lies above z_k".  That test is monotone in z_k
// (n.(a - q) changes sign once along the column; the perturbation decides the tie the
// same way at every point), so a binary search over the sorted z coordinates with the
// exact per-point predicate finds the first cell the triangle no longer counts for,
// k_T.  Then chi(z_k) = sum over the column's triangles with k < k_T of sign(n_z).
// Every decision is taken by the same predicate call the per-query traversal makes at
// the same point, so the result is bit-identical to it.
//
// The triangles are rasterised onto the columns instead of walking the tree for every
// column: each triangle finds the columns inside its xy box by searching the sorted
// axes (the same candidates a column's walk reaches) and adds its sign at cell
// k_T - 1 of a column's difference array; a suffix sum up the column gives the counts.
// The triangles stream through once (48 bytes each) and thousands of columns' serial
// walks become independent (triangle, column) tests: 256 x 240 columns of a closed
// 655k-triangle mesh 776 us -> 97 us, 60^2 columns of a rough field 5.6 ms -> 62 us.  Bound by memory: the difference array is cleared,
// read once and replaced by the outputs.
#include <algorithm>

#include "gwn_internal.cuh"
#include "predicates.cuh"

namespace gwn {

namespace {

constexpr int kRasterThreads = 128;
// A triangle over more columns than this is left to k_grid_big, where 8 blocks share
// its columns, so that no warp works through one alone.
constexpr int kRasterMax = 1024;

// first index with a[i] >= v (strict = false) or a[i] > v (strict = true)
__device__ __forceinline__ int axis_bound(const float *__restrict__ a, int n, float v, bool strict) {
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        const float t = __ldg(a + mid);
        if (t < v || (strict && t == v)) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// One (triangle, column) test: the triangle's sign at the last cell it counts for.
__device__ __forceinline__ void raster_test(const GridDev &g, float3 a, float3 b, float3 c, int si, int sj,
                                            int32_t *__restrict__ diff, LocalCount ce, LocalCount cp) {
    const float px = __ldg(g.xs + si), py = __ldg(g.ys + sj);
    const int s0 = edge_sos(px, py, a.x, a.y, b.x, b.y, ce);
    const int s1 = edge_sos(px, py, b.x, b.y, c.x, c.y, ce);
    if (s0 == 0 || s0 != s1) return;
    const int s2 = edge_sos(px, py, c.x, c.y, a.x, a.y, ce);
    if (s2 != s0) return;
    // first cell the triangle does not count for: counts(k) is true, then false
    const float zmax = fmaxf(a.z, fmaxf(b.z, c.z));
    int lo = 0, hi = g.nz;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        const float z = __ldg(g.z + mid);
        const bool counts = z < zmax && plane_sos(make_float3(px, py, z), a, b, c, s0, cp) == s0;
        if (counts) lo = mid + 1;
        else hi = mid;
    }
    if (lo == 0) return;
    const int64_t col = (int64_t)__ldg(g.yi + sj) * g.nx + __ldg(g.xi + si);
    atomicAdd(&diff[(int64_t)(lo - 1) * g.nx * g.ny + col], s0);
}

// 32 triangles per warp; their candidate columns are dealt out to the lanes in one
// sequence, so that lanes stay busy whatever each triangle covers.
__global__ void __launch_bounds__(kRasterThreads) k_grid_raster(GridDev g, const float4 *__restrict__ tri, int64_t nt,
                                                                int32_t *__restrict__ diff, int32_t *__restrict__ big,
                                                                unsigned *__restrict__ n_big,
                                                                unsigned long long *__restrict__ counters) {
    __shared__ float s_t[kRasterThreads][9];
    __shared__ int s_r[kRasterThreads][4];   // first column and row of the range, its width, and pairs before
    const int lane = threadIdx.x & 31, w0 = threadIdx.x & ~31;
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int count = 0;
    if (t < nt) {
        const float4 a = __ldg(tri + 3 * t), b = __ldg(tri + 3 * t + 1), c = __ldg(tri + 3 * t + 2);
        if (__ldg(g.z) < fmaxf(a.z, fmaxf(b.z, c.z))) {   // else at or below every cell
            const int i0 = axis_bound(g.xs, g.nx, fminf(a.x, fminf(b.x, c.x)), false),
                      i1 = axis_bound(g.xs, g.nx, fmaxf(a.x, fmaxf(b.x, c.x)), true);
            if (i0 < i1) {
                const int j0 = axis_bound(g.ys, g.ny, fminf(a.y, fminf(b.y, c.y)), false),
                          j1 = axis_bound(g.ys, g.ny, fmaxf(a.y, fmaxf(b.y, c.y)), true);
                const int64_t n = (int64_t)(i1 - i0) * (j1 - j0);
                if (n > kRasterMax) {
                    big[atomicAdd(n_big, 1u)] = (int32_t)t;
                } else if (n > 0) {
                    count = (int)n;
                    float *T = s_t[threadIdx.x];
                    T[0] = a.x; T[1] = a.y; T[2] = a.z; T[3] = b.x; T[4] = b.y; T[5] = b.z; T[6] = c.x; T[7] = c.y; T[8] = c.z;
                    s_r[threadIdx.x][0] = i0;
                    s_r[threadIdx.x][1] = j0;
                    s_r[threadIdx.x][2] = i1 - i0;
                }
            }
        }
    }
    int incl = count;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    s_r[threadIdx.x][3] = incl - count;
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    __syncwarp();
    unsigned ce = 0, cp = 0;   // exact decisions
    for (int p = lane; p < total; p += 32) {
        int o = 0;   // the last triangle of the warp with at most p pairs before it
#pragma unroll
        for (int step = 16; step > 0; step >>= 1)
            if (s_r[w0 + o + step][3] <= p) o += step;
        const int *r = s_r[w0 + o];
        const float *T = s_t[w0 + o];
        const int q = p - r[3];
        raster_test(g, make_float3(T[0], T[1], T[2]), make_float3(T[3], T[4], T[5]), make_float3(T[6], T[7], T[8]),
                    r[0] + q % r[2], r[1] + q / r[2], diff, LocalCount{&ce}, LocalCount{&cp});
    }
    __syncwarp();
    flush_count(ce, &counters[CNT_EXACT_EDGE]);
    flush_count(cp, &counters[CNT_EXACT_PLANE]);
}

// The listed triangles: blocks (b, y) share triangle b's columns.
__global__ void __launch_bounds__(256) k_grid_big(GridDev g, const float4 *__restrict__ tri, const int32_t *__restrict__ big,
                                                  const unsigned *__restrict__ n_big, int32_t *__restrict__ diff,
                                                  unsigned long long *__restrict__ counters) {
    const unsigned n = *n_big;
    unsigned ce = 0, cp = 0;   // exact decisions
    for (unsigned k = blockIdx.x; k < n; k += gridDim.x) {
        const int64_t t = big[k];
        const float4 A = __ldg(tri + 3 * t), B = __ldg(tri + 3 * t + 1), C = __ldg(tri + 3 * t + 2);
        const float3 a = make_float3(A.x, A.y, A.z), b = make_float3(B.x, B.y, B.z), c = make_float3(C.x, C.y, C.z);
        const int i0 = axis_bound(g.xs, g.nx, fminf(a.x, fminf(b.x, c.x)), false),
                  w = axis_bound(g.xs, g.nx, fmaxf(a.x, fmaxf(b.x, c.x)), true) - i0,
                  j0 = axis_bound(g.ys, g.ny, fminf(a.y, fminf(b.y, c.y)), false),
                  h = axis_bound(g.ys, g.ny, fmaxf(a.y, fmaxf(b.y, c.y)), true) - j0;
        const int64_t cols = (int64_t)w * h;
        for (int64_t q = (int64_t)blockIdx.y * blockDim.x + threadIdx.x; q < cols; q += (int64_t)gridDim.y * blockDim.x)
            raster_test(g, a, b, c, i0 + (int)(q % w), j0 + (int)(q / w), diff, LocalCount{&ce}, LocalCount{&cp});
    }
    __syncwarp();
    flush_count(ce, &counters[CNT_EXACT_EDGE]);
    flush_count(cp, &counters[CNT_EXACT_PLANE]);
}

// Suffix sum up every column (one thread each, neighbouring columns in a warp): chi in
// place, or for a closed mesh (w = chi) the outputs w and label in its stead.
template <bool Outputs>
__global__ void __launch_bounds__(128) k_grid_sum(int32_t *__restrict__ chi, int64_t plane, int nz, float *__restrict__ w,
                                                  uint8_t *__restrict__ label) {
    const int64_t col = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (col >= plane) return;
    constexpr int U = 16;   // loads in flight
    int c = 0;
    for (int k1 = nz; k1 > 0; k1 -= U) {
        int v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) v[u] = k1 - 1 - u >= 0 ? chi[(int64_t)(k1 - 1 - u) * plane + col] : 0;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (k1 - 1 - u < 0) break;
            const int64_t o = (int64_t)(k1 - 1 - u) * plane + col;
            c += v[u];
            if (Outputs) {
                if (w) w[o] = (float)c;
                label[o] = c > 0 ? 1 : 0;
            } else {
                chi[o] = c;
            }
        }
    }
}

// Materialise the grid points ([(k ny + j) nx + i][3]) for the per-point kernels.
__global__ void k_grid_points(const float *__restrict__ gx, int nx, const float *__restrict__ gy, int ny,
                              const float *__restrict__ gz, int64_t n, float *__restrict__ pts) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n) return;
    const int i = (int)(c % nx);
    const int64_t r = c / nx;
    const int j = (int)(r % ny), k = (int)(r / ny);
    pts[3 * c] = gx[i];
    pts[3 * c + 1] = gy[j];
    pts[3 * c + 2] = gz[k];
}

}  // namespace

// The difference array of every column (chi: [nz][ny][nx], overwritten).
static gwn_status grid_diff(const gwn_mesh *m, const GridDev &g, int32_t *chi, cudaStream_t s) {
    const int64_t n = (int64_t)g.nx * g.ny * g.nz;
    int32_t *big = nullptr;
    unsigned *n_big = nullptr;
    GWN_CUDA_TRY(cudaMemsetAsync(chi, 0, sizeof(int32_t) * n, s));
    if (m->nt == 0) return GWN_OK;
    GWN_CUDA_TRY(dev_alloc(&big, sizeof(int32_t) * m->nt, s));
    GWN_CUDA_TRY(dev_alloc(&n_big, sizeof(unsigned), s));
    GWN_CUDA_TRY(cudaMemsetAsync(n_big, 0, sizeof(unsigned), s));
    k_grid_raster<<<grid_for(m->nt, kRasterThreads), kRasterThreads, 0, s>>>(g, m->leaf_tri, m->nt, chi, big, n_big,
                                                                            m->counters);
    k_grid_big<<<dim3(608, 8), 256, 0, s>>>(g, m->leaf_tri, big, n_big, chi, m->counters);
    note_launches(2);
    cudaFreeAsync(big, s);
    cudaFreeAsync(n_big, s);
    GWN_LAUNCH_CHECK("k_grid_raster");
    return GWN_OK;
}

// chi of every cell of the grid (gz non-decreasing).
gwn_status launch_grid_chi(const gwn_mesh *m, const GridDev &g, int32_t *chi, cudaStream_t s) {
    const int64_t plane = (int64_t)g.nx * g.ny;
    if (plane == 0 || g.nz == 0) return GWN_OK;
    ProfScope prof("grid_chi", s);
    gwn_status st = grid_diff(m, g, chi, s);
    if (st != GWN_OK) return st;
    k_grid_sum<false><<<grid_for(plane, 128), 128, 0, s>>>(chi, plane, g.nz, nullptr, nullptr);
    note_launches(1);
    GWN_LAUNCH_CHECK("k_grid_sum");
    return GWN_OK;
}

// Labels (and w) of every cell: chi by ray reuse, then the boundary sum and the
// FP64 re-evaluation near 1/2 on the materialised grid points (a closed mesh
// needs neither: w = chi).
gwn_status launch_classify_grid(const gwn_mesh *m, const GridDev &g, uint8_t *label, float *w, cudaStream_t s) {
    const int64_t plane = (int64_t)g.nx * g.ny, n = plane * g.nz;
    if (n == 0) return GWN_OK;
    int32_t *chi = nullptr;
    GWN_CUDA_TRY(dev_alloc(&chi, sizeof(int32_t) * n, s));
    gwn_status st = GWN_OK;
    if (m->npts < 2) {
        ProfScope prof("grid_chi", s);
        if ((st = grid_diff(m, g, chi, s)) == GWN_OK)
            k_grid_sum<true><<<grid_for(plane, 128), 128, 0, s>>>(chi, plane, g.nz, w, label);
        note_launches(1);
    } else if ((st = launch_grid_chi(m, g, chi, s)) == GWN_OK) {
        float *pts = nullptr, *wt = w;
        int32_t *list = nullptr;
        unsigned long long *len = nullptr;
        if ((st = [&]() -> gwn_status {
                 GWN_CUDA_TRY(dev_alloc(&pts, sizeof(float) * 3 * n, s));
                 GWN_CUDA_TRY(dev_alloc(&list, sizeof(int32_t) * n, s));
                 GWN_CUDA_TRY(dev_alloc(&len, sizeof(unsigned long long), s));
                 if (!wt) GWN_CUDA_TRY(dev_alloc(&wt, sizeof(float) * n, s));
                 return GWN_OK;
             }()) == GWN_OK) {
            cudaMemsetAsync(len, 0, sizeof(unsigned long long), s);
            k_grid_points<<<grid_for(n, 256), 256, 0, s>>>(g.x, g.nx, g.y, g.ny, g.z, n, pts);
            if ((st = launch_boundary_sum_list(m, pts, n, chi, wt, label, true, list, len, SumOrder::kCaller, s)) == GWN_OK)
                st = launch_fp64_fix_list(m, pts, chi, wt, label, list, len, s);
        }
        for (void *p : {(void *)pts, (void *)list, (void *)len}) if (p) cudaFreeAsync(p, s);
        if (wt && wt != w) cudaFreeAsync(wt, s);
    }
    cudaFreeAsync(chi, s);
    if (st != GWN_OK) return st;
    GWN_LAUNCH_CHECK("classify grid");
    return GWN_OK;
}

}  // namespace gwn
