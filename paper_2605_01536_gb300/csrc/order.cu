// Spatial order of a query batch.  The crossing count walks the BVH once per
// query, the boundary hierarchy's walk takes the union over a warp, and the boundary
// kernel decides per warp and boundary tile whether its cancellation test is
// needed; all do best when the queries of a warp lie close together.  Large batches are
// therefore evaluated cell by cell along a Hilbert curve over the mesh's box (a counting
// sort), and the results are scattered back to the caller's order.  Places come from
// atomics: the order inside a cell, and which queries share a warp, differ from run to
// run.  Each query's arithmetic does not depend on its neighbours, so no result does.
// Lists of queries and the queries of many meshes (within each mesh's range) are
// put in the order of their Hilbert keys by the build's radix sort, which is stable.
#include <algorithm>

#include "farfield.cuh"
#include "gwn_internal.cuh"

namespace gwn {

namespace {

constexpr int TB = 256;

// Radix-sorted keys of 24 bits (256 cells per axis of the box's cube): as coherent for a
// warp as 30 and one pass fewer.
constexpr int kOrderBits = 24;

// Hilbert key of p in the cube at the low corner of box = (min x, min y, min z,
// max x, max y, max z) with the box's longest side; points outside are clamped
// onto it (NaN coordinates count as the minimum).  The Hilbert order has no jumps
// (Morton order does), so the 64 queries of a warp stay closer together: 10% fewer
// hierarchy nodes per warp of the boundary sum.
__device__ __forceinline__ uint32_t order_key(const float *__restrict__ p, const float *__restrict__ box) {
    float ext = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) ext = fmaxf(ext, box[3 + k] - box[k]);
    const float inv = ext > 0.f ? 256.0f / ext : 0.f;
    uint32_t c[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float u = fminf(fmaxf((p[k] - box[k]) * inv, 0.f), 255.f);   // fmaxf(NaN, 0) = 0
        c[k] = (uint32_t)u;
    }
    return hilbert_key(c[0], c[1], c[2], 8);
}

// The order is a counting sort over the cells of the curve: only neighbourhood matters,
// so neither the order inside a cell nor the curve's global order has to be kept, and
// three kernels do it (a radix sort on 24 bits took 17 launches: 50k queries 110 ->
// 23 us, 2M queries 202 -> 103 us).  About one cell per query, at most 128^3.
__host__ __device__ __forceinline__ int cell_bits(int64_t n) {
    int b = 3;
    while (b < 7 && (int64_t(1) << (3 * b + 2)) <= n) ++b;
    return b;
}
constexpr int kCellChunk = 4096;   // cells a block of k_cell_offsets lays out

// cell of p on the curve with 2^bits cells per axis
__device__ __forceinline__ uint32_t order_cell(const float *__restrict__ p, const float *__restrict__ box, int bits) {
    float ext = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) ext = fmaxf(ext, box[3 + k] - box[k]);
    const float top = (float)((1 << bits) - 1), inv = ext > 0.f ? (float)(1 << bits) / ext : 0.f;
    uint32_t c[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) c[k] = (uint32_t)fminf(fmaxf((p[k] - box[k]) * inv, 0.f), top);   // fmaxf(NaN, 0) = 0
    return hilbert_key(c[0], c[1], c[2], bits);
}

// count[cell] and each query's rank in its cell; one atomic per cell and warp
__global__ void k_cell_count(const float *__restrict__ q, int64_t n, const float *__restrict__ box, int bits,
                             uint32_t *__restrict__ count, uint32_t *__restrict__ rank) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t cell = i < n ? order_cell(q + 3 * i, box, bits) : 0xffffffffu;
    const unsigned peers = __match_any_sync(0xffffffffu, cell);
    const int lane = threadIdx.x & 31, lead = __ffs(peers) - 1;
    uint32_t first = 0;
    if (lane == lead && i < n) first = atomicAdd(&count[cell], (uint32_t)__popc(peers));
    first = __shfl_sync(0xffffffffu, first, lead);
    if (i < n) rank[i] = first + __popc(peers & ((1u << lane) - 1u));
}

// count -> first place, in place: an exclusive scan over the block's cells from a base
// taken from the cursor (count[ncells]), so blocks need not wait for one another
__global__ void __launch_bounds__(256) k_cell_offsets(uint32_t *__restrict__ count, int64_t ncells) {
    __shared__ uint32_t s_warp[8], s_base;
    constexpr int kPer = kCellChunk / 256;
    const int64_t base = (int64_t)blockIdx.x * kCellChunk + (int64_t)threadIdx.x * kPer;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t v[kPer], sum = 0;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        v[k] = base + k < ncells ? count[base + k] : 0u;
        sum += v[k];
    }
    uint32_t x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t t = 0;
        for (int w = 0; w < 8; ++w) {
            const uint32_t c = s_warp[w];
            s_warp[w] = t;
            t += c;
        }
        s_base = atomicAdd(&count[ncells], t);
    }
    __syncthreads();
    uint32_t run = s_base + s_warp[warp] + x - sum;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        if (base + k < ncells) count[base + k] = run;
        run += v[k];
    }
}

__global__ void k_cell_place(const float *__restrict__ q, int64_t n, const float *__restrict__ box, int bits,
                             const uint32_t *__restrict__ first, const uint32_t *__restrict__ rank,
                             uint32_t *__restrict__ perm, float *__restrict__ qs) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float p[3] = {q[3 * i], q[3 * i + 1], q[3 * i + 2]};
    const int64_t o = (int64_t)first[order_cell(p, box, bits)] + rank[i];
    perm[o] = (uint32_t)i;
    qs[3 * o] = p[0];
    qs[3 * o + 1] = p[1];
    qs[3 * o + 2] = p[2];
}

// Batch key of query i: its mesh index (found in the meshes' query offsets)
// above the Hilbert key in that mesh's box, so that the sort keeps every mesh's
// queries together and orders each range in space.
__global__ void k_batch_keys(const float *__restrict__ q, int64_t n, const int64_t *__restrict__ mesh_off,
                             int n_mesh, const BatchMesh *__restrict__ meshes, uint64_t *__restrict__ keys,
                             uint32_t *__restrict__ ids) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int lo = 0, hi = n_mesh - 1;   // mesh_off[lo] <= i < mesh_off[lo + 1]
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (mesh_off[mid] <= i) lo = mid;
        else hi = mid - 1;
    }
    keys[i] = (uint64_t)lo << kOrderBits | order_key(q + 3 * i, meshes[lo].box);
    ids[i] = (uint32_t)i;
}

// keys of listed queries (list: indices into q)
__global__ void k_list_keys(const float *__restrict__ q, const int32_t *__restrict__ list, int64_t n,
                              const float *__restrict__ box, uint32_t *__restrict__ keys) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    keys[i] = order_key(q + 3 * (int64_t)list[i], box);
}

__global__ void k_gather_queries(const float *__restrict__ q, const uint32_t *__restrict__ perm, int64_t n,
                                 float *__restrict__ qs) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int64_t j = perm[i];
    qs[3 * i] = q[3 * j];
    qs[3 * i + 1] = q[3 * j + 1];
    qs[3 * i + 2] = q[3 * j + 2];
}

template <class T>
__global__ void k_scatter(const T *__restrict__ in, const uint32_t *__restrict__ perm, int64_t n, T *__restrict__ out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[perm[i]] = in[i];
}

// out[perm[i]] = in[i] for each given pair (all may be NULL but perm)
__global__ void k_scatter_results(const uint32_t *__restrict__ perm, int64_t n, const float *__restrict__ ws,
                                  float *__restrict__ w, const int32_t *__restrict__ cs, int32_t *__restrict__ chi,
                                  const uint8_t *__restrict__ ls, uint8_t *__restrict__ label) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint32_t o = perm[i];
    if (w) w[o] = ws[i];
    if (chi) chi[o] = cs[i];
    if (label) label[o] = ls[i];
}

__global__ void k_gather_i32_perm(const int32_t *__restrict__ in, const uint32_t *__restrict__ perm, int64_t n,
                                  int32_t *__restrict__ out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = in[perm[i]];
}

__global__ void k_map_list(int32_t *__restrict__ list, const unsigned long long *__restrict__ len,
                           const uint32_t *__restrict__ perm) {
    const unsigned long long n = *len;
    for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * blockDim.x)
        list[i] = (int32_t)perm[list[i]];
}

}  // namespace

gwn_status gather_i32(const int32_t *in, const uint32_t *perm, int64_t n, int32_t *out, cudaStream_t s) {
    if (n <= 0) return GWN_OK;
    k_gather_i32_perm<<<grid_for(n, TB), TB, 0, s>>>(in, perm, n, out);
    GWN_LAUNCH_CHECK("gather");
    return GWN_OK;
}

gwn_status map_list(int32_t *list, const unsigned long long *len, int64_t n, const uint32_t *perm, cudaStream_t s) {
    if (n <= 0) return GWN_OK;
    k_map_list<<<std::min<unsigned>(grid_for(n, TB), 304), TB, 0, s>>>(list, len, perm);
    GWN_LAUNCH_CHECK("list map");
    return GWN_OK;
}

size_t order_cells_bytes(int64_t n) { return sizeof(uint32_t) * ((size_t(1) << (3 * cell_bits(n))) + 1); }

gwn_status order_queries_on(const gwn_mesh *m, const float *q, int64_t n, uint32_t *rank, uint32_t *perm, float *qs,
                            uint32_t *cells, cudaStream_t s) {
    if (n <= 0) return GWN_OK;
    if (n > (int64_t)0x7fffffff) return set_error(GWN_ERR_INVALID_ARG, "too many queries to order");
    ProfScope prof("query_order", s);
    const int bits = cell_bits(n);
    const int64_t ncells = int64_t(1) << (3 * bits);
    GWN_CUDA_TRY(cudaMemsetAsync(cells, 0, sizeof(uint32_t) * (ncells + 1), s));
    k_cell_count<<<grid_for(n, TB), TB, 0, s>>>(q, n, m->box, bits, cells, rank);
    k_cell_offsets<<<grid_for(ncells, kCellChunk), 256, 0, s>>>(cells, ncells);
    k_cell_place<<<grid_for(n, TB), TB, 0, s>>>(q, n, m->box, bits, cells, rank, perm, qs);
    note_launches(3);
    GWN_LAUNCH_CHECK("query order");
    return GWN_OK;
}

gwn_status order_queries(const gwn_mesh *m, const float *q, int64_t n, uint32_t *rank, uint32_t *perm, float *qs,
                         cudaStream_t s) {
    if (n <= 0) return GWN_OK;
    uint32_t *cells = nullptr;
    GWN_CUDA_TRY(dev_alloc(&cells, order_cells_bytes(n), s));
    const gwn_status st = order_queries_on(m, q, n, rank, perm, qs, cells, s);
    cudaFreeAsync(cells, s);
    return st;
}

gwn_status order_query_list(const gwn_mesh *m, const float *q, int32_t *list, int64_t n, cudaStream_t s) {
    if (n < kOrderMinQueries) return GWN_OK;
    if (n > (int64_t)0x7fffffff) return set_error(GWN_ERR_INVALID_ARG, "too many queries to order");
    ProfScope prof("query_order", s);
    uint32_t *keys = nullptr;
    GWN_CUDA_TRY(dev_alloc(&keys, sizeof(uint32_t) * n, s));
    k_list_keys<<<grid_for(n, TB), TB, 0, s>>>(q, list, n, m->box, keys);
    note_launches(1);
    gwn_status st = radix_sort_u32(keys, reinterpret_cast<uint32_t *>(list), n, kOrderBits, s);
    cudaFreeAsync(keys, s);
    if (st != GWN_OK) return st;
    GWN_LAUNCH_CHECK("query list order");
    return GWN_OK;
}

gwn_status order_batch_queries(const float *q, int64_t n, const int64_t *mesh_off, int n_mesh,
                               const BatchMesh *meshes, uint64_t *keys, uint32_t *perm, float *qs, cudaStream_t s) {
    if (n <= 0 || n_mesh <= 0) return GWN_OK;
    if (n > (int64_t)0x7fffffff) return set_error(GWN_ERR_INVALID_ARG, "too many queries to order");
    int mbits = 0;
    while ((1 << mbits) < n_mesh) ++mbits;
    k_batch_keys<<<grid_for(n, TB), TB, 0, s>>>(q, n, mesh_off, n_mesh, meshes, keys, perm);
    gwn_status st = radix_sort_u64(keys, perm, n, kOrderBits + mbits, s);
    if (st != GWN_OK) return st;
    k_gather_queries<<<grid_for(n, TB), TB, 0, s>>>(q, perm, n, qs);
    GWN_LAUNCH_CHECK("batch query order");
    return GWN_OK;
}

gwn_status scatter_f32(const float *in, const uint32_t *perm, int64_t n, float *out, cudaStream_t s) {
    if (n <= 0 || !out) return GWN_OK;
    ProfScope prof("scatter", s);
    k_scatter<float><<<grid_for(n, TB), TB, 0, s>>>(in, perm, n, out);
    GWN_LAUNCH_CHECK("scatter");
    return GWN_OK;
}

gwn_status scatter_i32(const int32_t *in, const uint32_t *perm, int64_t n, int32_t *out, cudaStream_t s) {
    if (n <= 0 || !out) return GWN_OK;
    ProfScope prof("scatter", s);
    k_scatter<int32_t><<<grid_for(n, TB), TB, 0, s>>>(in, perm, n, out);
    GWN_LAUNCH_CHECK("scatter");
    return GWN_OK;
}

gwn_status scatter_results(const uint32_t *perm, int64_t n, const float *ws, float *w, const int32_t *cs, int32_t *chi,
                           const uint8_t *ls, uint8_t *label, cudaStream_t s) {
    if (n <= 0) return GWN_OK;
    ProfScope prof("scatter", s);
    k_scatter_results<<<grid_for(n, TB), TB, 0, s>>>(perm, n, ws, w, cs, chi, ls, label);
    GWN_LAUNCH_CHECK("scatter");
    return GWN_OK;
}

}  // namespace gwn
