// Acceleration build: oriented boundary extraction + chaining, and the LBVH.
//
// Boundary (Sec. 4.1, Eq. 9): the auxiliary triangles of an interior edge cancel
// in pairs, so only the oriented boundary dM contributes.  Treated as a 1-chain:
// every face contributes its three directed edges; an undirected edge {u, v}
// (matched by vertex index) has net multiplicity m = #(u->v) - #(v->u) and
// appears |m| times in its net direction.  Steps: the half-edges are put into a bucket per
// smaller vertex and netted out there, in ascending order of the other vertex (a mesh with
// a vertex of very many half-edges: sort of the 3 nt half-edge keys, segmented sum of the
// signs, compaction).  Edges are then chained into closed
// loops (the boundary of a 2-chain is a cycle: in-degree = out-degree at every
// vertex) so that consecutive edges share their common point in the query
// kernel.
//
// LBVH (replaces the paper's Embree BVH, Sec. 5): 30-bit Morton codes of the
// triangle centroids, radix sort, Karras' binary radix tree (Karras 2012),
// bottom-up box refit, and depth-first escape links for stackless traversal.
#include <algorithm>

#include "farfield.cuh"
#include "gwn_internal.cuh"

namespace gwn {

namespace {

constexpr int TB = 256;

// Blocks of a grid-stride bounds kernel: with one thread per element and atomics per
// warp, the atomics on six addresses took 158 us for 330k vertices (now 5 us).
constexpr unsigned kBoundsBlocks = 304;

__device__ __forceinline__ int ordered_key(float f) {
    int i = __float_as_int(f);
    return i >= 0 ? i : i ^ 0x7fffffff;
}
__device__ __forceinline__ float from_ordered_key(int k) {
    return __int_as_float(k >= 0 ? k : k ^ 0x7fffffff);
}

// Bounds of point(i), i < n, over the block's grid-stride share, merged into bounds
// (6: min xyz, max xyz as ordered ints) with one atomic per bound.
template <class Point>
__device__ __forceinline__ void block_bounds(int64_t n, Point &&point, int *__restrict__ bounds) {
    __shared__ int s_b[8][6];
    int v[6] = {0x7fffffff, 0x7fffffff, 0x7fffffff, (int)0x80000000, (int)0x80000000, (int)0x80000000};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float3 p = point(i);
        const int k[3] = {ordered_key(p.x), ordered_key(p.y), ordered_key(p.z)};
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            v[d] = min(v[d], k[d]);
            v[3 + d] = max(v[3 + d], k[d]);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int d = 0; d < 6; ++d) {
            const int w = __shfl_xor_sync(0xffffffffu, v[d], o);
            v[d] = d < 3 ? min(v[d], w) : max(v[d], w);
        }
    const int warp = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0)
        for (int d = 0; d < 6; ++d) s_b[warp][d] = v[d];
    __syncthreads();
    if (threadIdx.x < 6) {
        const int d = threadIdx.x;
        int r = s_b[0][d];
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) r = d < 3 ? min(r, s_b[w][d]) : max(r, s_b[w][d]);
        if (d < 3) atomicMin(&bounds[d], r);
        else atomicMax(&bounds[d], r);
    }
}

// ------------------------------------------------------------ boundary ----

__global__ void k_halfedge_keys(const int32_t *__restrict__ F, int64_t nt, int64_t nv,
                                uint64_t *__restrict__ keys, uint32_t *__restrict__ vals) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 3 * nt) return;
    int64_t t = i / 3;
    int e = (int)(i % 3);
    int64_t u = F[3 * t + e], v = F[3 * t + (e + 1) % 3];
    int64_t lo = u < v ? u : v, hi = u < v ? v : u;
    // a half-edge from a vertex to itself (repeated index in a degenerate face)
    // is a zero chain and contributes nothing: mark it with sign code 2
    keys[i] = (uint64_t)(lo * nv + hi);
    vals[i] = (u == v) ? 2u : (u < v ? 1u : 0u);
}

__global__ void k_seg_heads(const uint64_t *__restrict__ keys, int64_t n, uint32_t *__restrict__ head) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    head[i] = (i == 0 || keys[i] != keys[i - 1]) ? 1u : 0u;
}

__global__ void k_seg_sum(const uint64_t *__restrict__ keys, const uint32_t *__restrict__ vals,
                          const uint32_t *__restrict__ head, const uint32_t *__restrict__ head_scan,
                          int64_t n, int32_t *__restrict__ mult, uint64_t *__restrict__ seg_key) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint32_t seg = head_scan[i] + head[i] - 1u;
    if (head[i]) seg_key[seg] = keys[i];
    uint32_t v = vals[i];
    if (v != 2u) atomicAdd(&mult[seg], v ? 1 : -1);
}

__global__ void k_abs(const int32_t *__restrict__ mult, int64_t nseg, uint32_t *__restrict__ cnt) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nseg) return;
    int32_t m = mult[i];
    cnt[i] = (uint32_t)(m < 0 ? -m : m);
}

__global__ void k_emit_edges(const int32_t *__restrict__ mult, const uint64_t *__restrict__ seg_key,
                             const uint32_t *__restrict__ off, int64_t nseg, int64_t nv,
                             int32_t *__restrict__ edges) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nseg) return;
    int32_t m = mult[i];
    if (m == 0) return;
    int64_t key = (int64_t)seg_key[i];
    int32_t lo = (int32_t)(key / nv), hi = (int32_t)(key % nv);
    int32_t a = m > 0 ? lo : hi, b = m > 0 ? hi : lo;
    int32_t c = m < 0 ? -m : m;
    for (int32_t r = 0; r < c; ++r) {
        edges[2 * (off[i] + r)] = a;
        edges[2 * (off[i] + r) + 1] = b;
    }
}

// Boundary edges by buckets of the smaller vertex: half-edges are counted and placed
// per vertex (entry: larger vertex << 1 | direction), and each vertex's few entries are
// netted out against one another.  A vertex with more than kBucketMax entries sets *overflow and
// the sort above takes over (one such vertex beside a 642k-triangle mesh, buckets / sort: 200
// entries 1.78 / 1.98 ms for the whole build, 400 entries 2.04 / 1.99, 1,000 entries 3.80 / 2.00;
// alone 0.61 / 0.59, 0.90 / 0.64, 2.86 / 0.85).  A half-edge from a vertex to itself (repeated index in a
// degenerate face) is a zero chain and contributes nothing.
constexpr uint32_t kBucketMax = 128;
__global__ void k_bucket_count(const int32_t *__restrict__ F, int64_t nh, uint32_t *__restrict__ count,
                               uint32_t *__restrict__ rank, uint32_t *__restrict__ overflow) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nh) return;
    const int64_t t = i / 3;
    const int e = (int)(i - 3 * t);
    const int32_t u = F[i], v = F[3 * t + (e == 2 ? 0 : e + 1)];
    if (u == v) return;
    const uint32_t r = atomicAdd(&count[min(u, v)], 1u);
    rank[i] = r;
    if (r >= kBucketMax) *overflow = 1u;
}

__global__ void k_bucket_place(const int32_t *__restrict__ F, int64_t nh, const uint32_t *__restrict__ first,
                               const uint32_t *__restrict__ rank, uint32_t *__restrict__ entry) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nh) return;
    const int64_t t = i / 3;
    const int e = (int)(i - 3 * t);
    const int32_t u = F[i], v = F[3 * t + (e == 2 ? 0 : e + 1)];
    if (u == v) return;
    entry[first[min(u, v)] + rank[i]] = (uint32_t)max(u, v) << 1 | (u < v ? 1u : 0u);
}

// Net multiplicity of entry i's edge if i is its first entry in [b, e), else 0.
__device__ __forceinline__ int bucket_net(const uint32_t *__restrict__ entry, uint32_t b, uint32_t e, uint32_t i) {
    const uint32_t hi = entry[i] >> 1;
    int m = 0;
    for (uint32_t j = b; j < e; ++j) {
        const uint32_t x = entry[j];
        if (x >> 1 != hi) continue;
        if (j < i) return 0;
        m += x & 1u ? 1 : -1;
    }
    return m;
}

// The copies of entry i's edge (net[i] != 0) at their place: after the copies of the vertex's
// edges with a smaller other vertex, which begin at base
__device__ __forceinline__ void bucket_emit(const uint32_t *__restrict__ entry, const int32_t *__restrict__ net, uint32_t b,
                                            uint32_t e, uint32_t i, int32_t v, uint32_t base, int32_t *__restrict__ edges) {
    const int m = net[i];
    if (m == 0) return;
    const int32_t hi = (int32_t)(entry[i] >> 1);
    for (uint32_t j = b; j < e; ++j)
        if ((int32_t)(entry[j] >> 1) < hi) base += (uint32_t)abs(net[j]);
    for (int r = 0; r < abs(m); ++r) {
        edges[2 * (base + r)] = m > 0 ? v : hi;
        edges[2 * (base + r) + 1] = m > 0 ? hi : v;
    }
}

// edges NULL: every entry's net multiplicity into net and each vertex's number of edges
// into out; else the edges themselves, each vertex's from out[v] on in ascending order of
// the other vertex.  A thread per vertex; buckets of more than kBucketSerial entries, whose
// cost goes with the square of their size, are taken by the warp together (one thread and
// nothing kept between the passes: a vertex of 126 unmatched half-edges 55 ms).
constexpr uint32_t kBucketSerial = 16;
__global__ void k_bucket_net(const uint32_t *__restrict__ entry, const uint32_t *__restrict__ first,
                             const uint32_t *__restrict__ count, int64_t nv, int32_t *__restrict__ net,
                             uint32_t *__restrict__ out, int32_t *__restrict__ edges,
                             const uint32_t *__restrict__ overflow) {
    if (*overflow) return;
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31;
    const uint32_t b = v < nv ? first[v] : 0u, e = v < nv ? b + count[v] : 0u;
    uint32_t total = 0;
    if (e - b <= kBucketSerial) {
        for (uint32_t i = b; i < e; ++i) {
            if (edges) {
                bucket_emit(entry, net, b, e, i, (int32_t)v, out[v], edges);
            } else {
                net[i] = bucket_net(entry, b, e, i);
                total += (uint32_t)abs(net[i]);
            }
        }
    }
    for (unsigned big = __ballot_sync(0xffffffffu, e - b > kBucketSerial); big; big &= big - 1) {
        const int src = __ffs(big) - 1;
        const uint32_t wb = __shfl_sync(0xffffffffu, b, src), we = __shfl_sync(0xffffffffu, e, src);
        const int64_t wv = v - lane + src;
        uint32_t sum = 0;
        for (uint32_t i = wb + lane; i < we; i += 32) {
            if (edges) {
                bucket_emit(entry, net, wb, we, i, (int32_t)wv, out[wv], edges);
            } else {
                net[i] = bucket_net(entry, wb, we, i);
                sum += (uint32_t)abs(net[i]);
            }
        }
        sum = __reduce_add_sync(0xffffffffu, sum);
        if (lane == src) total = sum;
    }
    if (!edges && v < nv) out[v] = total;
}

// keys for sorting edges by start (which = 0) or end (which = 1) vertex
__global__ void k_edge_vertex_keys(const int32_t *__restrict__ edges, int64_t nb, int which,
                                   uint32_t *__restrict__ keys, uint32_t *__restrict__ ids) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nb) return;
    keys[i] = (uint32_t)edges[2 * i + which];
    ids[i] = (uint32_t)i;
}

// in-degree = out-degree at every vertex, so the vertex segments of the two
// sorted lists start at the same positions: pair the p-th incoming edge with
// the p-th outgoing edge.
__global__ void k_pair_succ(const uint32_t *__restrict__ in_ids, const uint32_t *__restrict__ out_ids,
                            int64_t nb, uint32_t *__restrict__ succ) {
    int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= nb) return;
    succ[in_ids[p]] = out_ids[p];
}

__global__ void k_init_rep(const uint32_t *__restrict__ succ, int64_t nb, uint32_t *rep, uint32_t *nxt) {
    int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= nb) return;
    rep[e] = (uint32_t)e;
    nxt[e] = succ[e];
}

// one pointer-jumping round of the cycle minimum
__global__ void k_jump_min(const uint32_t *__restrict__ rep_in, const uint32_t *__restrict__ nxt_in, int64_t nb,
                           uint32_t *__restrict__ rep_out, uint32_t *__restrict__ nxt_out) {
    int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= nb) return;
    uint32_t n = nxt_in[e];
    rep_out[e] = min(rep_in[e], rep_in[n]);
    nxt_out[e] = nxt_in[n];
}

// list ranking: cut each cycle in front of its representative
__global__ void k_init_rank(const uint32_t *__restrict__ succ, const uint32_t *__restrict__ rep, int64_t nb,
                            uint32_t *dist, int32_t *nxt) {
    int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= nb) return;
    uint32_t s = succ[e];
    bool last = (s == rep[e]);
    nxt[e] = last ? -1 : (int32_t)s;
    dist[e] = last ? 0u : 1u;
}

__global__ void k_jump_rank(const uint32_t *__restrict__ dist_in, const int32_t *__restrict__ nxt_in, int64_t nb,
                            uint32_t *__restrict__ dist_out, int32_t *__restrict__ nxt_out) {
    int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= nb) return;
    int32_t n = nxt_in[e];
    if (n < 0) {
        dist_out[e] = dist_in[e];
        nxt_out[e] = -1;
    } else {
        dist_out[e] = dist_in[e] + dist_in[n];
        nxt_out[e] = nxt_in[n];
    }
}

// Representative (smallest edge) and rank of every edge of a loop of at most kWalkMax
// edges, by walking it; a longer loop sets *longer and pointer jumping takes over.
constexpr int kWalkMax = 48;
__global__ void k_walk_loops(const uint32_t *__restrict__ succ, int64_t nb, uint32_t *__restrict__ rep,
                             uint32_t *__restrict__ dist, uint32_t *__restrict__ longer) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= nb) return;
    uint32_t at = succ[e], least = (uint32_t)e;
    int len = 1, to_least = 0;   // steps from e to the smallest edge
    while (at != (uint32_t)e && len < kWalkMax) {
        if (at < least) {
            least = at;
            to_least = len;
        }
        at = succ[at];
        ++len;
    }
    if (at != (uint32_t)e) *longer = 1u;
    rep[e] = least;
    dist[e] = (uint32_t)((to_least == 0 ? len : to_least) - 1);
}

// Pointer jumping of k_jump_min and k_jump_rank in one block, for few edges
__global__ void __launch_bounds__(1024) k_jump_small(const uint32_t *__restrict__ succ, int nb, int rounds, uint32_t *rep0,
                                                     uint32_t *rep1, uint32_t *nx0, uint32_t *nx1, uint32_t *dist0,
                                                     uint32_t *dist1, int32_t *rn0, int32_t *rn1) {
    for (int e = threadIdx.x; e < nb; e += blockDim.x) {
        rep0[e] = (uint32_t)e;
        nx0[e] = succ[e];
    }
    for (int r = 0; r < rounds; ++r) {
        __syncthreads();
        const uint32_t *ri = r & 1 ? rep1 : rep0, *ni = r & 1 ? nx1 : nx0;
        uint32_t *ro = r & 1 ? rep0 : rep1, *no = r & 1 ? nx0 : nx1;
        for (int e = threadIdx.x; e < nb; e += blockDim.x) {
            const uint32_t n = ni[e];
            ro[e] = min(ri[e], ri[n]);
            no[e] = ni[n];
        }
    }
    __syncthreads();
    const uint32_t *rep = rounds & 1 ? rep1 : rep0;
    for (int e = threadIdx.x; e < nb; e += blockDim.x) {
        const bool last = succ[e] == rep[e];
        rn0[e] = last ? -1 : (int32_t)succ[e];
        dist0[e] = last ? 0u : 1u;
    }
    for (int r = 0; r < rounds; ++r) {
        __syncthreads();
        const uint32_t *di = r & 1 ? dist1 : dist0;
        uint32_t *dt = r & 1 ? dist0 : dist1;
        const int32_t *ni = r & 1 ? rn1 : rn0;
        int32_t *no = r & 1 ? rn0 : rn1;
        for (int e = threadIdx.x; e < nb; e += blockDim.x) {
            const int32_t n = ni[e];
            dt[e] = n < 0 ? di[e] : di[e] + di[n];
            no[e] = n < 0 ? -1 : ni[n];
        }
    }
}
// Edges k_jump_small takes.  Build of a rim, one block / a launch per round: 100 edges 500 / 565
// us, 4,000 970 / 1057, 16,000 1173 / 1200, 17,000 1228 / 1229, 60,000 2059 / 1517.
constexpr int64_t kJumpSmall = 16384;

// points per loop (length + 1 closing point), stored at the representative
__global__ void k_loop_sizes(const uint32_t *__restrict__ rep, const uint32_t *__restrict__ dist, int64_t nb,
                             uint32_t *__restrict__ size) {
    int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= nb) return;
    size[e] = (rep[e] == (uint32_t)e) ? dist[e] + 2u : 0u;   // dist at the head = length - 1
}

__global__ void k_emit_chained(const int32_t *__restrict__ edges, const uint32_t *__restrict__ rep,
                               const uint32_t *__restrict__ dist, const uint32_t *__restrict__ loop_off,
                               const float4 *__restrict__ V, int64_t nb, int64_t npts,
                               float4 *__restrict__ pts, uint2 *__restrict__ ends) {
    int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= nb) return;
    uint32_t r = rep[e];
    if (r >= nb) return;
    uint32_t len = dist[r] + 1u;
    uint32_t pos = len - 1u - dist[e];
    uint32_t base = loop_off[r];
    if ((int64_t)base + len >= npts || pos >= len) return;   // never write outside the point array
    float4 p = V[edges[2 * e]];
    p.w = 1.0f;
    pts[base + pos] = p;
    ends[base + pos] = make_uint2(base, base + len);   // the loop's first and closing points
    if (e == (int64_t)r) {   // closing point: back to the loop's first vertex
        float4 c = V[edges[2 * e]];
        c.w = 0.0f;
        pts[base + len] = c;
        ends[base + len] = make_uint2(base, base + len);
    }
}

__global__ void k_emit_unchained(const int32_t *__restrict__ edges, const float4 *__restrict__ V, int64_t nb,
                                 float4 *__restrict__ pts) {
    int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= nb) return;
    float4 a = V[edges[2 * e]], b = V[edges[2 * e + 1]];
    a.w = 1.0f;
    b.w = 0.0f;
    pts[2 * e] = a;
    pts[2 * e + 1] = b;
}

// Loops are laid out in the order of the Morton code (in the box of the
// boundary's points) of their first point, so that a tile of consecutive
// points covers a compact region and the boundary kernel can skip its
// cancellation test for the many queries far from it.

__global__ void k_gather_sizes(const uint32_t *__restrict__ ids, const uint32_t *__restrict__ size, int64_t nb,
                               uint32_t *__restrict__ out) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nb) return;
    out[i] = size[ids[i]];
}

__global__ void k_scatter_offsets(const uint32_t *__restrict__ ids, const uint32_t *__restrict__ off, int64_t nb,
                                  uint32_t *__restrict__ loop_off) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nb) return;
    loop_off[ids[i]] = off[i];
}

// count[0]: loops, count[1]: of them with three edges
__global__ void k_count_heads(const uint32_t *__restrict__ rep, const uint32_t *__restrict__ dist, int64_t nb,
                              unsigned long long *count) {
    int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool head = e < nb && rep[e] == (uint32_t)e;
    const unsigned heads = __ballot_sync(0xffffffffu, head), tris = __ballot_sync(0xffffffffu, head && dist[e] == 2u);
    if ((threadIdx.x & 31) == 0 && heads) {
        atomicAdd(count, (unsigned long long)__popc(heads));
        if (tris) atomicAdd(count + 1, (unsigned long long)__popc(tris));
    }
}

// 1 at the first point of every loop of three edges (ends: per point the first and
// closing point of its loop)
__global__ void k_tri_heads(const uint2 *__restrict__ ends, int64_t npts, uint32_t *__restrict__ head) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= npts) return;
    head[i] = ends[i].x == (uint32_t)i && ends[i].y - ends[i].x == 3u;
}

// Splits the chained points into triangle loops (5 float4 each, TriLoop) and the points
// of the other loops; before: the triangle loops that start before each point (each
// takes four points)
__global__ void k_split_loops(const float4 *__restrict__ pts, const uint2 *__restrict__ ends,
                              const uint32_t *__restrict__ before, int64_t npts, float4 *__restrict__ tri,
                              float4 *__restrict__ rest) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= npts) return;
    if (ends[i].y - ends[i].x != 3u) {
        rest[i - 4 * (int64_t)before[i]] = pts[i];
        return;
    }
    if (ends[i].x != (uint32_t)i) return;
    float4 a = pts[i], b = pts[i + 1], c = pts[i + 2], *T = tri + 5 * (int64_t)before[i];
    const double ux = (double)b.x - a.x, uy = (double)b.y - a.y, uz = (double)b.z - a.z;
    const double vx = (double)c.x - a.x, vy = (double)c.y - a.y, vz = (double)c.z - a.z;
    a.w = fmaxf(a.z, fmaxf(b.z, c.z));
    b.w = c.w = 0.f;
    T[0] = a;
    T[1] = b;
    T[2] = c;
    // the normal as a power of two times a vector of magnitude about 1 (0 if it vanishes)
    const double nx = uy * vz - uz * vy, ny = uz * vx - ux * vz, nz = ux * vy - uy * vx;
    const double top = fmax(fabs(nx), fmax(fabs(ny), fabs(nz)));
    const int e = top > 0.0 ? ilogb(top) : 0;
    T[3] = make_float4((float)scalbn(nx, -e), (float)scalbn(ny, -e), (float)scalbn(nz, -e),
                       top > 0.0 ? (float)scalbn(1.0, e) : 0.f);
    T[4] = make_float4(fminf(a.x, fminf(b.x, c.x)), fmaxf(a.x, fmaxf(b.x, c.x)), fminf(a.y, fminf(b.y, c.y)),
                       fmaxf(a.y, fmaxf(b.y, c.y)));
}

// ------------------------------------------------------------------ BVH ----

__global__ void __launch_bounds__(256) k_centroid_bounds(const float4 *__restrict__ V, const int32_t *__restrict__ F,
                                                         int64_t nt, int *__restrict__ bounds) {
    block_bounds(nt, [&](int64_t t) {
        const float4 a = V[F[3 * t]], b = V[F[3 * t + 1]], d = V[F[3 * t + 2]];
        return make_float3((a.x + b.x + d.x) * (1.0f / 3.0f), (a.y + b.y + d.y) * (1.0f / 3.0f),
                           (a.z + b.z + d.z) * (1.0f / 3.0f));
    }, bounds);
}

__device__ __forceinline__ uint32_t spread10(uint32_t v) {
    v &= 0x3ffu;
    v = (v | (v << 16)) & 0x030000ffu;
    v = (v | (v << 8)) & 0x0300f00fu;
    v = (v | (v << 4)) & 0x030c30c3u;
    v = (v | (v << 2)) & 0x09249249u;
    return v;
}

__device__ __forceinline__ uint32_t morton30(float x, float y, float z, const int *__restrict__ bounds) {
    const float c[3] = {x, y, z};
    uint32_t q[3];
    for (int k = 0; k < 3; ++k) {
        const float lo = from_ordered_key(bounds[k]), hi = from_ordered_key(bounds[3 + k]);
        const float ext = hi - lo;
        float u = ext > 0.f ? (c[k] - lo) / ext : 0.f;
        u = fminf(fmaxf(u, 0.f), 1.f);
        q[k] = min((uint32_t)(u * 1024.0f), 1023u);
    }
    return (spread10(q[0]) << 2) | (spread10(q[1]) << 1) | spread10(q[2]);
}

__global__ void __launch_bounds__(256) k_edge_start_bounds(const int32_t *__restrict__ edges, const float4 *__restrict__ V,
                                                           int64_t nb, int *__restrict__ bounds) {
    block_bounds(nb, [&](int64_t e) {
        const float4 p = V[edges[2 * e]];
        return make_float3(p.x, p.y, p.z);
    }, bounds);
}

// 30-bit Hilbert key in the cube over the bounds
__device__ __forceinline__ uint32_t hilbert30(float x, float y, float z, const int *__restrict__ bounds) {
    const float c[3] = {x, y, z};
    float ext = 0.f;
    for (int k = 0; k < 3; ++k) ext = fmaxf(ext, from_ordered_key(bounds[3 + k]) - from_ordered_key(bounds[k]));
    uint32_t q[3];
    for (int k = 0; k < 3; ++k) {
        const float u = ext > 0.f ? (c[k] - from_ordered_key(bounds[k])) / ext : 0.f;
        q[k] = min((uint32_t)(fminf(fmaxf(u, 0.f), 1.f) * 1024.0f), 1023u);
    }
    return hilbert_key(q[0], q[1], q[2], 10);
}

// key of a loop's representative edge: the Morton code or Hilbert key of its start
// point; every other edge sorts after all loops (bit 30)
__global__ void k_loop_keys(const uint32_t *__restrict__ rep, const int32_t *__restrict__ edges,
                            const float4 *__restrict__ V, int64_t nb, const int *__restrict__ bounds, int hilbert,
                            uint32_t *__restrict__ keys, uint32_t *__restrict__ ids) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= nb) return;
    uint32_t key = 1u << 30;
    if (rep[e] == (uint32_t)e) {
        const float4 p = V[edges[2 * e]];
        key = hilbert ? hilbert30(p.x, p.y, p.z, bounds) : morton30(p.x, p.y, p.z, bounds);
    }
    keys[e] = key;
    ids[e] = (uint32_t)e;
}

__device__ __forceinline__ uint32_t spread15(uint32_t v) {
    v &= 0x7fffu;
    v = (v | (v << 8)) & 0x00ff00ffu;
    v = (v | (v << 4)) & 0x0f0f0f0fu;
    v = (v | (v << 2)) & 0x33333333u;
    v = (v | (v << 1)) & 0x55555555u;
    return v;
}

// 30-bit Morton code of each triangle's centroid in the centroids' box: over x,
// y and z (dims = 3), or over x and y only (dims = 2: a tree of columns, which
// +z rays from neighbouring queries walk alike)
__global__ void k_morton(const float4 *__restrict__ V, const int32_t *__restrict__ F, int64_t nt,
                         const int *__restrict__ bounds, int dims, uint32_t *__restrict__ codes,
                         uint32_t *__restrict__ ids) {
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nt) return;
    float4 a = V[F[3 * t]], b = V[F[3 * t + 1]], d = V[F[3 * t + 2]];
    float c[3] = {(a.x + b.x + d.x) * (1.0f / 3.0f), (a.y + b.y + d.y) * (1.0f / 3.0f),
                  (a.z + b.z + d.z) * (1.0f / 3.0f)};
    const float cells = dims == 2 ? 32768.0f : 1024.0f;
    const uint32_t top = dims == 2 ? 32767u : 1023u;
    uint32_t q[3];
    for (int k = 0; k < 3; ++k) {
        float lo = from_ordered_key(bounds[k]), hi = from_ordered_key(bounds[3 + k]);
        float ext = hi - lo;
        float u = ext > 0.f ? (c[k] - lo) / ext : 0.f;
        u = fminf(fmaxf(u, 0.f), 1.f);
        q[k] = min((uint32_t)(u * cells), top);
    }
    codes[t] = dims == 2 ? (spread15(q[0]) << 1) | spread15(q[1])
                         : (spread10(q[0]) << 2) | (spread10(q[1]) << 1) | spread10(q[2]);
    ids[t] = (uint32_t)t;
}

// Expected node tests of the +z walk from a point uniform in the mesh's vertex box, the
// cost the two candidate trees are compared by: a walk tests the root and both children
// of every internal node it hits, it hits a node iff the point's xy lies in the node's
// box and its z below the top (its ancestors' boxes contain it), and the three are
// independent.  So the expectation is 1 + 2 sum over the internal nodes of (x share)
// (y share) (z share); the sum goes to *cost.  (4,096 sampled walks, serial chains of
// hundreds of loads, took 130 us a tree on soup7 and 530 us on 30,000 random triangles.)
__global__ void __launch_bounds__(256) k_tree_cost(const gwn::BvhNode *__restrict__ nodes, int64_t ninternal,
                                                   const float *__restrict__ box, double *__restrict__ cost) {
    __shared__ double s_c[8];
    const float ex = box[3] - box[0], ey = box[4] - box[1], ez = box[5] - box[2];
    const float ix = ex > 0.f ? 1.f / ex : 0.f, iy = ey > 0.f ? 1.f / ey : 0.f, iz = ez > 0.f ? 1.f / ez : 0.f;
    double c = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < ninternal; i += (int64_t)gridDim.x * blockDim.x) {
        const float4 b0 = __ldg(reinterpret_cast<const float4 *>(nodes + i));
        const float zmax = __ldg(&nodes[i].zmax);
        const float fx = ex > 0.f ? (b0.y - b0.x) * ix : 1.f, fy = ey > 0.f ? (b0.w - b0.z) * iy : 1.f,
                    fz = ez > 0.f ? (zmax - box[2]) * iz : 1.f;
        c += (double)(fx * fy) * fz;
    }
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if ((threadIdx.x & 31) == 0) s_c[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) c += s_c[w];
        atomicAdd(cost, c);
    }
}

__device__ __forceinline__ int delta(const uint32_t *codes, int64_t n, int64_t i, int64_t j) {
    if (j < 0 || j >= n) return -1;
    uint32_t a = codes[i], b = codes[j];
    if (a != b) return __clz(a ^ b);
    return 32 + __clz((uint32_t)i ^ (uint32_t)j);
}

// Karras 2012: internal node i covers leaves [min(i,j), max(i,j)]; its split
// gamma gives children gamma (left) and gamma + 1 (right), leaves when the
// child's range is a single leaf.  Node numbering: internal i -> i, leaf k ->
// (n - 1) + k.
__global__ void k_karras(const uint32_t *__restrict__ codes, int64_t n, int32_t *__restrict__ left,
                         int32_t *__restrict__ right, int32_t *__restrict__ parent, int32_t *__restrict__ first,
                         int32_t *__restrict__ last) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n - 1) return;
    int d = (delta(codes, n, i, i + 1) - delta(codes, n, i, i - 1)) >= 0 ? 1 : -1;
    int dmin = delta(codes, n, i, i - d);
    int64_t lmax = 2;
    while (delta(codes, n, i, i + lmax * d) > dmin) lmax <<= 1;
    int64_t l = 0;
    for (int64_t t = lmax >> 1; t >= 1; t >>= 1)
        if (delta(codes, n, i, i + (l + t) * d) > dmin) l += t;
    int64_t j = i + l * d;
    int dnode = delta(codes, n, i, j);
    int64_t s = 0, div = 2, t;
    do {
        t = (l + div - 1) / div;
        if (delta(codes, n, i, i + (s + t) * d) > dnode) s += t;
        div <<= 1;
    } while (t > 1);
    int64_t gamma = i + s * d + (d < 0 ? -1 : 0);
    int64_t lo = i < j ? i : j, hi = i < j ? j : i;
    int32_t lc = (lo == gamma) ? (int32_t)(n - 1 + gamma) : (int32_t)gamma;
    int32_t rc = (hi == gamma + 1) ? (int32_t)(n - 1 + gamma + 1) : (int32_t)(gamma + 1);
    left[i] = lc;
    right[i] = rc;
    parent[lc] = (int32_t)i;
    parent[rc] = (int32_t)i;
    first[i] = (int32_t)lo;
    last[i] = (int32_t)hi;
}

__global__ void k_leaves(const float4 *__restrict__ V, const int32_t *__restrict__ F, const uint32_t *__restrict__ ids,
                         int64_t n, gwn::BvhNode *__restrict__ nodes, float4 *__restrict__ leaf_tri) {
    int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    int64_t t = ids[k];
    float4 a = V[F[3 * t]], b = V[F[3 * t + 1]], c = V[F[3 * t + 2]];
    a.w = b.w = c.w = 0.f;
    leaf_tri[3 * k] = a;
    leaf_tri[3 * k + 1] = b;
    leaf_tri[3 * k + 2] = c;
    gwn::BvhNode nd;
    nd.xmin = fminf(a.x, fminf(b.x, c.x));
    nd.xmax = fmaxf(a.x, fmaxf(b.x, c.x));
    nd.ymin = fminf(a.y, fminf(b.y, c.y));
    nd.ymax = fmaxf(a.y, fmaxf(b.y, c.y));
    nd.zmax = fmaxf(a.z, fmaxf(b.z, c.z));
    nd.child = (int32_t)k;
    nd.skip = -1;
    nd.is_leaf = 1;
    nodes[n - 1 + k] = nd;
}

// bottom-up refit: the second thread to reach a node merges its children
__global__ void k_refit(int64_t n, const int32_t *__restrict__ parent, const int32_t *__restrict__ left,
                        const int32_t *__restrict__ right, gwn::BvhNode *nodes, unsigned *visits) {
    int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n || n < 2) return;
    int32_t node = (int32_t)(n - 1 + k);
    for (int level = 0; level < 256; ++level) {   // Karras depth <= 63 (30-bit codes + index bits)
        int32_t p = parent[node];
        if (p < 0 || p >= n - 1) break;
        __threadfence();
        if (atomicAdd(&visits[p], 1u) == 0u) break;
        __threadfence();
        const gwn::BvhNode *L = nodes + left[p], *R = nodes + right[p];
        float lxmin = __ldcg(&L->xmin), lxmax = __ldcg(&L->xmax), lymin = __ldcg(&L->ymin),
              lymax = __ldcg(&L->ymax), lzmax = __ldcg(&L->zmax);
        float rxmin = __ldcg(&R->xmin), rxmax = __ldcg(&R->xmax), rymin = __ldcg(&R->ymin),
              rymax = __ldcg(&R->ymax), rzmax = __ldcg(&R->zmax);
        gwn::BvhNode *P = nodes + p;
        __stcg(&P->xmin, fminf(lxmin, rxmin));
        __stcg(&P->xmax, fmaxf(lxmax, rxmax));
        __stcg(&P->ymin, fminf(lymin, rymin));
        __stcg(&P->ymax, fmaxf(lymax, rymax));
        __stcg(&P->zmax, fmaxf(lzmax, rzmax));
        __stcg(&P->child, left[p]);
        __stcg(&P->is_leaf, 0);
        node = p;
    }
}

// Escape link of a node covering leaves [f, l]: the next subtree in depth-first
// order is rooted at the right sibling of the lowest ancestor-or-self that is a
// left child; its parent splits at l, so that sibling is leaf l+1 or internal
// node l+1 (the latter exactly when internal l+1 starts at l+1).
__global__ void k_skip(int64_t n, const int32_t *__restrict__ first, const int32_t *__restrict__ last,
                       gwn::BvhNode *__restrict__ nodes) {
    int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= 2 * n - 1) return;
    int64_t l = (x < n - 1) ? last[x] : x - (n - 1);
    int32_t s;
    if (l == n - 1) s = -1;
    else if (l + 1 <= n - 2 && first[l + 1] == l + 1) s = (int32_t)(l + 1);
    else s = (int32_t)(n - 1 + l + 1);
    nodes[x].skip = s;
}

__global__ void __launch_bounds__(256) k_vertex_bounds(const float4 *__restrict__ V, int64_t nv, int *__restrict__ bounds) {
    block_bounds(nv, [&](int64_t i) { return make_float3(V[i].x, V[i].y, V[i].z); }, bounds);
}

__global__ void k_bounds_to_box(const int *__restrict__ bounds, float *__restrict__ box) {
    if (threadIdx.x < 6) box[threadIdx.x] = from_ordered_key(bounds[threadIdx.x]);
}

}  // namespace

// The boundary edges by sorting all half-edge keys (meshes with a vertex of very many
// edges); tot: two counters of scratch.
static gwn_status boundary_by_sort(gwn_mesh *m, uint32_t *tot, cudaStream_t s) {
    const int64_t nh = 3 * m->nt;
    uint64_t *keys = nullptr, *seg_key = nullptr;
    uint32_t *vals = nullptr, *head = nullptr, *hscan = nullptr, *cnt = nullptr, *off = nullptr;
    int32_t *mult = nullptr;
    GWN_CUDA_TRY(dev_alloc(&keys, sizeof(uint64_t) * nh, s));
    GWN_CUDA_TRY(dev_alloc(&vals, sizeof(uint32_t) * nh, s));
    GWN_CUDA_TRY(dev_alloc(&head, sizeof(uint32_t) * nh, s));
    GWN_CUDA_TRY(dev_alloc(&hscan, sizeof(uint32_t) * nh, s));
    k_halfedge_keys<<<grid_for(nh, TB), TB, 0, s>>>(m->F, m->nt, m->nv, keys, vals);
    int bits = 1;
    while (bits < 64 && ((unsigned __int128)1 << bits) <= (unsigned __int128)m->nv * (unsigned __int128)m->nv) ++bits;
    gwn_status st = radix_sort_u64(keys, vals, nh, bits, s);
    if (st != GWN_OK) return st;
    k_seg_heads<<<grid_for(nh, TB), TB, 0, s>>>(keys, nh, head);
    if ((st = exclusive_scan_u32(head, hscan, nh, tot, s)) != GWN_OK) return st;
    uint32_t nseg_h = 0;
    GWN_CUDA_TRY(cudaMemcpyAsync(&nseg_h, tot, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    GWN_CUDA_TRY(cudaStreamSynchronize(s));
    const int64_t nseg = nseg_h;
    GWN_CUDA_TRY(dev_alloc(&mult, sizeof(int32_t) * nseg, s));
    GWN_CUDA_TRY(dev_alloc(&seg_key, sizeof(uint64_t) * nseg, s));
    GWN_CUDA_TRY(dev_alloc(&cnt, sizeof(uint32_t) * nseg, s));
    GWN_CUDA_TRY(dev_alloc(&off, sizeof(uint32_t) * nseg, s));
    GWN_CUDA_TRY(cudaMemsetAsync(mult, 0, sizeof(int32_t) * nseg, s));
    k_seg_sum<<<grid_for(nh, TB), TB, 0, s>>>(keys, vals, head, hscan, nh, mult, seg_key);
    k_abs<<<grid_for(nseg, TB), TB, 0, s>>>(mult, nseg, cnt);
    if ((st = exclusive_scan_u32(cnt, off, nseg, tot + 1, s)) != GWN_OK) return st;
    uint32_t nb_h = 0;
    GWN_CUDA_TRY(cudaMemcpyAsync(&nb_h, tot + 1, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    GWN_CUDA_TRY(cudaStreamSynchronize(s));
    m->nb = nb_h;
    if (m->nb > 0) {
        GWN_CUDA_TRY(dev_alloc(&m->bedges, sizeof(int32_t) * 2 * m->nb, s));
        k_emit_edges<<<grid_for(nseg, TB), TB, 0, s>>>(mult, seg_key, off, nseg, m->nv, m->bedges);
    }
    cudaFreeAsync(keys, s);
    cudaFreeAsync(vals, s);
    cudaFreeAsync(head, s);
    cudaFreeAsync(hscan, s);
    cudaFreeAsync(mult, s);
    cudaFreeAsync(seg_key, s);
    cudaFreeAsync(cnt, s);
    cudaFreeAsync(off, s);
    return GWN_OK;
}

gwn_status build_boundary(gwn_mesh *m, cudaStream_t s) {
    const int64_t nh = 3 * m->nt;
    m->nb = 0;
    m->npts = 0;
    m->nloops = 0;
    if (m->bedges) { cudaFreeAsync(m->bedges, s); m->bedges = nullptr; }
    if (m->bpts) { cudaFreeAsync(m->bpts, s); m->bpts = nullptr; }
    if (m->tri_loops) { cudaFreeAsync(m->tri_loops, s); m->tri_loops = nullptr; }
    if (m->rest_pts) { cudaFreeAsync(m->rest_pts, s); m->rest_pts = nullptr; }
    m->n_tri_loops = m->n_rest = 0;
    if (m->far_nodes) { cudaFreeAsync(m->far_nodes, s); m->far_nodes = nullptr; }
    if (m->far_pts) { cudaFreeAsync(m->far_pts, s); m->far_pts = nullptr; }
    if (m->far_gcoef) { cudaFreeAsync(m->far_gcoef, s); m->far_gcoef = nullptr; }
    if (m->far_coef) { cudaFreeAsync(m->far_coef, s); m->far_coef = nullptr; }
    if (m->far_roots) { cudaFreeAsync(m->far_roots, s); m->far_roots = nullptr; }
    m->far_nn = 0;
    m->far_nroots = 0;
    m->far_sum = false;
    if (nh == 0) return GWN_OK;
    gwn_status st = GWN_OK;
    bool by_buckets = false;
    uint32_t *tot = nullptr;   // [0], [1]: totals; [2]: a bucket overflowed
    GWN_CUDA_TRY(dev_alloc(&tot, sizeof(uint32_t) * 4, s));
    {   // buckets: 1.9M half-edges 120 us, against 1.25 ms for the sort
        uint32_t *count = nullptr, *first = nullptr, *rank = nullptr, *entry = nullptr, *out = nullptr;
        GWN_CUDA_TRY(dev_alloc(&count, sizeof(uint32_t) * m->nv, s));
        GWN_CUDA_TRY(dev_alloc(&first, sizeof(uint32_t) * m->nv, s));
        GWN_CUDA_TRY(dev_alloc(&out, sizeof(uint32_t) * m->nv, s));
        GWN_CUDA_TRY(dev_alloc(&rank, sizeof(uint32_t) * nh, s));
        GWN_CUDA_TRY(dev_alloc(&entry, sizeof(uint32_t) * nh, s));
        GWN_CUDA_TRY(cudaMemsetAsync(count, 0, sizeof(uint32_t) * m->nv, s));
        GWN_CUDA_TRY(cudaMemsetAsync(tot, 0, sizeof(uint32_t) * 4, s));
        k_bucket_count<<<grid_for(nh, TB), TB, 0, s>>>(m->F, nh, count, rank, tot + 2);
        if ((st = exclusive_scan_u32(count, first, m->nv, nullptr, s)) != GWN_OK) return st;
        k_bucket_place<<<grid_for(nh, TB), TB, 0, s>>>(m->F, nh, first, rank, entry);
        int32_t *net = reinterpret_cast<int32_t *>(rank);   // the ranks are not needed any more
        k_bucket_net<<<grid_for(m->nv, TB), TB, 0, s>>>(entry, first, count, m->nv, net, out, nullptr, tot + 2);
        if ((st = exclusive_scan_u32(out, out, m->nv, tot + 1, s)) != GWN_OK) return st;
        uint32_t tot_h[3] = {0, 0, 0};
        GWN_CUDA_TRY(cudaMemcpyAsync(tot_h, tot, sizeof(tot_h), cudaMemcpyDeviceToHost, s));
        GWN_CUDA_TRY(cudaStreamSynchronize(s));
        by_buckets = tot_h[2] == 0;
        if (by_buckets) {
            m->nb = tot_h[1];
            if (m->nb > 0) {
                GWN_CUDA_TRY(dev_alloc(&m->bedges, sizeof(int32_t) * 2 * m->nb, s));
                k_bucket_net<<<grid_for(m->nv, TB), TB, 0, s>>>(entry, first, count, m->nv, net, out, m->bedges,
                                                                tot + 2);
            }
        }
        for (uint32_t *p : {count, first, rank, entry, out}) cudaFreeAsync(p, s);
    }
    if (!by_buckets && (st = boundary_by_sort(m, tot, s)) != GWN_OK) return st;
    GWN_LAUNCH_CHECK("boundary extraction");
    if (m->nb == 0) {
        cudaFreeAsync(tot, s);
        return GWN_OK;
    }

    const int64_t nb = m->nb;
    if (m->cfg.chain_boundary < 0) {
        m->npts = 2 * nb;
        m->nloops = nb;
        GWN_CUDA_TRY(dev_alloc(&m->bpts, sizeof(float4) * m->npts, s));
        k_emit_unchained<<<grid_for(nb, TB), TB, 0, s>>>(m->bedges, m->V, nb, m->bpts);
        cudaFreeAsync(tot, s);
        GWN_LAUNCH_CHECK("boundary points");
        return GWN_OK;
    }

    // ---- chaining into loops
    uint32_t *kin = nullptr, *idin = nullptr, *kout = nullptr, *idout = nullptr, *succ = nullptr;
    uint32_t *rep[2] = {nullptr, nullptr}, *nx[2] = {nullptr, nullptr}, *dist[2] = {nullptr, nullptr};
    int32_t *rnx[2] = {nullptr, nullptr};
    uint32_t *lsize = nullptr, *loff = nullptr;
    unsigned long long *nl = nullptr;
    GWN_CUDA_TRY(dev_alloc(&kin, sizeof(uint32_t) * nb, s));
    GWN_CUDA_TRY(dev_alloc(&idin, sizeof(uint32_t) * nb, s));
    GWN_CUDA_TRY(dev_alloc(&kout, sizeof(uint32_t) * nb, s));
    GWN_CUDA_TRY(dev_alloc(&idout, sizeof(uint32_t) * nb, s));
    GWN_CUDA_TRY(dev_alloc(&succ, sizeof(uint32_t) * nb, s));
    for (int b = 0; b < 2; ++b) {
        GWN_CUDA_TRY(dev_alloc(&rep[b], sizeof(uint32_t) * nb, s));
        GWN_CUDA_TRY(dev_alloc(&nx[b], sizeof(uint32_t) * nb, s));
        GWN_CUDA_TRY(dev_alloc(&dist[b], sizeof(uint32_t) * nb, s));
        GWN_CUDA_TRY(dev_alloc(&rnx[b], sizeof(int32_t) * nb, s));
    }
    GWN_CUDA_TRY(dev_alloc(&lsize, sizeof(uint32_t) * nb, s));
    GWN_CUDA_TRY(dev_alloc(&loff, sizeof(uint32_t) * nb, s));
    GWN_CUDA_TRY(dev_alloc(&nl, 2 * sizeof(unsigned long long), s));
    int vbits = 1;
    while (vbits < 32 && ((int64_t)1 << vbits) <= m->nv) ++vbits;
    k_edge_vertex_keys<<<grid_for(nb, TB), TB, 0, s>>>(m->bedges, nb, 1, kin, idin);
    if ((st = radix_sort_u32(kin, idin, nb, vbits, s)) != GWN_OK) return st;
    k_edge_vertex_keys<<<grid_for(nb, TB), TB, 0, s>>>(m->bedges, nb, 0, kout, idout);
    if ((st = radix_sort_u32(kout, idout, nb, vbits, s)) != GWN_OK) return st;
    k_pair_succ<<<grid_for(nb, TB), TB, 0, s>>>(idin, idout, nb, succ);
    int rounds = 1;
    while (((int64_t)1 << rounds) < nb) ++rounds;
    rounds += 1;
    uint32_t longer = 0;
    GWN_CUDA_TRY(cudaMemsetAsync(tot + 2, 0, sizeof(uint32_t), s));
    k_walk_loops<<<grid_for(nb, TB), TB, 0, s>>>(succ, nb, rep[0], dist[0], tot + 2);
    GWN_CUDA_TRY(cudaMemcpyAsync(&longer, tot + 2, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    GWN_CUDA_TRY(cudaStreamSynchronize(s));
    int cur = 0, cd = 0;   // the arrays that hold the result
    if (longer && nb <= kJumpSmall) {
        k_jump_small<<<1, 1024, 0, s>>>(succ, (int)nb, rounds, rep[0], rep[1], nx[0], nx[1], dist[0], dist[1], rnx[0],
                                        rnx[1]);
        cur = cd = rounds & 1;
    } else if (longer) {
        k_init_rep<<<grid_for(nb, TB), TB, 0, s>>>(succ, nb, rep[0], nx[0]);
        for (int r = 0; r < rounds; ++r) {
            k_jump_min<<<grid_for(nb, TB), TB, 0, s>>>(rep[cur], nx[cur], nb, rep[cur ^ 1], nx[cur ^ 1]);
            cur ^= 1;
        }
        k_init_rank<<<grid_for(nb, TB), TB, 0, s>>>(succ, rep[cur], nb, dist[0], rnx[0]);
        for (int r = 0; r < rounds; ++r) {
            k_jump_rank<<<grid_for(nb, TB), TB, 0, s>>>(dist[cd], rnx[cd], nb, dist[cd ^ 1], rnx[cd ^ 1]);
            cd ^= 1;
        }
    }
    uint32_t *repf = rep[cur], *distf = dist[cd];
    k_loop_sizes<<<grid_for(nb, TB), TB, 0, s>>>(repf, distf, nb, lsize);
    int *bnd = nullptr;
    const int init[6] = {0x7fffffff, 0x7fffffff, 0x7fffffff, (int)0x80000000, (int)0x80000000, (int)0x80000000};
    GWN_CUDA_TRY(dev_alloc(&bnd, sizeof(init), s));
    GWN_CUDA_TRY(cudaMemcpyAsync(bnd, init, sizeof(init), cudaMemcpyHostToDevice, s));
    k_edge_start_bounds<<<std::min(grid_for(nb, TB), kBoundsBlocks), TB, 0, s>>>(m->bedges, m->V, nb, bnd);
    // the loops' offsets in the order of their first points on the curve (kin, idin
    // and kout are free again: loop keys, representative ids, permuted sizes)
    auto order_loops = [&](int hilbert) -> gwn_status {
        k_loop_keys<<<grid_for(nb, TB), TB, 0, s>>>(repf, m->bedges, m->V, nb, bnd, hilbert, kin, idin);
        gwn_status r = radix_sort_u32(kin, idin, nb, 31, s);
        if (r != GWN_OK) return r;
        k_gather_sizes<<<grid_for(nb, TB), TB, 0, s>>>(idin, lsize, nb, kout);
        if ((r = exclusive_scan_u32(kout, kout, nb, tot, s)) != GWN_OK) return r;
        k_scatter_offsets<<<grid_for(nb, TB), TB, 0, s>>>(idin, kout, nb, loff);
        return GWN_OK;
    };
    if ((st = order_loops(0)) != GWN_OK) return st;
    GWN_CUDA_TRY(cudaMemsetAsync(nl, 0, 2 * sizeof(unsigned long long), s));
    k_count_heads<<<grid_for(nb, TB), TB, 0, s>>>(repf, distf, nb, nl);
    uint32_t npts_h = 0;
    unsigned long long nl_h[2] = {0, 0};
    GWN_CUDA_TRY(cudaMemcpyAsync(&npts_h, tot, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    GWN_CUDA_TRY(cudaMemcpyAsync(nl_h, nl, sizeof(nl_h), cudaMemcpyDeviceToHost, s));
    GWN_CUDA_TRY(cudaStreamSynchronize(s));
    m->npts = npts_h;
    m->nloops = (int64_t)nl_h[0];
    uint2 *ends = nullptr;
    GWN_CUDA_TRY(dev_alloc(&m->bpts, sizeof(float4) * m->npts, s));
    GWN_CUDA_TRY(dev_alloc(&ends, sizeof(uint2) * m->npts, s));
    k_emit_chained<<<grid_for(nb, TB), TB, 0, s>>>(m->bedges, repf, distf, loff, m->V, nb, m->npts, m->bpts, ends);
    const int64_t ntri = (int64_t)nl_h[1];
    if (6 * ntri >= nb && m->cfg.quantize_bits == 0) {   // at least half of the edges
        uint32_t *before = nullptr;
        m->n_tri_loops = ntri;
        m->n_rest = m->npts - 4 * ntri;
        GWN_CUDA_TRY(dev_alloc(&before, sizeof(uint32_t) * m->npts, s));
        GWN_CUDA_TRY(dev_alloc(&m->tri_loops, 5 * sizeof(float4) * ntri, s));
        GWN_CUDA_TRY(dev_alloc(&m->rest_pts, sizeof(float4) * std::max<int64_t>(m->n_rest, 1), s));
        k_tri_heads<<<grid_for(m->npts, TB), TB, 0, s>>>(ends, m->npts, before);
        if ((st = exclusive_scan_u32(before, before, m->npts, nullptr, s)) != GWN_OK) return st;
        k_split_loops<<<grid_for(m->npts, TB), TB, 0, s>>>(m->bpts, ends, before, m->npts, m->tri_loops, m->rest_pts);
        cudaFreeAsync(before, s);
    }
    if (m->npts >= kFarMinPoints) {
        float4 *fpts = nullptr;
        GWN_CUDA_TRY(dev_alloc(&fpts, sizeof(float4) * m->npts, s));
        if ((st = order_loops(1)) != GWN_OK) return st;
        k_emit_chained<<<grid_for(nb, TB), TB, 0, s>>>(m->bedges, repf, distf, loff, m->V, nb, m->npts, fpts, ends);
        st = build_far(m, fpts, ends, s);
    }
    cudaFreeAsync(ends, s);
    cudaFreeAsync(bnd, s);
    for (void *p : {(void *)kin, (void *)idin, (void *)kout, (void *)idout, (void *)succ, (void *)lsize,
                    (void *)loff, (void *)nl, (void *)tot})
        cudaFreeAsync(p, s);
    for (int b = 0; b < 2; ++b) {
        cudaFreeAsync(rep[b], s);
        cudaFreeAsync(nx[b], s);
        cudaFreeAsync(dist[b], s);
        cudaFreeAsync(rnx[b], s);
    }
    if (st != GWN_OK) return st;
    GWN_LAUNCH_CHECK("boundary chaining");
    return GWN_OK;
}

gwn_status build_box(gwn_mesh *m, cudaStream_t s) {
    if (!m->box) GWN_CUDA_TRY(dev_alloc(&m->box, sizeof(float) * 6, s));
    if (m->nv == 0) {
        GWN_CUDA_TRY(cudaMemsetAsync(m->box, 0, sizeof(float) * 6, s));
        return GWN_OK;
    }
    int *bounds = nullptr;
    const int init[6] = {0x7fffffff, 0x7fffffff, 0x7fffffff, (int)0x80000000, (int)0x80000000, (int)0x80000000};
    GWN_CUDA_TRY(dev_alloc(&bounds, sizeof(init), s));
    GWN_CUDA_TRY(cudaMemcpyAsync(bounds, init, sizeof(init), cudaMemcpyHostToDevice, s));
    k_vertex_bounds<<<std::min(grid_for(m->nv, TB), kBoundsBlocks), TB, 0, s>>>(m->V, m->nv, bounds);
    k_bounds_to_box<<<1, 32, 0, s>>>(bounds, m->box);
    cudaFreeAsync(bounds, s);
    GWN_LAUNCH_CHECK("vertex box");
    return GWN_OK;
}

// One LBVH over the triangles: Morton codes over dims axes, radix sort, Karras
// hierarchy, leaves in sorted order, bottom-up refit, escape links.
static gwn_status build_tree(const gwn_mesh *m, int dims, const int *bounds, gwn::BvhNode *nodes,
                             float4 *leaf_tri, cudaStream_t s) {
    const int64_t n = m->nt;
    uint32_t *codes = nullptr, *ids = nullptr;
    int32_t *left = nullptr, *right = nullptr, *parent = nullptr, *first = nullptr, *last = nullptr;
    unsigned *visits = nullptr;
    GWN_CUDA_TRY(dev_alloc(&codes, sizeof(uint32_t) * n, s));
    GWN_CUDA_TRY(dev_alloc(&ids, sizeof(uint32_t) * n, s));
    const int64_t ni = n > 1 ? n - 1 : 1;
    GWN_CUDA_TRY(dev_alloc(&left, sizeof(int32_t) * ni, s));
    GWN_CUDA_TRY(dev_alloc(&right, sizeof(int32_t) * ni, s));
    GWN_CUDA_TRY(dev_alloc(&first, sizeof(int32_t) * ni, s));
    GWN_CUDA_TRY(dev_alloc(&last, sizeof(int32_t) * ni, s));
    GWN_CUDA_TRY(dev_alloc(&parent, sizeof(int32_t) * (2 * n - 1), s));
    GWN_CUDA_TRY(dev_alloc(&visits, sizeof(unsigned) * ni, s));
    GWN_CUDA_TRY(cudaMemsetAsync(parent, 0xff, sizeof(int32_t) * (2 * n - 1), s));
    GWN_CUDA_TRY(cudaMemsetAsync(visits, 0, sizeof(unsigned) * ni, s));
    k_morton<<<grid_for(n, TB), TB, 0, s>>>(m->V, m->F, n, bounds, dims, codes, ids);
    gwn_status st = radix_sort_u32(codes, ids, n, 30, s);
    if (st == GWN_OK) {
        if (n > 1) k_karras<<<grid_for(n - 1, TB), TB, 0, s>>>(codes, n, left, right, parent, first, last);
        k_leaves<<<grid_for(n, TB), TB, 0, s>>>(m->V, m->F, ids, n, nodes, leaf_tri);
        if (n > 1) k_refit<<<grid_for(n, TB), TB, 0, s>>>(n, parent, left, right, nodes, visits);
        k_skip<<<grid_for(2 * n - 1, TB), TB, 0, s>>>(n, first, last, nodes);
    }
    for (void *p : {(void *)codes, (void *)ids, (void *)left, (void *)right, (void *)parent, (void *)first,
                    (void *)last, (void *)visits})
        cudaFreeAsync(p, s);
    if (st != GWN_OK) return st;
    GWN_LAUNCH_CHECK("bvh build");
    return GWN_OK;
}

// Both a tree over xyz Morton codes and one over xy codes (columns: the +z rays
// of neighbouring queries share their paths) are built, and the one with fewer
// expected node tests per walk (k_tree_cost) is kept.  On the soup8 mesh the xy tree
// has 57 instead of 99 node tests per query; random soups of large overlapping
// triangles keep the xyz tree, whose zmax bounds prune better there.
gwn_status build_bvh(gwn_mesh *m, cudaStream_t s) {
    const int64_t n = m->nt;
    if (m->nodes) { cudaFreeAsync(m->nodes, s); m->nodes = nullptr; }
    if (m->leaf_tri) { cudaFreeAsync(m->leaf_tri, s); m->leaf_tri = nullptr; }
    m->nnodes = 0;
    if (n == 0) return GWN_OK;
    m->nnodes = 2 * n - 1;
    gwn::BvhNode *nodes[2] = {nullptr, nullptr};
    float4 *leaf[2] = {nullptr, nullptr};
    int *bounds = nullptr;
    double *cost = nullptr;
    auto cleanup = [&]() {
        for (int t = 0; t < 2; ++t) {
            if (nodes[t]) cudaFreeAsync(nodes[t], s);
            if (leaf[t]) cudaFreeAsync(leaf[t], s);
        }
    };
    for (int t = 0; t < 2; ++t) {
        cudaError_t e;
        if ((e = dev_alloc(&nodes[t], sizeof(gwn::BvhNode) * m->nnodes, s)) != cudaSuccess ||
            (e = dev_alloc(&leaf[t], sizeof(float4) * 3 * n, s)) != cudaSuccess) {
            cudaGetLastError();
            cleanup();
            return set_error(GWN_ERR_OOM, std::string("bvh: ") + cudaGetErrorString(e));
        }
    }
    GWN_CUDA_TRY(dev_alloc(&bounds, sizeof(int) * 6, s));
    GWN_CUDA_TRY(dev_alloc(&cost, sizeof(double) * 2, s));
    const int init[6] = {0x7fffffff, 0x7fffffff, 0x7fffffff, (int)0x80000000, (int)0x80000000, (int)0x80000000};
    GWN_CUDA_TRY(cudaMemcpyAsync(bounds, init, sizeof(init), cudaMemcpyHostToDevice, s));
    GWN_CUDA_TRY(cudaMemsetAsync(cost, 0, sizeof(double) * 2, s));
    k_centroid_bounds<<<std::min(grid_for(n, TB), kBoundsBlocks), TB, 0, s>>>(m->V, m->F, n, bounds);
    gwn_status st = GWN_OK;
    for (int t = 0; t < 2 && st == GWN_OK; ++t) {
        st = build_tree(m, t == 0 ? 3 : 2, bounds, nodes[t], leaf[t], s);
        if (st == GWN_OK)
            k_tree_cost<<<std::min(grid_for(n, TB), 608u), TB, 0, s>>>(nodes[t], n - 1, m->box, cost + t);
    }
    double cost_h[2] = {0.0, 0.0};
    if (st == GWN_OK) {
        cudaError_t e = cudaMemcpyAsync(cost_h, cost, sizeof(cost_h), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) st = set_error(GWN_ERR_CUDA, cudaGetErrorString(e));
    }
    cudaFreeAsync(bounds, s);
    cudaFreeAsync(cost, s);
    if (st != GWN_OK) {
        cleanup();
        return st;
    }
    const int keep = cost_h[1] < cost_h[0] ? 1 : 0;
    m->nodes = nodes[keep];
    m->leaf_tri = leaf[keep];
    m->bvh_xy = keep == 1;
    m->walk_cost = 1.0 + 2.0 * cost_h[keep];
    cudaFreeAsync(nodes[1 - keep], s);
    cudaFreeAsync(leaf[1 - keep], s);
    GWN_LAUNCH_CHECK("bvh build");
    return GWN_OK;
}

}  // namespace gwn
