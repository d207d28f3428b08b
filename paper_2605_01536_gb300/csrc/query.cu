// Query kernels: crossing number (BVH traversal), boundary-curve sum, combine /
// classify with FP64 re-evaluation, and the direct solid-angle sum.
//
// Antipodal evaluation (Eq. 9, Algorithm 1 with x0 = +z, x1 = -z):
//   w(q) = chi(q) + (1/2pi) * sum_{(a,b) in dM} atan2(n_ab, d_ab)
// since Area(A, B, x1) = 2 atan2(n, d).  With a = p_a - q, b = p_b - q,
// l = |a|, the van Oosterom-Strackee numerator and denominator scaled by the
// positive factor l_a l_b are
//   n = x1 . (a x b) = a_y b_x - a_x b_y
//   d = l_a l_b + l_b x1.a + l_a x1.b + a.b = h_a h_b + a_x b_x + a_y b_y,
//   h = l - a_z,
// (the denominator of Supp. S4's Algorithm 3 rearranged).  h is computed as
// (a_x^2 + a_y^2) / (l + a_z) when a_z > 0, which keeps d accurate when a vertex
// lies nearly straight above the query, where the plain form cancels.
#include <algorithm>
#include <type_traits>

#include "gwn_internal.cuh"
#include "predicates.cuh"
#include "bterms.cuh"
#include "traverse.cuh"

namespace gwn {

namespace {


// Launched in blocks of 128 threads (compiled for up to 256): finer tails than
// 256 (measured 5.6% faster on 2M soup8 queries, bit-identical).
constexpr int kChiThreads = 128;
// Leaves k_small tests one by one (64 per lane); a call of 500 queries on closed spheres, one
// by one / walking: 320 leaves 21.6 / 24.3 us, 1,280 20.4 / 22.5, 5,120 38.9 / 23.1.
constexpr int64_t kSmallTris = 2048;

// Fixed selects the predicate mode at compile time (the host knows the mesh's
// quantize_bits), so the exact kernel carries none of the fixed-point code.
// Limited: a query whose walk is longer than kWalkLimit nodes is listed with its partial
// count (in chi) and the node it stands at, and finished by a warp of its own
// (k_chi_rest).  Rays along a rough surface or through random triangles test up to tens
// of thousands of nodes, and the slowest lane held the launch: 1,000 queries on a
// 319k-triangle height field 3.61 -> 0.33 ms, 6,000 on 44k random triangles 1.45 -> 0.31.
// Where walks are short the test costs up to 13% (soup8, 57 nodes a walk), so it is
// compiled in only for meshes whose expected walk is long.
template <bool Fixed, bool Limited>
__global__ void __launch_bounds__(256, 4) k_chi(const float *__restrict__ q, int64_t n,
                                             const BvhNode *__restrict__ nodes, int64_t nnodes,
                                             const float4 *__restrict__ tri, int32_t *__restrict__ chi,
                                             int32_t *__restrict__ rest_q, int32_t *__restrict__ rest_node,
                                             unsigned long long *__restrict__ rest_len,
                                             unsigned long long *__restrict__ counters) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if constexpr (Fixed) {
        if (i >= n) return;
        const float3 p = make_float3(q[3 * i], q[3 * i + 1], q[3 * i + 2]);
        chi[i] = chi_one_q(p, nodes, nnodes, tri, counters, qframe(counters));
    } else {   // the warp walks together (bvh_walk_up_warp): every lane stays to the end
        __shared__ unsigned s_cnt[8][2];   // exact decisions of each warp
        unsigned *cnt = s_cnt[threadIdx.x >> 5];
        const bool active = i < n;
        const float3 p = active ? make_float3(q[3 * i], q[3 * i + 1], q[3 * i + 2]) : make_float3(0.f, 0.f, 0.f);
        int c = 0, rest = -1;
        warp_count_begin(cnt);
        const bool ok = bvh_walk_up_warp<Limited>(active, p, nodes, nnodes, tri, counters,
                                                  [&](int, float3 a, float3 b, float3 cc) {
                                                      c += tri_crossing(p, a, b, cc, WarpCount{cnt}, WarpCount{cnt + 1});
                                                  }, &rest);
        warp_count_end(cnt, counters);
        if (active) chi[i] = ok ? c : INT32_MIN;
        if (Limited && ok && rest >= 0) {
            const unsigned long long slot = atomicAdd(rest_len, 1ull);
            rest_q[slot] = (int32_t)i;
            rest_node[slot] = rest;
        }
    }
}

// The listed long walks, one warp each.
__global__ void __launch_bounds__(128) k_chi_rest(const float *__restrict__ q, const BvhNode *__restrict__ nodes,
                                                  int64_t nnodes, const float4 *__restrict__ tri,
                                                  int32_t *__restrict__ chi, const int32_t *__restrict__ rest_q,
                                                  const int32_t *__restrict__ rest_node,
                                                  const unsigned long long *__restrict__ rest_len,
                                                  unsigned long long *__restrict__ counters) {
    __shared__ unsigned long long s_stack[4][kFrontierCap];
    __shared__ unsigned s_cnt[4][2];   // exact decisions of each warp
    unsigned *cnt = s_cnt[threadIdx.x >> 5];
    const unsigned long long len = *rest_len;
    for (unsigned long long k = (unsigned long long)blockIdx.x * 4 + (threadIdx.x >> 5); k < len;
         k += (unsigned long long)gridDim.x * 4) {
        const int64_t i = rest_q[k];
        const float3 p = make_float3(q[3 * i], q[3 * i + 1], q[3 * i + 2]);
        int c = 0;
        warp_count_begin(cnt);
        const bool ok = bvh_frontier_warp(p, rest_node[k], 2, nodes, nnodes, tri, counters, s_stack[threadIdx.x >> 5],
                                          [&](int, float3 a, float3 b, float3 cc) {
                                              c += tri_crossing(p, a, b, cc, WarpCount{cnt}, WarpCount{cnt + 1});
                                          });
        warp_count_end(cnt, counters);
        c = __reduce_add_sync(0xffffffffu, c);
        if ((threadIdx.x & 31) == 0) chi[i] = ok ? chi[i] + c : INT32_MIN;
    }
}

// The crossing count of k_chi<false>, instrumented: the BVH nodes read and the
// triangles tested, summed over the queries into visits[0] and visits[1].
__global__ void __launch_bounds__(256) k_chi_visits(const float *__restrict__ q, int64_t n,
                                                    const BvhNode *__restrict__ nodes, int64_t nnodes,
                                                    const float4 *__restrict__ tri, int32_t *__restrict__ chi,
                                                    unsigned long long *__restrict__ counters,
                                                    unsigned long long *__restrict__ visits) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    unsigned nv = 0, nt = 0;
    if (i < n) {
        const float3 p = make_float3(q[3 * i], q[3 * i + 1], q[3 * i + 2]);
        int c = 0;
        const bool ok = bvh_walk_up<false, true>(
            p, nodes, nnodes, tri, counters,
            [&](int, float3 a, float3 b, float3 cc) {
                ++nt;
                c += tri_crossing(p, a, b, cc, &counters[CNT_EXACT_EDGE], &counters[CNT_EXACT_PLANE]);
            },
            0.f, &nv);
        chi[i] = ok ? c : INT32_MIN;
    }
    unsigned long long a = nv, b = nt;
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&visits[0], a);
        atomicAdd(&visits[1], b);
    }
}

// Boundary terms of the edges starting at points [e_begin, e_end) for the
// block's 2 KP queries per thread, added to the thread's FP64 accumulators in
// shared memory, s_acc[k * blockDim.x + threadIdx.x] (touched once per tile, so
// they need not occupy registers).  The
// block streams the chained points through shared memory (tile + 1 points);
// point j carries flag w = 1 when an edge runs from it to point j+1.  Every
// thread of the block must call it.
template <int KP, bool Defer = false, bool Cond = false, bool Running = false>
__device__ __forceinline__ void bsum_accumulate(const float4 *__restrict__ pts, int64_t e_begin, int64_t e_end,
                                                int tile, float4 *s_pts, const float2 (&nqx)[KP],
                                                const float2 (&nqy)[KP], const float2 (&nqz)[KP],
                                                double *s_acc, unsigned long long *counters, CancelQ cq,
                                                BsumDefer dq = BsumDefer{}) {
    constexpr int KQ = 2 * KP;
    static_assert(!(Defer || Cond) || KQ <= 4, "queue entries hold a 2-bit query slot");
    BsumState<KP> st;
    int q_count = 0;   // entries in this warp's queue (warp-uniform)
    if constexpr (Defer || Cond) {
#pragma unroll
        for (int k = 0; k < KQ; ++k) cq.fix[k * blockDim.x + threadIdx.x] = 0;
        if ((threadIdx.x & 31) == 0) *cq.count = 0;
        __syncwarp();
    }
#pragma unroll
    for (int k = 0; k < KP; ++k) {
        st.re[k] = bc2(1.f);
        st.im[k] = bc2(0.f);
        st.part[k] = bc2(0.f);
        st.comp[k] = bc2(0.f);
    }
    int g_count = 0;
    // close the current group: one atan2 of each query's product
    auto finalize = [&]() {
#pragma unroll
        for (int k = 0; k < KP; ++k) {
            two_sum_acc2(st.part[k], st.comp[k], fast_atan2_2(st.im[k], st.re[k]));
            st.re[k] = bc2(1.f);
            st.im[k] = bc2(0.f);
        }
        g_count = 0;
    };

    // the edge point j -> j+1 with unit-vector data A (point j) and B (point j+1);
    // cond (std::true_type / std::false_type) selects the cancellation test
    auto add_edge = [&](auto cond, const PointRel2 *A, const PointRel2 *B, int j) {
        constexpr bool C = decltype(cond)::value;
        unsigned fail = 0;   // bit 2k + h: query half h of pair k takes its own atan2
        float2 en[KP], ed[KP];
#pragma unroll
        for (int k = 0; k < KP; ++k) {
            en[k] = fma2(A[k].ay, B[k].ax, neg2(mul2(A[k].ax, B[k].ay)));
            const float2 pl = fma2(A[k].ax, B[k].ax, mul2(A[k].ay, B[k].ay));   // planar part of d
            ed[k] = fma2(A[k].h, B[k].h, pl);
            // a NaN (a padding query past n) counts as accepted: its sum is never read
            bool px, py;
            float2 nre, nim;
            if constexpr (Running) {
                nre = fma2(st.re[k], ed[k], neg2(mul2(st.im[k], en[k])));
                nim = fma2(st.re[k], en[k], mul2(st.im[k], ed[k]));
                px = !(ed[k].x <= kMinD) && !(nre.x <= 0.f);
                py = !(ed[k].y <= kMinD) && !(nre.y <= 0.f);
            } else {
                const float2 v = fma2(bc2(kTanGroup), ed[k], neg2(make_float2(fabsf(en[k].x), fabsf(en[k].y))));
                px = !(v.x <= kAccept);
                py = !(v.y <= kAccept);
            }
            if constexpr (C) {   // and the term must not be ill-conditioned (cancels(), paired)
                const float2 t = mul2(bc2(kCancel), mul2(A[k].h, B[k].h));
                const float2 m2 = fma2(en[k], en[k], mul2(ed[k], ed[k]));
                const float2 t2 = mul2(t, t);
                px = px && !(m2.x < t2.x);
                py = py && !(m2.y < t2.y);
            }
            if constexpr (Running) {
                st.re[k] = make_float2(px ? nre.x : st.re[k].x, py ? nre.y : st.re[k].y);
                st.im[k] = make_float2(px ? nim.x : st.im[k].x, py ? nim.y : st.im[k].y);
            } else {
                const float2 fd = make_float2(px ? ed[k].x : 1.f, py ? ed[k].y : 1.f);
                const float2 fn = make_float2(px ? en[k].x : 0.f, py ? en[k].y : 0.f);
                nre = fma2(st.re[k], fd, neg2(mul2(st.im[k], fn)));
                nim = fma2(st.re[k], fn, mul2(st.im[k], fd));
                st.re[k] = nre;
                st.im[k] = nim;
            }
            fail |= (px ? 0u : 1u << (2 * k)) | (py ? 0u : 2u << (2 * k));
        }
        if constexpr (Defer) {
            // every lane of the warp is here (the loop and the edge flags are block-uniform)
            if (__any_sync(0xffffffffu, fail)) {
                const unsigned lane = threadIdx.x & 31u, below = (1u << lane) - 1u;
#pragma unroll
                for (int k = 0; k < KQ; ++k) {
                    const bool mine = fail >> k & 1u;
                    const unsigned b = __ballot_sync(0xffffffffu, mine);
                    if (mine) dq.queue[q_count + __popc(b & below)] = (unsigned)j << 7 | (unsigned)k << 5 | lane;
                    q_count += __popc(b);
                }
                if (q_count >= 32 * KQ) {
                    __syncwarp();
                    bsum_drain<Cond>(dq.queue, q_count, s_pts, dq.q, dq.fix, cq, counters);
                    q_count = 0;
                }
            }
        } else if (C ? __any_sync(0xffffffffu, fail) : fail != 0) {   // rare: the failing terms one by one
            const float4 Pa = s_pts[j], Pb = s_pts[j + 1];
#pragma unroll
            for (int k = 0; k < KQ; ++k) {
                if (!(fail >> k & 1u)) continue;
                const int kp = k >> 1;
                const bool hi = k & 1;
                const PointRel a = {hi ? A[kp].ax.y : A[kp].ax.x, hi ? A[kp].ay.y : A[kp].ay.x,
                                    hi ? A[kp].h.y : A[kp].h.x};
                const PointRel b = {hi ? B[kp].ax.y : B[kp].ax.x, hi ? B[kp].ay.y : B[kp].ay.x,
                                    hi ? B[kp].h.y : B[kp].h.x};
                const float qx = -(hi ? nqx[kp].y : nqx[kp].x), qy = -(hi ? nqy[kp].y : nqy[kp].x),
                            qz = -(hi ? nqz[kp].y : nqz[kp].x);
                const float nk = hi ? en[kp].y : en[kp].x, dk = hi ? ed[kp].y : ed[kp].x;
                // a queued ill-conditioned term is added later, in FP64.  Only
                // the loop for warps near the tile tests: no query outside the
                // tile's widened box has such a term, so a query's terms do not
                // depend on its warp
                float t = 0.f;
                if (C && cancels(nk, dk, a.h, b.h)) cancel_push(cq, (unsigned)j << 7 | (unsigned)k << 5 | (threadIdx.x & 31u));
                else t = fallback_term(nk, dk, a, b, Pa, Pb, qx, qy, qz, counters);
                if (hi) two_sum_acc(st.part[kp].y, st.comp[kp].y, t);
                else two_sum_acc(st.part[kp].x, st.comp[kp].x, t);
            }
            if constexpr (C) {   // (the whole warp is here)
                if (cancel_count(cq.count) > kCancelCap - 32 * KQ) cancel_drain(cq, s_pts, counters);
            }
        }
        if (++g_count == GROUP) finalize();
    };

    auto run_edges = [&](auto cond, int cnt) {
        PointRel2 ra[KP], rb[KP];
#pragma unroll
        for (int k = 0; k < KP; ++k) ra[k] = point_rel2(s_pts[0], nqx[k], nqy[k], nqz[k]);
        for (int j = 0; j < cnt; j += 2) {
            const float4 P0 = s_pts[j], P1 = s_pts[j + 1];
#pragma unroll
            for (int k = 0; k < KP; ++k) rb[k] = point_rel2(P1, nqx[k], nqy[k], nqz[k]);
            if (P0.w != 0.f) add_edge(cond, ra, rb, j);
            if (j + 1 < cnt) {
                const float4 P2 = s_pts[j + 2];
#pragma unroll
                for (int k = 0; k < KP; ++k) ra[k] = point_rel2(P2, nqx[k], nqy[k], nqz[k]);
                if (P1.w != 0.f) add_edge(cond, rb, ra, j + 1);
            }
        }
    };

    for (int64_t t0 = e_begin; t0 < e_end; t0 += tile) {
        const int cnt = (int)min((int64_t)tile, e_end - t0);   // edge start points in this tile
        __syncthreads();
        for (int i = threadIdx.x; i <= cnt; i += blockDim.x) s_pts[i] = __ldg(pts + t0 + i);
        __syncthreads();
        bool near = false;
        if constexpr (Cond) {
            // A term can be ill-conditioned only if its edge subtends nearly pi at
            // the query, which needs the query within a small fraction of the
            // edge's length of the edge.  The tile's widened box (tile_box) holds
            // every such query; for a warp with no query in it no term is
            // ill-conditioned, so the loop without the test takes the same
            // decisions (bit-identical results).
            float box[6];
            tile_box(s_pts, cnt, box);
#pragma unroll
            for (int k = 0; k < KP; ++k) {
                near |= in_box(box, -nqx[k].x, -nqy[k].x, -nqz[k].x) || in_box(box, -nqx[k].y, -nqy[k].y, -nqz[k].y);
            }
            near = __any_sync(0xffffffffu, near);
            if (near) cancel_tile<KQ>(cq);
        }
        if (near) run_edges(std::true_type{}, cnt);
        else run_edges(std::false_type{}, cnt);
        if (g_count > 0) finalize();
        if constexpr (Defer) {
            if (q_count > 0) {   // the entries index this tile's points
                __syncwarp();
                bsum_drain<Cond>(dq.queue, q_count, s_pts, dq.q, dq.fix, cq, counters);
                q_count = 0;
            }
        }
        if constexpr (Cond) {   // the queued cancelling terms of this tile, in FP64
            if (cancel_count(cq.count) > 0) cancel_drain(cq, s_pts, counters);
        }
#pragma unroll
        for (int k = 0; k < KP; ++k) {
            s_acc[(2 * k) * blockDim.x + threadIdx.x] += (double)st.part[k].x + (double)st.comp[k].x;
            s_acc[(2 * k + 1) * blockDim.x + threadIdx.x] += (double)st.part[k].y + (double)st.comp[k].y;
            st.part[k] = bc2(0.f);
            st.comp[k] = bc2(0.f);
        }
    }
    if constexpr (Defer || Cond) {   // the warp's own drains wrote these sums
        __syncwarp();
#pragma unroll
        for (int k = 0; k < KQ; ++k)
            s_acc[k * blockDim.x + threadIdx.x] += (double)cq.fix[k * blockDim.x + threadIdx.x] * kFixUnit;
    }
}

// One thread holds 2*KP queries as KP float2 pairs (strided by the block size).
// Blocks of 128 threads, 4 resident per SM (at most 128 registers): the same 16 warps
// per SM as 2 blocks of 256, but with finer-grained scheduling, measured 2%
// faster on 2M queries x 154k edges.
// Block (x, y) covers queries of tile x and the edges starting in point chunk y;
// with more than one chunk it writes FP64 partial sums [chunk][query] that
// k_boundary_combine adds, otherwise it combines with chi itself.
constexpr int kBsumThreads = 128;

template <int KP, bool Cond = false, bool Running = false>
__global__ void __launch_bounds__(kBsumThreads, 4) k_boundary_sum(const float *__restrict__ q, int64_t n,
                                                      const float4 *__restrict__ pts, int64_t npts, int tile,
                                                      const TriLoop *__restrict__ tris, int64_t ntri,
                                                      int64_t chunk_len, double *__restrict__ partial,
                                                      const int32_t *__restrict__ chi, float *__restrict__ w,
                                                      uint8_t *__restrict__ label, int classify, float margin,
                                                      int32_t *__restrict__ list,
                                                      unsigned long long *__restrict__ list_len,
                                                      unsigned *__restrict__ listed,
                                                      unsigned long long *__restrict__ counters) {
    // dynamic shared memory (bsum_smem): tile + 1 points | 2 KP x blockDim FP64 sums |
    // (Cond) 2 KP x blockDim fixed-point sums, per warp kCancelCap queue entries, per warp
    // a count per query, per warp a count
    extern __shared__ float4 s_pts[];
    double *s_acc = reinterpret_cast<double *>(s_pts + tile + 1);
    constexpr int KQ = 2 * KP;
    const int64_t qblock = (int64_t)blockIdx.x * blockDim.x * KQ;
    const int64_t base = qblock + threadIdx.x;
    // chunk of the boundary: the triangle loops, two units each, then the edge start points
    const int64_t c0 = (int64_t)blockIdx.y * chunk_len, c1 = c0 + chunk_len;
    const int64_t e_begin = max((int64_t)0, c0 - 2 * ntri);
    const int64_t e_end = min(npts - 1, c1 - 2 * ntri);
    CancelQ cq{};
    unsigned *tri_queue = nullptr;   // with triangle loops, after the counts: per warp 64 KQ entries
    if constexpr (Cond) {
        const int warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
        cq.fix = reinterpret_cast<long long *>(s_acc + KQ * blockDim.x);
        unsigned *queues = reinterpret_cast<unsigned *>(cq.fix + KQ * blockDim.x);
        cq.queue = queues + warp * kCancelCap;
        cq.own = reinterpret_cast<int *>(queues + nwarps * kCancelCap) + warp * 32 * KQ;
        cq.count = reinterpret_cast<int *>(queues + nwarps * (kCancelCap + 32 * KQ)) + warp;
        tri_queue = queues + nwarps * (kCancelCap + 32 * KQ + 1) + warp * 64 * KQ;
        cq.q = q + 3 * qblock;
        cq.qbase = qblock;
        cq.list = list;
        cq.list_len = list_len;
        cq.listed = listed;
    }
    float2 nqx[KP], nqy[KP], nqz[KP];
    load_query_pairs<KP>(q, base, n, nqx, nqy, nqz);
#pragma unroll
    for (int k = 0; k < KQ; ++k) s_acc[k * blockDim.x + threadIdx.x] = 0.0;
    if constexpr (Cond)
        tri_accumulate<KP>(tris, min(ntri, c0 / 2), min(ntri, c1 / 2), (tile + 1) / 5, reinterpret_cast<TriLoop *>(s_pts),
                           nqx, nqy, nqz, s_acc, counters, cq, tri_queue);
    bsum_accumulate<KP, false, Cond, Running>(pts, e_begin, e_end, tile, s_pts, nqx, nqy, nqz, s_acc, counters, cq);
    double acc[KQ];
#pragma unroll
    for (int k = 0; k < KQ; ++k) acc[k] = s_acc[k * blockDim.x + threadIdx.x];
#pragma unroll
    for (int k = 0; k < KQ; ++k) {
        const int64_t idx = base + (int64_t)k * blockDim.x;
        if (idx >= n) continue;
        if (partial) {
            partial[(int64_t)blockIdx.y * n + idx] = acc[k];
            continue;
        }
        const double wv = (double)chi[idx] + acc[k] * kInv2Pi;
        w[idx] = (float)wv;
        if (classify) {
            label[idx] = wv > 0.5 ? 1 : 0;
            if (fabs(wv - 0.5) <= (double)margin) list_query(idx, list, list_len, listed);
        }
    }
}

// Bytes of k_boundary_sum's dynamic shared memory.
static size_t bsum_smem(int kp, int tile, bool cond, bool tris) {
    const size_t kq = 2 * (size_t)kp, threads = kBsumThreads;
    size_t b = sizeof(float4) * (tile + 1) + sizeof(double) * kq * threads;
    if (cond) b += sizeof(long long) * kq * threads + sizeof(unsigned) * (kCancelCap + 32 * kq + 1) * (threads / 32);
    if (tris) b += sizeof(unsigned) * 64 * kq * (threads / 32);
    return b;
}

// Persistent kernel over the work queue of a batch of meshes.  Each block
// repeatedly takes the next item (items are sorted by estimated cost, largest
// first): a crossing item computes chi for its tile's queries; a boundary item
// adds the tile's boundary terms of one point chunk into the FP64 accumulators
// (atomically, so the FP64 summation order of chunks is not fixed).  The block
// that completes a tile's last item combines w = chi + acc / 2pi for that tile
// (the writers fence before counting), so no grid-wide barrier is needed.
template <int KP>
__global__ void __launch_bounds__(256, 2) k_batch(const BatchMesh *__restrict__ meshes,
                                               const BatchTile *__restrict__ tiles,
                                               const BatchItem *__restrict__ items, int64_t n_items,
                                               const float *__restrict__ q, int32_t *chi, double *acc,
                                               float *__restrict__ w, unsigned *tile_done,
                                               unsigned long long *head, int tile_pts, int32_t *list,
                                               unsigned long long *list_len, unsigned *listed) {
    extern __shared__ float4 s_pts[];
    __shared__ long long s_item;
    __shared__ int s_last;
    __shared__ unsigned s_cnt[8][2];   // exact decisions of each warp
    unsigned *cnt = s_cnt[threadIdx.x >> 5];
    constexpr int KQ = 2 * KP;
    while (true) {
        if (threadIdx.x == 0) s_item = (long long)atomicAdd(head, 1ull);
        __syncthreads();
        const long long it = s_item;
        __syncthreads();
        if (it >= n_items) break;
        const BatchItem wi = items[it];
        const BatchTile tl = tiles[wi.tile];
        const BatchMesh mh = meshes[tl.mesh];
        if (wi.kind == 0) {
            // the crossing numbers of the tile: in exact mode the warp walks
            // together (bvh_walk_up_warp), so every lane takes every round
            const bool fixed = qframe(mh.counters)->bits != 0;
            for (int64_t base = wi.p_begin; base < wi.p_end; base += blockDim.x) {
                const int64_t i = base + threadIdx.x;
                const bool active = i < wi.p_end;
                const int64_t g = tl.q_begin + (active ? i : 0);
                const float3 p = active ? make_float3(q[3 * g], q[3 * g + 1], q[3 * g + 2]) : make_float3(0.f, 0.f, 0.f);
                int c = 0;
                warp_count_begin(cnt);
                if (fixed) {
                    if (active) c = chi_one(p, mh.nodes, mh.nnodes, mh.tri, mh.counters);
                } else {
                    const bool ok = bvh_walk_up_warp(active, p, mh.nodes, mh.nnodes, mh.tri, mh.counters,
                                                     [&](int, float3 a, float3 b, float3 cc) {
                                                         c += tri_crossing(p, a, b, cc, WarpCount{cnt},
                                                                           WarpCount{cnt + 1});
                                                     });
                    warp_count_end(cnt, mh.counters);
                    if (!ok) c = INT32_MIN;
                }
                if (active) chi[g] = c;
            }
        } else {
            float2 nqx[KP], nqy[KP], nqz[KP];
            double *s_acc = reinterpret_cast<double *>(s_pts + tile_pts + 1);
            const int warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
            BsumDefer dq;
            dq.q = q + 3 * tl.q_begin;
            dq.fix = reinterpret_cast<long long *>(s_acc + KQ * blockDim.x);
            unsigned *queues = reinterpret_cast<unsigned *>(dq.fix + KQ * blockDim.x);
            dq.queue = queues + warp * (64 * KQ);
            CancelQ cq;
            cq.fix = dq.fix;
            cq.queue = queues + nwarps * (64 * KQ) + warp * kCancelCap;
            cq.own = reinterpret_cast<int *>(queues + nwarps * (64 * KQ + kCancelCap)) + warp * 32 * KQ;
            cq.count = reinterpret_cast<int *>(queues + nwarps * (96 * KQ + kCancelCap)) + warp;
            cq.q = dq.q;
            cq.qbase = tl.q_begin;
            cq.list = list;
            cq.list_len = list_len;
            cq.listed = listed;
            load_query_pairs<KP>(dq.q, threadIdx.x, tl.q_count, nqx, nqy, nqz);
#pragma unroll
            for (int k = 0; k < KQ; ++k) s_acc[k * blockDim.x + threadIdx.x] = 0.0;
            if (wi.kind == 2)
                tri_accumulate<KP>(reinterpret_cast<const TriLoop *>(mh.tri_loops), wi.p_begin, wi.p_end,
                                   (tile_pts + 1) / 5, reinterpret_cast<TriLoop *>(s_pts), nqx, nqy, nqz, s_acc,
                                   mh.counters, cq, dq.queue);
            else
                bsum_accumulate<KP, true, true, true>(mh.rest_pts, wi.p_begin, wi.p_end, tile_pts, s_pts, nqx, nqy, nqz, s_acc,
                                            mh.counters, cq, dq);
#pragma unroll
            for (int k = 0; k < KQ; ++k) {
                const int local = threadIdx.x + k * blockDim.x;
                if (local < tl.q_count) atomicAdd(&acc[tl.q_begin + local], s_acc[k * blockDim.x + threadIdx.x]);
            }
        }
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) s_last = atomicAdd(&tile_done[wi.tile], 1u) == (unsigned)(tl.n_items - 1);
        __syncthreads();
        if (s_last) {
            __threadfence();
            for (int i = threadIdx.x; i < tl.q_count; i += blockDim.x) {
                const int64_t g = tl.q_begin + i;
                w[g] = (float)((double)__ldcg(chi + g) + __ldcg(acc + g) * kInv2Pi);
            }
        }
    }
}

// w = chi + (sum over chunks, in chunk order) / 2pi, then the labels
__global__ void k_boundary_combine(const double *__restrict__ partial, int64_t first, int64_t n, int chunks,
                                   const int32_t *__restrict__ chi, float *__restrict__ w,
                                   uint8_t *__restrict__ label, int classify, float margin,
                                   int32_t *__restrict__ list, unsigned long long *__restrict__ list_len,
                                   unsigned *__restrict__ listed) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, idx = first + i;
    if (i >= n) return;
    double s = 0.0;
    for (int c = 0; c < chunks; ++c) s += partial[(int64_t)c * n + i];
    const double wv = (double)chi[idx] + s * kInv2Pi;
    w[idx] = (float)wv;
    if (classify) {
        label[idx] = wv > 0.5 ? 1 : 0;
        if (fabs(wv - 0.5) <= (double)margin) list_query(idx, list, list_len, listed);
    }
}

// One block per listed query (grid-stride over the list): FP64 boundary sum,
// fixed-order block reduction, then w and the label are rewritten.
__global__ void __launch_bounds__(256) k_fp64_fix(const float *__restrict__ q, const float4 *__restrict__ pts,
                                                  int64_t npts, const int32_t *__restrict__ chi,
                                                  float *__restrict__ w, uint8_t *__restrict__ label,
                                                  const int32_t *__restrict__ list,
                                                  const unsigned long long *__restrict__ list_len,
                                                  unsigned long long *__restrict__ counters) {
    __shared__ double red[256];
    const unsigned long long len = *list_len;
    for (unsigned long long li = blockIdx.x; li < len; li += gridDim.x) {
        const int64_t idx = list[li];
        const float qx = q[3 * idx], qy = q[3 * idx + 1], qz = q[3 * idx + 2];
        // thread t: the edges starting at points [t c, (t + 1) c), c = ceil((npts - 1) / blockDim)
        const int64_t nstart = npts > 0 ? npts - 1 : 0, per = (nstart + blockDim.x - 1) / blockDim.x;
        const int64_t j0 = min((int64_t)threadIdx.x * per, nstart), j1 = min(j0 + per, nstart);
        red[threadIdx.x] = bsum64_range(pts, j0, j1, qx, qy, qz, counters);
        __syncthreads();
        for (int o = 128; o > 0; o >>= 1) {
            if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            const double wv = (double)chi[idx] + red[0] * kInv2Pi;
            w[idx] = (float)wv;
            if (label) label[idx] = wv > 0.5 ? 1 : 0;
            atomicAdd(&counters[CNT_FP64], 1ull);
        }
        __syncthreads();
    }
}

// The batched launch's FP64 re-evaluation: one block per listed query (more than
// kCancelOwn cancelling terms in a tile); the mesh is found by binary
// search in the meshes' query offsets.
__global__ void __launch_bounds__(256) k_batch_fp64_fix(const BatchMesh *__restrict__ meshes,
                                                        const int64_t *__restrict__ mesh_off, int n_mesh,
                                                        const float *__restrict__ q, const int32_t *__restrict__ chi,
                                                        float *__restrict__ w, const int32_t *__restrict__ list,
                                                        const unsigned long long *__restrict__ list_len) {
    __shared__ double red[256];
    const unsigned long long len = *list_len;
    for (unsigned long long li = blockIdx.x; li < len; li += gridDim.x) {
        const int64_t g = list[li];
        int lo = 0, hi = n_mesh - 1;   // the mesh with mesh_off[mi] <= g < mesh_off[mi + 1]
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (mesh_off[mid] <= g) lo = mid;
            else hi = mid - 1;
        }
        const BatchMesh mh = meshes[lo];
        const float qx = q[3 * g], qy = q[3 * g + 1], qz = q[3 * g + 2];
        const int64_t nstart = mh.npts > 0 ? mh.npts - 1 : 0, per = (nstart + blockDim.x - 1) / blockDim.x;
        const int64_t j0 = min((int64_t)threadIdx.x * per, nstart), j1 = min(j0 + per, nstart);
        red[threadIdx.x] = bsum64_range(mh.pts, j0, j1, qx, qy, qz, mh.counters);
        __syncthreads();
        for (int o = 128; o > 0; o >>= 1) {
            if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            w[g] = (float)((double)chi[g] + red[0] * kInv2Pi);
            atomicAdd(&mh.counters[CNT_FP64], 1ull);
        }
        __syncthreads();
    }
}

// ------------------------------------------------------- small calls ----

// A call of few queries against few boundary points, whole: one warp per query counts
// the crossings (every leaf box by all lanes on a small mesh, else all lanes walk the
// tree: bvh_frontier_warp), sums the edge terms lane by lane in FP64, and re-evaluates the sum in FP64 where
// classify needs it.  The general path's kernels each leave the GPU nearly idle for a
// serial chain (64 queries on a 36-edge boundary: crossings 22 us, boundary 20 us, FP64
// check 4 us, with five allocations and two memsets); this is one launch of about 8 us
// and no scratch.  Bound by latency: the chain of one warp.
constexpr int kSmallThreads = 128;
__global__ void __launch_bounds__(kSmallThreads) k_small(const float *__restrict__ q, int64_t n,
                                                         const BvhNode *__restrict__ nodes, int64_t nnodes,
                                                         const float4 *__restrict__ tri, const float4 *__restrict__ pts,
                                                         int64_t npts, float *__restrict__ w, int32_t *__restrict__ chi,
                                                         uint8_t *__restrict__ label, float margin,
                                                         unsigned long long *__restrict__ counters) {
    __shared__ unsigned long long s_stack[kSmallThreads / 32][kFrontierCap];
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (i >= n) return;
    const float qx = q[3 * i], qy = q[3 * i + 1], qz = q[3 * i + 2];
    const float3 p = make_float3(qx, qy, qz);
    const int64_t nt = (nnodes + 1) / 2;
    int c = 0;
    bool ok = true;
    if (nt <= kSmallTris) {
        for (int64_t t = lane; t < nt; t += 32) {
            const float4 *np = reinterpret_cast<const float4 *>(nodes + (nt - 1) + t);   // leaf t of the tree
            const float4 b0 = __ldg(np), b1 = __ldg(np + 1);
            if (!(qx >= b0.x && qx <= b0.y && qy >= b0.z && qy <= b0.w && qz <= b1.x)) continue;
            const float4 a = __ldg(tri + 3 * t), b = __ldg(tri + 3 * t + 1), d = __ldg(tri + 3 * t + 2);
            c += tri_crossing(p, make_float3(a.x, a.y, a.z), make_float3(b.x, b.y, b.z), make_float3(d.x, d.y, d.z),
                              &counters[CNT_EXACT_EDGE], &counters[CNT_EXACT_PLANE]);
        }
    } else {
        ok = bvh_frontier_warp(p, 0, 0, nodes, nnodes, tri, counters, s_stack[threadIdx.x >> 5],
                               [&](int, float3 a, float3 b, float3 d) {
                                   c += tri_crossing(p, a, b, d, &counters[CNT_EXACT_EDGE], &counters[CNT_EXACT_PLANE]);
                               });
    }
    c = __reduce_add_sync(0xffffffffu, c);
    if (!__all_sync(0xffffffffu, ok)) c = INT32_MIN;
    double s = 0.0;
    int cancelled = 0;
    for (int64_t j = lane; j + 1 < npts; j += 32) {
        const float4 Pa = __ldg(pts + j), Pb = __ldg(pts + j + 1);
        if (Pa.w == 0.f) continue;
        const PointRel A = point_rel_twin(Pa, qx, qy, qz), B = point_rel_twin(Pb, qx, qy, qz);
        const float en = __fmaf_rn(A.ay, B.ax, -__fmul_rn(A.ax, B.ay));
        const float ed = __fmaf_rn(A.h, B.h, __fmaf_rn(A.ax, B.ax, __fmul_rn(A.ay, B.ay)));
        if (cancels(en, ed, A.h, B.h)) {
            s += edge_angle64(Pa, Pb, qx, qy, qz, counters);
            ++cancelled;
        } else {
            s += edge_term(en, ed, A, B, Pa, Pb, qx, qy, qz, counters);
        }
    }
    cancelled = __reduce_add_sync(0xffffffffu, cancelled);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    double wv = (double)c + s * kInv2Pi;
    if (label && fabs(wv - 0.5) <= (double)margin) {   // warp-uniform
        s = 0.0;
        for (int64_t j = lane; j + 1 < npts; j += 32) {
            const float4 Pa = __ldg(pts + j);
            if (Pa.w != 0.f) s += edge_angle64(Pa, __ldg(pts + j + 1), qx, qy, qz, counters);
        }
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        wv = (double)c + s * kInv2Pi;
        if (lane == 0) atomicAdd(&counters[CNT_FP64], 1ull);
    }
    if (lane != 0) return;
    if (cancelled) atomicAdd(&counters[CNT_CANCEL], (unsigned long long)cancelled);
    if (w) w[i] = (float)wv;
    if (chi) chi[i] = c;
    if (label) label[i] = wv > 0.5 ? 1 : 0;
}

// ------------------------------------------------------------- direct ----

// Direct sum (Eq. 2, each area by Eq. 6): per triangle 2 atan2(det, den) with unit vectors
// A, B, C toward the vertices, den = 1 + A.B + A.C + B.C and det = (A . N') (h / (|b| |c|)),
// N = h N' the triangle's normal vector as for triangle loops (bterms.cuh; computed once
// per block when the triangle is staged, as accurate as the FP32 vertices allow: a slim
// triangle's normal is small against the products it is made of).
// Terms are multiplied into a group's complex product like the boundary sum's (one atan2
// per 8 triangles) under the triangle loops' test: an angle below pi/8, well-conditioned;
// nearer triangles take their own, for the pair of queries at once and with the determinant
// of the unit vectors, which is as accurate beside every vertex (the nearest vertex against
// N' for each query that failed: 200k queries beside the 200 slim triangles of a fan 196
// us, now 149; every term by itself 139).  a is the vertex opposite the longest edge, so
// that b and c are far apart and few terms of slim triangles fail.  Each thread holds 2 KP queries as float2 pairs.  The
// triangle range is split into gridDim.y chunks so that any query count fills the GPU:
// with one chunk the kernel writes w, otherwise FP64 partial sums [chunk][query] that
// k_direct_reduce adds in chunk order.  Bound by the FP32 pipe (77% of its cycles): 49 paired
// operations a term (75 with an atan2 and a 3 x 3 determinant each): 30k queries x 40k
// triangles 2.54 -> 1.97 ms.  Errors above 1e-5 beside surfaces, edges and vertices (132 sets
// of queries against FP64) 29.7k -> 11.8k against that determinant's.
template <int KP>
__global__ void __launch_bounds__(256, 2) k_direct(const float *__restrict__ q, int64_t n, const float *__restrict__ tri9,
                                                   int64_t nt, int tile, int64_t chunk_len, float *__restrict__ w,
                                                   double *__restrict__ partial) {
    extern __shared__ float4 s_dir[];   // per triangle: (a, N'.x), (b, N'.y), (c, N'.z); then their h
    float *s_h = reinterpret_cast<float *>(s_dir + 3 * tile);
    constexpr int KQ = 2 * KP;
    const int64_t base = (int64_t)blockIdx.x * blockDim.x * KQ + threadIdx.x;
    const int64_t t_begin = (int64_t)blockIdx.y * chunk_len;
    const int64_t t_end = min(nt, t_begin + chunk_len);
    float2 nqx[KP], nqy[KP], nqz[KP], part[KP], re[KP], im[KP];
    double acc[KQ];
#pragma unroll
    for (int k = 0; k < KQ; ++k) {
        const int64_t idx = base + (int64_t)k * blockDim.x;
        const bool ok = idx < n;
        const float x = ok ? -q[3 * idx] : 0.f, y = ok ? -q[3 * idx + 1] : 0.f, z = ok ? -q[3 * idx + 2] : 0.f;
        if (k & 1) { nqx[k >> 1].y = x; nqy[k >> 1].y = y; nqz[k >> 1].y = z; }
        else       { nqx[k >> 1].x = x; nqy[k >> 1].x = y; nqz[k >> 1].x = z; }
        acc[k] = 0.0;
    }
#pragma unroll
    for (int k = 0; k < KP; ++k) {
        part[k] = im[k] = bc2(0.f);
        re[k] = bc2(1.f);
    }
    int g = 0;
    auto close = [&]() {
#pragma unroll
        for (int k = 0; k < KP; ++k) {
            part[k] = add2(part[k], fast_atan2_2(im[k], re[k]));
            re[k] = bc2(1.f);
            im[k] = bc2(0.f);
        }
        g = 0;
    };
    for (int64_t t0 = t_begin; t0 < t_end; t0 += tile) {
        const int cnt = (int)min((int64_t)tile, t_end - t0);
        __syncthreads();
        for (int i = threadIdx.x; i < cnt; i += blockDim.x) {
            const float *T = tri9 + 9 * (t0 + i);
            float ax = __ldg(T), ay = __ldg(T + 1), az = __ldg(T + 2), bx = __ldg(T + 3), by = __ldg(T + 4),
                  bz = __ldg(T + 5), cx = __ldg(T + 6), cy = __ldg(T + 7), cz = __ldg(T + 8);
            auto len2 = [](float x, float y, float z) { return x * x + y * y + z * z; };
            auto turn = [](float &x, float &y, float &z) {   // (x, y, z) -> (y, z, x)
                const float t = x;
                x = y;
                y = z;
                z = t;
            };
            // a opposite the longest edge
            const float la = len2(cx - bx, cy - by, cz - bz), lb = len2(ax - cx, ay - cy, az - cz),
                        lc = len2(bx - ax, by - ay, bz - az);
            for (int turns = lb > fmaxf(la, lc) ? 1 : lc > la ? 2 : 0; turns > 0; --turns) {
                turn(ax, bx, cx);
                turn(ay, by, cy);
                turn(az, bz, cz);
            }
            float u[3], v[3], ul[3], vl[3], N[3];   // the edges as exact sums of two floats
            two_diff32(bx, ax, u[0], ul[0]);
            two_diff32(by, ay, u[1], ul[1]);
            two_diff32(bz, az, u[2], ul[2]);
            two_diff32(cx, ax, v[0], vl[0]);
            two_diff32(cy, ay, v[1], vl[1]);
            two_diff32(cz, az, v[2], vl[2]);
            float top = 0.f;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int k1 = (k + 1) % 3, k2 = (k + 2) % 3;
                // u1 v2 - u2 v1 with the rounding of the second product made good, and the low parts
                const float m = u[k2] * v[k1];
                N[k] = (fmaf(u[k1], v[k2], -m) + fmaf(-u[k2], v[k1], m)) +
                       (fmaf(u[k1], vl[k2], ul[k1] * v[k2]) - fmaf(u[k2], vl[k1], ul[k2] * v[k1]));
                top = fmaxf(top, fabsf(N[k]));
            }
            const int e = __float_as_int(top) & 0x7f800000;   // h = 2^floor(log2 top), or 0
            const float r = e ? __int_as_float((254 << 23) - e) : 0.f;
            s_dir[3 * i] = make_float4(ax, ay, az, N[0] * r);
            s_dir[3 * i + 1] = make_float4(bx, by, bz, N[1] * r);
            s_dir[3 * i + 2] = make_float4(cx, cy, cz, N[2] * r);
            s_h[i] = __int_as_float(e);
        }
        __syncthreads();
        for (int j = 0; j < cnt; ++j) {
            const float4 A = s_dir[3 * j], B = s_dir[3 * j + 1], C = s_dir[3 * j + 2];
            const float h = s_h[j];
#pragma unroll
            for (int k = 0; k < KP; ++k) {
                const float2 ax = add2(bc2(A.x), nqx[k]), ay = add2(bc2(A.y), nqy[k]), az = add2(bc2(A.z), nqz[k]);
                const float2 bx = add2(bc2(B.x), nqx[k]), by = add2(bc2(B.y), nqy[k]), bz = add2(bc2(B.z), nqz[k]);
                const float2 cx = add2(bc2(C.x), nqx[k]), cy = add2(bc2(C.y), nqy[k]), cz = add2(bc2(C.z), nqz[k]);
                const float2 la = fma2(ax, ax, fma2(ay, ay, mul2(az, az)));
                const float2 lb = fma2(bx, bx, fma2(by, by, mul2(bz, bz)));
                const float2 lc = fma2(cx, cx, fma2(cy, cy, mul2(cz, cz)));
                const float2 ia = make_float2(sfu_rsqrt(la.x), sfu_rsqrt(la.y)), ib = make_float2(sfu_rsqrt(lb.x), sfu_rsqrt(lb.y)),
                             ic = make_float2(sfu_rsqrt(lc.x), sfu_rsqrt(lc.y));
                const float2 ab = fma2(ax, bx, fma2(ay, by, mul2(az, bz)));
                const float2 ac = fma2(ax, cx, fma2(ay, cy, mul2(az, cz)));
                const float2 bc = fma2(bx, cx, fma2(by, cy, mul2(bz, cz)));
                const float2 ibc = mul2(ib, ic);
                const float2 den = fma2(bc, ibc, fma2(mul2(ac, ia), ic, fma2(mul2(ab, ia), ib, bc2(1.f))));
                const float2 dn = fma2(ax, bc2(A.w), fma2(ay, bc2(B.w), mul2(az, bc2(C.w))));
                const float2 g = mul2(bc2(h), ibc);
                const float2 det = mul2(mul2(dn, ia), g);
                const float2 v = fma2(bc2(-kTriSpread), g,
                                      fma2(bc2(kTanGroup), den, neg2(make_float2(fabsf(det.x), fabsf(det.y)))));
                const bool px = v.x > kTriAccept, py = v.y > kTriAccept;   // (not if NaN, at a vertex)
                if (!(px && py)) {   // an atan2 of the pair's own, by the determinant of the unit vectors
                    float2 ja = ia, jb = ib, jc = ic, oe = den;
                    if (!(v.x > -1e30f && v.y > -1e30f)) {   // at a vertex: finite reciprocal lengths
                        auto finite = [](float2 i) { return make_float2(fminf(i.x, 3.1e18f), fminf(i.y, 3.1e18f)); };
                        ja = finite(ia);
                        jb = finite(ib);
                        jc = finite(ic);
                        oe = fma2(bc, mul2(jb, jc), fma2(mul2(ac, ja), jc, fma2(mul2(ab, ja), jb, bc2(1.f))));
                    }
                    const float2 Ax = mul2(ax, ja), Ay = mul2(ay, ja), Az = mul2(az, ja), Bx = mul2(bx, jb),
                                 By = mul2(by, jb), Bz = mul2(bz, jb), Cx = mul2(cx, jc), Cy = mul2(cy, jc), Cz = mul2(cz, jc);
                    const float2 od = fma2(Ax, fma2(By, Cz, neg2(mul2(Bz, Cy))),
                                           fma2(Ay, fma2(Bz, Cx, neg2(mul2(Bx, Cz))), mul2(Az, fma2(Bx, Cy, neg2(mul2(By, Cx))))));
                    const float2 t = fast_atan2_2(od, oe);
                    part[k] = add2(part[k], make_float2(px ? 0.f : t.x, py ? 0.f : t.y));
                }
                const float2 fd = make_float2(px ? den.x : 1.f, py ? den.y : 1.f);
                const float2 fn = make_float2(px ? det.x : 0.f, py ? det.y : 0.f);
                const float2 r = fma2(re[k], fd, neg2(mul2(im[k], fn)));
                im[k] = fma2(re[k], fn, mul2(im[k], fd));
                re[k] = r;
            }
            if (++g == GROUP) close();
        }
        if (g > 0) close();
#pragma unroll
        for (int k = 0; k < KP; ++k) {
            acc[2 * k] += (double)part[k].x;
            acc[2 * k + 1] += (double)part[k].y;
            part[k] = bc2(0.f);
        }
    }
#pragma unroll
    for (int k = 0; k < KQ; ++k) {
        const int64_t idx = base + (int64_t)k * blockDim.x;
        if (idx >= n) continue;
        if (partial) partial[(int64_t)blockIdx.y * n + idx] = acc[k];
        else w[idx] = (float)(acc[k] * kInv2Pi);
    }
}

__global__ void k_direct_reduce(const double *__restrict__ partial, int64_t n, int chunks, float *__restrict__ w) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double s = 0.0;
    for (int c = 0; c < chunks; ++c) s += partial[(int64_t)c * n + i];
    w[i] = (float)(s * kInv2Pi);
}

}  // namespace

// Where k_chi cuts walks: on meshes above twice soup8's 57 expected node tests, for calls
// whose slowest walk holds the launch.  A warp of its own per long walk does more work in
// all, so many queries are better left to fill the GPU.  Crossing counts on a 319k-triangle
// height field, cut / whole: 1k queries 179 / 826 us, 16k 313 / 865, 32k 603 / 1020,
// 100k 1265 / 1052, 1M 11.2 / 5.6 ms; on an 80k one 32k 454 / 434 us, 64k 366 / 259.
constexpr double kLongWalk = 128.0;
constexpr int64_t kLongWalkQueries = 32768;
static bool long_walks(const gwn_mesh *m, int64_t n) {
    return m->cfg.quantize_bits == 0 && m->walk_cost >= kLongWalk && m->nnodes > kWalkLimit && n <= kLongWalkQueries;
}

// rest_len, rest_q, rest_node: scratch for the long walks (a counter and n entries each),
// used if long_walks(m, n)
static gwn_status chi_on(const gwn_mesh *m, const float *q, int64_t n, int32_t *chi, unsigned long long *rest_len,
                         int32_t *rest_q, int32_t *rest_node, cudaStream_t s) {
    const unsigned blocks = grid_for(n, kChiThreads);
    if (m->cfg.quantize_bits) {
        k_chi<true, false><<<blocks, kChiThreads, 0, s>>>(q, n, m->nodes, m->nnodes, m->leaf_tri, chi, nullptr, nullptr,
                                                          nullptr, m->counters);
    } else if (!long_walks(m, n)) {
        k_chi<false, false><<<blocks, kChiThreads, 0, s>>>(q, n, m->nodes, m->nnodes, m->leaf_tri, chi, nullptr, nullptr,
                                                           nullptr, m->counters);
    } else {
        GWN_CUDA_TRY(cudaMemsetAsync(rest_len, 0, sizeof(unsigned long long), s));
        k_chi<false, true><<<blocks, kChiThreads, 0, s>>>(q, n, m->nodes, m->nnodes, m->leaf_tri, chi, rest_q, rest_node,
                                                          rest_len, m->counters);
        k_chi_rest<<<std::min(grid_for(n, 4), 1216u), 128, 0, s>>>(q, m->nodes, m->nnodes, m->leaf_tri, chi, rest_q,
                                                                   rest_node, rest_len, m->counters);
        note_launches(1);
    }
    note_launches(1);
    GWN_LAUNCH_CHECK("k_chi");
    return GWN_OK;
}

gwn_status launch_chi(const gwn_mesh *m, const float *q, int64_t n, int32_t *chi, cudaStream_t s) {
    if (n <= 0) return GWN_OK;
    ProfScope prof("chi_traversal", s);
    if (!long_walks(m, n)) return chi_on(m, q, n, chi, nullptr, nullptr, nullptr, s);
    unsigned long long *len = nullptr;
    GWN_CUDA_TRY(dev_alloc(&len, sizeof(unsigned long long) + 2 * sizeof(int32_t) * n, s));
    int32_t *rest_q = reinterpret_cast<int32_t *>(len + 1);
    const gwn_status st = chi_on(m, q, n, chi, len, rest_q, rest_q + n, s);
    cudaFreeAsync(len, s);
    return st;
}

// Few queries (a warp each), few points (a lane takes npts / 32 of them) and little
// work in all: 2^20 terms of about 150 instructions are 4 us of the whole GPU.  Explicit
// schedules and the plain FP32 or fixed-point forms keep the general path.
bool small_call(const gwn_mesh *m, int64_t n) {
    return n <= 4096 && m->npts <= 4096 && n * m->npts <= (int64_t(1) << 20) && m->cfg.quantize_bits == 0 &&
           m->cfg.queries_per_thread == 0 && m->cfg.boundary_tile == 0 && m->cfg.group_test == 0 &&
           m->cfg.fp64_cancel >= 0;
}

gwn_status launch_small(const gwn_mesh *m, const float *q, int64_t n, float *w, int32_t *chi, uint8_t *label,
                        cudaStream_t s) {
    if (n <= 0) return GWN_OK;
    ProfScope prof("small_call", s);
    const float margin = m->cfg.classify_margin > 0.f ? m->cfg.classify_margin : 1e-4f;
    k_small<<<grid_for(32 * n, kSmallThreads), kSmallThreads, 0, s>>>(q, n, m->nodes, m->nnodes, m->leaf_tri, m->bpts,
                                                                      m->npts, w, chi, label, margin, m->counters);
    GWN_LAUNCH_CHECK("k_small");
    return GWN_OK;
}

gwn_status launch_chi_visits(const gwn_mesh *m, const float *q, int64_t n, int32_t *chi,
                             unsigned long long *visits, cudaStream_t s) {
    if (n <= 0) return GWN_OK;
    k_chi_visits<<<grid_for(n, 256), 256, 0, s>>>(q, n, m->nodes, m->nnodes, m->leaf_tri, chi, m->counters, visits);
    GWN_LAUNCH_CHECK("k_chi_visits");
    return GWN_OK;
}

void launch_boundary_combine(const double *partial, int64_t first, int64_t n, int chunks, const int32_t *chi, float *w,
                             uint8_t *label, bool classify, float margin, int32_t *list,
                             unsigned long long *list_len, unsigned *listed, cudaStream_t s) {
    k_boundary_combine<<<grid_for(n, 256), 256, 0, s>>>(partial, first, n, chunks, chi, w, label, classify ? 1 : 0, margin,
                                                        list, list_len, listed);
    note_launches(1);
}

// The edges (with triangle loops apart: the other edges and two halves per triangle) that
// the direct boundary sum splits into parts
static bool split_triangles(const gwn_mesh *m, bool cond, bool plain) {
    const int tile = m->cfg.boundary_tile > 0 ? m->cfg.boundary_tile : 512;
    return cond && !plain && m->n_tri_loops > 0 && tile >= 64;
}
static int64_t edge_points(const gwn_mesh *m, bool split) {
    const int64_t npts = split ? m->n_rest : m->npts;
    return (npts > 0 ? npts - 1 : 0) + 2 * (split ? m->n_tri_loops : 0);
}

// Into how many parts a call of n queries splits them when the query tiles alone cannot
// fill the GPU.  A function of the mesh and n only: a query's FP32 groups, and with them
// the bits of w, follow it (the slices of gwn_classify_static pass the whole call's n).
// 48 blocks per SM: a grid of 1.6 waves, 500k queries x 797 points, took 575 us instead of
// 490, 100k queries 123 instead of 87, and near triangle loops make blocks uneven; the
// surrogate's labels keep 8, and with it their bits.
static int64_t direct_parts(const gwn_mesh *m, int64_t n, int kp, bool cond, bool plain) {
    const int tile = m->cfg.boundary_tile > 0 ? m->cfg.boundary_tile : 512;
    const int64_t per_block = kBsumThreads * 2 * kp, qblocks = (n + per_block - 1) / per_block;
    const int64_t nedge_pts = edge_points(m, split_triangles(m, cond, plain));
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int64_t parts = ((plain ? 8 : 48) * (int64_t)(sms > 0 ? sms : 148) + qblocks - 1) / qblocks;
    // (a part of 128 points still pays for its partial sums: 64 queries against
    // 9.8k edges take 47 us instead of 200 us with parts of 1024 points)
    const int64_t min_part = n < kOrderMinQueries || !plain ? std::min<int64_t>(128, 2 * tile) : 2 * tile;
    parts = std::max<int64_t>(1, std::min<int64_t>(parts, (nedge_pts + min_part - 1) / min_part));
    return std::min<int64_t>(parts, 65535);
}

template <int KP, bool Cond = false, bool Running = false>
static gwn_status launch_bsum_kp(const gwn_mesh *m, const float *q, int64_t n, const int32_t *chi, float *w,
                                 uint8_t *label, bool classify, int32_t *list, unsigned long long *list_len,
                                 unsigned *listed, double *partial_buf, int64_t call_n, bool plain,
                                 cudaStream_t s) {
    const int tile = m->cfg.boundary_tile > 0 ? m->cfg.boundary_tile : 512;
    const float margin = m->cfg.classify_margin > 0.f ? m->cfg.classify_margin : 1e-4f;
    const int64_t per_block = kBsumThreads * 2 * KP;
    const int64_t qblocks = (n + per_block - 1) / per_block;
    // triangle loops as one term each (tri_accumulate; the FP64 test of their edges needs Cond)
    const bool split = split_triangles(m, Cond, plain);
    const float4 *pts = split ? m->rest_pts : m->bpts;
    const int64_t npts = split ? m->n_rest : m->npts, ntri = split ? m->n_tri_loops : 0;
    const int64_t nedge_pts = edge_points(m, split);
    const size_t smem = bsum_smem(KP, tile, Cond, ntri > 0);
    if (smem > 48 * 1024)
        cudaFuncSetAttribute(k_boundary_sum<KP, Cond, Running>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem);
    const int64_t chunks = direct_parts(m, call_n, KP, Cond, plain);
    int64_t chunk_len = chunks > 1 ? (nedge_pts + chunks - 1) / chunks : std::max<int64_t>(nedge_pts, 1);
    if (ntri > 0) chunk_len += chunk_len & 1;   // whole triangles
    double *partial = chunks > 1 ? partial_buf : nullptr;
    const bool own = chunks > 1 && !partial_buf;
    if (own) GWN_CUDA_TRY(dev_alloc(&partial, sizeof(double) * chunks * n, s));
    dim3 grid((unsigned)qblocks, (unsigned)chunks);
    k_boundary_sum<KP, Cond, Running><<<grid, kBsumThreads, smem, s>>>(q, n, pts, npts, tile,
                                                                      reinterpret_cast<const TriLoop *>(m->tri_loops),
                                                                      ntri, chunk_len, partial, chi, w, label, classify ? 1 : 0,
                                                                      margin, list, list_len, listed, m->counters);
    note_launches(1);
    if (partial) {
        launch_boundary_combine(partial, 0, n, (int)chunks, chi, w, label, classify, margin, list, list_len, listed, s);
        if (own) cudaFreeAsync(partial, s);
    }
    GWN_LAUNCH_CHECK("k_boundary_sum");
    return GWN_OK;
}

// The group acceptance test of a mesh (gwn_config.group_test): the running
// test where the boundary is dense, at least one boundary edge per two
// triangles (random soups, 3 per triangle), else the per-term test.
static bool group_test_running(const gwn_mesh *m) {
    if (m->cfg.group_test == 1) return false;
    if (m->cfg.group_test == 2) return true;
    return 2 * m->nb >= m->nt && m->nb > 0;
}

// The boundary sum with the scratch it needs provided: list (n entries), a
// zeroed list_len and zeroed listed bits (n / 32 words, rounded up); the parts' partial
// sums in partial_buf (n times boundary_parts(m, call_n, far) doubles), or allocated as
// needed when it is null.  call_n: the queries of the whole call.
static gwn_status boundary_sum_on(const gwn_mesh *m, const float *q, int64_t n, const int32_t *chi, float *w,
                                  uint8_t *label, bool classify, int32_t *list, unsigned long long *list_len,
                                  unsigned *listed, double *partial_buf, int64_t call_n, bool far,
                                  bool plain, cudaStream_t s) {
    const int kq = m->cfg.queries_per_thread > 0 ? m->cfg.queries_per_thread : 4;
    ProfScope prof("boundary_sum", s);
    const bool running = group_test_running(m);
    if (far)
        return launch_boundary_far(m, q, n, chi, w, label, classify, running, list, list_len, listed, partial_buf, call_n, s);
#define GWN_BSUM(KP, C, R) \
    launch_bsum_kp<KP, C, R>(m, q, n, chi, w, label, classify, list, list_len, listed, partial_buf, call_n, plain, s)
    if (m->cfg.fp64_cancel >= 0) {   // the default: cancelling terms in FP64
        const bool small = kq == 1 || kq == 2;   // 8 queries per thread: the queue holds 2-bit slots
        if (running) return small ? GWN_BSUM(1, true, true) : GWN_BSUM(2, true, true);
        return small ? GWN_BSUM(1, true, false) : GWN_BSUM(2, true, false);
    }
    switch (kq) {
        case 1:
        case 2: return running ? GWN_BSUM(1, false, true) : GWN_BSUM(1, false, false);
        case 8: return GWN_BSUM(4, false, false);
        default: return running ? GWN_BSUM(2, false, true) : GWN_BSUM(2, false, false);
    }
#undef GWN_BSUM
}

int64_t boundary_parts(const gwn_mesh *m, int64_t n, bool far) {
    if (far) return far_parts(m, n);
    const int kq = m->cfg.queries_per_thread > 0 ? m->cfg.queries_per_thread : 4;
    const bool cond = m->cfg.fp64_cancel >= 0;
    return direct_parts(m, n, kq <= 2 ? 1 : (kq == 8 && !cond ? 4 : 2), cond, false);
}

gwn_status launch_boundary_sum_list(const gwn_mesh *m, const float *q, int64_t n, const int32_t *chi, float *w,
                                    uint8_t *label, bool classify, int32_t *list, unsigned long long *list_len,
                                    SumOrder order, cudaStream_t s) {
    if (n <= 0) return GWN_OK;
    if (order == SumOrder::kCaller && far_pays(m, n)) {
        // the hierarchy wants neighbours in a warp: evaluate in spatial order, scatter back
        uint32_t *keys = nullptr, *perm = nullptr;
        float *qs = nullptr, *ws = nullptr;
        int32_t *cs = nullptr;
        uint8_t *ls = nullptr;
        gwn_status st = [&]() -> gwn_status {
            GWN_CUDA_TRY(dev_alloc(&keys, sizeof(uint32_t) * n, s));
            GWN_CUDA_TRY(dev_alloc(&perm, sizeof(uint32_t) * n, s));
            GWN_CUDA_TRY(dev_alloc(&qs, sizeof(float) * 3 * n, s));
            GWN_CUDA_TRY(dev_alloc(&ws, sizeof(float) * n, s));
            GWN_CUDA_TRY(dev_alloc(&cs, sizeof(int32_t) * n, s));
            if (label) GWN_CUDA_TRY(dev_alloc(&ls, n, s));
            return GWN_OK;
        }();
        if (st == GWN_OK && (st = order_queries(m, q, n, keys, perm, qs, s)) == GWN_OK &&
            (st = gather_i32(chi, perm, n, cs, s)) == GWN_OK &&
            (st = launch_boundary_sum_list(m, qs, n, cs, ws, ls, classify, list, list_len, SumOrder::kSpatial, s)) == GWN_OK &&
            (st = scatter_results(perm, n, ws, w, nullptr, nullptr, ls, label, s)) == GWN_OK && list)
            st = map_list(list, list_len, n, perm, s);
        for (void *p : {(void *)keys, (void *)perm, (void *)qs, (void *)ws, (void *)cs, (void *)ls})
            if (p) cudaFreeAsync(p, s);
        return st;
    }
    const size_t words = (size_t)((n + 31) / 32);
    unsigned *listed = nullptr;
    GWN_CUDA_TRY(dev_alloc(&listed, sizeof(unsigned) * words, s));
    GWN_CUDA_TRY(cudaMemsetAsync(listed, 0, sizeof(unsigned) * words, s));
    // without a caller list (no labels wanted), queries with more cancelling terms in
    // a tile than kCancelOwn still need their FP64 re-evaluation
    const bool own_list = list == nullptr;
    if (own_list) {
        GWN_CUDA_TRY(dev_alloc(&list, sizeof(int32_t) * n, s));
        GWN_CUDA_TRY(dev_alloc(&list_len, sizeof(unsigned long long), s));
        GWN_CUDA_TRY(cudaMemsetAsync(list_len, 0, sizeof(unsigned long long), s));
    }
    gwn_status st = boundary_sum_on(m, q, n, chi, w, label, classify, list, list_len, listed, nullptr, n,
                                    order == SumOrder::kSpatial && far_pays(m, n), order == SumOrder::kDirect, s);
    if (st == GWN_OK && own_list) st = launch_fp64_fix_list(m, q, chi, w, nullptr, list, list_len, s);
    cudaFreeAsync(listed, s);
    if (own_list) {
        cudaFreeAsync(list, s);
        cudaFreeAsync(list_len, s);
    }
    return st;
}

// The classify sequence on caller-provided scratch (allocates nothing): chi_tmp
// [n] int32, list [n] int32, list_len one zeroed counter, listed (n + 31) / 32
// zeroed words, partial n times boundary_parts(m, call_n, far) doubles (unused where
// that is 1), call_n the queries of the whole call.
gwn_status launch_classify_on_scratch(const gwn_mesh *m, const float *q, int64_t n, uint8_t *label, float *w,
                                      int32_t *chi_tmp, int32_t *list, unsigned long long *list_len,
                                      unsigned *listed, double *partial, int64_t call_n, bool far,
                                      cudaStream_t s) {
    if (n <= 0) return GWN_OK;
    // (the FP64 list and w are free until the boundary sum: the long walks' list)
    gwn_status st = chi_on(m, q, n, chi_tmp, list_len, list, reinterpret_cast<int32_t *>(w), s);
    if (st != GWN_OK) return st;
    if (long_walks(m, n)) GWN_CUDA_TRY(cudaMemsetAsync(list_len, 0, sizeof(unsigned long long), s));
    st = boundary_sum_on(m, q, n, chi_tmp, w, label, true, list, list_len, listed, partial, call_n, far, false, s);
    if (st != GWN_OK) return st;
    return launch_fp64_fix_list(m, q, chi_tmp, w, label, list, list_len, s);
}

// k_batch's dynamic shared memory: tile + 1 points, then per query slot an FP64
// sum and a fixed-point sum, then per warp one deferred-term queue of 64 KQ
// entries, then per warp a cancelling-term queue, its queries' counts and its own.
static size_t batch_smem(int kp, int tile_pts) {
    const size_t kq = 2 * (size_t)kp, threads = 256, warps = threads / 32;
    return sizeof(float4) * (tile_pts + 1) + (sizeof(double) + sizeof(long long)) * kq * threads +
           sizeof(unsigned) * (96 * kq + kCancelCap + 1) * warps;
}

template <int KP>
static gwn_status launch_batch_kp(int grid, int tile_pts, const BatchMesh *meshes, const BatchTile *tiles,
                                  const BatchItem *items, int64_t n_items, const float *q, int32_t *chi, double *acc,
                                  float *w, unsigned *tile_done, unsigned long long *head, int32_t *list,
                                  unsigned long long *list_len, unsigned *listed, cudaStream_t s) {
    const size_t smem = batch_smem(KP, tile_pts);
    if (smem > 48 * 1024)
        cudaFuncSetAttribute(k_batch<KP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k_batch<KP><<<grid, 256, smem, s>>>(meshes, tiles, items, n_items, q, chi, acc, w, tile_done, head, tile_pts,
                                        list, list_len, listed);
    GWN_LAUNCH_CHECK("k_batch");
    return GWN_OK;
}

gwn_status launch_batch_kernel(int kp, int grid, int tile_pts, const BatchMesh *meshes, const BatchTile *tiles,
                               const BatchItem *items, int64_t n_items, const float *q, int32_t *chi, double *acc,
                               float *w, unsigned *tile_done, unsigned long long *head, int32_t *list,
                               unsigned long long *list_len, unsigned *listed, cudaStream_t s) {
    ProfScope prof("batch", s);
    if (kp == 1)
        return launch_batch_kp<1>(grid, tile_pts, meshes, tiles, items, n_items, q, chi, acc, w, tile_done, head,
                                  list, list_len, listed, s);
    return launch_batch_kp<2>(grid, tile_pts, meshes, tiles, items, n_items, q, chi, acc, w, tile_done, head, list,
                              list_len, listed, s);
}

int batch_blocks_per_sm(int kp, int tile_pts) {
    int nb = 0;
    const size_t smem = batch_smem(kp == 1 ? 1 : 2, tile_pts);
    if (kp == 1) {
        if (smem > 48 * 1024)
            cudaFuncSetAttribute(k_batch<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_batch<1>, 256, smem);
    } else {
        if (smem > 48 * 1024)
            cudaFuncSetAttribute(k_batch<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_batch<2>, 256, smem);
    }
    return nb > 0 ? nb : 1;
}

gwn_status launch_batch_fp64_fix(const BatchMesh *meshes, const int64_t *mesh_off, int n_mesh, const float *q,
                                 const int32_t *chi, float *w, const int32_t *list,
                                 const unsigned long long *list_len, cudaStream_t s) {
    if (n_mesh <= 0) return GWN_OK;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    k_batch_fp64_fix<<<(unsigned)(sms > 0 ? 2 * sms : 128), 256, 0, s>>>(meshes, mesh_off, n_mesh, q, chi, w, list,
                                                                          list_len);
    GWN_LAUNCH_CHECK("k_batch_fp64_fix");
    return GWN_OK;
}

gwn_status launch_fp64_fix_list(const gwn_mesh *m, const float *q, const int32_t *chi, float *w, uint8_t *label,
                                const int32_t *list, const unsigned long long *list_len, cudaStream_t s) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    ProfScope prof("fp64_fix", s);
    k_fp64_fix<<<(unsigned)(sms > 0 ? 2 * sms : 128), 256, 0, s>>>(q, m->bpts, m->npts, chi, w, label, list,
                                                                    list_len, m->counters);
    GWN_LAUNCH_CHECK("k_fp64_fix");
    return GWN_OK;
}

gwn_status launch_direct(const gwn_mesh *m, const float *q, int64_t n, float *w, cudaStream_t s) {
    if (n <= 0) return GWN_OK;
    if (m->nt == 0) {
        GWN_CUDA_TRY(cudaMemsetAsync(w, 0, sizeof(float) * n, s));
        return GWN_OK;
    }
    constexpr int KP = 2;
    const int tile = 256;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t qblocks = (n + 256 * 2 * KP - 1) / (256 * 2 * KP);
    // about eight waves of two resident blocks per SM; a chunk of 128 triangles still
    // pays for its partial sums (64 queries x 40k triangles: 300 us in chunks of 1024)
    int64_t chunks = (16 * (int64_t)(sms > 0 ? sms : 148) + qblocks - 1) / qblocks;
    chunks = std::max<int64_t>(1, std::min<int64_t>(chunks, (m->nt + 127) / 128));
    chunks = std::min<int64_t>(chunks, 65535);
    const int64_t chunk_len = (m->nt + chunks - 1) / chunks;
    double *partial = nullptr;
    if (chunks > 1) GWN_CUDA_TRY(dev_alloc(&partial, sizeof(double) * chunks * n, s));
    {
        ProfScope prof("direct_sum", s);
        dim3 grid((unsigned)qblocks, (unsigned)chunks);
        k_direct<KP><<<grid, 256, (sizeof(float4) * 3 + sizeof(float)) * tile, s>>>(q, n, m->tri9, m->nt, tile, chunk_len, w, partial);
        if (partial) k_direct_reduce<<<grid_for(n, 256), 256, 0, s>>>(partial, n, (int)chunks, w);
    }
    if (partial) cudaFreeAsync(partial, s);
    GWN_LAUNCH_CHECK("k_direct");
    return GWN_OK;
}

}  // namespace gwn
