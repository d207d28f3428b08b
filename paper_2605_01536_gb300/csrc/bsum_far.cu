// Boundary sum over the boundary hierarchy (farfield.cuh): each warp walks the
// preorder nodes for its 64 queries (a float2 pair per lane) together.  A query takes a node's expansion
// when it lies outside the node's error radius and its ray misses the node's box,
// and the edges of a leaf one by one otherwise; a query that has taken a node
// skips its subtree (resume).  The decisions, the order of a query's sums and the
// grouping of its terms depend on the query and the mesh alone, so its result does
// not depend on the queries beside it.
//
// Bound by the FP32 pipe while its walks last (a query of the soup8 mesh, 202k
// boundary points, takes about 270 expansions of 250 paired operations and 360 edges;
// a warp takes the union over its queries, 1.8 times as many), and by the walks'
// latency where warps are few, hence the split over subtrees.  96 registers, 20 warps
// per SM.  Boundary sum, direct -> hierarchy: soup8 with 2M queries 383.5 -> 11.4 ms,
// 200k 42.1 -> 2.3 ms; soup6 (12k points) with 50k queries 0.80 -> 0.31 ms.  Maximum
// error against FP64 on soup8 1.3e-6 -> 2.0e-7 (fewer FP32 terms).  Four queries per
// lane instead of two: equal at 2M queries, 15% slower at 200k.
#include <algorithm>

#include "bterms.cuh"
#include "farfield.cuh"

namespace gwn {

namespace {

constexpr int kFarThreads = 128;

// Value of a node's expansion (in units of the sum of atan2 terms) for KP query
// pairs at (x, y, z) from its centre in units of its radius.
template <int KP>
__device__ __forceinline__ void far_eval(const float *__restrict__ coef, const float2 (&x)[KP], const float2 (&y)[KP],
                                         const float2 (&z)[KP], float2 (&phi)[KP]) {
    constexpr int P = kFarP;
    float2 Z[KP], nU[KP], ex[KP], ey[KP], er[KP], ei[KP];
#pragma unroll
    for (int k = 0; k < KP; ++k) {
        const float2 r2 = fma2(x[k], x[k], fma2(y[k], y[k], mul2(z[k], z[k])));
        const float2 ir = make_float2(sfu_rsqrt(r2.x), sfu_rsqrt(r2.y));
        const float2 U = mul2(ir, ir);
        nU[k] = neg2(U);
        Z[k] = mul2(z[k], U);
        ex[k] = mul2(x[k], U);
        ey[k] = mul2(y[k], U);
        er[k] = ir;
        ei[k] = bc2(0.f);
    }
    const float2 *c2 = reinterpret_cast<const float2 *>(coef);
    float2 A[KP], B[KP], t1[KP], t2[KP];
    // column m = 0: real coefficients of l = 1..P
#pragma unroll
    for (int k = 0; k < KP; ++k) { t2[k] = bc2(0.f); t1[k] = bc2(1.f); A[k] = bc2(0.f); }
#pragma unroll
    for (int l = 1; l <= P; l += 2) {
        const float2 c = __ldg(c2 + (l - 1) / 2);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
#pragma unroll
            for (int k = 0; k < KP; ++k) {
                const float2 t = l + h == 1 ? Z[k] : fma2(Z[k], t1[k], mul2(mul2(bc2(far_beta(l + h, 0)), nU[k]), t2[k]));
                t2[k] = t1[k];
                t1[k] = t;
                A[k] = fma2(bc2(h ? c.y : c.x), t, A[k]);
            }
        }
    }
#pragma unroll
    for (int k = 0; k < KP; ++k) phi[k] = mul2(er[k], A[k]);
#pragma unroll
    for (int m = 1; m <= P; ++m) {
#pragma unroll
        for (int k = 0; k < KP; ++k) {
            const float2 nr = fma2(er[k], ex[k], neg2(mul2(ei[k], ey[k])));
            ei[k] = fma2(er[k], ey[k], mul2(ei[k], ex[k]));
            er[k] = nr;
        }
#pragma unroll
        for (int l = m; l <= P; ++l) {
            const float2 c = __ldg(c2 + far_col(m) / 2 + (l - m));
#pragma unroll
            for (int k = 0; k < KP; ++k) {
                if (l == m) {
                    t1[k] = bc2(1.f);
                    A[k] = bc2(c.x);
                    B[k] = bc2(c.y);
                } else {
                    const float2 t = l == m + 1 ? Z[k] : fma2(Z[k], t1[k], mul2(mul2(bc2(far_beta(l, m)), nU[k]), t2[k]));
                    t2[k] = t1[k];
                    t1[k] = t;
                    A[k] = fma2(bc2(c.x), t, A[k]);
                    B[k] = fma2(bc2(c.y), t, B[k]);
                }
            }
        }
#pragma unroll
        for (int k = 0; k < KP; ++k) phi[k] = fma2(er[k], A[k], fma2(ei[k], B[k], phi[k]));
    }
}

// The warp's queue of ill-conditioned terms (bterms.cuh): entry
// (edge of the leaf) << 7 | (query slot) << 5 | lane, evaluated in FP64 after the leaf.  It
// has room for kFarOwn terms of every query; a query with more in one leaf (several loops
// on one another) is listed for a full FP64 re-evaluation, so that its result does not
// depend on its neighbours' terms.  (A call that empties the queue inside the edge loop
// instead spills there: 2M queries on soup8 12.3 -> 13.4 ms.)
constexpr unsigned kFarOwn = 4;
struct FarQueue {
    unsigned *queue;
    int *count;
    long long *fix;   // fixed-point sums, fix[slot 32 + lane]
};

__device__ __noinline__ void far_drain(const FarQueue fq, const float4 *__restrict__ pts, const float *__restrict__ q,
                                       unsigned long long *counters) {
    const int lane = threadIdx.x & 31;
    const int count = *fq.count;
    for (int r = lane; r < count; r += 32) {
        const unsigned e = fq.queue[r];
        const int slot = (int)(e & 127u), j = (int)(e >> 7);
        const double t = edge_angle64(pts[j], pts[j + 1], q[3 * slot], q[3 * slot + 1], q[3 * slot + 2], counters);
        atomicAdd(reinterpret_cast<unsigned long long *>(fq.fix + slot), (unsigned long long)__double2ll_rn(t * kFixScale64));
    }
    if (lane == 0 && count > 0) atomicAdd(&counters[CNT_CANCEL], (unsigned long long)count);
    __syncwarp();
    if (lane == 0) *fq.count = 0;
    __syncwarp();
}

template <bool Running>
__global__ void __launch_bounds__(kFarThreads, 5)
    k_boundary_far(const float *__restrict__ q, int64_t first, int64_t n, const FarNode *__restrict__ nodes,
                   const int32_t *__restrict__ roots, int nroots, double *__restrict__ partial,
                   const float *__restrict__ coef, const float4 *__restrict__ pts, const int32_t *__restrict__ chi,
                   float *__restrict__ w, uint8_t *__restrict__ label, int classify, float margin,
                   int32_t *__restrict__ list, unsigned long long *__restrict__ list_len,
                   unsigned *__restrict__ listed, unsigned long long *__restrict__ counters) {
    constexpr int KP = 1, KQ = 2 * KP, kWarps = kFarThreads / 32;
    __shared__ long long s_fix[kWarps][32 * KQ];
    __shared__ unsigned s_queue[kWarps][32 * KQ * kFarOwn];
    __shared__ int s_count[kWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t qbase = first + ((int64_t)blockIdx.x * kWarps + warp) * (32 * KQ);   // queries [first, n)
    if (qbase >= n) return;
    const FarQueue fq{s_queue[warp], &s_count[warp], s_fix[warp]};
    float2 nqx[KP], nqy[KP], nqz[KP], part[KP], comp[KP];
    double acc[KQ];
    int resume[KQ];   // first preorder node the query has not skipped
#pragma unroll
    for (int k = 0; k < KQ; ++k) {
        const int64_t idx = qbase + lane + 32 * k;
        const bool ok = idx < n;
        const float x = ok ? -q[3 * idx] : 0.f, y = ok ? -q[3 * idx + 1] : 0.f, z = ok ? -q[3 * idx + 2] : 0.f;
        if (k & 1) { nqx[k >> 1].y = x; nqy[k >> 1].y = y; nqz[k >> 1].y = z; }
        else       { nqx[k >> 1].x = x; nqy[k >> 1].x = y; nqz[k >> 1].x = z; }
        resume[k] = ok ? 0 : 0x7fffffff;
        acc[k] = 0.0;
        fq.fix[32 * k + lane] = 0;
    }
    if (lane == 0) *fq.count = 0;
#pragma unroll
    for (int k = 0; k < KP; ++k) part[k] = comp[k] = bc2(0.f);
    __syncwarp();

    // this block row's subtrees; each one's sum is closed in FP64 before the next
    const int root0 = (int)((int64_t)nroots * blockIdx.y / gridDim.y),
              root1 = (int)((int64_t)nroots * (blockIdx.y + 1) / gridDim.y);
    int root = root0, node = 0, end = 0;
    while (true) {
        if (node >= end) {
#pragma unroll
            for (int k = 0; k < KQ; ++k)
                acc[k] += k & 1 ? (double)part[k >> 1].y + (double)comp[k >> 1].y
                                : (double)part[k >> 1].x + (double)comp[k >> 1].x;
#pragma unroll
            for (int k = 0; k < KP; ++k) part[k] = comp[k] = bc2(0.f);
            if (root == root1) break;
            node = __ldg(roots + root);
            ++root;
            end = __ldg(&nodes[node].skip);
        }
        const float4 *np = reinterpret_cast<const float4 *>(nodes + node);
        const float4 h0 = __ldg(np), h1 = __ldg(np + 1), h2 = __ldg(np + 2);
        const int skip = __float_as_int(h2.z), nchord = __float_as_int(h2.w);
        float2 x[KP], y[KP], z[KP];
        unsigned take = 0, into = 0;   // query slots that take the expansion / need the node's parts
#pragma unroll
        for (int k = 0; k < KP; ++k) {
            x[k] = add2(bc2(-h0.x), neg2(nqx[k]));
            y[k] = add2(bc2(-h0.y), neg2(nqy[k]));
            z[k] = add2(bc2(-h0.z), neg2(nqz[k]));
            const float2 r2 = fma2(x[k], x[k], fma2(y[k], y[k], mul2(z[k], z[k])));
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float qx = -(h ? nqx[k].y : nqx[k].x), qy = -(h ? nqy[k].y : nqy[k].x),
                            qz = -(h ? nqz[k].y : nqz[k].x);
                const bool active = node >= resume[2 * k + h];
                const bool hit = qx >= h1.x && qx <= h1.y && qy >= h1.z && qy <= h1.w && qz <= h2.x;
                const bool far = (h ? r2.y : r2.x) > h0.w && !hit;
                if (active) {
                    if (far) { take |= 1u << (2 * k + h); resume[2 * k + h] = skip; }
                    else into |= 1u << (2 * k + h);
                }
            }
        }
        if (__any_sync(0xffffffffu, take != 0)) {
            float2 v[KP];
#pragma unroll
            for (int k = 0; k < KP; ++k) {
                x[k] = mul2(x[k], bc2(h2.y));
                y[k] = mul2(y[k], bc2(h2.y));
                z[k] = mul2(z[k], bc2(h2.y));
            }
            far_eval<KP>(coef + (int64_t)node * kFarCoef, x, y, z, v);
            for (int c = 0; c < nchord; ++c) {   // the chords that close the node's cut loops
                const int4 ch = __ldg(reinterpret_cast<const int4 *>(np + 4));
                const float4 Pa = __ldg(pts + (c ? ch.z : ch.x)), Pb = __ldg(pts + (c ? ch.w : ch.y));
#pragma unroll
                for (int k = 0; k < KP; ++k) {
                    const PointRel2 A = point_rel2(Pa, nqx[k], nqy[k], nqz[k]), B = point_rel2(Pb, nqx[k], nqy[k], nqz[k]);
                    const float2 en = fma2(A.ay, B.ax, neg2(mul2(A.ax, B.ay)));
                    const float2 ed = fma2(A.h, B.h, fma2(A.ax, B.ax, mul2(A.ay, B.ay)));
                    v[k] = add2(v[k], fast_atan2_2(en, ed));
                }
            }
#pragma unroll
            for (int k = 0; k < KP; ++k) {
                const float2 a = make_float2(take >> (2 * k) & 1u ? v[k].x : 0.f, take >> (2 * k + 1) & 1u ? v[k].y : 0.f);
                two_sum_acc2(part[k], comp[k], a);
            }
        }
        if (!__any_sync(0xffffffffu, into != 0)) {
            node = skip;
            continue;
        }
        if (skip == node + 1) {   // a leaf: its edges one by one
            const float4 h3 = __ldg(np + 3);
            const int begin = __float_as_int(h3.x), count = __float_as_int(h3.y);
            if (count == 0) {
                ++node;
                continue;
            }
            const float4 *lp = pts + begin;
            float2 re[KP], im[KP];
            int g = 0;
            unsigned own = 0;   // queued terms of this leaf, a byte per query slot
#pragma unroll
            for (int k = 0; k < KP; ++k) { re[k] = bc2(1.f); im[k] = bc2(0.f); }
            auto close = [&]() {
#pragma unroll
                for (int k = 0; k < KP; ++k) {
                    const float2 t = fast_atan2_2(im[k], re[k]);
                    two_sum_acc2(part[k], comp[k], make_float2(into >> (2 * k) & 1u ? t.x : 0.f,
                                                               into >> (2 * k + 1) & 1u ? t.y : 0.f));
                    re[k] = bc2(1.f);
                    im[k] = bc2(0.f);
                }
                g = 0;
            };
            PointRel2 A[KP], B[KP];
            float4 Pa = __ldg(lp);
#pragma unroll
            for (int k = 0; k < KP; ++k) A[k] = point_rel2(Pa, nqx[k], nqy[k], nqz[k]);
            for (int j = 0; j < count; ++j) {
                if (Pa.w == 0.f) {   // a loop's closing point: the next one starts another loop
                    if (j + 1 < count) {
                        Pa = __ldg(lp + j + 1);
#pragma unroll
                        for (int k = 0; k < KP; ++k) A[k] = point_rel2(Pa, nqx[k], nqy[k], nqz[k]);
                    }
                    continue;
                }
                const float4 Pb = __ldg(lp + j + 1);
                unsigned fail = 0;
                float2 en[KP], ed[KP];
#pragma unroll
                for (int k = 0; k < KP; ++k) {
                    B[k] = point_rel2(Pb, nqx[k], nqy[k], nqz[k]);
                    en[k] = fma2(A[k].ay, B[k].ax, neg2(mul2(A[k].ax, B[k].ay)));
                    ed[k] = fma2(A[k].h, B[k].h, fma2(A[k].ax, B[k].ax, mul2(A[k].ay, B[k].ay)));
                    bool px, py;
                    float2 nre, nim;
                    if constexpr (Running) {
                        nre = fma2(re[k], ed[k], neg2(mul2(im[k], en[k])));
                        nim = fma2(re[k], en[k], mul2(im[k], ed[k]));
                        px = !(ed[k].x <= kMinD) && !(nre.x <= 0.f);
                        py = !(ed[k].y <= kMinD) && !(nre.y <= 0.f);
                    } else {
                        const float2 v = fma2(bc2(kTanGroup), ed[k], neg2(make_float2(fabsf(en[k].x), fabsf(en[k].y))));
                        px = !(v.x <= kAccept);
                        py = !(v.y <= kAccept);
                    }
                    {   // ill-conditioned terms leave the product (cancels(), paired)
                        const float2 t = mul2(bc2(kCancel), mul2(A[k].h, B[k].h));
                        const float2 m2 = fma2(en[k], en[k], mul2(ed[k], ed[k])), t2 = mul2(t, t);
                        px = px && !(m2.x < t2.x);
                        py = py && !(m2.y < t2.y);
                    }
                    if constexpr (Running) {
                        re[k] = make_float2(px ? nre.x : re[k].x, py ? nre.y : re[k].y);
                        im[k] = make_float2(px ? nim.x : im[k].x, py ? nim.y : im[k].y);
                    } else {
                        const float2 fd = make_float2(px ? ed[k].x : 1.f, py ? ed[k].y : 1.f);
                        const float2 fn = make_float2(px ? en[k].x : 0.f, py ? en[k].y : 0.f);
                        nre = fma2(re[k], fd, neg2(mul2(im[k], fn)));
                        nim = fma2(re[k], fn, mul2(im[k], fd));
                        re[k] = nre;
                        im[k] = nim;
                    }
                    fail |= (px ? 0u : 1u << (2 * k)) | (py ? 0u : 2u << (2 * k));
                }
                fail &= into;
                if (fail) {
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
                        if (cancels(nk, dk, a.h, b.h)) {
                            if ((own >> (8 * k) & 255u) < kFarOwn) {
                                own += 1u << (8 * k);
                                fq.queue[atomicAdd(fq.count, 1)] = (unsigned)j << 7 | (unsigned)k << 5 | (unsigned)lane;
                                continue;
                            }
                            list_query(qbase + lane + 32 * k, list, list_len, listed);
                        }
                        const float t = fallback_term(nk, dk, a, b, Pa, Pb, qx, qy, qz, counters);
                        if (hi) two_sum_acc(part[kp].y, comp[kp].y, t);
                        else two_sum_acc(part[kp].x, comp[kp].x, t);
                    }
                }
                if (++g == GROUP) close();
                Pa = Pb;
#pragma unroll
                for (int k = 0; k < KP; ++k) A[k] = B[k];
            }
            if (g > 0) close();
            if (cancel_count(fq.count) > 0) far_drain(fq, lp, q + 3 * qbase, counters);
        }
        ++node;
    }
    __syncwarp();
#pragma unroll
    for (int k = 0; k < KQ; ++k) {
        const int64_t idx = qbase + lane + 32 * k;
        if (idx >= n) continue;
        const double sum = acc[k] + (double)fq.fix[32 * k + lane] * kFixUnit;
        if (partial) {
            partial[(int64_t)blockIdx.y * (n - first) + (idx - first)] = sum;
            continue;
        }
        const double wv = (double)chi[idx] + sum * kInv2Pi;
        w[idx] = (float)wv;
        if (classify) {
            label[idx] = wv > 0.5 ? 1 : 0;
            if (fabs(wv - 0.5) <= (double)margin) list_query(idx, list, list_len, listed);
        }
    }
}

}  // namespace

// Calls of the default schedule (an explicit queries_per_thread, boundary_tile or
// fp64_cancel = -1 asks for the direct sum's own) large enough to be ordered in space.  The
// limit is the order's; direct / hierarchy where an order and the hierarchy begin at 1,024
// queries, query: soup6 (12k points) 3k queries 133 / 158 us, 16k 234 / 268; soup7 (51k) 6k
// 321 / 474, 12k 509 / 500, 16k 656 / 532; soup8 (203k) 6k 915 / 1322, 12k 1614 / 1355, 16k
// 2103 / 1392; gradient: soup6 6k 263 / 183, soup7 582 / 502, soup8 1936 / 1783, 12k 3850 / 1834.
bool far_pays_gradient(const gwn_mesh *m, int64_t n) {
    return m->far_nodes && n >= kOrderMinQueries && m->cfg.queries_per_thread == 0 && m->cfg.boundary_tile == 0 &&
           m->cfg.fp64_cancel >= 0;
}

// The boundary sum, moreover, where the direct sum has 5e9 operations to do (about 220
// us): below, the walks' latency shows (12k points of small holes: 16k queries 180
// against 161 us, 25k 216 against 221).
bool far_pays(const gwn_mesh *m, int64_t n) {
    return m->far_sum && far_pays_gradient(m, n) && (double)n * direct_cost(m) >= 5e9;
}

// One walk is a serial chain of about 600 nodes: split it over the subtrees until there
// are 320 blocks per SM (soup8, 200k queries: unsplit 4.0 ms, 16 parts 2.6, 64 parts 2.3;
// 2M queries: 4 parts 11.4, 64 parts 11.5)
int64_t far_parts(const gwn_mesh *m, int64_t n) {
    const int64_t blocks = (n + kFarThreads * 2 - 1) / (kFarThreads * 2);
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t parts = (320 * (int64_t)(sms > 0 ? sms : 148) + blocks - 1) / blocks;
    return std::max<int64_t>(1, std::min<int64_t>(parts, m->far_nroots));
}

gwn_status launch_boundary_far(const gwn_mesh *m, const float *q, int64_t n, const int32_t *chi, float *w,
                               uint8_t *label, bool classify, bool running, int32_t *list,
                               unsigned long long *list_len, unsigned *listed, double *partial_buf,
                               int64_t call_n, cudaStream_t s) {
    const float margin = m->cfg.classify_margin > 0.f ? m->cfg.classify_margin : 1e-4f;
    const int64_t split = far_parts(m, call_n);
    double *partial = split > 1 ? partial_buf : nullptr;
    const bool own = split > 1 && !partial_buf;
    const int64_t slice = own ? query_slice(n, sizeof(double) * split) : n;
    if (own) GWN_CUDA_TRY(dev_alloc(&partial, sizeof(double) * split * slice, s));
#define GWN_FAR(R)                                                                                                    \
    k_boundary_far<R><<<grid, kFarThreads, 0, s>>>(q, at, end, m->far_nodes, m->far_roots, m->far_nroots, partial,           \
                                                   m->far_coef, m->far_pts, chi, w, label, classify ? 1 : 0, margin,   \
                                                   list, list_len, listed, m->counters)
    for (int64_t at = 0; at < n; at += slice) {
        const int64_t end = std::min(n, at + slice);
        const dim3 grid((unsigned)((end - at + kFarThreads * 2 - 1) / (kFarThreads * 2)), (unsigned)split);
        if (running) GWN_FAR(true);
        else GWN_FAR(false);
        note_launches(1);
        if (partial)
            launch_boundary_combine(partial, at, end - at, (int)split, chi, w, label, classify, margin, list, list_len,
                                    listed, s);
    }
#undef GWN_FAR
    if (own) cudaFreeAsync(partial, s);
    GWN_LAUNCH_CHECK("k_boundary_far");
    return GWN_OK;
}

}  // namespace gwn
