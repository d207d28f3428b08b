// Gradient of the winding number with respect to the query point (Supp. S4,
// Algorithm 3).  The crossing count is piecewise constant, so only the boundary
// terms carry a gradient:
//   grad w = (1/4pi) sum_{(a,b) in dM} (c_n g_n + c_d g_d),
//   c_n = 2 d / (n^2 + d^2),  c_d = -2 n / (n^2 + d^2),
// with n, d the (unnormalised) van Oosterom-Strackee pair of the edge seen from
// the query and g_n = dn/dp, g_d = dd/dp.  With x1 = -z and r0 = a - p,
// r1 = b - p, l = |r|, v = r / l, h = l - r_z (= l (1 + x1.v)):
//   n   = r0_y r1_x - r0_x r1_y
//   d   = h0 h1 + r0_x r1_x + r0_y r1_y
//   g_n = (b_y - a_y, a_x - b_x, 0)                 (-(r1 x x1 + x1 x r0))
//   g_d = (l0 + l1) z - (r0 + r1 + h1 v0 + h0 v1)    (-(t1 + t2) of Algorithm 3)
// h is computed as (r_x^2 + r_y^2) / (l + |r_z|) + (|r_z| - r_z), which avoids the
// cancellation of l - r_z for a point nearly straight above the query.  A term
// whose n^2 + d^2 underflows (the query on the boundary curve, or a boundary
// point exactly straight above or below it, where the term is singular) is
// skipped and counted.
//
// Layout and schedule follow the boundary-sum kernel: each thread holds 2 KP
// queries as float2 pairs (one Blackwell paired instruction per step for two
// queries), the chained boundary points stream through shared memory in tiles,
// FP32 partial sums are flushed into FP64 accumulators (shared memory) every
// 64 edges, and small query batches split the boundary into chunks whose FP64
// partials are added in chunk order.
#include <algorithm>

#include "farfield.cuh"
#include "gwn_internal.cuh"
#include "fp32x2.cuh"

namespace gwn {

namespace {

constexpr double kInv4Pi = 0.079577471545947667884;
constexpr int kGradThreads = 128;
constexpr int kFlushEdges = 64;
constexpr float kMinModulus2 = 1e-30f;

// Per-point data of two queries: r = P - q, l = |r|, v = r / l, h = l - r_z.
struct GradPoint2 {
    float2 rx, ry, rz, l, h, vx, vy, vz;
};

__device__ __forceinline__ GradPoint2 grad_point2(float4 P, float2 nqx, float2 nqy, float2 nqz) {
    GradPoint2 g;
    g.rx = add2(bc2(P.x), nqx);
    g.ry = add2(bc2(P.y), nqy);
    g.rz = add2(bc2(P.z), nqz);
    const float2 s = fma2(g.rx, g.rx, mul2(g.ry, g.ry));
    const float2 r2 = add2(fma2(g.rz, g.rz, s), bc2(1e-37f));   // > 0 for a coincident point
    const float2 il = make_float2(sfu_rsqrt(r2.x), sfu_rsqrt(r2.y));
    g.l = mul2(r2, il);
    g.vx = mul2(g.rx, il);
    g.vy = mul2(g.ry, il);
    g.vz = mul2(g.rz, il);
    const float2 az = make_float2(fabsf(g.rz.x), fabsf(g.rz.y));
    const float2 den = add2(g.l, az);
    g.h = fma2(s, make_float2(sfu_rcp(den.x), sfu_rcp(den.y)), add2(az, neg2(g.rz)));
    return g;
}

// Adds the edge term (point A -> point B) of two queries to (gx, gy, gz).
// ex, ey: the query-independent edge vector a - b.  skipped counts lanes whose
// term was dropped as singular (count_x, count_y: of the first and second query).
__device__ __forceinline__ void grad_edge2(const GradPoint2 &A, const GradPoint2 &B, float ex, float ey, float2 &gx,
                                           float2 &gy, float2 &gz, unsigned &skipped, bool count_x = true,
                                           bool count_y = true) {
    const float2 n = fma2(A.ry, B.rx, neg2(mul2(A.rx, B.ry)));
    const float2 d = fma2(A.h, B.h, fma2(A.rx, B.rx, mul2(A.ry, B.ry)));
    const float2 m2 = fma2(n, n, mul2(d, d));
    const bool okx = m2.x > kMinModulus2, oky = m2.y > kMinModulus2;
    skipped += (okx || !count_x ? 0u : 1u) + (oky || !count_y ? 0u : 1u);
    const float2 t = make_float2(okx ? 2.f * sfu_rcp(m2.x) : 0.f, oky ? 2.f * sfu_rcp(m2.y) : 0.f);
    const float2 cn = mul2(d, t);
    const float2 cd = neg2(mul2(n, t));
    // u = r0 + r1 + h1 v0 + h0 v1, so that g_d = (l0 + l1) z - u
    const float2 ux = fma2(A.h, B.vx, fma2(B.h, A.vx, add2(A.rx, B.rx)));
    const float2 uy = fma2(A.h, B.vy, fma2(B.h, A.vy, add2(A.ry, B.ry)));
    const float2 uz = fma2(A.h, B.vz, fma2(B.h, A.vz, add2(A.rz, B.rz)));
    // c_n g_n + c_d g_d with g_n = (-e_y, e_x, 0)
    gx = add2(gx, neg2(fma2(cn, bc2(ey), mul2(cd, ux))));
    gy = fma2(cn, bc2(ex), add2(gy, neg2(mul2(cd, uy))));
    gz = fma2(cd, add2(add2(A.l, B.l), neg2(uz)), gz);
}

template <int KP>
__global__ void __launch_bounds__(kGradThreads) k_gradient(const float *__restrict__ q, int64_t n,
                                                           const float4 *__restrict__ pts, int64_t npts, int tile,
                                                           int64_t chunk_len, double *__restrict__ partial,
                                                           float *__restrict__ grad,
                                                           unsigned long long *__restrict__ counters) {
    extern __shared__ float4 s_pts[];   // tile + 1 points, then 3 x 2 KP x blockDim doubles
    double *s_acc = reinterpret_cast<double *>(s_pts + tile + 1);
    constexpr int KQ = 2 * KP;
    const int64_t base = (int64_t)blockIdx.x * blockDim.x * KQ + threadIdx.x;
    const int64_t e_begin = (int64_t)blockIdx.y * chunk_len;
    const int64_t e_end = min(npts - 1, e_begin + chunk_len);   // edge start points
    float2 nqx[KP], nqy[KP], nqz[KP];
#pragma unroll
    for (int k = 0; k < KQ; ++k) {
        const int64_t idx = base + (int64_t)k * blockDim.x;
        const bool ok = idx < n;
        // queries past n sit far away (their n^2 + d^2 overflows to +inf, so they are
        // never counted as singular); their results are discarded
        const float x = ok ? -q[3 * idx] : 1e15f, y = ok ? -q[3 * idx + 1] : 1e15f, z = ok ? -q[3 * idx + 2] : 1e15f;
        if (k & 1) { nqx[k >> 1].y = x; nqy[k >> 1].y = y; nqz[k >> 1].y = z; }
        else       { nqx[k >> 1].x = x; nqy[k >> 1].x = y; nqz[k >> 1].x = z; }
    }
#pragma unroll
    for (int k = 0; k < 3 * KQ; ++k) s_acc[k * blockDim.x + threadIdx.x] = 0.0;
    float2 gx[KP], gy[KP], gz[KP];
#pragma unroll
    for (int k = 0; k < KP; ++k) gx[k] = gy[k] = gz[k] = bc2(0.f);
    unsigned skipped = 0;
    int since_flush = 0;
    auto flush = [&]() {
#pragma unroll
        for (int k = 0; k < KP; ++k) {
            double *a = s_acc + (6 * k) * blockDim.x + threadIdx.x;
            a[0 * blockDim.x] += (double)gx[k].x;
            a[1 * blockDim.x] += (double)gy[k].x;
            a[2 * blockDim.x] += (double)gz[k].x;
            a[3 * blockDim.x] += (double)gx[k].y;
            a[4 * blockDim.x] += (double)gy[k].y;
            a[5 * blockDim.x] += (double)gz[k].y;
            gx[k] = gy[k] = gz[k] = bc2(0.f);
        }
        since_flush = 0;
    };
    for (int64_t t0 = e_begin; t0 < e_end; t0 += tile) {
        const int cnt = (int)min((int64_t)tile, e_end - t0);
        __syncthreads();
        for (int i = threadIdx.x; i <= cnt; i += blockDim.x) s_pts[i] = __ldg(pts + t0 + i);
        __syncthreads();
        GradPoint2 ga[KP];
#pragma unroll
        for (int k = 0; k < KP; ++k) ga[k] = grad_point2(s_pts[0], nqx[k], nqy[k], nqz[k]);
        for (int j = 0; j < cnt; ++j) {
            const float4 Pa = s_pts[j], Pb = s_pts[j + 1];
            GradPoint2 gb[KP];
#pragma unroll
            for (int k = 0; k < KP; ++k) gb[k] = grad_point2(Pb, nqx[k], nqy[k], nqz[k]);
            if (Pa.w != 0.f) {
                const float ex = Pa.x - Pb.x, ey = Pa.y - Pb.y;
#pragma unroll
                for (int k = 0; k < KP; ++k) grad_edge2(ga[k], gb[k], ex, ey, gx[k], gy[k], gz[k], skipped);
                if (++since_flush == kFlushEdges) flush();
            }
#pragma unroll
            for (int k = 0; k < KP; ++k) ga[k] = gb[k];
        }
    }
    flush();
    if (skipped) atomicAdd(&counters[CNT_GRAD_SKIPPED], (unsigned long long)skipped);
#pragma unroll
    for (int k = 0; k < KQ; ++k) {
        const int64_t idx = base + (int64_t)k * blockDim.x;
        if (idx >= n) continue;
        const int kp = k >> 1, lane = k & 1;
        const double *a = s_acc + (6 * kp + 3 * lane) * blockDim.x + threadIdx.x;
        for (int c = 0; c < 3; ++c) {
            const double v = a[c * blockDim.x];
            if (partial) partial[((int64_t)blockIdx.y * n + idx) * 3 + c] = v;
            else grad[3 * idx + c] = (float)(v * kInv4Pi);
        }
    }
}

// place: the queries' places in grad, or NULL: as they come
__global__ void k_gradient_combine(const double *__restrict__ partial, const uint32_t *__restrict__ place, int64_t n,
                                   int chunks, double scale, float *__restrict__ grad) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 3 * n) return;
    double s = 0.0;
    for (int c = 0; c < chunks; ++c) s += partial[(int64_t)c * 3 * n + i];
    const int64_t o = place ? 3 * (int64_t)place[i / 3] + i % 3 : i;
    grad[o] = (float)(s * scale);
}

// Gradient of a node's expansion for two queries at (x, y, z) from its centre in
// units of its radius, in those units (far_eval in three components).
__device__ __forceinline__ void far_grad_eval(const float *__restrict__ gcoef, float2 x, float2 y, float2 z, float2 &gx,
                                              float2 &gy, float2 &gz) {
    constexpr int L = kFarP + 1, kComp = kFarGradCoef / 3;
    const float2 r2 = fma2(x, x, fma2(y, y, mul2(z, z)));
    const float2 ir = make_float2(sfu_rsqrt(r2.x), sfu_rsqrt(r2.y));
    const float2 U = mul2(ir, ir), nU = neg2(U), Z = mul2(z, U), ex = mul2(x, U), ey = mul2(y, U);
    const float2 *cx = reinterpret_cast<const float2 *>(gcoef), *cy = reinterpret_cast<const float2 *>(gcoef + kComp),
                 *cz = reinterpret_cast<const float2 *>(gcoef + 2 * kComp);
    float2 er = ir, ei = bc2(0.f);
    {   // column 0, degrees 2..L: T_0 = 1, T_1 = Z
        float2 t2 = bc2(1.f), t1 = Z, ax = bc2(0.f), ay = bc2(0.f), az = bc2(0.f);
#pragma unroll
        for (int l = 2; l <= L; ++l) {
            const float2 t = fma2(Z, t1, mul2(mul2(bc2(far_beta(l, 0)), nU), t2));
            t2 = t1;
            t1 = t;
            const int i = (l - 2) / 2, h = (l - 2) & 1;
            const float2 vx = __ldg(cx + i), vy = __ldg(cy + i), vz = __ldg(cz + i);
            ax = fma2(bc2(h ? vx.y : vx.x), t, ax);
            ay = fma2(bc2(h ? vy.y : vy.x), t, ay);
            az = fma2(bc2(h ? vz.y : vz.x), t, az);
        }
        gx = mul2(er, ax);
        gy = mul2(er, ay);
        gz = mul2(er, az);
    }
#pragma unroll
    for (int m = 1; m <= L; ++m) {
        const float2 nr = fma2(er, ex, neg2(mul2(ei, ey)));
        ei = fma2(er, ey, mul2(ei, ex));
        er = nr;
        float2 t1 = bc2(1.f), t2 = bc2(0.f);
        float2 ax = bc2(0.f), bx = bc2(0.f), ay = bc2(0.f), by = bc2(0.f), az = bc2(0.f), bz = bc2(0.f);
#pragma unroll
        for (int l = m; l <= L; ++l) {
            if (l > m) {
                const float2 t = l == m + 1 ? Z : fma2(Z, t1, mul2(mul2(bc2(far_beta(l, m)), nU), t2));
                t2 = t1;
                t1 = t;
            }
            if (l < 2) continue;
            const int i = kFarP / 2 + far_grad_col(m) + (l - far_grad_first(m));
            const float2 vx = __ldg(cx + i), vy = __ldg(cy + i), vz = __ldg(cz + i);
            ax = fma2(bc2(vx.x), t1, ax);
            bx = fma2(bc2(vx.y), t1, bx);
            ay = fma2(bc2(vy.x), t1, ay);
            by = fma2(bc2(vy.y), t1, by);
            az = fma2(bc2(vz.x), t1, az);
            bz = fma2(bc2(vz.y), t1, bz);
        }
        gx = fma2(er, ax, fma2(ei, bx, gx));
        gy = fma2(er, ay, fma2(ei, by, gy));
        gz = fma2(er, az, fma2(ei, bz, gz));
    }
}

// part + x with the rounding error kept in comp (Knuth's TwoSum), for two queries
__device__ __forceinline__ void two_sum2(float2 &part, float2 &comp, float2 x) {
    const float2 s = add2(part, x), bv = add2(s, neg2(part)), av = add2(s, neg2(bv));
    comp = add2(comp, add2(add2(part, neg2(av)), add2(x, neg2(bv))));
    part = s;
}

// The gradient over the boundary hierarchy, walked as in k_boundary_far: a node's
// closed curves by the gradient of their expansion (outside its radius and where the
// query's ray misses its box, so that no term of theirs is singular), its chords and
// the near edges by Algorithm 3's terms.  The ray test has a margin of 1/128 of the
// mesh's longest side (gpad): Algorithm 3's terms lose up to u h / rho^2 where a
// boundary point h above the query stands rho beside its ray, and inside that margin
// the terms are kept, so that the results differ from the direct sum's by rounding
// everywhere.  perm: the queries' places in the output; partial sums are in the queries' order.
// Bound by issue (an expansion's gradient is about 560 instructions for two queries per
// lane).  soup8, 200k queries: 59.3 -> 5.4 ms; soup6 (12k points), 100k: 1.98 -> 0.93 ms;
// median error against FP64 on soup8 1.9e-5 -> 5.6e-6.  A truncation bound of 4e-6
// instead of 2e-6: 5% faster.
__global__ void __launch_bounds__(kGradThreads, 4)
    k_gradient_far(const float *__restrict__ q, const uint32_t *__restrict__ perm, int64_t first, int64_t n,
                   const FarNode *__restrict__ nodes, const int32_t *__restrict__ roots, int nroots,
                   double *__restrict__ partial, const float *__restrict__ gcoef, const float4 *__restrict__ pts,
                   float *__restrict__ grad, unsigned long long *__restrict__ counters) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t qbase = first + ((int64_t)blockIdx.x * (kGradThreads / 32) + warp) * 64;   // queries [first, n)
    if (qbase >= n) return;
    const int64_t i0 = qbase + lane, i1 = i0 + 32;
    const bool ok0 = i0 < n, ok1 = i1 < n;
    float2 nqx = bc2(0.f), nqy = bc2(0.f), nqz = bc2(0.f);
    if (ok0) { nqx.x = -q[3 * i0]; nqy.x = -q[3 * i0 + 1]; nqz.x = -q[3 * i0 + 2]; }
    if (ok1) { nqx.y = -q[3 * i1]; nqy.y = -q[3 * i1 + 1]; nqz.y = -q[3 * i1 + 2]; }
    int res0 = ok0 ? 0 : 0x7fffffff, res1 = ok1 ? 0 : 0x7fffffff;   // first preorder node not skipped
    double acc[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    float2 px = bc2(0.f), py = bc2(0.f), pz = bc2(0.f), kx = bc2(0.f), ky = bc2(0.f), kz = bc2(0.f);
    unsigned skipped = 0;
    const int root1 = (int)((int64_t)nroots * (blockIdx.y + 1) / gridDim.y);
    int root = (int)((int64_t)nroots * blockIdx.y / gridDim.y), node = 0, end = 0;
    while (true) {
        if (node >= end) {
            acc[0] += (double)px.x + (double)kx.x; acc[1] += (double)py.x + (double)ky.x; acc[2] += (double)pz.x + (double)kz.x;
            acc[3] += (double)px.y + (double)kx.y; acc[4] += (double)py.y + (double)ky.y; acc[5] += (double)pz.y + (double)kz.y;
            px = py = pz = kx = ky = kz = bc2(0.f);
            if (root == root1) break;
            node = __ldg(roots + root);
            ++root;
            end = __ldg(&nodes[node].skip);
        }
        const float4 *np = reinterpret_cast<const float4 *>(nodes + node);
        const float4 h0 = __ldg(np), h1 = __ldg(np + 1), h2 = __ldg(np + 2), h3 = __ldg(np + 3);
        const int skip = __float_as_int(h2.z), nchord = __float_as_int(h2.w);
        float2 x = add2(bc2(-h0.x), neg2(nqx)), y = add2(bc2(-h0.y), neg2(nqy)), z = add2(bc2(-h0.z), neg2(nqz));
        const float2 r2 = fma2(x, x, fma2(y, y, mul2(z, z)));
        const float bx0 = h1.x - h3.w, bx1 = h1.y + h3.w, by0 = h1.z - h3.w, by1 = h1.w + h3.w, bz1 = h2.x + h3.w;
        const bool hit0 = -nqx.x >= bx0 && -nqx.x <= bx1 && -nqy.x >= by0 && -nqy.x <= by1 && -nqz.x <= bz1;
        const bool hit1 = -nqx.y >= bx0 && -nqx.y <= bx1 && -nqy.y >= by0 && -nqy.y <= by1 && -nqz.y <= bz1;
        const bool act0 = node >= res0, act1 = node >= res1;
        const bool far0 = r2.x > h3.z && !hit0, far1 = r2.y > h3.z && !hit1;
        const bool take0 = act0 && far0, take1 = act1 && far1, into0 = act0 && !far0, into1 = act1 && !far1;
        if (take0) res0 = skip;
        if (take1) res1 = skip;
        if (__any_sync(0xffffffffu, take0 || take1)) {
            float2 gx, gy, gz;
            const float2 is = bc2(h2.y);
            far_grad_eval(gcoef + (int64_t)node * kFarGradCoef, mul2(x, is), mul2(y, is), mul2(z, is), gx, gy, gz);
            gx = mul2(gx, is);
            gy = mul2(gy, is);
            gz = mul2(gz, is);
            float2 cx = bc2(0.f), cy = bc2(0.f), cz = bc2(0.f);
            unsigned none = 0;
            for (int c = 0; c < nchord; ++c) {
                const int4 ch = __ldg(reinterpret_cast<const int4 *>(np + 4));
                const float4 Pa = __ldg(pts + (c ? ch.z : ch.x)), Pb = __ldg(pts + (c ? ch.w : ch.y));
                const GradPoint2 A = grad_point2(Pa, nqx, nqy, nqz), B = grad_point2(Pb, nqx, nqy, nqz);
                grad_edge2(A, B, Pa.x - Pb.x, Pa.y - Pb.y, cx, cy, cz, none);
            }
            const float2 s4 = bc2((float)kInv4Pi);
            gx = fma2(cx, s4, gx);
            gy = fma2(cy, s4, gy);
            gz = fma2(cz, s4, gz);
            two_sum2(px, kx, make_float2(take0 ? gx.x : 0.f, take1 ? gx.y : 0.f));
            two_sum2(py, ky, make_float2(take0 ? gy.x : 0.f, take1 ? gy.y : 0.f));
            two_sum2(pz, kz, make_float2(take0 ? gz.x : 0.f, take1 ? gz.y : 0.f));
        }
        if (!__any_sync(0xffffffffu, into0 || into1)) {
            node = skip;
            continue;
        }
        const int begin = __float_as_int(h3.x), count = __float_as_int(h3.y);
        if (skip == node + 1 && count > 0) {   // a leaf: its edges one by one
            const float4 *lp = pts + begin;
            float2 gx = bc2(0.f), gy = bc2(0.f), gz = bc2(0.f);
            float4 Pa = __ldg(lp);
            GradPoint2 A = grad_point2(Pa, nqx, nqy, nqz);
            for (int j = 0; j < count; ++j) {
                if (Pa.w == 0.f) {   // a loop's closing point
                    if (j + 1 < count) {
                        Pa = __ldg(lp + j + 1);
                        A = grad_point2(Pa, nqx, nqy, nqz);
                    }
                    continue;
                }
                const float4 Pb = __ldg(lp + j + 1);
                const GradPoint2 B = grad_point2(Pb, nqx, nqy, nqz);
                unsigned sk = 0;
                grad_edge2(A, B, Pa.x - Pb.x, Pa.y - Pb.y, gx, gy, gz, sk, into0, into1);
                skipped += sk;
                Pa = Pb;
                A = B;
            }
            const float2 s4 = bc2((float)kInv4Pi);
            two_sum2(px, kx, mul2(s4, make_float2(into0 ? gx.x : 0.f, into1 ? gx.y : 0.f)));
            two_sum2(py, ky, mul2(s4, make_float2(into0 ? gy.x : 0.f, into1 ? gy.y : 0.f)));
            two_sum2(pz, kz, mul2(s4, make_float2(into0 ? gz.x : 0.f, into1 ? gz.y : 0.f)));
        }
        ++node;
    }
    if (skipped) atomicAdd(&counters[CNT_GRAD_SKIPPED], (unsigned long long)skipped);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int64_t i = h ? i1 : i0;
        if (!(h ? ok1 : ok0)) continue;
        const int64_t o = perm[i];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if (partial) partial[((int64_t)blockIdx.y * (n - first) + (i - first)) * 3 + c] = acc[3 * h + c];
            else grad[3 * o + c] = (float)acc[3 * h + c];
        }
    }
}

}  // namespace

gwn_status launch_gradient(const gwn_mesh *m, const float *q, int64_t n, float *grad, cudaStream_t s) {
    if (n <= 0) return GWN_OK;
    const int64_t nedge_pts = m->npts > 0 ? m->npts - 1 : 0;
    if (nedge_pts == 0) {   // no boundary: the gradient vanishes almost everywhere
        GWN_CUDA_TRY(cudaMemsetAsync(grad, 0, sizeof(float) * 3 * n, s));
        return GWN_OK;
    }
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 148;
    if (far_pays_gradient(m, n)) {   // the boundary hierarchy, in spatial order
        uint32_t *keys = nullptr, *perm = nullptr;
        float *qs = nullptr;
        double *partial = nullptr;
        const int64_t blocks = (n + 2 * kGradThreads - 1) / (2 * kGradThreads);
        const int64_t split = std::max<int64_t>(1, std::min<int64_t>((320 * (int64_t)sms + blocks - 1) / blocks, m->far_nroots));
        const int64_t slice = split > 1 ? query_slice(n, sizeof(double) * 3 * split) : n;
        gwn_status st = [&]() -> gwn_status {
            GWN_CUDA_TRY(dev_alloc(&keys, sizeof(uint32_t) * n, s));
            GWN_CUDA_TRY(dev_alloc(&perm, sizeof(uint32_t) * n, s));
            GWN_CUDA_TRY(dev_alloc(&qs, sizeof(float) * 3 * n, s));
            if (split > 1) GWN_CUDA_TRY(dev_alloc(&partial, sizeof(double) * 3 * split * slice, s));
            return order_queries(m, q, n, keys, perm, qs, s);
        }();
        if (st == GWN_OK) {
            ProfScope prof("gradient", s);
            for (int64_t at = 0; at < n; at += slice) {
                const int64_t end = std::min(n, at + slice), count = end - at;
                const dim3 grid((unsigned)((count + 2 * kGradThreads - 1) / (2 * kGradThreads)), (unsigned)split);
                k_gradient_far<<<grid, kGradThreads, 0, s>>>(qs, perm, at, end, m->far_nodes, m->far_roots, m->far_nroots,
                                                             partial, m->far_gcoef, m->far_pts, grad, m->counters);
                note_launches(1);
                if (!partial) continue;
                k_gradient_combine<<<grid_for(3 * count, 256), 256, 0, s>>>(partial, perm + at, count, (int)split, 1.0, grad);
                note_launches(1);
            }
        }
        for (void *p : {(void *)keys, (void *)perm, (void *)qs, (void *)partial})
            if (p) cudaFreeAsync(p, s);
        if (st != GWN_OK) return st;
        GWN_LAUNCH_CHECK("k_gradient_far");
        return GWN_OK;
    }
    constexpr int KP = 2;
    const int tile = m->cfg.boundary_tile > 0 ? m->cfg.boundary_tile : 512;
    const size_t smem = sizeof(float4) * (tile + 1) + sizeof(double) * 3 * 2 * KP * kGradThreads;
    if (smem > 48 * 1024)
        cudaFuncSetAttribute(k_gradient<KP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    const int64_t per_block = kGradThreads * 2 * KP;
    const int64_t qblocks = (n + per_block - 1) / per_block;
    int64_t chunks = (8 * (int64_t)sms + qblocks - 1) / qblocks;
    chunks = std::max<int64_t>(1, std::min<int64_t>(chunks, (nedge_pts + 2 * tile - 1) / (2 * tile)));
    chunks = std::min<int64_t>(chunks, 65535);
    const int64_t chunk_len = chunks > 1 ? (nedge_pts + chunks - 1) / chunks : nedge_pts;
    double *partial = nullptr;
    if (chunks > 1) GWN_CUDA_TRY(dev_alloc(&partial, sizeof(double) * 3 * chunks * n, s));
    {
        ProfScope prof("gradient", s);
        dim3 grid((unsigned)qblocks, (unsigned)chunks);
        k_gradient<KP><<<grid, kGradThreads, smem, s>>>(q, n, m->bpts, m->npts, tile, chunk_len, partial, grad,
                                                        m->counters);
        if (partial)
            k_gradient_combine<<<grid_for(3 * n, 256), 256, 0, s>>>(partial, nullptr, n, (int)chunks, kInv4Pi, grad);
    }
    if (partial) cudaFreeAsync(partial, s);
    GWN_LAUNCH_CHECK("k_gradient");
    return GWN_OK;
}

}  // namespace gwn
