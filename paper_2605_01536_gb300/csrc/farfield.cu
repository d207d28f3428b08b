// Build of the boundary hierarchy (farfield.cuh): leaf cuts, boxes and error
// radii, moments of the leaves, moments translated up level by level, and the
// packed coefficients the query kernels read.
#include <algorithm>
#include <cmath>

#include "farfield.cuh"

namespace gwn {

namespace {

constexpr int P = kFarP;

// Levels of the hierarchy: level l has ceil(nleaf / 2^l) nodes, node (l, i)
// covers leaves [i 2^l, (i + 1) 2^l); one node at the top level.
struct FarShape {
    int64_t nleaf;
    int top;
    int64_t off[32];   // first node of each level in level-major order
    int64_t total;
};

__host__ __device__ __forceinline__ int64_t far_level_count(const FarShape &sh, int l) {
    return (sh.nleaf + (int64_t(1) << l) - 1) >> l;
}

// Preorder index of the highest subtree that starts at leaf x: every node whose
// first leaf lies before x comes first.
__device__ __forceinline__ int64_t far_before(const FarShape &sh, int64_t x) {
    if (x >= sh.nleaf) return sh.total;
    int64_t s = 0;
    for (int l = 0; l <= sh.top; ++l) s += (x + (int64_t(1) << l) - 1) >> l;
    return s;
}
__device__ __forceinline__ int64_t far_preorder(const FarShape &sh, int l, int64_t i) {
    const int64_t x = i << l;
    int64_t s = far_before(sh, x);
    for (int k = l + 1; k <= sh.top; ++k) s += (x & ((int64_t(1) << k) - 1)) == 0;   // ancestors starting there
    return s;
}
__device__ __forceinline__ void far_level_of(const FarShape &sh, int64_t t, int &l, int64_t &i) {
    l = 0;
    while (l < sh.top && t >= sh.off[l + 1]) ++l;
    i = t - sh.off[l];
}

// Leaf cuts near every kFarLeaf-th point: at the end of the loop there if it closes
// within kFarLeaf points, else inside the loop.
__global__ void k_far_cuts(const uint2 *__restrict__ ends, int64_t npts, int64_t nleaf, int32_t *__restrict__ cut) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i > nleaf) return;
    const int64_t pos = i * kFarLeaf;
    int64_t c = pos;
    if (pos >= npts) c = npts;
    else if (i > 0 && (int64_t)ends[pos].x != pos && (int64_t)ends[pos].y < pos + kFarLeaf) c = (int64_t)ends[pos].y + 1;
    cut[i] = (int32_t)c;
}

// Geometry of nodes [t0, t0 + gridDim.x) in level-major order, one block each: box,
// radius, chords, the error coefficient and from it the acceptance radius.  Nodes
// from level kFarWideLevel up get blocks of 1024 threads: their passes over the points are
// the kernel's critical path.
constexpr int kFarWideLevel = 7;   // 128 leaves, about 2048 points
template <int Threads>
__global__ void __launch_bounds__(Threads) k_far_geom(FarShape sh, int64_t t0, const int32_t *__restrict__ cut,
                                                  const uint2 *__restrict__ ends, const float4 *__restrict__ pts,
                                                  int64_t npts, const float *__restrict__ mesh_box, float eps,
                                                  FarNode *__restrict__ nodes) {
    constexpr int kWarps = Threads / 32;
    __shared__ float s_red[kWarps][8];
    int l;
    int64_t i;
    far_level_of(sh, t0 + blockIdx.x, l, i);
    const int64_t first = i << l, past = min(sh.nleaf, (i + 1) << l);
    const int a = cut[first], b = cut[past];
    const bool a_mid = a < b && (int)ends[a].x < a;
    const bool b_mid = a < b && b < npts && (int)ends[b].x < b;
    const int last = b_mid ? b : b - 1;   // last point of the node's closed curves
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float v[6] = {INFINITY, INFINITY, INFINITY, -INFINITY, -INFINITY, -INFINITY};
    for (int j = a + (int)threadIdx.x; j <= last; j += blockDim.x) {
        const float4 p = pts[j];
        v[0] = fminf(v[0], p.x); v[1] = fminf(v[1], p.y); v[2] = fminf(v[2], p.z);
        v[3] = fmaxf(v[3], p.x); v[4] = fmaxf(v[4], p.y); v[5] = fmaxf(v[5], p.z);
    }
    for (int o = 16; o > 0; o >>= 1)
        for (int k = 0; k < 6; ++k) {
            const float w = __shfl_xor_sync(0xffffffffu, v[k], o);
            v[k] = k < 3 ? fminf(v[k], w) : fmaxf(v[k], w);
        }
    if (lane == 0)
        for (int k = 0; k < 6; ++k) s_red[warp][k] = v[k];
    __syncthreads();
    for (int k = 0; k < 6; ++k) {
        v[k] = s_red[0][k];
        for (int w = 1; w < kWarps; ++w) v[k] = k < 3 ? fminf(v[k], s_red[w][k]) : fmaxf(v[k], s_red[w][k]);
    }
    __syncthreads();
    // (a cut at the end of a loop can leave a leaf without points)
    const float cx = a < b ? 0.5f * v[0] + 0.5f * v[3] : 0.f, cy = a < b ? 0.5f * v[1] + 0.5f * v[4] : 0.f,
                cz = a < b ? 0.5f * v[2] + 0.5f * v[5] : 0.f;
    float r2 = 0.f;
    for (int j = a + (int)threadIdx.x; j <= last; j += blockDim.x) {
        const float4 p = pts[j];
        const float dx = p.x - cx, dy = p.y - cy, dz = p.z - cz;
        r2 = fmaxf(r2, dx * dx + dy * dy + dz * dz);
    }
    for (int o = 16; o > 0; o >>= 1) r2 = fmaxf(r2, __shfl_xor_sync(0xffffffffu, r2, o));
    if (lane == 0) s_red[warp][6] = r2;
    __syncthreads();
    for (int w = 0; w < kWarps; ++w) r2 = fmaxf(r2, s_red[w][6]);
    const float s = 1.0001f * sqrtf(r2);   // rounded up: the ball contains every point
    const float inv_s = s > 0.f ? 1.f / s : 0.f;
    // E / s^(P+2): each edge's fan triangle from the start of its piece
    float e = 0.f, edges = 0.f;
    for (int j = a + (int)threadIdx.x; j < b; j += blockDim.x) {
        const float4 p = pts[j];
        if (p.w == 0.f) continue;
        const float4 q = pts[j + 1], o = pts[max(a, (int)ends[j].x)];
        const float px = (p.x - cx) * inv_s, py = (p.y - cy) * inv_s, pz = (p.z - cz) * inv_s;
        const float qx = (q.x - cx) * inv_s, qy = (q.y - cy) * inv_s, qz = (q.z - cz) * inv_s;
        const float ox = (o.x - cx) * inv_s, oy = (o.y - cy) * inv_s, oz = (o.z - cz) * inv_s;
        const float ux = px - ox, uy = py - oy, uz = pz - oz, wx = qx - ox, wy = qy - oy, wz = qz - oz;
        const float nx = uy * wz - uz * wy, ny = uz * wx - ux * wz, nz = ux * wy - uy * wx;
        const float m2 = fmaxf(fmaxf(px * px + py * py + pz * pz, qx * qx + qy * qy + qz * qz),
                               ox * ox + oy * oy + oz * oz);
        float m = 1.f;
        for (int k = 0; k < P / 2; ++k) m *= m2;
        e += 0.5f * sqrtf(nx * nx + ny * ny + nz * nz) * m;
        edges += 1.f;
    }
    for (int o = 16; o > 0; o >>= 1) {
        e += __shfl_xor_sync(0xffffffffu, e, o);
        edges += __shfl_xor_sync(0xffffffffu, edges, o);
    }
    __syncthreads();
    if (lane == 0) { s_red[warp][0] = e; s_red[warp][1] = edges; }
    __syncthreads();
    if (threadIdx.x != 0) return;
    e = edges = 0.f;
    for (int w = 0; w < kWarps; ++w) {
        e += s_red[w][0];
        edges += s_red[w][1];
    }
    e *= 1.001f * 0.0795774715f;
    FarNode nd;
    nd.cx = cx; nd.cy = cy; nd.cz = cz;
    // smallest x = r / s in [1.5, 2^14] with the truncation bound <= eps
    auto bound = [&](float x) {
        const float y = 1.f / x, g = 1.f / (1.f - y);
        return e * exp2f(-(P + 2) * log2f(x)) * ((P + 1) * g + y * g * g);
    };
    float lo = 1.5f, hi = 16384.f;
    if (bound(lo) <= eps) hi = lo;
    else
        for (int it = 0; it < 30; ++it) {
            const float mid = sqrtf(lo * hi);
            if (bound(mid) <= eps) hi = mid;
            else lo = mid;
        }
    const bool leaf = l == 0;
    const bool use = s > 0.f && hi < 16384.f && !(leaf && edges < (float)kFarMinEdges);
    nd.r2acc = use ? (hi * s) * (hi * s) * 1.0001f : INFINITY;
    // margin of the ray test: above one quantum of the fixed-point grid (at most
    // the box's longest side / 2^28), so that a snapped ray misses the hull too
    const float ext = fmaxf(mesh_box[3] - mesh_box[0], fmaxf(mesh_box[4] - mesh_box[1], mesh_box[5] - mesh_box[2]));
    const float pad = ext * 0x1p-26f;
    nd.xmin = v[0] - pad; nd.xmax = v[3] + pad; nd.ymin = v[1] - pad; nd.ymax = v[4] + pad;
    nd.zmax = v[5] + pad;
    nd.inv_s = inv_s;
    nd.skip = (int32_t)far_before(sh, past);
    nd.begin = a;
    nd.count = b - a;
    // the gradient's radius: bound E / r^(P+3) (P+1)(P+2) / (1-y)^3 <= kFarGradEps / ext
    auto gbound = [&](float x) {
        const float g = 1.f / (1.f - 1.f / x);
        return e * exp2f(-(P + 3) * log2f(x)) * ((P + 1) * (P + 2)) * g * g * g;
    };
    const float geps = ext > 0.f ? kFarGradEps * (s / ext) : 0.f;
    lo = 1.5f;
    hi = 16384.f;
    if (gbound(lo) <= geps) hi = lo;
    else
        for (int it = 0; it < 30; ++it) {
            const float mid = sqrtf(lo * hi);
            if (gbound(mid) <= geps) hi = mid;
            else lo = mid;
        }
    nd.r2grad = use && hi < 16384.f ? (hi * s) * (hi * s) * 1.0001f : INFINITY;
    nd.gpad = ext * 0x1p-7f;
    nd.nchord = 0;
    nd.ch[0] = nd.ch[1] = nd.ch[2] = nd.ch[3] = 0;
    if (a_mid) {   // the piece of a loop that began before a
        nd.ch[0] = a;
        nd.ch[1] = min((int)ends[a].y, b);
        nd.nchord = 1;
    }
    if (b_mid && (int)ends[b].x >= a) {   // the piece of a loop that goes on after b
        nd.ch[2 * nd.nchord] = (int)ends[b].x;
        nd.ch[2 * nd.nchord + 1] = b;
        ++nd.nchord;
    }
    nodes[far_preorder(sh, l, i)] = nd;
}

struct Cplx {
    float r, i;
};
__device__ __forceinline__ Cplx cmul(Cplx a, Cplx b) { return {a.r * b.r - a.i * b.i, a.r * b.i + a.i * b.r}; }

// R_l^m (degrees up to L, m >= 0) of (x, y, z): r^l P_l^m e^(i m phi) / (l + m)!
template <int L>
__device__ __forceinline__ void solid_regular(float x, float y, float z, Cplx (&R)[(L + 1) * (L + 2) / 2]) {
    const float r2 = x * x + y * y + z * z;
    R[0] = {1.f, 0.f};
#pragma unroll
    for (int m = 0; m <= L; ++m) {
        if (m > 0) {
            const float k = -0.5f / m;
            R[far_idx(m, m)] = cmul(R[far_idx(m - 1, m - 1)], {k * x, k * y});
        }
        if (m + 1 <= L) R[far_idx(m + 1, m)] = {z * R[far_idx(m, m)].r, z * R[far_idx(m, m)].i};
#pragma unroll
        for (int l = m + 2; l <= L; ++l) {
            const float f = 1.f / (float)((l + m) * (l - m)), g = (2 * l - 1) * f * z, h = f * r2;
            R[far_idx(l, m)] = {g * R[far_idx(l - 1, m)].r - h * R[far_idx(l - 2, m)].r,
                                g * R[far_idx(l - 1, m)].i - h * R[far_idx(l - 2, m)].i};
        }
    }
}

// Adds the cone over the edge a -> b (relative to the centre, in units of s) to M.
// The integrand has degree P - 1 along the edge: 4-point Gauss-Legendre is exact.
__device__ __forceinline__ void edge_moments(float3 a, float3 b, Cplx (&M)[kFarRaw]) {
    static_assert(P <= 8, "4 Gauss points integrate degree 7");
    const float vx = a.y * b.z - a.z * b.y, vy = a.z * b.x - a.x * b.z, vz = a.x * b.y - a.y * b.x;
    const float gx[4] = {0.0694318442f, 0.3300094782f, 0.6699905218f, 0.9305681558f};
    const float gw[4] = {0.1739274226f, 0.3260725774f, 0.3260725774f, 0.1739274226f};
    for (int g = 0; g < 4; ++g) {
        Cplx R[P * (P + 1) / 2];
        solid_regular<P - 1>(a.x + gx[g] * (b.x - a.x), a.y + gx[g] * (b.y - a.y), a.z + gx[g] * (b.z - a.z), R);
#pragma unroll
        for (int l = 1; l <= P; ++l) {
            const float k = gw[g] / (float)(l + 1);
#pragma unroll
            for (int m = 0; m <= l; ++m) {
                // grad R_l^m: d/dz = R_(l-1)^m, d/dx + i d/dy = R_(l-1)^(m+1), d/dx - i d/dy = -R_(l-1)^(m-1)
                Cplx G = {0.f, 0.f};
                if (m <= l - 1) G = {vz * R[far_idx(l - 1, m)].r, vz * R[far_idx(l - 1, m)].i};
                if (m + 1 <= l - 1) {
                    const Cplx t = cmul({vx, -vy}, R[far_idx(l - 1, m + 1)]);
                    G.r += 0.5f * t.r;
                    G.i += 0.5f * t.i;
                }
                if (m >= 1) {
                    const Cplx t = cmul({vx, vy}, R[far_idx(l - 1, m - 1)]);
                    G.r -= 0.5f * t.r;
                    G.i -= 0.5f * t.i;
                } else if (l >= 2) {   // R_(l-1)^(-1) = -conj(R_(l-1)^1)
                    const Cplx t = cmul({vx, vy}, {R[far_idx(l - 1, 1)].r, -R[far_idx(l - 1, 1)].i});
                    G.r += 0.5f * t.r;
                    G.i += 0.5f * t.i;
                }
                M[far_idx(l, m)].r += k * G.r;
                M[far_idx(l, m)].i += k * G.i;
            }
        }
    }
}

__device__ __forceinline__ float3 rel_point(const float4 *pts, int j, const FarNode &nd) {
    const float4 p = pts[j];
    return make_float3((p.x - nd.cx) * nd.inv_s, (p.y - nd.cy) * nd.inv_s, (p.z - nd.cz) * nd.inv_s);
}

// Sums M over the warp and lets lane 0 store it to out.
__device__ __forceinline__ void warp_store_moments(Cplx (&M)[kFarRaw], Cplx *out, bool add) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 1; k < kFarRaw; ++k) {
        float r = M[k].r, i = M[k].i;
        for (int o = 16; o > 0; o >>= 1) {
            r += __shfl_xor_sync(0xffffffffu, r, o);
            i += __shfl_xor_sync(0xffffffffu, i, o);
        }
        if (lane == (k & 31)) {
            if (add) { out[k].r += r; out[k].i += i; }
            else out[k] = {r, i};
        }
    }
}

// Moments of the leaves, one warp each: lanes take the leaf's edges and the
// reversed chords that close its pieces.
__global__ void __launch_bounds__(64) k_far_leaf_moments(FarShape sh, const FarNode *__restrict__ nodes,
                                                         const float4 *__restrict__ pts, Cplx *__restrict__ raw) {
    const int64_t i = (int64_t)blockIdx.x * 2 + (threadIdx.x >> 5);
    if (i >= sh.nleaf) return;
    const FarNode nd = nodes[far_preorder(sh, 0, i)];
    Cplx M[kFarRaw];
#pragma unroll
    for (int k = 0; k < kFarRaw; ++k) M[k] = {0.f, 0.f};
    for (int t = threadIdx.x & 31; t < nd.count + nd.nchord; t += 32) {
        int ja, jb;
        if (t < nd.count) {
            ja = nd.begin + t;
            jb = ja + 1;
            if (pts[ja].w == 0.f) continue;
        } else {
            ja = nd.ch[2 * (t - nd.count) + 1];
            jb = nd.ch[2 * (t - nd.count)];
        }
        edge_moments(rel_point(pts, ja, nd), rel_point(pts, jb, nd), M);
    }
    warp_store_moments(M, raw + i * kFarRaw, false);
}

// Moments of the nodes of level l > 0, one block each: the children's moments
// translated to the node's centre,
//   M_lm += sum_{l' <= l, m'} R_(l-l')^(m-m')(d) M_l'm',  d = the child's centre,
// plus the closed polygons by which the children's chords differ from the node's.
// The levels follow one another, so the latency of one node counts: thread (child,
// output) sums one child's part of one moment, and the columns of R are made by one
// thread each (one warp per node with R made by one lane: 24 us a level, now 7).
constexpr int kUpThreads = 96;
__global__ void __launch_bounds__(kUpThreads) k_far_up(FarShape sh, int l, const FarNode *__restrict__ nodes,
                                                       const float4 *__restrict__ pts, Cplx *__restrict__ raw) {
    __shared__ Cplx s_R[2][kFarRaw], s_M[2][kFarRaw], s_part[kFarRaw];
    __shared__ int s_chords;
    const int64_t i = blockIdx.x;
    const FarNode *nd = nodes + far_preorder(sh, l, i);
    const FarNode *ch[2] = {nullptr, nullptr};   // the children that have points
#pragma unroll
    for (int c = 0; c < 2; ++c)
        if (2 * i + c < far_level_count(sh, l - 1)) {
            const FarNode *p = nodes + far_preorder(sh, l - 1, 2 * i + c);
            if (p->count > 0) ch[c] = p;
        }
    const int t = threadIdx.x;
    if (t == 0) s_chords = nd->nchord + (ch[0] ? ch[0]->nchord : 0) + (ch[1] ? ch[1]->nchord : 0);
    const float is = nd->inv_s;
    if (t < 2 * (P + 1)) {   // column m of R at child c's centre
        const int c = t / (P + 1), m = t % (P + 1);
        if (ch[c]) {
            const float x = (ch[c]->cx - nd->cx) * is, y = (ch[c]->cy - nd->cy) * is, z = (ch[c]->cz - nd->cz) * is,
                        r2 = x * x + y * y + z * z;
            Cplx a = {1.f, 0.f}, b = {0.f, 0.f};
            for (int k = 1; k <= m; ++k) {
                const float f = -0.5f / k;
                a = cmul(a, {f * x, f * y});
            }
            s_R[c][far_idx(m, m)] = a;
            for (int L = m + 1; L <= P; ++L) {
                const float f = 1.f / (float)((L + m) * (L - m)), g = (2 * L - 1) * f * z, h = L == m + 1 ? 0.f : f * r2;
                const Cplx n = {g * a.r - h * b.r, g * a.i - h * b.i};
                b = a;
                a = n;
                s_R[c][far_idx(L, m)] = n;
            }
        }
    }
    for (int k = t; k < 2 * kFarRaw; k += kUpThreads) {   // the children's moments in units of this node
        const int c = k / kFarRaw, j = k % kFarRaw;
        if (!ch[c] || j == 0) continue;
        int L = 1;
        while (far_idx(L + 1, 0) <= j) ++L;
        const float ratio = ch[c]->inv_s > 0.f ? is / ch[c]->inv_s : 0.f;   // s_child / s
        float f = ratio;
        for (int q = 0; q < L; ++q) f *= ratio;
        const Cplx v = raw[(sh.off[l - 1] + 2 * i + c) * kFarRaw + j];
        s_M[c][j] = {f * v.r, f * v.i};
    }
    __syncthreads();
    const int c = t / (kFarRaw - 1), o = 1 + t % (kFarRaw - 1);   // child, output
    Cplx acc = {0.f, 0.f};
    if (c < 2 && ch[c]) {
        int L = 1;
        while (far_idx(L + 1, 0) <= o) ++L;
        const int m = o - far_idx(L, 0);
        for (int lp = 1; lp <= L; ++lp)
            for (int mp = max(-lp, m - (L - lp)); mp <= min(lp, m + (L - lp)); ++mp) {
                const int mr = m - mp;
                Cplx a = s_M[c][far_idx(lp, abs(mp))], r = s_R[c][far_idx(L - lp, abs(mr))];
                // X_l^(-m) = (-1)^m conj(X_l^m)
                if (mp < 0) a = (mp & 1) ? Cplx{-a.r, a.i} : Cplx{a.r, -a.i};
                if (mr < 0) r = (mr & 1) ? Cplx{-r.r, r.i} : Cplx{r.r, -r.i};
                const Cplx p = cmul(r, a);
                acc.r += p.r;
                acc.i += p.i;
            }
    }
    if (c == 1) s_part[o] = acc;
    __syncthreads();
    Cplx *out = raw + (sh.off[l] + i) * kFarRaw;
    if (c == 0) out[o] = {acc.r + s_part[o].r, acc.i + s_part[o].i};
    if (s_chords == 0) return;
    __syncthreads();
    if (t >= 32) return;
    Cplx M[kFarRaw];
#pragma unroll
    for (int k = 0; k < kFarRaw; ++k) M[k] = {0.f, 0.f};
    // lanes 0-3: the children's chords (start -> end); 4, 5: the node's own, reversed
    int ja = -1, jb = -1;
    if (t < 4) {
        const FarNode *p = ch[t >> 1];
        if (p && (t & 1) < p->nchord) {
            ja = p->ch[2 * (t & 1)];
            jb = p->ch[2 * (t & 1) + 1];
        }
    } else if (t < 6 && t - 4 < nd->nchord) {
        ja = nd->ch[2 * (t - 4) + 1];
        jb = nd->ch[2 * (t - 4)];
    }
    if (ja >= 0) edge_moments(rel_point(pts, ja, *nd), rel_point(pts, jb, *nd), M);
    warp_store_moments(M, out, true);
}

// Packed coefficients in preorder.  Folded in: -(1/4pi) for w, 2pi so that the
// value adds to the sum of atan2 terms, 2 for the conjugate pair m < 0, the basis
// constant (2l-1)!! of I_l^m against T_lm, and the phase (-1)^m.
__global__ void k_far_pack(FarShape sh, const Cplx *__restrict__ raw, float *__restrict__ coef) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= sh.total * kFarRaw) return;
    const int k = (int)(t % kFarRaw);
    if (k == 0) return;
    int l;
    int64_t i;
    far_level_of(sh, t / kFarRaw, l, i);
    int L = 1;
    while (far_idx(L + 1, 0) <= k) ++L;
    const int m = k - far_idx(L, 0);
    float f = -0.5f;
    for (int j = 2 * L - 1; j > 1; j -= 2) f *= (float)j;
    if (m > 0) f *= (m & 1) ? -2.f : 2.f;
    float *out = coef + far_preorder(sh, l, i) * kFarCoef;
    if (m == 0) {
        out[L - 1] = f * raw[t].r;
    } else {
        out[far_col(m) + 2 * (L - m)] = f * raw[t].r;
        out[far_col(m) + 2 * (L - m) + 1] = f * raw[t].i;
    }
}

// Packed coefficients of the gradient in preorder (layout in farfield.cuh), component
// by component, with -(1/4pi) for w, the basis constants and the phase folded in; the
// unit of length stays with the kernel.  With a = M_l^(m-1), b = M_l^(m+1):
//   d/dx: Re[conj(a - b) I_(l+1)^m], d/dy: Re[conj(i (a + b)) I_(l+1)^m],
//   d/dz: Re[conj(-2 M_l^m) I_(l+1)^m]  (m >= 1; for m = 0 half of each).
__global__ void k_far_pack_grad(FarShape sh, const Cplx *__restrict__ raw, float *__restrict__ gcoef) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    constexpr int kPer = kFarP + kFarGradCols;   // (l, m) entries of a component
    if (t >= sh.total * kPer) return;
    const int k = (int)(t % kPer);
    int lev;
    int64_t i;
    far_level_of(sh, t / kPer, lev, i);
    const Cplx *M = raw + (t / kPer) * kFarRaw;
    int m = 0, l;   // degree of the gradient's entry
    if (k < kFarP) {
        l = k + 2;
    } else {
        m = 1;
        while (far_grad_col(m + 1) <= k - kFarP) ++m;
        l = far_grad_first(m) + (k - kFarP - far_grad_col(m));
    }
    const int L = l - 1;   // degree of the moment
    auto mom = [&](int mm) -> Cplx { return mm > L ? Cplx{0.f, 0.f} : M[far_idx(L, mm)]; };
    float f = -0.0795774715f;
    for (int j = 2 * l - 1; j > 1; j -= 2) f *= (float)j;
    if (m & 1) f = -f;
    float *out = gcoef + far_preorder(sh, lev, i) * kFarGradCoef;
    constexpr int kComp = kFarGradCoef / 3;
    if (m == 0) {
        out[k] = -f * mom(1).r;
        out[kComp + k] = -f * mom(1).i;
        out[2 * kComp + k] = -f * mom(0).r;
    } else {
        const Cplx a = mom(m - 1), b = mom(m + 1), c = mom(m);
        const int at = kFarP + 2 * (k - kFarP);
        out[at] = f * (a.r - b.r);
        out[at + 1] = f * (a.i - b.i);
        out[kComp + at] = -f * (a.i + b.i);
        out[kComp + at + 1] = f * (a.r + b.r);
        out[2 * kComp + at] = -2.f * f * c.r;
        out[2 * kComp + at + 1] = -2.f * f * c.i;
    }
}

// Preorder index of each node of level l, and of the end.
__global__ void k_far_roots(FarShape sh, int l, int32_t *__restrict__ roots) {
    const int64_t i = threadIdx.x, n = far_level_count(sh, l);
    if (i <= n) roots[i] = (int32_t)(i < n ? far_preorder(sh, l, i) : sh.total);
}

// Cost of the hierarchical sum at sample points of the mesh's box (a fixed hash
// sequence), in the operation counts of the query kernel, summed into *cost, and the
// expansions each sample takes, added to taken[sample].  (The hash is the published
// 32-bit integer mixer "lowbias32" of C. Wellons' hash prospector.)
__device__ __forceinline__ float far_hash(uint32_t x) {
    x ^= x >> 16; x *= 0x7feb352du; x ^= x >> 15; x *= 0x846ca68bu; x ^= x >> 16;
    return (float)(x >> 8) * (1.0f / 16777216.0f);
}
constexpr int kFarVisitCost = 15, kFarEvalCost = 280, kFarChordCost = 80, kFarEdgeCost = 32;
__global__ void k_far_sample(const FarNode *__restrict__ nodes, const int32_t *__restrict__ roots, int nroots,
                             const float *__restrict__ box, int nsample, unsigned long long *__restrict__ cost,
                             uint32_t *__restrict__ taken) {
    // one thread per (sample, subtree): a whole walk is a serial chain of hundreds of loads
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int i = t / nroots;
    unsigned long long c = 0;
    if (i < nsample) {
        uint32_t expansions = 0;
        const float x = box[0] + (box[3] - box[0]) * far_hash(3u * i + 1u),
                    y = box[1] + (box[4] - box[1]) * far_hash(3u * i + 2u),
                    z = box[2] + (box[5] - box[2]) * far_hash(3u * i + 3u);
        int node = roots[t % nroots];
        const int end = nodes[node].skip;
        while (node < end) {
            const FarNode nd = nodes[node];
            const float dx = x - nd.cx, dy = y - nd.cy, dz = z - nd.cz;
            const bool hit = x >= nd.xmin && x <= nd.xmax && y >= nd.ymin && y <= nd.ymax && z <= nd.zmax;
            c += kFarVisitCost;
            if (dx * dx + dy * dy + dz * dz > nd.r2acc && !hit) {
                c += kFarEvalCost + kFarChordCost * nd.nchord;
                ++expansions;
                node = nd.skip;
            } else {
                if (nd.skip == node + 1) c += kFarEdgeCost * nd.count;
                ++node;
            }
        }
        if (expansions) atomicAdd(&taken[i], expansions);
    }
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(cost, c);
}

}  // namespace

gwn_status build_far(gwn_mesh *m, float4 *pts, const uint2 *ends, cudaStream_t s) {
    const int64_t npts = m->npts;
    FarShape sh{};
    sh.nleaf = (npts + kFarLeaf - 1) / kFarLeaf;
    while ((int64_t(1) << sh.top) < sh.nleaf) ++sh.top;
    for (int l = 0; l <= sh.top; ++l) {
        sh.off[l] = sh.total;
        sh.total += far_level_count(sh, l);
    }
    constexpr int kSamples = 1024;
    int rl = 0;
    while (far_level_count(sh, rl) > kFarRoots) ++rl;
    const int nroots = (int)far_level_count(sh, rl);
    int32_t *cut = nullptr, *roots = nullptr;
    Cplx *raw = nullptr;
    FarNode *nodes = nullptr;
    float *coef = nullptr;
    struct Sample {
        unsigned long long cost;
        uint32_t taken[kSamples];
    } *sample = nullptr, sample_h;
    GWN_CUDA_TRY(dev_alloc(&cut, sizeof(int32_t) * (sh.nleaf + 1), s));
    GWN_CUDA_TRY(dev_alloc(&sample, sizeof(Sample), s));
    GWN_CUDA_TRY(dev_alloc(&nodes, sizeof(FarNode) * sh.total, s));
    GWN_CUDA_TRY(dev_alloc(&roots, sizeof(int32_t) * (nroots + 1), s));
    k_far_cuts<<<grid_for(sh.nleaf + 1, 256), 256, 0, s>>>(ends, npts, sh.nleaf, cut);
    const int64_t wide = sh.top >= kFarWideLevel ? sh.off[kFarWideLevel] : sh.total;   // first wide node
    k_far_roots<<<1, kFarRoots + 32, 0, s>>>(sh, rl, roots);
    const double budget = 0.5 * (m->cfg.classify_margin > 0.f ? m->cfg.classify_margin : 1e-4f);
    double eps = kFarEps, first_cost = 0.0;
    bool held = false;   // the expansions' bounds add up to no more than the budget
    for (int round = 0; round < 4 && !held && eps >= kFarEpsMin; ++round) {
        if (wide < sh.total)
            k_far_geom<1024><<<(unsigned)(sh.total - wide), 1024, 0, s>>>(sh, wide, cut, ends, pts, npts, m->box, (float)eps,
                                                                         nodes);
        k_far_geom<64><<<(unsigned)wide, 64, 0, s>>>(sh, 0, cut, ends, pts, npts, m->box, (float)eps, nodes);
        GWN_CUDA_TRY(cudaMemsetAsync(sample, 0, sizeof(Sample), s));
        k_far_sample<<<grid_for((int64_t)kSamples * nroots, 128), 128, 0, s>>>(nodes, roots, nroots, m->box, kSamples,
                                                                              &sample->cost, sample->taken);
        GWN_CUDA_TRY(cudaMemcpyAsync(&sample_h, sample, sizeof(Sample), cudaMemcpyDeviceToHost, s));
        GWN_CUDA_TRY(cudaStreamSynchronize(s));
        m->far_cost = (double)sample_h.cost / kSamples;
        if (round == 0) first_cost = m->far_cost;
        if (m->far_cost > kFarWorth * 28.0 * (double)npts) break;
        const double most = *std::max_element(sample_h.taken, sample_h.taken + kSamples);
        held = most * eps <= budget;
        if (!held) eps *= 0.9 * std::pow(budget / (most * eps), 1.25);   // (expansions grow like eps^-0.2)
    }
    // (the gradient's radii have a bound of their own: first_cost decides whether it gets the hierarchy)
    if (first_cost <= kFarWorth * 28.0 * (double)npts) {
        GWN_CUDA_TRY(dev_alloc(&raw, sizeof(Cplx) * kFarRaw * sh.total, s));
        GWN_CUDA_TRY(dev_alloc(&coef, sizeof(float) * kFarCoef * sh.total, s));
        k_far_leaf_moments<<<grid_for(sh.nleaf, 2), 64, 0, s>>>(sh, nodes, pts, raw);
        for (int l = 1; l <= sh.top; ++l)
            k_far_up<<<(unsigned)far_level_count(sh, l), kUpThreads, 0, s>>>(sh, l, nodes, pts, raw);
        GWN_CUDA_TRY(dev_alloc(&m->far_gcoef, sizeof(float) * kFarGradCoef * sh.total, s));
        k_far_pack<<<grid_for(sh.total * kFarRaw, 256), 256, 0, s>>>(sh, raw, coef);
        k_far_pack_grad<<<grid_for(sh.total * (kFarP + kFarGradCols), 256), 256, 0, s>>>(sh, raw, m->far_gcoef);
        cudaFreeAsync(raw, s);
        m->far_pts = pts;
        m->far_nodes = nodes;
        m->far_coef = coef;
        m->far_nn = sh.total;
        m->far_roots = roots;
        m->far_nroots = nroots;
        m->far_sum = held && m->far_cost <= kFarWorth * direct_cost(m);
    } else {
        cudaFreeAsync(nodes, s);
        cudaFreeAsync(pts, s);
        cudaFreeAsync(roots, s);
    }
    cudaFreeAsync(cut, s);
    cudaFreeAsync(sample, s);
    GWN_LAUNCH_CHECK("boundary hierarchy");
    return GWN_OK;
}

}  // namespace gwn
