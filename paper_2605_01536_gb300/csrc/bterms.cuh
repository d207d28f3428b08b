// Boundary terms of the antipodal sum, shared by the boundary-sum kernels:
// unit vectors to boundary points, the edge term atan2(n, d) with its exact rare
// cases, grouped products, queues for ill-conditioned terms, and the FP64 forms.
#pragma once

#include "atan_poly.cuh"
#include "fp32x2.cuh"
#include "gwn_internal.cuh"
#include "predicates.cuh"
#include "quant.cuh"

namespace gwn {

namespace {

constexpr double kInv2Pi = 0.15915494309189533577;
constexpr float kPiF = 3.14159265358979f;

// ------------------------------------------------------ boundary terms ----

// atan2 for the hot loops: octant reduction to t = min/max in [0, 1], then
// atan(t) = t P(t^2) with the minimax polynomial of atan_poly.cuh (fitted by
// fit_atan.py), then the octant is undone.  Branch-free.  Callers never pass
// (0, 0).  The larger magnitude is clamped to the smallest normal float only
// to keep the approximate reciprocal finite; every operand the kernels pass is
// a normal number (an accepted group product is at least (4.9e-5)^8 ~ 3e-35),
// so the clamp never changes a result.
constexpr float kFltMin = 1.17549435e-38f;
__device__ __forceinline__ float fast_atan2(float y, float x) {
    const float ax = fabsf(x), ay = fabsf(y);
    const float mx = fmaxf(fmaxf(ax, ay), kFltMin), mn = fminf(ax, ay);
    const float t = mn * sfu_rcp(mx);
    const float s = t * t;
    float r = gwn_atan_poly(s) * t;
    r = ay > ax ? 1.57079632679489662f - r : r;
    r = x < 0.f ? 3.14159265358979324f - r : r;
    return copysignf(r, y);
}

// Unit vector from the query to a boundary point, kept as (A_x, A_y, H) with
// H = 1 - A_z computed without cancellation: (A_x^2 + A_y^2) / (1 + A_z) when
// A_z > 0.  The point coincident with the query gives (0, 0, 0).  With two such
// vectors A, B the van Oosterom-Strackee numerator and denominator of
// Area(A, B, x1) / 2 for x1 = (0, 0, -1) are
//   n = A.(B x x1) = A_y B_x - A_x B_y,
//   d = 1 + A.B + A.x1 + B.x1 = H_a H_b + A_x B_x + A_y B_y.
struct PointRel {
    float ax, ay, h;
};

// Limit of atan2(n, d) for the edge (u, v) when u lies exactly on the query's
// vertical ray (u - q = (0, 0, h), h > 0): the perturbed unit vector to u is
// (-e1/h, -e2/h, 1), so n ~ e1 r_y - e2 r_x and d ~ -e1 r_x - e2 r_y with
// r = v - q; hence atan2(r_y, -r_x), and for r_y = 0 the e2 order gives -pi
// (r_x > 0) or 0 (r_x < 0).
__device__ __forceinline__ float apex_angle(float rx, float ry, bool &degenerate) {
    if (ry != 0.f) return atan2f(ry, -rx);
    if (rx > 0.f) return -kPiF;
    if (rx < 0.f) return 0.f;
    degenerate = true;
    return 0.f;
}

// Rare path of one edge term: n = d = 0 (a boundary vertex straight above the
// query, or the query on the edge), or d <= 0 with |n| within its rounding
// bound (the atan2 branch cut, where the sign of n is the exact perturbed sign
// of the 2-D edge classification, Supp. S2.1).
__device__ __noinline__ float edge_angle_slow(float4 Pa, float4 Pb, float qx, float qy, float qz, float n, float d,
                                               unsigned long long *counters) {
    if (n == 0.f && d == 0.f) {
        const float ax = Pa.x - qx, ay = Pa.y - qy, az = Pa.z - qz;
        const float bx = Pb.x - qx, by = Pb.y - qy, bz = Pb.z - qz;
        bool deg = false;
        float t;
        const bool a_up = ax == 0.f && ay == 0.f, b_up = bx == 0.f && by == 0.f;
        if (a_up && !b_up && az > 0.f) {
            t = apex_angle(bx, by, deg);
        } else if (b_up && !a_up && bz > 0.f) {
            t = -apex_angle(ax, ay, deg);
        } else {
            deg = true;
            t = 0.f;
        }
        atomicAdd(&counters[deg ? CNT_DEGENERATE : CNT_APEX], 1ull);
        return t;
    }
    atomicAdd(&counters[CNT_EXACT_BRANCH], 1ull);
    const int s = branch_sos(qx, qy, Pa.x, Pa.y, Pb.x, Pb.y, counters);   // n ~ -classification
    const float mag = fabsf(n);
    return atan2f(s > 0 ? -mag : mag, d);
}

// One edge term atan2(n, d).  |n - n_exact| <= ~4u (|A_y B_x| + |A_x B_y|) + the
// rounding of the unit vectors; 1e-6 (|A_y B_x| + |A_x B_y|) + 1e-30 covers it
// with margin, so outside that band the FP32 sign of n is the exact one.
__device__ __forceinline__ float edge_term(float n, float d, const PointRel &A, const PointRel &B, float4 Pa,
                                           float4 Pb, float qx, float qy, float qz, unsigned long long *counters) {
    if (d <= 0.f && fabsf(n) <= fmaf(1e-6f, fabsf(A.ay * B.ax) + fabsf(A.ax * B.ay), 1e-30f))
        return edge_angle_slow(Pa, Pb, qx, qy, qz, n, d, counters);
    return fast_atan2(n, d);
}

struct PointRel2 {
    float2 ax, ay, h;
};

// point_rel for two queries (nqx, nqy, nqz hold minus the query coordinates).
// H = 1 - A_z without a select: with g = 1 + |A_z|, hh = (A_x^2 + A_y^2) / g
// equals 1 - |A_z| (no cancellation), and H = hh + (|A_z| - A_z).
__device__ __forceinline__ PointRel2 point_rel2(float4 P, float2 nqx, float2 nqy, float2 nqz) {
    const float2 dx = add2(bc2(P.x), nqx), dy = add2(bc2(P.y), nqy), dz = add2(bc2(P.z), nqz);
    const float2 s = fma2(dx, dx, mul2(dy, dy));
    const float2 r2 = add2(fma2(dz, dz, s), bc2(1e-37f));    // > 0 even for a coincident point
    const float2 inv = make_float2(sfu_rsqrt(r2.x), sfu_rsqrt(r2.y));
    PointRel2 r;
    r.ax = mul2(dx, inv);
    r.ay = mul2(dy, inv);
    const float2 az = mul2(dz, inv);
    const float2 aaz = make_float2(fabsf(az.x), fabsf(az.y));
    const float2 g = add2(bc2(1.0f), aaz);
    const float2 hh = mul2(mul2(mul2(s, inv), inv), make_float2(sfu_rcp(g.x), sfu_rcp(g.y)));
    r.h = add2(hh, add2(aaz, neg2(az)));
    return r;
}


// fast_atan2 for two (y, x) pairs at once
__device__ __forceinline__ float2 fast_atan2_2(float2 y, float2 x) {
    const float axx = fabsf(x.x), axy = fabsf(x.y), ayx = fabsf(y.x), ayy = fabsf(y.y);
    const float mxx = fmaxf(fmaxf(axx, ayx), kFltMin), mxy = fmaxf(fmaxf(axy, ayy), kFltMin);
    const float2 t = mul2(make_float2(fminf(axx, ayx), fminf(axy, ayy)), make_float2(sfu_rcp(mxx), sfu_rcp(mxy)));
    const float2 s = mul2(t, t);
    float2 p = bc2(GWN_ATAN_C8);
    p = fma2(p, s, bc2(GWN_ATAN_C7));
    p = fma2(p, s, bc2(GWN_ATAN_C6));
    p = fma2(p, s, bc2(GWN_ATAN_C5));
    p = fma2(p, s, bc2(GWN_ATAN_C4));
    p = fma2(p, s, bc2(GWN_ATAN_C3));
    p = fma2(p, s, bc2(GWN_ATAN_C2));
    p = fma2(p, s, bc2(GWN_ATAN_C1));
    p = fma2(p, s, bc2(GWN_ATAN_C0));
    const float2 r = mul2(p, t);
    // undo the octant reduction: r -> A + B r with (A, B) from (|y| > |x|, x < 0)
    const bool fx1 = ayx > axx, fy1 = ayy > axy, fx2 = x.x < 0.f, fy2 = x.y < 0.f;
    const float2 A = make_float2(fx1 ? 1.57079632679489662f : (fx2 ? 3.14159265358979324f : 0.f),
                                 fy1 ? 1.57079632679489662f : (fy2 ? 3.14159265358979324f : 0.f));
    const float2 B = make_float2((fx1 != fx2) ? -1.f : 1.f, (fy1 != fy2) ? -1.f : 1.f);
    const float2 o = fma2(B, r, A);
    return make_float2(copysignf(o.x, y.x), copysignf(o.y, y.y));
}

// Terms are grouped GROUP edges at a time: each term's (d + i n) is multiplied
// into a running product, one atan2 per group.  The product's argument equals
// the sum of the accepted angles as long as it never passes +-pi, which either
// of two acceptance tests guarantees:
// - per term (the default for sparse boundaries): |n| < tan(pi/GROUP) d -
//   kAccept, each angle below pi/8 in magnitude, so 8 of them sum to less
//   than pi.  The test depends on the term alone, off the product's chain.
// - running (dense boundaries, where many terms are steep: on random soups
//   2.5% fail the per-term test, 0.35% this one): d > kMinD and the product
//   with the term keeps a positive real part.  By induction the argument
//   stays in (-pi/2, pi/2): an accepted angle is below pi/2 in magnitude
//   (d > 0), so the new argument lies in (-pi, pi), and a positive real part
//   puts it in (-pi/2, pi/2).  Rounding can only matter where the real part is
//   near zero, an argument near +-pi/2, where atan2 is continuous.  The test
//   sits on the product's chain (compare, then select), which costs 9% where
//   nearly every term passes either test.
// Both margins keep every accepted factor's modulus above 4.9e-5, so a product
// of 8 factors of modulus at most 4 neither underflows nor overflows.  A term
// that is not accepted (an edge seen steeply from the query, the atan2 branch
// cut, a vertex straight above) leaves the product unchanged and takes its own
// atan2, with the exact branch-cut sign and apex limit where they apply.
constexpr int GROUP = 8;
constexpr float kTanGroup = 0.41f;     // < tan(pi/8) = 0.41421
constexpr float kAccept = 2e-5f;
constexpr float kMinD = 5e-5f;

template <int KP>
struct BsumState {
    float2 re[KP], im[KP], part[KP], comp[KP];
};

// part + x as an unevaluated sum part + comp (Knuth's TwoSum, error folded into
// comp): keeps the FP32 running sum of group angles accurate to about one
// rounding however many groups a tile holds.
__device__ __forceinline__ void two_sum_acc2(float2 &part, float2 &comp, float2 x) {
    const float2 s = add2(part, x);
    const float2 bv = add2(s, neg2(part));
    const float2 av = add2(s, neg2(bv));
    const float2 err = add2(add2(part, neg2(av)), add2(x, neg2(bv)));
    comp = add2(comp, err);
    part = s;
}

__device__ __forceinline__ void two_sum_acc(float &part, float &comp, float x) {
    const float s = part + x;
    const float bv = s - part;
    const float av = s - bv;
    comp += (part - av) + (x - bv);
    part = s;
}

// Load the block's queries: thread t holds queries base + t + k * blockDim.x,
// k < 2 KP, as KP float2 pairs of negated coordinates (NaN past n).
template <int KP>
__device__ __forceinline__ void load_query_pairs(const float *__restrict__ q, int64_t base, int64_t n,
                                                 float2 (&nqx)[KP], float2 (&nqy)[KP], float2 (&nqz)[KP]) {
#pragma unroll
    for (int k = 0; k < 2 * KP; ++k) {
        const int64_t idx = base + (int64_t)k * blockDim.x;
        const bool ok = idx < n;
        const float nan = __int_as_float(0x7fc00000);
        const float x = ok ? -q[3 * idx] : nan, y = ok ? -q[3 * idx + 1] : nan, z = ok ? -q[3 * idx + 2] : nan;
        if (k & 1) { nqx[k >> 1].y = x; nqy[k >> 1].y = y; nqz[k >> 1].y = z; }
        else       { nqx[k >> 1].x = x; nqy[k >> 1].x = y; nqz[k >> 1].x = z; }
    }
}

// Deferred fallback terms (the batched kernel's variant).  Where many terms
// fail the group test (dense soups: about 1 in 40), nearly every warp-edge has
// some failing lane, and computing the failing terms in place runs the scalar
// path once per query slot with most lanes idle.  Instead each warp appends its
// failing (query, edge) pairs to a queue in shared memory, entry
// j << 7 | k << 5 | lane (edge j of the tile, query slot k of that lane), and
// drains it with all 32 lanes once it holds 32 KQ entries and at the end of
// every tile.  Drained terms are added to per-query 64-bit fixed-point sums
// (units of 2^-40 rad) with integer atomics: exact, so the result does not
// depend on the order of the drain.
constexpr float kFixScale = 0x1p40f;

// Scalar twins of point_rel2 and edge_nd2: the same operations in the same
// order with explicit rounding (no contraction), so a drained term is computed
// from bit-identical n and d to the ones the group test saw.  Near n = d = 0
// (an apex seen almost head-on) atan2 is ill-conditioned enough that another
// rounding of the unit vectors moves the term by ~1e-5 rad.
__device__ __forceinline__ PointRel point_rel_twin(float4 P, float qx, float qy, float qz) {
    const float dx = __fadd_rn(P.x, -qx), dy = __fadd_rn(P.y, -qy), dz = __fadd_rn(P.z, -qz);
    const float s = __fmaf_rn(dx, dx, __fmul_rn(dy, dy));
    const float r2 = __fadd_rn(__fmaf_rn(dz, dz, s), 1e-37f);
    const float inv = sfu_rsqrt(r2);
    PointRel r;
    r.ax = __fmul_rn(dx, inv);
    r.ay = __fmul_rn(dy, inv);
    const float az = __fmul_rn(dz, inv);
    const float aaz = fabsf(az);
    const float g = __fadd_rn(1.0f, aaz);
    const float hh = __fmul_rn(__fmul_rn(__fmul_rn(s, inv), inv), sfu_rcp(g));
    r.h = __fadd_rn(hh, __fadd_rn(aaz, -az));
    return r;
}

// Ill-conditioned terms: |d + i n| < 2^-6 H_a H_b.  A term's FP32 rounding
// error is a few units of rounding of the products that make up n and d,
// whose size is about H_a H_b where the term is ill-conditioned (the unit
// vectors to the edge's ends nearly opposite: the query close to the edge),
// divided by |d + i n|; below 2^-6 H_a H_b the amplification exceeds 64 and
// the term is recomputed in FP64 from the FP32 inputs, where the differences
// to the query are exact.  |d + i n|^2 = 2 (1 + A.B) H_a H_b for unit A, B, so
// this needs 1 + A.B < H_a H_b / 8192: A and B within 1/45 rad of opposite.
// The hot loop tests it (paired, the same arithmetic) only in warps near the
// boundary tile, and keeps such terms out of the group products.
constexpr float kCancel = 0x1p-6f;
__device__ __forceinline__ bool cancels(float n, float d, float ha, float hb) {
    const float t = kCancel * (ha * hb);
    return fmaf(n, n, d * d) < t * t;
}
__device__ double edge_angle64(float4 Pa, float4 Pb, float qx, float qy, float qz,
                               const unsigned long long *counters);

// The FP64 evaluation does not run inside the edge loop: its registers would
// crowd the loop's (a call to it from there cost 9% of the kernel).  A
// cancelling term found in the loop is put on a per-warp queue in shared
// memory, entry j << 7 | k << 5 | lane (edge j of the tile, query slot k of that
// lane), and the warp evaluates the queue in FP64 after the tile's edges, where
// the loop's registers are free; the results go to per-query 64-bit
// fixed-point sums (units of 2^-40 rad) with integer atomics, exact and
// independent of the order.  A queue without room for what comes next is evaluated and
// emptied on the spot, so that a query's sum does not depend on how many terms its
// neighbours in the warp queue.  A query with more than kCancelOwn such terms in one tile
// is listed for a full FP64 re-evaluation (k_fp64_fix), once (the listed bits).
constexpr int kCancelCap = 256;   // room for a warp's 128 queries' terms of one edge, twice
constexpr int kCancelOwn = 64;
constexpr double kFixUnit = 0x1p-40;
constexpr double kFixScale64 = 0x1p40;

struct CancelQ {
    unsigned *queue;            // this warp's queue, kCancelCap entries
    int *count;                 // this warp's entry count
    int *own;                   // terms per query of the warp in this tile, own[32 slot + lane]
    long long *fix;             // fixed-point sums, fix[k blockDim.x + t]
    const float *q;             // the block's queries: slot k of thread t at q[3 (t + k blockDim.x)]
    int64_t qbase;              // caller's index of the block's query slot 0 of thread 0 (for the list)
    int32_t *list;              // queries for a full FP64 re-evaluation
    unsigned long long *list_len;
    unsigned *listed;           // one bit per query: already listed
};

// Put query idx on the FP64 re-evaluation list unless it is there already.
__device__ __forceinline__ void list_query(int64_t idx, int32_t *list, unsigned long long *list_len,
                                           unsigned *listed) {
    const unsigned bit = 1u << (idx & 31);
    if (atomicOr(&listed[idx >> 5], bit) & bit) return;
    list[atomicAdd(list_len, 1ull)] = (int32_t)idx;
}

// Queue a term (the caller has made sure of room).
__device__ __forceinline__ void cancel_push(const CancelQ &cq, unsigned entry) {
    cq.queue[atomicAdd(cq.count, 1)] = entry;
}

// The entries of the warp's queue; every lane of the warp calls it.
__device__ __forceinline__ int cancel_count(const int *count) {
    __syncwarp();
    return __shfl_sync(0xffffffffu, *count, 0);
}

// Start of a tile: no terms of this tile yet.
template <int KQ>
__device__ __forceinline__ void cancel_tile(const CancelQ &cq) {
#pragma unroll
    for (int k = 0; k < KQ; ++k) cq.own[32 * k + (threadIdx.x & 31)] = 0;
    __syncwarp();
}

// FP64 evaluation of this warp's queued terms; edge(j) gives the two points of entry j's
// edge.  All 32 lanes of the warp call it, with the loop's registers out of use.
template <class Edge>
__device__ __forceinline__ void cancel_drain_edges(const CancelQ &cq, unsigned long long *counters, Edge &&edge) {
    __syncwarp();
    const int lane = threadIdx.x & 31, warp0 = threadIdx.x & ~31;
    const int count = *cq.count;
    for (int r = lane; r < count; r += 32) {
        const unsigned e = cq.queue[r];
        const int slot = (int)(e & 127u), owner = warp0 + (slot & 31), k = slot >> 5;
        const int local = owner + k * (int)blockDim.x;
        float4 Pa, Pb;
        edge((int)(e >> 7), Pa, Pb);
        const double t = edge_angle64(Pa, Pb, cq.q[3 * local], cq.q[3 * local + 1], cq.q[3 * local + 2], counters);
        atomicAdd(reinterpret_cast<unsigned long long *>(cq.fix + (k * (int)blockDim.x + owner)),
                  (unsigned long long)__double2ll_rn(t * kFixScale64));
        if (atomicAdd(&cq.own[slot], 1) == kCancelOwn) list_query(cq.qbase + local, cq.list, cq.list_len, cq.listed);
    }
    if (lane == 0 && count > 0) atomicAdd(&counters[CNT_CANCEL], (unsigned long long)count);
    __syncwarp();
    if (lane == 0) *cq.count = 0;
    __syncwarp();
}
// entries: edges of the staged points
__device__ __noinline__ void cancel_drain(const CancelQ &cq, const float4 *s_pts, unsigned long long *counters) {
    cancel_drain_edges(cq, counters, [&](int j, float4 &Pa, float4 &Pb) {
        Pa = s_pts[j];
        Pb = s_pts[j + 1];
    });
}

// A term that failed the group test and does not cancel, from the n and d the
// test saw.  Out of line: it runs for a few terms in a thousand, and inlined its
// registers would crowd the group loop.
__device__ __noinline__ float fallback_term(float n, float d, PointRel a, PointRel b, float4 Pa, float4 Pb, float qx,
                                            float qy, float qz, unsigned long long *counters) {
    return edge_term(n, d, a, b, Pa, Pb, qx, qy, qz, counters);
}

struct BsumDefer {
    const float *q;            // the block's queries: query slot k of thread t at q[3 (t + k blockDim.x)]
    unsigned *queue;           // this warp's queue, 64 KQ entries
    long long *fix;            // fixed-point sums, fix[k blockDim.x + t]
};

// The deferred terms of the batched kernel, drained by all 32 lanes.  With
// Cond, a term whose d cancels goes on the cancellation queue (FP64 after the
// tile, or as soon as the queue may be short of room) instead.
template <bool Cond>
__device__ __noinline__ void bsum_drain(const unsigned *queue, int count, const float4 *s_pts, const float *q,
                                        long long *fix, CancelQ cq, unsigned long long *counters) {
    const int lane = threadIdx.x & 31, warp0 = threadIdx.x & ~31;
    for (int r0 = 0; r0 < count; r0 += 32) {
        if (r0 + lane < count) {
            const unsigned e = queue[r0 + lane];
            const int owner = warp0 + (int)(e & 31u), k = (int)(e >> 5 & 3u), j = (int)(e >> 7);
            const int local = owner + k * (int)blockDim.x;
            const float4 Pa = s_pts[j], Pb = s_pts[j + 1];
            const float qx = q[3 * local], qy = q[3 * local + 1], qz = q[3 * local + 2];
            const PointRel A = point_rel_twin(Pa, qx, qy, qz), B = point_rel_twin(Pb, qx, qy, qz);
            const float n = __fmaf_rn(A.ay, B.ax, -__fmul_rn(A.ax, B.ay));
            const float d = __fmaf_rn(A.h, B.h, __fmaf_rn(A.ax, B.ax, __fmul_rn(A.ay, B.ay)));
            if (Cond && cancels(n, d, A.h, B.h)) {
                cancel_push(cq, e);
            } else {
                const float t = edge_term(n, d, A, B, Pa, Pb, qx, qy, qz, counters);
                atomicAdd(reinterpret_cast<unsigned long long *>(fix + (k * (int)blockDim.x + owner)),
                          (unsigned long long)__float2ll_rn(t * kFixScale));
            }
        }
        if (Cond && cancel_count(cq.count) > kCancelCap - 32) cancel_drain(cq, s_pts, counters);
    }
    __syncwarp();
}

// Box of the staged tile's points (points 0..cnt) widened on every side by a
// tenth of its longest edge, into box[0..5] = (min x, max x, min y, max y,
// min z, max z) for every thread of the block.  An ill-conditioned term,
// |d + i n| < H_a H_b / 64, has |d + i n|^2 = 2 (1 + A.B) H_a H_b below
// (H_a H_b)^2 / 4096, so 1 + A.B < H_a H_b / 8192 <= 4.9e-4 (H_a H_b <= 4): the
// edge subtends an angle within 0.032 rad of pi, which puts the query within
// 0.032 L of the edge (L its length).  A tenth of the longest edge leaves a
// factor of three for rounding.  Contains barriers: every thread of the block
// must call it.
__device__ __noinline__ void tile_box(const float4 *s_pts, int cnt, float *box) {
    __shared__ float s_red[8][8];   // up to 8 warps x (3 minima, 3 maxima, edge length^2)
    float v[7] = {INFINITY, INFINITY, INFINITY, -INFINITY, -INFINITY, -INFINITY, 0.f};
    for (int i = threadIdx.x; i <= cnt; i += blockDim.x) {
        const float4 P = s_pts[i];
        v[0] = fminf(v[0], P.x); v[1] = fminf(v[1], P.y); v[2] = fminf(v[2], P.z);
        v[3] = fmaxf(v[3], P.x); v[4] = fmaxf(v[4], P.y); v[5] = fmaxf(v[5], P.z);
        if (i < cnt && P.w != 0.f) {
            const float4 Q = s_pts[i + 1];
            const float dx = Q.x - P.x, dy = Q.y - P.y, dz = Q.z - P.z;
            v[6] = fmaxf(v[6], dx * dx + dy * dy + dz * dz);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int k = 0; k < 3; ++k) v[k] = fminf(v[k], __shfl_xor_sync(0xffffffffu, v[k], o));
#pragma unroll
        for (int k = 3; k < 7; ++k) v[k] = fmaxf(v[k], __shfl_xor_sync(0xffffffffu, v[k], o));
    }
    const int warp = threadIdx.x >> 5, nwarps = (blockDim.x + 31) >> 5;
    if ((threadIdx.x & 31) == 0) {
#pragma unroll
        for (int k = 0; k < 7; ++k) s_red[warp][k] = v[k];
    }
    __syncthreads();
    float r[7];
#pragma unroll
    for (int k = 0; k < 7; ++k) r[k] = s_red[0][k];
    for (int w = 1; w < nwarps; ++w) {
#pragma unroll
        for (int k = 0; k < 3; ++k) r[k] = fminf(r[k], s_red[w][k]);
#pragma unroll
        for (int k = 3; k < 7; ++k) r[k] = fmaxf(r[k], s_red[w][k]);
    }
    __syncthreads();   // s_red is reused by the next tile
    const float L = 0.1f * sqrtf(r[6]);
    box[0] = r[0] - L; box[1] = r[3] + L;
    box[2] = r[1] - L; box[3] = r[4] + L;
    box[4] = r[2] - L; box[5] = r[5] + L;
}

__device__ __forceinline__ bool in_box(const float *b, float x, float y, float z) {
    return x >= b[0] && x <= b[1] && y >= b[2] && y <= b[3] && z >= b[4] && z <= b[5];
}

// --------------------------------------------------- FP64 re-evaluation ----

__device__ double apex_angle64(double rx, double ry, bool &degenerate) {
    if (ry != 0.0) return atan2(ry, -rx);
    if (rx > 0.0) return -3.14159265358979323846;
    if (rx < 0.0) return 0.0;
    degenerate = true;
    return 0.0;
}

__device__ double edge_angle64(float4 Pa, float4 Pb, float qx, float qy, float qz,
                               const unsigned long long *counters) {
    const double ax = (double)Pa.x - qx, ay = (double)Pa.y - qy, az = (double)Pa.z - qz;
    const double bx = (double)Pb.x - qx, by = (double)Pb.y - qy, bz = (double)Pb.z - qz;
    const double sa = ax * ax + ay * ay, sb = bx * bx + by * by;
    const double la = sqrt(sa + az * az), lb = sqrt(sb + bz * bz);
    const double ha = az > 0.0 ? sa / (la + az) : la - az;
    const double hb = bz > 0.0 ? sb / (lb + bz) : lb - bz;
    const double n = ay * bx - ax * by;
    const double d = ha * hb + ax * bx + ay * by;
    if (n == 0.0 && d == 0.0) {
        bool deg = false;
        if (ax == 0.0 && ay == 0.0 && ha == 0.0 && !(bx == 0.0 && by == 0.0)) return apex_angle64(bx, by, deg);
        if (bx == 0.0 && by == 0.0 && hb == 0.0 && !(ax == 0.0 && ay == 0.0)) return -apex_angle64(ax, ay, deg);
        return 0.0;
    }
    if (d < 0.0) {
        const int s = branch_sos(qx, qy, Pa.x, Pa.y, Pb.x, Pb.y, counters);
        return atan2(s > 0 ? -fabs(n) : fabs(n), d);
    }
    return atan2(n, d);
}


// FP64 boundary sum of one query over the edges that start at points
// [j0, j1) of a chained point stream, for the re-evaluation kernels.  FP64 runs
// at 1/64 of the FP32 rate here, so the terms are grouped like the FP32 path:
// each point's unnormalised relative vector (l, and h = l - z without
// cancellation) is formed once and shared by its two edges, and a term with
// 0 < |n| / d < 0.41 (angle below pi/8) is multiplied into a complex product,
// one atan2 per 8 edges.  1e-30 < d < 1e30 keeps a product of 8 such factors
// inside the FP64 range whatever the coordinates' scale.  Every other term
// (steep, on the branch cut, degenerate) is edge_angle64's, exactly as before.
__device__ double bsum64_range(const float4 *__restrict__ pts, int64_t j0, int64_t j1, float qx, float qy, float qz,
                               const unsigned long long *counters) {
    if (j0 >= j1) return 0.0;
    double acc = 0.0, re = 1.0, im = 0.0;
    int g = 0;
    float4 P = pts[j0];
    double ax = (double)P.x - qx, ay = (double)P.y - qy, az = (double)P.z - qz;
    double sa = ax * ax + ay * ay;
    double la = sqrt(sa + az * az);
    double ha = az > 0.0 ? sa / (la + az) : la - az;
    for (int64_t j = j0; j < j1; ++j) {
        const float4 Q = pts[j + 1];
        const double bx = (double)Q.x - qx, by = (double)Q.y - qy, bz = (double)Q.z - qz;
        const double sb = bx * bx + by * by, lb = sqrt(sb + bz * bz);
        const double hb = bz > 0.0 ? sb / (lb + bz) : lb - bz;
        if (P.w != 0.f) {
            const double n = ay * bx - ax * by, d = ha * hb + ax * bx + ay * by;
            if (d > 1e-30 && d < 1e30 && fabs(n) < 0.41 * d) {
                const double r = re * d - im * n;
                im = re * n + im * d;
                re = r;
            } else {
                acc += edge_angle64(P, Q, qx, qy, qz, counters);
            }
            if (++g == GROUP) {
                acc += atan2(im, re);
                re = 1.0;
                im = 0.0;
                g = 0;
            }
        }
        P = Q;
        ax = bx;
        ay = by;
        az = bz;
        ha = hb;
    }
    if (g > 0) acc += atan2(im, re);
    return acc;
}

// ------------------------------------------------------- triangle loops ----
//
// A loop of three edges a -> b -> c bounds the triangle T = (a, b, c), and its
// three antipodal terms sum to (Eq. 9 for T alone)
//   2 pi S_T = atan2(det, den) - 2 pi cross(q, T),
// half T's solid angle (van Oosterom-Strackee) minus the signed crossing of the
// ray with T.  One such term costs 45 paired operations against 3 edges of about 60
// each (random soups, whose every loop is a triangle, and small holes), and its
// rounding is relative to the triangle's solid angle, not to the edges' steep angles.
// With unit vectors A, B, C toward the vertices, N the triangle's normal vector:
//   den = 1 + A.B + A.C + B.C,  det = (a . N) / (|a| |b| |c|) = (A . N') (h / (|b| |c|)),
// N = h N' with h a power of two and N' of magnitude about 1: a . N and 1 / (|a| |b| |c|)
// alone go with the cube of the coordinates, and FP32 holds neither beyond 2^42 or below
// 2^-43 (A . N' and h / (|b| |c|) it holds wherever it holds the squared distances).
// The rounding of A . N' reaches det times g = h / (|b| |c|), which is large beside b or c
// (an edge length L over the distance) and along a triangle's short edge opposite a.
// The term enters the group product if 0.41 den - |det| - g / 8 > 0.05: its angle is below
// pi/8 (8 factors stay below pi), away from the cut at +-pi, den > 0.12 and g < 13 bound
// the amplification of rounding (at most 1e-7 of w a term, in an emulation over random
// and slim triangles at 3 to 1e-5 edge lengths; without g 8e-3 at 1e-5, and 1e-4 at one
// edge length of a triangle with one edge a thousandth of the others).  Otherwise (the
// query within about an edge's length) it takes its own atan2, with the nearest vertex in
// the place of a (then |N| <= 4 times the product of the two other distances, at most
// 6e-7 of w), or, close to T, its three edges' terms.  A ray that meets the
// triangle's box takes the crossing predicate; every other ray misses T.  Both are
// deferred like the batched kernel's failing terms: about 3% of a warp's triangles have
// such a lane (random soup, 100k queries), and done in place, with most lanes idle,
// they cost more than all the rest.  Measured, edges -> triangles: soup8's direct sum with
// 2M queries 383 -> 228 ms; 3,000 random triangles with 20k queries 0.53 -> 0.18 ms,
// 20,000 with 50k 5.6 -> 2.2 ms, with 100k 10.8 -> 4.3 ms (4.0 without the test on g); the
// maximum error against FP64 on soup8 1.3e-6 -> 6.0e-7.  Bound by the FP32 pipe (62% of
// its cycles; issue 65%).
struct __align__(16) TriLoop {
    float4 a, b, c;   // the vertices; a.w = max z
    float4 n;         // (b - a) x (c - a) = n.w (n.x, n.y, n.z), n.w a power of two
    float4 box;       // min x, max x, min y, max y
};
static_assert(sizeof(TriLoop) == 80, "TriLoop must be 80 bytes");
constexpr float kTriAccept = 0.05f;
constexpr float kTriSpread = 0.125f;   // weight of g

// A triangle's term by itself, det from the nearest vertex; a, b, c: the relative vectors.
// The unit vectors are exact down to lengths of 3e-19 (a distance that something is added
// to, as the edge terms' 1e-37, is no harm there, where n and d shrink alike, but den
// is 1 plus products of unit vectors: w off by 0.1 at 1e-18).  Returns the smallest squared length.
__device__ __forceinline__ float tri_own(float4 n, float3 a, float3 b, float3 c, float &det, float &den) {
    const float la = a.x * a.x + a.y * a.y + a.z * a.z, lb = b.x * b.x + b.y * b.y + b.z * b.z,
                lc = c.x * c.x + c.y * c.y + c.z * c.z;
    float ia = sfu_rsqrt(fmaxf(la, 1e-37f)), ib = sfu_rsqrt(fmaxf(lb, 1e-37f)), ic = sfu_rsqrt(fmaxf(lc, 1e-37f));
    den = 1.f + (a.x * b.x + a.y * b.y + a.z * b.z) * (ia * ib) + (a.x * c.x + a.y * c.y + a.z * c.z) * (ia * ic) +
          (b.x * c.x + b.y * c.y + b.z * c.z) * (ib * ic);
    if (ib >= fmaxf(ia, ic)) {
        const float i = ia;
        a = b;
        ia = ib;
        ib = i;
    } else if (ic >= ia) {
        const float i = ia;
        a = c;
        ia = ic;
        ic = i;
    }
    det = (a.x * n.x + a.y * n.y + a.z * n.z) * ia * (n.w * (ib * ic));
    return fminf(la, fminf(lb, lc));
}

// The exact predicate, where the FP32 filter of tri_cross cannot decide.
__device__ __noinline__ int tri_cross_exact(const TriLoop &T, float qx, float qy, float qz,
                                            unsigned long long *counters) {
    return tri_crossing(make_float3(qx, qy, qz), make_float3(T.a.x, T.a.y, T.a.z), make_float3(T.b.x, T.b.y, T.b.z),
                        make_float3(T.c.x, T.c.y, T.c.z), &counters[CNT_EXACT_EDGE], &counters[CNT_EXACT_PLANE]);
}

// Signed crossing of the ray of a query inside the triangle's box.  The signs of the
// three projected edge functions and of the plane side are those of the exact values
// where they exceed 1e-6 of the sum of their products' magnitudes (16 units of
// rounding; at most 4 to 6 occur).  *vertex is set when the query coincides with a
// vertex (the term is then degenerate: its edges decide).
__device__ __forceinline__ int tri_cross(const TriLoop &T, float qx, float qy, float qz, bool *vertex,
                                         unsigned long long *counters) {
    const float ax = T.a.x - qx, ay = T.a.y - qy, az = T.a.z - qz, bx = T.b.x - qx, by = T.b.y - qy, bz = T.b.z - qz,
                cx = T.c.x - qx, cy = T.c.y - qy, cz = T.c.z - qz;
    *vertex = (ax == 0.f && ay == 0.f && az == 0.f) || (bx == 0.f && by == 0.f && bz == 0.f) ||
              (cx == 0.f && cy == 0.f && cz == 0.f);
    const float p0 = ax * by, m0 = ay * bx, p1 = bx * cy, m1 = by * cx, p2 = cx * ay, m2 = cy * ax;
    const float e0 = p0 - m0, e1 = p1 - m1, e2 = p2 - m2;
    const bool clear = fabsf(e0) > fmaf(1e-6f, fabsf(p0) + fabsf(m0), 1e-30f) &&
                       fabsf(e1) > fmaf(1e-6f, fabsf(p1) + fabsf(m1), 1e-30f) &&
                       fabsf(e2) > fmaf(1e-6f, fabsf(p2) + fabsf(m2), 1e-30f);
    if (clear) {
        if ((e0 > 0.f) != (e1 > 0.f) || (e0 > 0.f) != (e2 > 0.f)) return 0;
        const float nx = ax * T.n.x, ny = ay * T.n.y, nz = az * T.n.z, side = nx + ny + nz;
        if (fabsf(side) > fmaf(1e-6f, fabsf(nx) + fabsf(ny) + fabsf(nz), 1e-30f))
            return (side > 0.f) == (e0 > 0.f) ? (e0 > 0.f ? 1 : -1) : 0;
    }
    return tri_cross_exact(T, qx, qy, qz, counters);
}

__device__ __forceinline__ float4 tri_vertex(const TriLoop &T, int e) { return e == 0 ? T.a : e == 1 ? T.b : T.c; }

// The three edge terms of triangle j (of the staged tile) for the query of slot (32 k +
// lane); ill-conditioned ones go on the warp's FP64 queue (entry 3 j + edge).
__device__ __noinline__ float tri_edges(const TriLoop &T, int j, unsigned slot, float qx, float qy, float qz, const CancelQ &cq,
                                        unsigned long long *counters) {
    float sum = 0.f;
    for (int e = 0; e < 3; ++e) {
        const float4 Pa = tri_vertex(T, e), Pb = tri_vertex(T, e == 2 ? 0 : e + 1);
        const PointRel A = point_rel_twin(Pa, qx, qy, qz), B = point_rel_twin(Pb, qx, qy, qz);
        const float n = __fmaf_rn(A.ay, B.ax, -__fmul_rn(A.ax, B.ay));
        const float d = __fmaf_rn(A.h, B.h, __fmaf_rn(A.ax, B.ax, __fmul_rn(A.ay, B.ay)));
        if (cancels(n, d, A.h, B.h)) cancel_push(cq, (unsigned)(3 * j + e) << 7 | slot);
        else sum += edge_term(n, d, A, B, Pa, Pb, qx, qy, qz, counters);
    }
    return sum;
}

// entries: edges of the staged triangles
__device__ __noinline__ void tri_drain(const CancelQ &cq, const TriLoop *s_tri, unsigned long long *counters) {
    cancel_drain_edges(cq, counters, [&](int j, float4 &Pa, float4 &Pb) {
        const TriLoop &T = s_tri[j / 3];
        Pa = tri_vertex(T, j % 3);
        Pb = tri_vertex(T, j % 3 == 2 ? 0 : j % 3 + 1);
    });
}

// The warp's deferred triangle terms, drained by all 32 lanes: entry
// fail << 31 | triangle of the tile << 7 | query slot << 5 | lane.  fail: the term is not
// in the group product.  Sums go to the fixed-point accumulators (order-independent).
__device__ __noinline__ void tri_deferred(const unsigned *queue, int count, const TriLoop *s_tri, const CancelQ &cq,
                                          unsigned long long *counters) {
    const int lane = threadIdx.x & 31, warp0 = threadIdx.x & ~31;
    for (int r0 = 0; r0 < count; r0 += 32) {
        if (r0 + lane < count) {
            const unsigned e = queue[r0 + lane];
            const int owner = warp0 + (int)(e & 31u), k = (int)(e >> 5 & 3u), j = (int)(e >> 7 & 0xffffffu);
            const bool fail = e >> 31;
            const int local = owner + k * (int)blockDim.x;
            const float qx = cq.q[3 * local], qy = cq.q[3 * local + 1], qz = cq.q[3 * local + 2];
            const TriLoop &T = s_tri[j];
            bool edges = false;
            const bool inbox = qx >= T.box.x && qx <= T.box.y && qy >= T.box.z && qy <= T.box.w && qz <= T.a.w;
            const int cr = inbox ? tri_cross(T, qx, qy, qz, &edges, counters) : 0;
            float t = 0.f;
            if (fail && !edges) {   // a well-conditioned angle away from the cut takes its own atan2
                float det, den;
                const float least = tri_own(T.n, make_float3(T.a.x - qx, T.a.y - qy, T.a.z - qz),
                                            make_float3(T.b.x - qx, T.b.y - qy, T.b.z - qz),
                                            make_float3(T.c.x - qx, T.c.y - qy, T.c.z - qz), det, den);
                if (den * den + det * det > 0.01f && (den > 0.f || fabsf(det) > 0.1f) && least > 1e-37f) t = fast_atan2(det, den);
                else edges = true;
            }
            const double sum = edges ? (double)tri_edges(T, j, e & 127u, qx, qy, qz, cq, counters)
                                     : (double)t - 6.28318530717958647693 * cr;
            if (sum != 0.0)
                atomicAdd(reinterpret_cast<unsigned long long *>(cq.fix + (k * (int)blockDim.x + owner)),
                          (unsigned long long)__double2ll_rn(sum * kFixScale64));
        }
        if (cancel_count(cq.count) > kCancelCap - 96) tri_drain(cq, s_tri, counters);   // 3 edges a lane
    }
    __syncwarp();
}

// Terms of triangle loops [t_begin, t_end) for the block's 2 KP queries per thread,
// added to s_acc as in bsum_accumulate (which the caller runs after this, for the
// other loops); s_tri holds cap triangles, queue 64 KQ entries of this warp.  Every
// thread of the block must call it.
template <int KP>
__device__ __forceinline__ void tri_accumulate(const TriLoop *__restrict__ tris, int64_t t_begin, int64_t t_end, int cap,
                                               TriLoop *s_tri, const float2 (&nqx)[KP], const float2 (&nqy)[KP],
                                               const float2 (&nqz)[KP], double *s_acc, unsigned long long *counters,
                                               const CancelQ &cq, unsigned *queue) {
    constexpr int KQ = 2 * KP;
    if (t_begin >= t_end) return;
#pragma unroll
    for (int k = 0; k < KQ; ++k) cq.fix[k * blockDim.x + threadIdx.x] = 0;
    if ((threadIdx.x & 31) == 0) *cq.count = 0;
    __syncwarp();
    float2 re[KP], im[KP], part[KP], comp[KP];
    unsigned live = 0;   // query slots that are not padding past n (NaN), whose sums are never read
#pragma unroll
    for (int k = 0; k < KP; ++k)
        live |= (nqx[k].x == nqx[k].x ? 1u : 0u) << (2 * k) | (nqx[k].y == nqx[k].y ? 2u : 0u) << (2 * k);
    int q_count = 0;   // entries in the warp's queue
#pragma unroll
    for (int k = 0; k < KP; ++k) {
        re[k] = bc2(1.f);
        im[k] = bc2(0.f);
        part[k] = comp[k] = bc2(0.f);
    }
    int g = 0;
    auto close = [&]() {
#pragma unroll
        for (int k = 0; k < KP; ++k) {
            two_sum_acc2(part[k], comp[k], fast_atan2_2(im[k], re[k]));
            re[k] = bc2(1.f);
            im[k] = bc2(0.f);
        }
        g = 0;
    };
    for (int64_t t0 = t_begin; t0 < t_end; t0 += cap) {
        const int cnt = (int)min((int64_t)cap, t_end - t0);
        __syncthreads();
        const float4 *src = reinterpret_cast<const float4 *>(tris + t0);
        for (int i = threadIdx.x; i < 5 * cnt; i += blockDim.x) reinterpret_cast<float4 *>(s_tri)[i] = __ldg(src + i);
        cancel_tile<KQ>(cq);
        __syncthreads();
        for (int j = 0; j < cnt; ++j) {
            const float4 a = s_tri[j].a, b = s_tri[j].b, c = s_tri[j].c, N = s_tri[j].n, bx = s_tri[j].box;
            unsigned fail = 0, inbox = 0;
            float2 den[KP], det[KP];
#pragma unroll
            for (int k = 0; k < KP; ++k) {
                const float2 ax = add2(bc2(a.x), nqx[k]), ay = add2(bc2(a.y), nqy[k]), az = add2(bc2(a.z), nqz[k]);
                const float2 px = add2(bc2(b.x), nqx[k]), py = add2(bc2(b.y), nqy[k]), pz = add2(bc2(b.z), nqz[k]);
                const float2 cx = add2(bc2(c.x), nqx[k]), cy = add2(bc2(c.y), nqy[k]), cz = add2(bc2(c.z), nqz[k]);
                const float2 la = fma2(ax, ax, fma2(ay, ay, mul2(az, az)));
                const float2 lb = fma2(px, px, fma2(py, py, mul2(pz, pz)));
                const float2 lc = fma2(cx, cx, fma2(cy, cy, mul2(cz, cz)));
                const float2 ia = make_float2(sfu_rsqrt(la.x), sfu_rsqrt(la.y)), ib = make_float2(sfu_rsqrt(lb.x), sfu_rsqrt(lb.y)),
                             ic = make_float2(sfu_rsqrt(lc.x), sfu_rsqrt(lc.y));
                const float2 ab = fma2(ax, px, fma2(ay, py, mul2(az, pz)));
                const float2 ac = fma2(ax, cx, fma2(ay, cy, mul2(az, cz)));
                const float2 bc = fma2(px, cx, fma2(py, cy, mul2(pz, cz)));
                const float2 ibc = mul2(ib, ic);
                den[k] = fma2(bc, ibc, fma2(mul2(ac, ia), ic, fma2(mul2(ab, ia), ib, bc2(1.f))));
                const float2 dn = fma2(ax, bc2(N.x), fma2(ay, bc2(N.y), mul2(az, bc2(N.z))));
                const float2 g = mul2(bc2(N.w), ibc);
                det[k] = mul2(mul2(dn, ia), g);
                // (an infinite reciprocal length, at a vertex, makes v NaN or -infinity: not accepted)
                const float2 v = fma2(bc2(-kTriSpread), g,
                                      fma2(bc2(kTanGroup), den[k], neg2(make_float2(fabsf(det[k].x), fabsf(det[k].y)))));
                fail |= (v.x > kTriAccept ? 0u : 1u) << (2 * k) | (v.y > kTriAccept ? 0u : 2u) << (2 * k);
                inbox |= (-nqx[k].x >= bx.x && -nqx[k].x <= bx.y && -nqy[k].x >= bx.z && -nqy[k].x <= bx.w && -nqz[k].x <= a.w ? 1u : 0u) << (2 * k) |
                         (-nqx[k].y >= bx.x && -nqx[k].y <= bx.y && -nqy[k].y >= bx.z && -nqy[k].y <= bx.w && -nqz[k].y <= a.w ? 2u : 0u) << (2 * k);
            }
            fail &= live;
            // near the triangle, or below its box (every lane of the warp is here)
            if (__any_sync(0xffffffffu, fail | inbox)) {
                const unsigned lane = threadIdx.x & 31u, below = (1u << lane) - 1u;
#pragma unroll
                for (int k = 0; k < KQ; ++k) {
                    const bool mine = (fail | inbox) >> k & 1u;
                    const unsigned m = __ballot_sync(0xffffffffu, mine);
                    if (mine)
                        queue[q_count + __popc(m & below)] = (fail >> k & 1u) << 31 | (unsigned)j << 7 | (unsigned)k << 5 | lane;
                    q_count += __popc(m);
                }
                if (q_count >= 32 * KQ) {
                    __syncwarp();
                    tri_deferred(queue, q_count, s_tri, cq, counters);
                    q_count = 0;
                }
            }
#pragma unroll
            for (int k = 0; k < KP; ++k) {
                const bool fx = fail >> (2 * k) & 1u, fy = fail >> (2 * k + 1) & 1u;
                const float2 fd = make_float2(fx ? 1.f : den[k].x, fy ? 1.f : den[k].y);
                const float2 fn = make_float2(fx ? 0.f : det[k].x, fy ? 0.f : det[k].y);
                const float2 r = fma2(re[k], fd, neg2(mul2(im[k], fn)));
                im[k] = fma2(re[k], fn, mul2(im[k], fd));
                re[k] = r;
            }
            if (++g == GROUP) close();
        }
        if (g > 0) close();
        __syncwarp();
        if (q_count > 0) {   // the entries index this tile's triangles
            tri_deferred(queue, q_count, s_tri, cq, counters);
            q_count = 0;
        }
        if (cancel_count(cq.count) > 0) tri_drain(cq, s_tri, counters);
#pragma unroll
        for (int k = 0; k < KP; ++k) {
            s_acc[(2 * k) * blockDim.x + threadIdx.x] += (double)part[k].x + (double)comp[k].x;
            s_acc[(2 * k + 1) * blockDim.x + threadIdx.x] += (double)part[k].y + (double)comp[k].y;
            part[k] = comp[k] = bc2(0.f);
        }
    }
    __syncwarp();
#pragma unroll
    for (int k = 0; k < KQ; ++k)
        s_acc[k * blockDim.x + threadIdx.x] += (double)cq.fix[k * blockDim.x + threadIdx.x] * kFixUnit;
}

}  // namespace

}  // namespace gwn
