// Far field of the boundary sum: a binary hierarchy over the chained boundary
// points whose nodes carry multipole moments, so that a query sums a distant part
// of dM with one expansion instead of one term per edge.
//
// A node covers a contiguous range of the chained points: whole loops, and at its
// ends at most two pieces of a loop that a cut divides.  Each such piece plus the
// chord from its end back to its start is closed, so
//   sum of the node's edge terms = w_N(q) + the chords' own terms,
// where w_N is the winding number of any surface that spans the closed curves
// inside their convex hull, provided the ray q + t z misses that hull (no
// crossing, so the antipodal sum of the closed curves is w_N itself, Eq. 9).
// w_N is harmonic outside the node's ball (centre c, radius s) and has the
// exterior expansion
//   w_N(q) = -(1/4pi) sum_{l,m} conj(M_lm) I_l^m(q - c),
//   M_lm = integral of n . grad R_l^m over the spanning surface
//        = 1/(l+1) sum over the edges of (a x b) . integral grad R_l^m ds
// (the cone over an edge from c; R, I the regular and irregular solid harmonics).
// Truncated at degree P the error is at most
//   E / r^(P+2) [(P+1)/(1-y) + y/(1-y)^2],  y = s/r,
//   E = (1/4pi) sum over fan triangles of area max|p - c|^P,
// so every node gets the smallest radius at which that bound is eps, and a
// query uses the node's expansion only outside that radius and only if its ray
// misses the node's box.  The choice depends on the query and the node alone.
// eps is kFarEps, or less where the expansions of a query (the most that any of 1,024
// sample points takes) would add up to more than half the mesh's classify_margin; the
// other half is left to FP32 rounding, so that labels stay exact.  A mesh whose margin
// would take eps below kFarEpsMin is summed directly.  With the default margin soup8 (at
// most 407 expansions a query) and smaller soups keep kFarEps; 200,000 small quads (1M
// points, 2249) take 1.4e-8 and half as many operations more.
//
// Degree 8 with leaves of 16 points: degrees 6 and 10 cost the same or more on soup8,
// leaves of 32 points 10% more.  Loops in Hilbert order instead of Morton order: 30%
// fewer expansions and 40% fewer near edges per query (no jumps inside a range).
// The hierarchy is used where its mean cost over sample points is at most kFarWorth
// of the direct sum's (a warp takes the union over its queries, 1.5 to 2 times the
// mean).  Random soups of large triangles overlap everywhere and stay with the direct
// sum; of small holes, 3.2k points (0.8 of the direct sum with triangle loops) are
// faster directly (200k queries: 413 against 506 us), 12k points (0.26) are not (1491
// against 831 us).
#pragma once

#include "gwn_internal.cuh"

namespace gwn {

constexpr int kFarP = 8;                                  // degree of the expansions
constexpr int kFarRaw = (kFarP + 1) * (kFarP + 2) / 2;    // complex moments (l, m >= 0), l = 0 unused
constexpr int kFarCoef = kFarP * (kFarP + 2);             // packed real coefficients (80)
constexpr float kFarEps = 1e-7f;                          // truncation bound of one expansion, in w (at most)
constexpr float kFarEpsMin = 1e-9f;                       // below an expansion's own rounding
constexpr int kFarLeaf = 16;                              // target points of a leaf (at most twice that)
constexpr float kFarGradEps = 2e-6f;                      // truncation bound of one gradient, times the box's side
constexpr int kFarGradCoef = 3 * (kFarP + 2 * (kFarP * (kFarP + 3) / 2));   // 288: x, y, z
constexpr double kFarWorth = 0.5;                         // used below this share of the direct sum's cost
// Built from this many points on.  (Wavy rims: of 150 to 1,000 points no hierarchy passes
// kFarWorth; of 1,500 one does, 1M queries 2.59 -> 1.60 ms.)
constexpr int kFarMinPoints = 1024;
constexpr int kFarRoots = 64;                             // subtrees a walk may be split into (at most)
// A leaf of fewer edges is summed directly.  Limits 1 / 10 / 17: query, soup6 with 100k
// queries 584 / 583 / 646 us, soup8 with 200k 2432 / 2413 / 2715; gradient 891 / 883 / 859 and
// 5682 / 5684 / 5117 us.
constexpr int kFarMinEdges = 10;

// Preorder node, 80 bytes.  A leaf's skip is its own index + 1.
struct __align__(16) FarNode {
    float cx, cy, cz, r2acc;            // centre; the expansion holds for |q - c|^2 > r2acc
    float xmin, xmax, ymin, ymax;       // box of the points: the ray test (with a small margin)
    float zmax, inv_s;                  // its top; 1 / radius, the expansion's unit of length
    int32_t skip, nchord;               // next node after the subtree; chords (0 to 2)
    int32_t begin, count;               // the points whose edges the node covers
    float r2grad, gpad;                 // the gradient's: |q - c|^2 > r2grad, the ray outside the box widened by gpad
    int32_t ch[4];                      // chords ch[0] -> ch[1], ch[2] -> ch[3] (point indices)
};
static_assert(sizeof(FarNode) == 80, "FarNode must be 80 bytes");

// The expansion's basis: with Z = z / r^2, U = 1 / r^2 (in units of s), T_mm = 1,
//   T_lm = Z T_(l-1)m - beta_lm U T_(l-2)m,  beta = ((l-1)^2 - m^2) / ((2l-1)(2l-3)),
//   value = sum_m Re[((x + i y) / r^2)^m / r * sum_l conj(C_lm) T_lm],
// C_lm = M_lm with the constants folded in (k_far_pack), packed m-major: the p
// coefficients of m = 0, then (re, im) for each m >= 1, l >= m.
__host__ __device__ constexpr float far_beta(int l, int m) {
    return (float)((l - 1) * (l - 1) - m * m) / (float)((2 * l - 1) * (2 * l - 3));
}
__host__ __device__ constexpr int far_idx(int l, int m) { return l * (l + 1) / 2 + m; }
// first packed coefficient of column m >= 1
__host__ __device__ constexpr int far_col(int m) { return kFarP + (m - 1) * (2 * kFarP + 2 - m); }

// The gradient of an expansion is one of degrees 2..P+1 in the same basis for each
// component (derivatives of I_l^m are I_(l+1)^(m-1..m+1)): P real coefficients for
// m = 0, then (re, im) for m = 1..P+1, l = max(m, 2)..P+1.
__host__ __device__ constexpr int far_grad_first(int m) { return m < 2 ? 2 : m; }   // lowest degree of column m
__host__ __device__ constexpr int far_grad_col(int m) {   // first entry (complex) of column m >= 1, after column 0
    int c = 0;
    for (int k = 1; k < m; ++k) c += kFarP + 2 - far_grad_first(k);
    return c;
}
constexpr int kFarGradCols = far_grad_col(kFarP + 2);   // 44 complex entries
static_assert(kFarGradCoef == 3 * (kFarP + 2 * kFarGradCols), "gradient coefficients");

// Position of cell (x, y, z), 2^bits cells per axis, on the Hilbert curve (Skilling
// 2004, "Programming the Hilbert curve").  Neighbours on the curve are neighbours in
// space, without the jumps of the Morton order.
__host__ __device__ inline uint32_t hilbert_key(uint32_t x, uint32_t y, uint32_t z, int bits) {
    uint32_t X[3] = {x, y, z};
    for (uint32_t Q = 1u << (bits - 1); Q > 1; Q >>= 1) {
        const uint32_t mask = Q - 1;
        for (int i = 0; i < 3; ++i) {
            if (X[i] & Q) {
                X[0] ^= mask;
            } else {
                const uint32_t t = (X[0] ^ X[i]) & mask;
                X[0] ^= t;
                X[i] ^= t;
            }
        }
    }
    X[1] ^= X[0];
    X[2] ^= X[1];
    uint32_t t = 0;
    for (uint32_t Q = 1u << (bits - 1); Q > 1; Q >>= 1)
        if (X[2] & Q) t ^= Q - 1;
    uint32_t key = 0;
    for (int b = bits - 1; b >= 0; --b)
        for (int i = 0; i < 3; ++i) key = key << 1 | ((X[i] ^ t) >> b & 1u);
    return key;
}

// farfield.cu: builds m->far_* for the chained points pts (loops in the order of
// the Hilbert keys of their first points, so that a range of points is compact)
// when the hierarchy is expected to pay, and takes ownership of pts; ends: per
// point (first, closing) point index of its loop
gwn_status build_far(gwn_mesh *m, float4 *pts, const uint2 *ends, cudaStream_t s);

}  // namespace gwn
