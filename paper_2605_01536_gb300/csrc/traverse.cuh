// Stackless walk of the escape-linked BVH for a +z ray, shared by the
// per-query crossing count and the grid (ray-reuse) kernels.
#pragma once

#include "gwn_internal.cuh"
#include "predicates.cuh"
#include "quant.cuh"

namespace gwn {

// Visit every leaf whose node box admits the +z ray from p (p.xy inside the
// closed xy box and p.z <= zmax, every bound widened by pad), in depth-first
// order, calling on_leaf(slot, a, b, c) with the leaf's triangle slot and
// vertices.  Returns false (and sets the traversal error flag) if the walk
// leaves the node array or exceeds its node budget (a corrupt tree), so it
// never loops or reads out of range.  Count = true adds the nodes read to
// *visits (the instrumented walk; the timed kernels compile without it);
// read_leaves = false skips the leaves' triangles (node counting only).
template <bool Padded = false, bool Count = false, class OnLeaf>
__device__ __forceinline__ bool bvh_walk_up(float3 p, const BvhNode *__restrict__ nodes, int64_t nnodes,
                                            const float4 *__restrict__ tri, unsigned long long *__restrict__ counters,
                                            OnLeaf &&on_leaf, float pad = 0.f, unsigned *visits = nullptr) {
    int node = nnodes > 0 ? 0 : -1;
    int64_t budget = nnodes + 1;   // depth-first order visits each node at most once
    while (node >= 0) {
        if constexpr (Count) ++*visits;
        if (--budget < 0 || node >= nnodes) {
            atomicOr(&counters[CNT_ERROR], (unsigned long long)ERR_TRAVERSAL_LIMIT);
            return false;
        }
        const float4 *np = reinterpret_cast<const float4 *>(nodes + node);
        const float4 b0 = __ldg(np);
        const float4 b1 = __ldg(np + 1);
        const int child = __float_as_int(b1.y), skip = __float_as_int(b1.z), leaf = __float_as_int(b1.w);
        const bool hit = Padded ? (p.x >= b0.x - pad && p.x <= b0.y + pad && p.y >= b0.z - pad &&
                                   p.y <= b0.w + pad && p.z <= b1.x + pad)
                                : (p.x >= b0.x && p.x <= b0.y && p.y >= b0.z && p.y <= b0.w && p.z <= b1.x);
        if (hit && leaf) {
            if ((unsigned)child >= (unsigned)((nnodes + 1) / 2)) {
                atomicOr(&counters[CNT_ERROR], (unsigned long long)ERR_TRAVERSAL_LIMIT);
                return false;
            }
            const float4 a = __ldg(tri + 3 * child), bb = __ldg(tri + 3 * child + 1),
                         cc = __ldg(tri + 3 * child + 2);
            on_leaf(child, make_float3(a.x, a.y, a.z), make_float3(bb.x, bb.y, bb.z), make_float3(cc.x, cc.y, cc.z));
            node = skip;
        } else {
            node = hit ? child : skip;
        }
    }
    return true;
}

// The walk of one ray by the 32 lanes of a warp together: the subtrees still to visit
// lie on a stack in shared memory and each round tests up to 32 of their roots.  A ray
// that runs along a surface tests tens of thousands of nodes, and as one lane's chain of
// dependent loads that takes milliseconds.  Items: node << 2 | follow; follow 1 adds the
// node's escape link as an item of its own (the sibling of a left child), 2 the whole
// chain of escape links (the rest of a depth-first walk that stands at the node).
// on_leaf runs on the lane that tests the leaf; the leaves are those of bvh_walk_up.
// Every lane must call it with the same arguments; stack: kFrontierCap entries of the warp.
constexpr int kFrontierCap = 512;
template <class OnLeaf>
__device__ __forceinline__ bool bvh_frontier_warp(float3 p, int start, int follow, const BvhNode *__restrict__ nodes,
                                                  int64_t nnodes, const float4 *__restrict__ tri,
                                                  unsigned long long *__restrict__ counters,
                                                  unsigned long long *stack, OnLeaf &&on_leaf) {
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    int count = start >= 0 && start < nnodes ? 1 : 0;
    if (lane == 0) stack[0] = (unsigned long long)start << 2 | (unsigned)follow;
    __syncwarp();
    int64_t budget = nnodes + 1;   // each node at most once
    while (count > 0) {
        // an item is replaced by at most two: near the stack's end one at a time, so that
        // it grows by at most the tree's depth (below 64 levels, two items each)
        const int k = count > kFrontierCap - 192 ? 1 : min(count, 32);
        budget -= k;
        if (budget < 0 || count > kFrontierCap - 2) {
            if (lane == 0) atomicOr(&counters[CNT_ERROR], (unsigned long long)ERR_TRAVERSAL_LIMIT);
            return false;
        }
        const bool mine = lane < k;
        const unsigned long long item = mine ? stack[count - 1 - lane] : 0ull;
        __syncwarp();
        count -= k;
        int child = -1, next = -1;
        const int follows = (int)(item & 3u);
        if (mine) {
            const int node = (int)(item >> 2);
            const float4 *np = reinterpret_cast<const float4 *>(nodes + node);
            const float4 b0 = __ldg(np), b1 = __ldg(np + 1);
            if (follows) next = __float_as_int(b1.z);
            if (p.x >= b0.x && p.x <= b0.y && p.y >= b0.z && p.y <= b0.w && p.z <= b1.x) {
                const int c = __float_as_int(b1.y);
                if (__float_as_int(b1.w)) {
                    const float4 a = __ldg(tri + 3 * (int64_t)c), bb = __ldg(tri + 3 * (int64_t)c + 1),
                                 cc = __ldg(tri + 3 * (int64_t)c + 2);
                    on_leaf(c, make_float3(a.x, a.y, a.z), make_float3(bb.x, bb.y, bb.z), make_float3(cc.x, cc.y, cc.z));
                } else {
                    child = c;
                }
            }
        }
        const unsigned mn = __ballot_sync(0xffffffffu, next >= 0), mc = __ballot_sync(0xffffffffu, child >= 0);
        if (next >= 0) stack[count + __popc(mn & below)] = (unsigned long long)next << 2 | (follows == 2 ? 2u : 0u);
        count += __popc(mn);
        if (child >= 0) stack[count + __popc(mc & below)] = (unsigned long long)child << 2 | 1u;
        count += __popc(mc);
        __syncwarp();
    }
    return true;
}

// The walk of bvh_walk_up taken by the 32 lanes of a warp together, with the
// leaves postponed so that the warp tests them in step: a lane that reaches a
// hit leaf holds it and walks on; reaching a second one it stops; the warp
// tests one held leaf per lane once the lanes holding a leaf are at least twice
// as many as those still looking for their first, or when no lane can walk
// (measured against 1x, 4x and "none looking": the leaf-heavy degenerate
// precision workload gains up to 25% with later phases, the node-heavy soup8
// walk loses up to 14%; 2x keeps soup8 and takes 9% of the gain).
// Each lane visits the same leaves in the same order as bvh_walk_up (on_leaf
// gets the same calls), and its node budget counts the same visits.  Every
// lane of the warp must call it; a lane without a query passes active = false.
// Limited: a lane that has tested kWalkLimit nodes stops after the leaves it holds and
// leaves the node it stands at in *rest (-1: done) for bvh_frontier_warp.
constexpr int kWalkLimit = 192;
template <bool Limited = false, class OnLeaf>
__device__ __forceinline__ bool bvh_walk_up_warp(bool active, float3 p, const BvhNode *__restrict__ nodes,
                                                 int64_t nnodes, const float4 *__restrict__ tri,
                                                 unsigned long long *__restrict__ counters, OnLeaf &&on_leaf,
                                                 int *rest = nullptr) {
    int left = kWalkLimit;
    if constexpr (Limited) *rest = -1;
    int node = active && nnodes > 0 ? 0 : -1;
    int held = -1, next = -1;   // the leaf to test next and the one after it
    int64_t budget = nnodes + 1;
    bool ok = true;
    const unsigned nleaves = (unsigned)((nnodes + 1) / 2);
    while (true) {
        const bool movable = node >= 0 && next < 0;
        const unsigned holders = __ballot_sync(0xffffffffu, held >= 0);
        const unsigned movers = __ballot_sync(0xffffffffu, movable);
        if (!holders && !movers) break;
        const unsigned searching = movers & ~holders;
        if (holders && (!searching || __popc(holders) >= 2 * __popc(searching))) {
            if (held >= 0) {
                const float4 a = __ldg(tri + 3 * held), bb = __ldg(tri + 3 * held + 1), cc = __ldg(tri + 3 * held + 2);
                on_leaf(held, make_float3(a.x, a.y, a.z), make_float3(bb.x, bb.y, bb.z),
                        make_float3(cc.x, cc.y, cc.z));
                held = next;
                next = -1;
            }
            continue;
        }
        if (!movable) continue;
        if constexpr (Limited) {
            if (--left < 0) {
                *rest = node;
                node = -1;
                continue;
            }
        }
        if (--budget < 0 || node >= nnodes) {
            atomicOr(&counters[CNT_ERROR], (unsigned long long)ERR_TRAVERSAL_LIMIT);
            ok = false;
            node = held = next = -1;
            continue;
        }
        const float4 *np = reinterpret_cast<const float4 *>(nodes + node);
        const float4 b0 = __ldg(np);
        const float4 b1 = __ldg(np + 1);
        const int child = __float_as_int(b1.y), skip = __float_as_int(b1.z), leaf = __float_as_int(b1.w);
        const bool hit = p.x >= b0.x && p.x <= b0.y && p.y >= b0.z && p.y <= b0.w && p.z <= b1.x;
        if (hit && leaf) {
            if ((unsigned)child >= nleaves) {
                atomicOr(&counters[CNT_ERROR], (unsigned long long)ERR_TRAVERSAL_LIMIT);
                ok = false;
                node = held = next = -1;
                continue;
            }
            if (held < 0) held = child;
            else next = child;
            node = skip;
        } else {
            node = hit ? child : skip;
        }
    }
    return ok;
}

// Signed +z crossing count of one query with the snapped (fixed-point)
// predicates of a mesh built with quantize_bits: the float boxes are widened by
// one quantum so that snapping never hides a crossing.
static __device__ __noinline__ int chi_one_q(float3 p, const BvhNode *__restrict__ nodes, int64_t nnodes,
                                      const float4 *__restrict__ tri, unsigned long long *__restrict__ counters,
                                      const QFrame *qf) {
    const long long qx = qcoord(p.x, qf->cx, qf->scale), qy = qcoord(p.y, qf->cy, qf->scale),
                    qz = qcoord(p.z, qf->cz, qf->scale);
    const int4 *lq = qf->leaf_q;
    int c = 0;
    const bool ok = bvh_walk_up<true>(
        p, nodes, nnodes, tri, counters,
        [&](int slot, float3, float3, float3) {
            c += tri_crossing_q(qx, qy, qz, lq[3 * slot], lq[3 * slot + 1], lq[3 * slot + 2]);
        },
        qf->pad);
    return ok ? c : INT32_MIN;
}

// Signed +z crossing count of one query with the predicates decided exactly on
// the FP32 inputs (Sec. 3.2, Supp. S2.1).  INT32_MIN on a corrupt tree.
__device__ __forceinline__ int chi_one_exact(float3 p, const BvhNode *__restrict__ nodes, int64_t nnodes,
                                             const float4 *__restrict__ tri,
                                             unsigned long long *__restrict__ counters) {
    int c = 0;
    const bool ok = bvh_walk_up(p, nodes, nnodes, tri, counters, [&](int, float3 a, float3 b, float3 cc) {
        c += tri_crossing(p, a, b, cc, &counters[CNT_EXACT_EDGE], &counters[CNT_EXACT_PLANE]);
    });
    return ok ? c : INT32_MIN;
}

// Signed +z crossing count of one query in the mesh's predicate mode (exact on
// the FP32 inputs, or fixed point), read from its status block.
__device__ __forceinline__ int chi_one(float3 p, const BvhNode *__restrict__ nodes, int64_t nnodes,
                                       const float4 *__restrict__ tri, unsigned long long *__restrict__ counters) {
    const QFrame *qf = qframe(counters);
    if (qf->bits) return chi_one_q(p, nodes, nnodes, tri, counters, qf);
    int c = 0;
    const bool ok = bvh_walk_up(p, nodes, nnodes, tri, counters, [&](int, float3 a, float3 b, float3 cc) {
        c += tri_crossing(p, a, b, cc, &counters[CNT_EXACT_EDGE], &counters[CNT_EXACT_PLANE]);
    });
    return ok ? c : INT32_MIN;
}

}  // namespace gwn
