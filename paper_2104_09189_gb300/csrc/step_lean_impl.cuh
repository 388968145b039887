// step_lean_impl.cuh -- the step kernel of the FP64 path where nothing is
// counted or reported: a lean pass per node, and the full node step
// (step_node) for the few nodes it leaves.
//
// step_node carries the state of Algorithm 1 through the exact stage, the
// hop cap and the fallback walk, and spills it on the path every node takes.  Here a node either finishes by
//   foot -> FP32 test of T^0 -> FP32 hops (from T^0, or from the jump table
//   when the foot is far) -> certified test -> value
// or is handed, with nothing kept, to step_node, which starts over.  What is
// left to it: signs the certified test cannot decide (the exact stage), a foot
// between triangles that a walk reached (which triangle it is depends on the
// path, and step_node's is the path from T^0), and walks that meet a
// boundary or do not settle in a few certified hops.  The foot, the numerators
// and the value are step_node's functions and the triangle that holds a foot
// in its inside is one, so the results are step_node's bit for bit.
#pragma once

#include "step_fast_impl.cuh"

namespace sl {

// The FP32 test of a triangle (A, B, C): the edge to cross (0, 1, 2: opposite
// A, B, C), the most negative of the orientations certainly below zero, or -1
// when none is.  Bounds as in step_node.
__device__ __forceinline__ int outside_edge(float4 A, float4 B, float4 C, float X, float Y)
{
    const float ax = A.x - C.x, ay = A.y - C.y, bx = B.x - C.x, by = B.y - C.y;
    const float xx = X - C.x, xy = Y - C.y;
    const float o1 = __fmaf_rn(xx, by, -__fmul_rn(xy, bx));
    const float o2 = __fmaf_rn(ax, xy, -__fmul_rn(ay, xx));
    const float dn = __fmaf_rn(ax, by, -__fmul_rn(ay, bx));
    const float o3 = dn - o1 - o2;
    const float S = fabsf(ax) + fabsf(ay) + fabsf(bx) + fabsf(by) + fabsf(xx) + fabsf(xy);
    const float e = hop_bound(S);
    const float e3 = 3.0f * e + 0x1p-23f * (fabsf(dn) + fabsf(o1) + fabsf(o2));
    int k = -1;
    float best = 0.0f;
    if (o1 < -e) { k = 0; best = o1; }
    if (o2 < -e && (k < 0 || o2 < best)) { k = 1; best = o2; }
    if (o3 < -e3 && (k < 0 || o3 < best)) k = 2;
    return k;
}

// FP32 hops from triangle (A, B, C) with start code e across its edge k to the
// triangle where no exit is certainly negative; returns a half-edge code of
// that triangle (of the start triangle when edge k is on the boundary).
template <bool kCompact>
__device__ __forceinline__ int32_t lean_hops_from(const FastArgs &a, int32_t e, int k, float4 A, float4 B, float4 C,
                                                  float X, float Y)
{
    // the next triangle: (W2, W1, Q), (W0, W2, Q) or (W1, W0, Q)
    const float p0x = k == 1 ? A.x : (k == 0 ? C.x : B.x), p0y = k == 1 ? A.y : (k == 0 ? C.y : B.y);
    const float p1x = k == 0 ? B.x : (k == 1 ? C.x : A.x), p1y = k == 0 ? B.y : (k == 1 ? C.y : A.y);
    uint32_t hops = 1;
    if (kCompact) {
        const uint2 R = __ldg(&a.he8[e + k]);
        int32_t e0 = he8_e0(R), d1 = he8_d1(R);
        if (tri_of(e0) == tri_of(e)) return e;
        const float2 Q = he8_vertex(R, p0x, p0y);
        lean_hops8(a.he8, __fsub_rn(p0x, X), __fsub_rn(p0y, Y), __fsub_rn(p1x, X), __fsub_rn(p1y, Y),
                   __fsub_rn(Q.x, X), __fsub_rn(Q.y, Y), e0, d1, hops, (uint32_t)a.walk_cap, a.hop_L);
        return e0;
    }
    const float4 R = __ldg(&a.he[e + k]);
    if (isnan(R.x)) return e;
    int32_t e0 = __float_as_int(R.z), e1 = __float_as_int(R.w);
    lean_hops(a, X, Y, p0x, p0y, p1x, p1y, R.x, R.y, e0, e1, hops, (uint32_t)a.walk_cap);
    return e0;
}

// The certified test's verdict on triangle j that the single-bound test left
// open: the signs as step_node takes them.  0..2: the edge to cross (the most
// negative barycentric coordinate); kIn: inside, perhaps on a boundary edge;
// kInShared: on a boundary vertex, between triangles; kOpen: a sign is left to
// the exact stage.
enum { kIn = 3, kInShared = 4, kOpen = 5 };
__device__ __forceinline__ int certified_verdict(const FastArgs &a, int32_t j, df X, df Y, const Numerators &t)
{
    const Certified u = certify_bounds(t);
    int s1 = u.n1.h > u.ea ? 1 : (u.n1.h < -u.ea ? -1 : 2);
    int s2 = u.n2.h > u.eb ? 1 : (u.n2.h < -u.eb ? -1 : 2);
    float n3h = u.n3h;
    int s3 = n3h > u.e3 ? 1 : (n3h < -u.e3 ? -1 : 2);
    if (s3 == 2) {
        const df n3 = df_sub(df_sub(u.den, u.n1), u.n2);
        const float ec = u.ed + u.ea + u.eb + 0x1p-45f * (fabsf(u.den.h) + fabsf(u.n1.h) + fabsf(u.n2.h));
        n3h = n3.h;
        s3 = n3.h > ec ? 1 : (n3.h < -ec ? -1 : 2);
    }
    if (s1 == 2 || s2 == 2 || s3 == 2) {
        const uint32_t fside = (df_is(X, 0.0f) ? 1u : 0u) | (df_is(X, 1.0f) ? 2u : 0u) |
                               (df_is(Y, 0.0f) ? 4u : 0u) | (df_is(Y, 1.0f) ? 8u : 0u);
        if (fside) {
            if (s1 == 2) { const int32_t nb = a.tn[0][j]; if (nb < 0 && (fside >> (-1 - nb) & 1u)) s1 = 0; }
            if (s2 == 2) { const int32_t nb = a.tn[1][j]; if (nb < 0 && (fside >> (-1 - nb) & 1u)) s2 = 0; }
            if (s3 == 2) { const int32_t nb = a.tn[2][j]; if (nb < 0 && (fside >> (-1 - nb) & 1u)) s3 = 0; }
        }
        if (s1 == 2 || s2 == 2 || s3 == 2) return kOpen;
    }
    if (s1 >= 0 && s2 >= 0 && s3 >= 0) return (s1 == 0) + (s2 == 0) + (s3 == 0) > 1 ? kInShared : kIn;
    int k = -1;
    float best = 0.0f;
    if (s1 < 0) { k = 0; best = u.n1.h; }
    if (s2 < 0 && (k < 0 || u.n2.h < best)) { k = 1; best = u.n2.h; }
    if (s3 < 0 && (k < 0 || n3h < best)) k = 2;
    return k;
}

// One node; false: nothing was written and the node is left to step_node.
template <bool kExt, bool kCompact, bool kSingle>
__device__ __forceinline__ bool lean_node(const FastArgs &a, int64_t i, int pi)
{
    const FastProb &P = kSingle ? a.prob0 : a.probs[pi];
    if (!kSingle && (P.flags & kFastUse)) {
        float2 v;
        if (!apply_weights(a, i, v)) return false;
        put_value(a, i, v);
        return true;
    }
    df X, Y;
    bool at_node, gone;
    float moves;
    const bool clipped = foot_pair<-1, kExt, true>(a, i, P, X, Y, at_node, gone, &moves);
    const float2 *vin = (const float2 *)a.vin;
    if (kExt && gone) {
        keep_value(a, i);
        return true;
    }
    bool moved = false, jumped = false;
    int4 tq;
    if (a.jump && !at_node && jump_moves(moves, P)) {
        tq = jump_start(a, P, X.h, Y.h);
        moved = jumped = true;
    } else {
        tq = kExt && a.grid_M > 0 ? __ldg(&a.grid_t0v[grid_slot(X.h, Y.h, a.grid_M)]) : a.t0v[i];
    }
    if (at_node) {
        // the foot is its own node: see step_node
        if (tq.y != (int32_t)i && tq.z != (int32_t)i && tq.w != (int32_t)i) return false;
        keep_value(a, i);
        if (P.flags & kFastEmit) emit_own(a, i);
        return true;
    }
    float4 A = a.xyq[tq.y], B = a.xyq[tq.z], C = a.xyq[tq.w];
    for (;;) {
        const int k = outside_edge(A, B, C, X.h, Y.h);
        if (k < 0) break;
        if (!jumped && a.jump && jump_far(X.h - C.x, Y.h - C.y, P)) {
            tq = jump_start(a, P, X.h, Y.h);
            A = a.xyq[tq.y];
            B = a.xyq[tq.z];
            C = a.xyq[tq.w];
            moved = jumped = true;
            continue;
        }
        const int32_t e = lean_hops_from<kCompact>(a, tq.x, k, A, B, C, X.h, Y.h);
        tq = __ldg(&a.tri[tri_of(e)]);
        A = a.xyq[tq.y];
        B = a.xyq[tq.z];
        C = a.xyq[tq.w];
        moved = true;
        break;
    }
    float2 V1, V2, V3;
    Numerators t;
    for (int n = 0;; ++n) {
        V1 = vin[tq.y];
        V2 = vin[tq.z];
        V3 = vin[tq.w];
        t = numerators(A, B, C, X.h, X.l, Y.h, Y.l);
        if (settle_test(t)) break;
        const int d = certified_verdict(a, tri_of(tq.x), X, Y, t);
        // between triangles the path decides: step_node's, as long as the FP32
        // walk from T^0 ended here
        if (d == kIn || (d == kInShared && !jumped && n == 0)) break;
        if (d >= kIn || n == a.lean_moves) return false;
        const int32_t u = a.tn[d][tri_of(tq.x)];
        if (u < 0) return false;
        tq = __ldg(&a.tri[u]);
        A = a.xyq[tq.y];
        B = a.xyq[tq.z];
        C = a.xyq[tq.w];
        moved = true;
    }
    if (a.io & kIoIn) {
        pair_in(a, V1);
        pair_in(a, V2);
        pair_in(a, V3);
    }
    float2 val;
    if (!clipped && steep(V1, V2, V3, t.den.h, a.steep_g2))
        val = precise_value(a.xyd, a.g1, a.g2, P, i, tq.y, tq.z, tq.w, V1, V2, V3);
    else
        val = p1_value_of(V1, V2, V3, t.n1, t.n2, t.den);
    put_value(a, i, val);
    if (P.flags & kFastEmit) emit_weights(a, i, tq.y, tq.z, tq.w, t.n1, t.n2, t.den, clipped);
    if (moved && !(kExt && a.keep_t0)) a.t0v[i] = tq;
    return true;
}

template <int kBlock, int kMinBlocks, bool kExt, bool kCompact, bool kSingle>
__global__ void __launch_bounds__(kBlock, kMinBlocks) k_lean_df(const __grid_constant__ FastArgs a)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    pdl_launch_dependents();
    pdl_wait();
    if (i >= a.N) return;
    const int pi = kSingle || a.nprob == 1 ? 0 : chunk_problem(a.chunk_prob, a.node_off, i);
    if (lean_node<kExt, kCompact, kSingle>(a, i, pi)) return;
    NodeCounters c;
    step_node<false, true, kExt, kCompact>(a, i, pi, c);
}

template <int kBlock, int kMinBlocks, bool kExt = false>
inline void launch_lean_df_cfg(const FastArgs &a, cudaStream_t s)
{
    const unsigned grid = (unsigned)((a.N + kBlock - 1) / kBlock);
    if (grid == 0) return;
    if (a.he8) {
        if (a.single) launch_step_kernel(k_lean_df<kBlock, kMinBlocks, kExt, true, true>, grid, kBlock, s, a);
        else launch_step_kernel(k_lean_df<kBlock, kMinBlocks, kExt, true, false>, grid, kBlock, s, a);
    } else {
        if (a.single) launch_step_kernel(k_lean_df<kBlock, kMinBlocks, kExt, false, true>, grid, kBlock, s, a);
        else launch_step_kernel(k_lean_df<kBlock, kMinBlocks, kExt, false, false>, grid, kBlock, s, a);
    }
}

}  // namespace sl
