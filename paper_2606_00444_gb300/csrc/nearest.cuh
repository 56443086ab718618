// NearestSurface on the device (Eq. 1 / Eq. 2, Sec. 3.3): the point-triangle and
// point-box distances, the tie rule's bookkeeping and the writing of a hit,
// shared by every search (query.cu, pool.cu), so that they all evaluate the same
// expressions and give the same answers, bit for bit.
#pragma once

#include <climits>
#include <math.h>

#include "common.cuh"

namespace meshgs {

constexpr int kQueryBlock = 128;
constexpr int kQueryMinBlocks = 8;    // 8 x 128 threads per SM: at most 64 registers
constexpr int kStackShared = 24;      // entries per thread in shared memory
constexpr int kStackTotal = kMaxTreeDepth;   // every tree is at most this deep: the Karras tree by
                                             // its bound (30 key bits + log2 nF + 1), the
                                             // agglomerative one by the build's depth check

__device__ __forceinline__ float box_d2(float3 q, float4 lo, float4 hi) {
    float dx = fmaxf(fmaxf(lo.x - q.x, q.x - hi.x), 0.0f);
    float dy = fmaxf(fmaxf(lo.y - q.y, q.y - hi.y), 0.0f);
    float dz = fmaxf(fmaxf(lo.z - q.z, q.z - hi.z), 0.0f);
    return dx * dx + dy * dy + dz * dz;
}

// MinMaxDist of Roussopoulos, Kelley & Vincent (1995) for a tight AABB: every
// face of the box touches the geometry inside it, so some primitive in the box
// lies within this distance of q.  It bounds the nearest distance from above
// before any triangle is tested and orders children whose boxes both contain q.
__device__ __forceinline__ float box_minmax_d2(float3 q, float4 lo, float4 hi) {
    float mx = 0.5f * (lo.x + hi.x), my = 0.5f * (lo.y + hi.y), mz = 0.5f * (lo.z + hi.z);
    float nx = q.x - (q.x <= mx ? lo.x : hi.x), fx = q.x - (q.x >= mx ? lo.x : hi.x);
    float ny = q.y - (q.y <= my ? lo.y : hi.y), fy = q.y - (q.y >= my ? lo.y : hi.y);
    float nz = q.z - (q.z <= mz ? lo.z : hi.z), fz = q.z - (q.z >= mz ? lo.z : hi.z);
    float f2x = fx * fx, f2y = fy * fy, f2z = fz * fz;
    float S = f2x + f2y + f2z;
    return fminf(fminf(S - f2x + nx * nx, S - f2y + ny * ny), S - f2z + nz * nz);
}

// The products and sums of a face's distance are rounded as written here, not as
// the compiler would contract them in each kernel: a computed distance decides
// ties, so every search must round it the same way.
__device__ __forceinline__ float dot3(float3 a, float3 b) {
    return __fmaf_rn(a.z, b.z, __fmaf_rn(a.x, b.x, __fmul_rn(a.y, b.y)));
}
// a b - c d
__device__ __forceinline__ float det2(float a, float b, float c, float d) { return __fmaf_rn(a, b, -__fmul_rn(c, d)); }
// x - t d
__device__ __forceinline__ float3 along(float3 x, float t, float3 d) {
    return make_float3(__fmaf_rn(-t, d.x, x.x), __fmaf_rn(-t, d.y, x.y), __fmaf_rn(-t, d.z, x.z));
}
// x - (v e + w f)
__device__ __forceinline__ float3 across(float3 x, float v, float3 e, float w, float3 f) {
    return make_float3(__fsub_rn(x.x, __fmaf_rn(e.x, v, __fmul_rn(f.x, w))),
                       __fsub_rn(x.y, __fmaf_rn(e.y, v, __fmul_rn(f.y, w))),
                       __fsub_rn(x.z, __fmaf_rn(e.z, v, __fmul_rn(f.z, w))));
}
__device__ __forceinline__ float3 sub3(float3 a, float3 b) {
    return make_float3(a.x - b.x, a.y - b.y, a.z - b.z);
}
__device__ __forceinline__ float3 xyz(float4 v) { return make_float3(v.x, v.y, v.z); }

// Closest point of segment xy to p: parameter t in [0, 1] and squared distance.
// The residual is formed from p - x (small when p is near the segment), never
// from absolute coordinates, so its rounding scales with the segment length.
__device__ __forceinline__ float seg_d2(float3 p, float3 x, float3 y, float &t) {
    float3 d = sub3(y, x), xp = sub3(p, x);
    float L = dot3(d, d);
    t = 0.0f;
    if (L > 0.0f) t = fminf(fmaxf(dot3(xp, d) / L, 0.0f), 1.0f);
    const float3 r = along(xp, t, d);
    return dot3(r, r);
}

// Closest point on triangle abc to p (Ericson, Real-Time Collision Detection
// 5.1.5: Voronoi regions of vertices, edges, face).  Faces flagged as exactly
// zero-area at build / refit use the nearest of their three edges instead.
// Returns the squared distance and the barycentric weights (u, v, w).  The
// residual p - closest point is assembled from the vertex-relative vectors
// (p - a, b - a, ...), so float32 rounding is relative to the triangle's size,
// not to the magnitude of the coordinates.
__device__ __forceinline__ float tri_closest(float3 p, float3 a, float3 b, float3 c, bool degenerate,
                                             float &u, float &v, float &w) {
    if (degenerate) {
        float t0, t1, t2;
        float s0 = seg_d2(p, a, b, t0), s1 = seg_d2(p, b, c, t1), s2 = seg_d2(p, c, a, t2);
        if (s0 <= s1 && s0 <= s2) { u = 1.0f - t0; v = t0; w = 0.0f; return s0; }
        if (s1 <= s2) { u = 0.0f; v = 1.0f - t1; w = t1; return s1; }
        u = t2; v = 0.0f; w = 1.0f - t2;
        return s2;
    }
    float3 ab = sub3(b, a), ac = sub3(c, a);
    float3 ap = sub3(p, a);
    float d1 = dot3(ab, ap), d2 = dot3(ac, ap);
    if (d1 <= 0.0f && d2 <= 0.0f) { u = 1.0f; v = 0.0f; w = 0.0f; return dot3(ap, ap); }
    float3 bp = sub3(p, b);
    float d3 = dot3(ab, bp), d4 = dot3(ac, bp);
    if (d3 >= 0.0f && d4 <= d3) { u = 0.0f; v = 1.0f; w = 0.0f; return dot3(bp, bp); }
    float vc = det2(d1, d4, d3, d2);
    float3 r;
    if (vc <= 0.0f && d1 >= 0.0f && d3 <= 0.0f) {
        float t = d1 / (d1 - d3);
        u = 1.0f - t; v = t; w = 0.0f;
        r = along(ap, t, ab);
    } else {
        float3 cp = sub3(p, c);
        float d5 = dot3(ab, cp), d6 = dot3(ac, cp);
        if (d6 >= 0.0f && d5 <= d6) { u = 0.0f; v = 0.0f; w = 1.0f; return dot3(cp, cp); }
        float vb = det2(d5, d2, d1, d6);
        if (vb <= 0.0f && d2 >= 0.0f && d6 <= 0.0f) {
            float t = d2 / (d2 - d6);
            u = 1.0f - t; v = 0.0f; w = t;
            r = along(ap, t, ac);
        } else {
            float va = det2(d3, d6, d5, d4);
            if (va <= 0.0f && (d4 - d3) >= 0.0f && (d5 - d6) >= 0.0f) {
                float t = (d4 - d3) / ((d4 - d3) + (d5 - d6));
                u = 0.0f; v = 1.0f - t; w = t;
                float3 bc = sub3(c, b);
                r = along(bp, t, bc);
            } else {
                float s = 1.0f / (va + vb + vc);
                v = vb * s;
                w = vc * s;
                u = 1.0f - v - w;
                r = across(ap, v, ab, w, ac);
            }
        }
    }
    return dot3(r, r);
}

// The squared distance of tri_closest alone, without its branches: the lanes of a
// warp hold triangles in different regions, and every region's code would run
// in turn.  The region is decided by the same tests in the same order, one
// quotient and one residual are formed from the operands it selects, and each
// is the expression of tri_closest, so the distance is the same, bit for bit.
__device__ __forceinline__ float tri_distance2(float3 p, float3 a, float3 b, float3 c, bool degenerate) {
    if (degenerate) {
        float u, v, w;
        return tri_closest(p, a, b, c, true, u, v, w);
    }
    const float3 ab = sub3(b, a), ac = sub3(c, a), bc = sub3(c, b);
    const float3 ap = sub3(p, a), bp = sub3(p, b), cp = sub3(p, c);
    const float d1 = dot3(ab, ap), d2 = dot3(ac, ap), d3 = dot3(ab, bp), d4 = dot3(ac, bp), d5 = dot3(ab, cp),
                d6 = dot3(ac, cp);
    const float vc = det2(d1, d4, d3, d2), vb = det2(d5, d2, d1, d6), va = det2(d3, d6, d5, d4);
    const float e43 = d4 - d3, e56 = d5 - d6;
    const bool inA = d1 <= 0.0f && d2 <= 0.0f;
    const bool inB = !inA && d3 >= 0.0f && d4 <= d3;
    const bool onAB = !inA && !inB && vc <= 0.0f && d1 >= 0.0f && d3 <= 0.0f;
    const bool pre = inA || inB || onAB;
    const bool inC = !pre && d6 >= 0.0f && d5 <= d6;
    const bool onAC = !pre && !inC && vb <= 0.0f && d2 >= 0.0f && d6 <= 0.0f;
    const bool onBC = !pre && !inC && !onAC && va <= 0.0f && e43 >= 0.0f && e56 >= 0.0f;
    const bool vertex = inA || inB || inC;
    float num = 1.0f, den = va + vb + vc;                     // the face's interior
    if (onBC) { num = e43; den = e43 + e56; }
    if (onAC) { num = d2; den = d2 - d6; }
    if (onAB) { num = d1; den = d1 - d3; }
    if (vertex) { num = 0.0f; den = 1.0f; }
    const float t = num / den;
    const float3 base = inB || onBC ? bp : inC ? cp : ap;
    const float3 dir = onBC ? bc : onAC ? ac : ab;
    const float3 re = along(base, t, dir), rf = across(ap, vb * t, ab, vc * t, ac);
    const float3 r = vertex || onAB || onAC || onBC ? re : rf;
    return dot3(r, r);
}

// The same region test in float64, used only to recompute the weights of the
// winning face when float32 would lose them: a query far from the face relative
// to its shortest edge (weight error grows like eps32 * d / edge) or a sliver.
struct D3 {
    double x, y, z;
};
__device__ __forceinline__ D3 dsub(D3 a, D3 b) { return D3{a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ double ddot(D3 a, D3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ D3 dof(float3 a) { return D3{a.x, a.y, a.z}; }

static __device__ __noinline__ void tri_weights_f64(float3 pf, float3 af, float3 bf, float3 cf,
                                             bool degenerate, float &u, float &v, float &w) {
    D3 p = dof(pf), a = dof(af), b = dof(bf), c = dof(cf);
    double U, V, W;
    if (degenerate) {
        D3 P[3] = {a, b, c};
        double best = 1e300, bt = 0.0;
        int be = 0;
        for (int e = 0; e < 3; ++e) {
            D3 x = P[e], d = dsub(P[(e + 1) % 3], x), xp = dsub(p, x);
            double L = ddot(d, d), t = 0.0;
            if (L > 0.0) t = fmin(fmax(ddot(xp, d) / L, 0.0), 1.0);
            D3 r = D3{xp.x - t * d.x, xp.y - t * d.y, xp.z - t * d.z};
            double s = ddot(r, r);
            if (s < best) { best = s; bt = t; be = e; }
        }
        if (be == 0) { U = 1.0 - bt; V = bt; W = 0.0; }
        else if (be == 1) { U = 0.0; V = 1.0 - bt; W = bt; }
        else { U = bt; V = 0.0; W = 1.0 - bt; }
    } else {
        D3 ab = dsub(b, a), ac = dsub(c, a), ap = dsub(p, a), bp = dsub(p, b), cp = dsub(p, c);
        double d1 = ddot(ab, ap), d2 = ddot(ac, ap), d3 = ddot(ab, bp), d4 = ddot(ac, bp);
        double d5 = ddot(ab, cp), d6 = ddot(ac, cp);
        double vc = d1 * d4 - d3 * d2, vb = d5 * d2 - d1 * d6, va = d3 * d6 - d5 * d4;
        if (d1 <= 0.0 && d2 <= 0.0) { U = 1.0; V = 0.0; W = 0.0; }
        else if (d3 >= 0.0 && d4 <= d3) { U = 0.0; V = 1.0; W = 0.0; }
        else if (vc <= 0.0 && d1 >= 0.0 && d3 <= 0.0) { double t = d1 / (d1 - d3); U = 1.0 - t; V = t; W = 0.0; }
        else if (d6 >= 0.0 && d5 <= d6) { U = 0.0; V = 0.0; W = 1.0; }
        else if (vb <= 0.0 && d2 >= 0.0 && d6 <= 0.0) { double t = d2 / (d2 - d6); U = 1.0 - t; V = 0.0; W = t; }
        else if (va <= 0.0 && (d4 - d3) >= 0.0 && (d5 - d6) >= 0.0) {
            double t = (d4 - d3) / ((d4 - d3) + (d5 - d6));
            U = 0.0; V = 1.0 - t; W = t;
        } else {
            double s = 1.0 / (va + vb + vc);
            V = vb * s; W = vc * s; U = 1.0 - V - W;
        }
    }
    u = (float)U; v = (float)V; w = (float)W;
}

// True when float32 weights of this face would be too coarse for the query.
// Their error grows like ~8 eps32 d / l_min (measured), so beyond 12 shortest
// edges it could approach 1e-5; slivers (altitude < 5% of the longest edge)
// are ill-conditioned at any distance.  Float64 is slow on this part, so the
// threshold keeps the float64 path off near-surface queries entirely.
__device__ __forceinline__ bool weights_need_f64(float3 a, float3 b, float3 c, float d2) {
    float3 ab = sub3(b, a), ac = sub3(c, a), bc = sub3(c, b);
    float l0 = dot3(ab, ab), l1 = dot3(ac, ac), l2 = dot3(bc, bc);
    float lmin = fminf(l0, fminf(l1, l2)), lmax = fmaxf(l0, fmaxf(l1, l2));
    float3 n = make_float3(ab.y * ac.z - ab.z * ac.y, ab.z * ac.x - ab.x * ac.z, ab.x * ac.y - ab.y * ac.x);
    return d2 > 144.0f * lmin || dot3(n, n) < 2.5e-3f * lmax * lmax;
}

struct Hit {
    int leaf;      // -1: nothing within the cutoff
    int face;
    float d2;
};

// Float32 error bound of a computed point-triangle or point-box distance for a
// query q on a mesh whose coordinates are at most vmax in magnitude.  Every
// difference such as q - a is below 2 s in magnitude, s = max(|q|_inf, vmax),
// and the residual assembled from such differences (and the box distance)
// carries at most about 30 eps32 s of rounding; 2^-18 s = 64 eps32 s covers
// it with a margin.  Pruning widened by this bound never skips a face whose
// computed distance lies inside the tie window, whatever the tree.
constexpr float kSlackScale = 0x1p-18f;

struct Traversal {
    const float4 *__restrict__ nodes;
    const float4 *__restrict__ tris;
    int n;
    float tau;     // absolute floor of the tie window (1e-12 of the box diagonal)
    float vmax;    // largest coordinate magnitude of the mesh box
    bool mmd;      // use MinMaxDist bounds (unbounded queries; a cutoff is tighter)
    const float4 *__restrict__ wide;   // the 4-wide records (traversal variant 13)
};

__device__ __forceinline__ float query_slack(const Traversal &T, float3 q) {
    return kSlackScale * fmaxf(fmaxf(fabsf(q.x), fabsf(q.y)), fmaxf(fabsf(q.z), T.vmax));
}

// The two thresholds of a nearest squared distance m: w2, the tie window (a
// face with d2 <= w2 counts as equally near), and p2, the pruning radius (the
// window widened by the float32 bound `slack`, so a box whose computed
// distance exceeds p2 holds no face whose computed distance is within w2).
__device__ __forceinline__ void windows(float m, float tau, float slack, float &w2, float &p2) {
    float r = sqrtf(m) * (1.0f + kTieRel) + tau;
    w2 = r * r;
    r += slack;
    p2 = r * r;
}

// Pruning radius implied by an upper bound u2 on the nearest squared distance
// (a MinMaxDist): some face lies within sqrt(u2) in exact arithmetic, so the
// final nearest computed distance is at most sqrt(u2) + slack; u2 itself is
// widened by 4e-5 relative for its own rounding.
__device__ __forceinline__ float bound_window2(float u2, float tau, float slack) {
    float r = (sqrtf(u2 * 1.00004f) + slack) * (1.0f + kTieRel) + tau + slack;
    return r * r;
}

// Pruning radius before any hit: the cutoff itself, widened the same way
// (faces just past the cutoff can still fall in the tie window of a hit).
__device__ __forceinline__ float cutoff_window2(float maxd2, float tau, float slack) {
    if (isinf(maxd2)) return INFINITY;
    float r = sqrtf(maxd2) * (1.0f + kTieRel) + tau + slack;
    return r * r;
}

// Candidate bookkeeping of the tie rule.  dmin is the nearest squared
// distance seen; the kept face (leaf `leaf`, its face id read back from the
// packed triangle when a tie needs it) is the lowest id among the faces seen
// within the window of dmin -- as long as every face seen inside the current
// window, other than the kept one, has a higher id.  `other` is the least
// squared distance of the faces seen and not kept; when the kept face leaves
// the shrinking window while `other` is still inside it, one of those faces
// may have the lowest id, and `other` is set to -1: the query is resolved at
// the end by one search with the final window fixed (resolve_ties).  The
// answer is therefore the lowest id within the final window, whatever the
// order in which faces were met.  Five registers, as the search carries them
// through every node visit.
struct Best {
    int leaf;
    float d2, dmin, thr, other;
};

__device__ __forceinline__ int face_of(const Traversal &T, int leaf) {
    return __float_as_int(ldg4(T.tris + 3 * (size_t)leaf).w);
}

__device__ __forceinline__ Best make_best(const Traversal &T, float3 q, float maxd2) {
    return Best{-1, INFINITY, INFINITY, cutoff_window2(maxd2, T.tau, query_slack(T, q)), INFINITY};
}

__device__ __forceinline__ void consider(const Traversal &T, Best &B, float3 q, int leaf, int face,
                                         float d2, float maxd2) {
    float nmin = fminf(B.dmin, d2);
    if (nmin > maxd2) {                       // no hit yet and this face is past the cutoff:
        B.other = fminf(B.other, d2);         // noted only (it may fall in a later hit's window)
        return;
    }
    float w2, p2;
    windows(nmin, T.tau, query_slack(T, q), w2, p2);
    if (d2 <= w2) {
        if (B.leaf >= 0 && B.d2 <= w2) {      // the kept face stays inside the window: a tie
            if (leaf != B.leaf) {
                if (face < face_of(T, B.leaf)) {
                    B.other = fminf(B.other, B.d2);
                    B.leaf = leaf; B.d2 = d2;
                } else {
                    B.other = fminf(B.other, d2);
                }
            }
        } else {                              // first hit, or the kept face left the window
            if (B.other <= w2) B.other = -1.0f;
            B.leaf = leaf; B.d2 = d2;
        }
    }
    B.dmin = nmin;
    B.thr = fminf(B.thr, p2);
}

__device__ __forceinline__ void test_leaf(const Traversal &T, Best &B, int leaf, float3 q,
                                          float maxd2) {
    const float4 *t = T.tris + 3 * (size_t)leaf;
    float4 a = ldg4(t), b = ldg4(t + 1), c = ldg4(t + 2);
    float u, v, w;
    float d2 = tri_closest(q, xyz(a), xyz(b), xyz(c), b.w != 0.0f, u, v, w);
    consider(T, B, q, leaf, __float_as_int(a.w), d2, maxd2);
}

// The faces of a leaf link: first = -link - 1, cnt from the record's hi.w (1
// without leaf collapse).  The first face's box is the link's box when cnt is
// 1; the others are tested against their own box first (computed from the
// corners just loaded), so a face far outside the window costs no region test.
// kRange = false (a tree without leaf collapse) compiles to the single face
// alone: the leaf-range loop costs the one-thread searches ~10 % even when
// every count is 1, so the kernels come in both forms and the host picks the
// plain one for leaf size 1.
template <bool kRange>
__device__ __forceinline__ void test_range(const Traversal &T, Best &B, int first, int cnt, float3 q,
                                           float maxd2) {
    if constexpr (!kRange) {
        test_leaf(T, B, first, q, maxd2);
        return;
    }
    // one call site of the region test; the per-face box test only runs for a
    // real range
#pragma unroll 1
    for (int k = 0; k < cnt; ++k) {
        const float4 *t = T.tris + 3 * (size_t)(first + k);
        float4 a = ldg4(t), b = ldg4(t + 1), c = ldg4(t + 2);
        if (cnt > 1) {
            float4 lo = make_float4(fminf(fminf(a.x, b.x), c.x), fminf(fminf(a.y, b.y), c.y),
                                    fminf(fminf(a.z, b.z), c.z), 0.0f);
            float4 hi = make_float4(fmaxf(fmaxf(a.x, b.x), c.x), fmaxf(fmaxf(a.y, b.y), c.y),
                                    fmaxf(fmaxf(a.z, b.z), c.z), 0.0f);
            if (box_d2(q, lo, hi) > B.thr) continue;
        }
        float u, v, w;
        float d2 = tri_closest(q, xyz(a), xyz(b), xyz(c), b.w != 0.0f, u, v, w);
        consider(T, B, q, first + k, __float_as_int(a.w), d2, maxd2);
    }
}

__device__ __forceinline__ int link_count(float4 hi) { return __float_as_int(hi.w); }

// The tie rule with the window fixed: one depth-first search that visits every
// box within the pruning radius of B.dmin and keeps the lowest face id whose
// distance lies within its window.  Run only for the rare queries whose online
// bookkeeping could not decide (three or more faces within about 2e-6 of one
// another, met in an order that moved the window past the kept one).
static __device__ __noinline__ void resolve_ties(const Traversal &T, Best &B, float3 q,
                                          unsigned int *status) {
    float w2, p2;
    windows(B.dmin, T.tau, query_slack(T, q), w2, p2);
    int bl = -1, bf = 0x7fffffff;
    float bd = INFINITY;
    auto test = [&](int leaf) {
        const float4 *t = T.tris + 3 * (size_t)leaf;
        float4 a = ldg4(t), b = ldg4(t + 1), c = ldg4(t + 2);
        float u, v, w;
        float d2 = tri_closest(q, xyz(a), xyz(b), xyz(c), b.w != 0.0f, u, v, w);
        int f = __float_as_int(a.w);
        if (d2 <= w2 && f < bf) { bl = leaf; bf = f; bd = d2; }
    };
    if (T.n == 1) {
        test(0);
    } else if (T.n > 1) {
        int stk[kStackTotal];
        int sp = 0, node = 0;
        while (true) {
            const float4 *r = T.nodes + 4 * (size_t)node;
            float4 l0 = ldg4(r), l1 = ldg4(r + 1), r0 = ldg4(r + 2), r1 = ldg4(r + 3);
            int cl = __float_as_int(l0.w), cr = __float_as_int(r0.w);
            bool il = box_d2(q, l0, l1) <= p2, ir = box_d2(q, r0, r1) <= p2;
            if (il && cl < 0)
                for (int k = 0; k < link_count(l1); ++k) test(-cl - 1 + k);
            if (ir && cr < 0)
                for (int k = 0; k < link_count(r1); ++k) test(-cr - 1 + k);
            bool gl = il && cl >= 0, gr = ir && cr >= 0;
            if (gl && gr) {
                if (sp < kStackTotal) stk[sp++] = cr;
                else atomicOr(status, (unsigned)MESH_DEV_STACK_OVERFLOW);
                node = cl;
                continue;
            }
            if (gl) { node = cl; continue; }
            if (gr) { node = cr; continue; }
            if (sp == 0) break;
            node = stk[--sp];
        }
    }
    if (bl >= 0) { B.leaf = bl; B.d2 = bd; }
    B.other = INFINITY;
}

__device__ __forceinline__ Hit finish(const Traversal &T, Best &B, float3 q, unsigned int *status) {
    if (B.other < 0.0f) resolve_ties(T, B, q, status);
    return Hit{B.leaf, B.leaf >= 0 ? face_of(T, B.leaf) : 0x7fffffff, B.d2};
}

// Per-mesh constants of the tie rule from the mesh box: the window's absolute
// floor (1e-12 of the box diagonal) and the largest coordinate magnitude.
__device__ __forceinline__ void set_scale(Traversal &T, float4 lo, float4 hi) {
    float dx = hi.x - lo.x, dy = hi.y - lo.y, dz = hi.z - lo.z;
    T.tau = kTieAbs * sqrtf(dx * dx + dy * dy + dz * dz);
    T.vmax = fmaxf(fmaxf(fmaxf(fabsf(lo.x), fabsf(hi.x)), fmaxf(fabsf(lo.y), fabsf(hi.y))),
                   fmaxf(fabsf(lo.z), fabsf(hi.z)));
    if (!(T.vmax < INFINITY)) T.vmax = 0.0f;   // empty mesh: an inverted (infinite) box
}
__device__ __forceinline__ void set_scale(Traversal &T, const Header *hdr) {
    set_scale(T, hdr->root_lo, hdr->root_hi);
}

// The weights and closest point of a hit on leaf `leaf` (squared distance d2),
// recomputed from the packed triangle.
__device__ __forceinline__ void write_weights(const Traversal &T, int leaf, float d2, float3 q, int64_t i,
                                              float *bary, float *point) {
    const float4 *t = T.tris + 3 * (size_t)leaf;
    float4 a = ldg4(t), b = ldg4(t + 1), c = ldg4(t + 2);
    float u, v, w;
    tri_closest(q, xyz(a), xyz(b), xyz(c), b.w != 0.0f, u, v, w);
    if (weights_need_f64(xyz(a), xyz(b), xyz(c), d2))
        tri_weights_f64(q, xyz(a), xyz(b), xyz(c), b.w != 0.0f, u, v, w);
    if (bary) { bary[3 * i] = u; bary[3 * i + 1] = v; bary[3 * i + 2] = w; }
    if (point) {
        point[3 * i] = u * a.x + v * b.x + w * c.x;
        point[3 * i + 1] = u * a.y + v * b.y + w * c.y;
        point[3 * i + 2] = u * a.z + v * b.z + w * c.z;
    }
}

// Writes the outputs of one query (recomputing the weights of the winning face).
__device__ __forceinline__ void write_hit(const Traversal &T, const Hit &h, float3 q, int64_t i,
                                          int *face, float *bary, float *point, float *dist2) {
    if (h.leaf < 0) {
        if (face) face[i] = -1;
        if (dist2) dist2[i] = INFINITY;
        if (bary) { bary[3 * i] = 0.0f; bary[3 * i + 1] = 0.0f; bary[3 * i + 2] = 0.0f; }
        if (point) { point[3 * i] = 0.0f; point[3 * i + 1] = 0.0f; point[3 * i + 2] = 0.0f; }
        return;
    }
    if (face) face[i] = h.face;
    if (dist2) dist2[i] = h.d2;
    if (bary || point) write_weights(T, h.leaf, h.d2, q, i, bary, point);
}

// The pooled search (pool.cu) with G lanes per query (a power of two from 2 to 32; the
// Chamfer kernel also 1, 32 queries per warp).  G = 0: the mesh has at most kFewFaces
// faces (a batch's scenes on average), each tested by a thread per query; the Chamfer
// kernel then takes 128 samples per block.
constexpr int kFewFaces = 24;
void pool_closest_point(const mesh_bvh *b, Traversal T, const float *Q, int64_t nQ, float maxd2, int G, int *face,
                        float *bary, float *point, float *dist2, const int *hint, cudaStream_t s);
void pool_signed(const mesh_bvh *b, Traversal T, const float *Q, int64_t nQ, float maxd2, int G, int *face, float *bary,
                 float *point, float *sdist, cudaStream_t s);

// One direction of the Chamfer distance: samples S searched on T's mesh.
struct ChamferSide {
    Traversal T;
    const Header *hdr;
    const float *S;
    int64_t n;
    int *face;
    float *bary, *dist2;
    const int *hint;               // warm start: a face id per sample (-1 = none), may alias face
    const int *iperm;              // face -> leaf of the mesh searched
};
// grid blocks of 128 / G samples, the first nbA of them a2b's.
void pool_chamfer(int G, bool range, const ChamferSide &a2b, const ChamferSide &b2a, unsigned nbA, unsigned grid,
                  unsigned *status, double *partial, unsigned *ticket, double *out, cudaStream_t s);
// Projection onto the k (1 to kKnnMax) nearest faces (mesh_knn_project).
constexpr int kKnnMax = 8;
void pool_knn(const mesh_bvh *b, Traversal T, const float *Q, int64_t nQ, int k, int G, const float *anchor,
              float anchor_w, float *point, int *face, float *d2, cudaStream_t s);
void pool_batch(const mesh_batch *b, const float *Q, const int *query_off, int64_t nQ, float maxd2, bool mmd, int G,
                int *face, float *bary, float *point, float *dist2, cudaStream_t s);

}  // namespace meshgs
