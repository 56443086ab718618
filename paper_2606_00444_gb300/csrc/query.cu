// NearestSurface queries (Eq. 1 / Eq. 2, Sec. 3.3): the entry points, the choice
// of search, and the one-thread searches (variants 1-13); the default is the
// pooled search of pool.cu.
//
// One thread per query.  A node record holds both children's boxes, so a
// visit is one 64-byte read that tests two boxes.  Leaf children (single
// faces) are tested on the spot; of two surviving internal children the
// nearer is entered and the farther pushed, with its box distance, on a
// per-thread stack kept in shared memory ([depth][thread], conflict free)
// that spills to a small local array.  Boxes are pruned against the tie
// window of the nearest distance found so far, widened by the float32 error
// bound of a computed distance, so no face whose computed distance could fall
// inside the final window is ever skipped.  The nearest face is the lowest id
// within that final window (see Best), the same for every tree, traversal
// order and warm start: a function of the query and the mesh alone.
#include <climits>
#include <math.h>

#include <mutex>

#include "common.cuh"
#include "nearest.cuh"

namespace meshgs {

// kSmem: stack entries per thread kept in shared memory (the rest spill to a
// local array; 0 = all local, leaving the SM's L1 to the node cache).
// kOneSite: leaf children are gathered and tested at one call site (the nearer
// first) instead of one site per child, so lanes testing a left and a right
// leaf in the same step run the same instructions together.
struct Counts {
    int visits, tests;
};

// hint_leaf >= 0: a leaf tested before the traversal (a warm start, e.g. the
// previous frame's nearest face); its distance bounds the search from the
// first node on.  Every leaf within the final tie window is still reached and
// the tie rule does not depend on the order, so the answer is the same as
// without the hint; only the work changes.
template <int kBlockT, int kSmem = kStackShared, bool kOneSite = false, bool kCount = false,
          bool kRange = false>
__device__ __forceinline__ Hit nearest(const Traversal &T, float3 q, float maxd2,
                                       int2 (*stk)[kBlockT], unsigned int *status,
                                       Counts *cnt = nullptr, int hint_leaf = -1) {
    Best B = make_best(T, q, maxd2);
    if (hint_leaf >= 0) test_leaf(T, B, hint_leaf, q, maxd2);
    if (T.n == 1) {
        if constexpr (kCount) cnt->tests++;
        test_leaf(T, B, 0, q, maxd2);
    } else if (T.n > 1) {
        int2 spill[kStackTotal - kSmem];
        int sp = 0;
        int node = 0;
        const int tid = threadIdx.x;
        while (true) {
            const float4 *r = T.nodes + 4 * (size_t)node;
            if constexpr (kCount) cnt->visits++;
            float4 l0 = ldg4(r), l1 = ldg4(r + 1), r0 = ldg4(r + 2), r1 = ldg4(r + 3);
            float dl = box_d2(q, l0, l1), dr = box_d2(q, r0, r1);
            float ml = 0.0f, mr = 0.0f;
            if (T.mmd) {
                ml = box_minmax_d2(q, l0, l1);
                mr = box_minmax_d2(q, r0, r1);
                B.thr = fminf(B.thr, bound_window2(fminf(ml, mr), T.tau, query_slack(T, q)));
            }
            int cl = __float_as_int(l0.w), cr = __float_as_int(r0.w);
            if constexpr (kCount)
                cnt->tests += (cl < 0 && dl <= B.thr ? link_count(l1) : 0) +
                              (cr < 0 && dr <= B.thr ? link_count(r1) : 0);
            if constexpr (kOneSite) {
                bool tl = cl < 0 && dl <= B.thr, tr = cr < 0 && dr <= B.thr;
                int la = tl ? -cl - 1 : -cr - 1, lb = -cr - 1;
                int na = tl ? link_count(l1) : link_count(r1), nb = link_count(r1);
                bool two = tl && tr;
                if (two && dr < dl) { int t = la; la = lb; lb = t; t = na; na = nb; nb = t; }
#pragma unroll 1
                for (int k = 0; k < 2; ++k) {
                    if (k == 0 ? !(tl || tr) : !two) break;
                    test_range<kRange>(T, B, k == 0 ? la : lb, k == 0 ? na : nb, q, maxd2);
                }
            } else {
                if (cl < 0 && dl <= B.thr) test_range<kRange>(T, B, -cl - 1, link_count(l1), q, maxd2);
                if (cr < 0 && dr <= B.thr) test_range<kRange>(T, B, -cr - 1, link_count(r1), q, maxd2);
            }
            bool gl = cl >= 0 && dl <= B.thr;
            bool gr = cr >= 0 && dr <= B.thr;
            if (gl && gr) {
                bool lfirst = dl < dr || (dl == dr && ml <= mr);
                int2 e = make_int2(lfirst ? cr : cl, __float_as_int(lfirst ? dr : dl));
                if (sp < kSmem) stk[sp][tid] = e;
                else if (sp < kStackTotal) spill[sp - kSmem] = e;
                else atomicOr(status, (unsigned)MESH_DEV_STACK_OVERFLOW);
                if (sp < kStackTotal) ++sp;
                node = lfirst ? cl : cr;
                continue;
            }
            if (gl) { node = cl; continue; }
            if (gr) { node = cr; continue; }
            bool found = false;
            while (sp > 0) {
                --sp;
                int2 e = sp < kSmem ? stk[sp][tid] : spill[sp - kSmem];
                if (__int_as_float(e.y) <= B.thr) { node = e.x; found = true; break; }
            }
            if (!found) break;
        }
    }
    return finish(T, B, q, status);
}

// Depth-first over the 4-wide records (variant 13): each visit tests up to four
// boxes -- the node's children, an internal child replaced by its own two --
// so a search takes about half the visits of the binary one, each reading one
// 128-byte record.  Leaf slots are tested first (they may shrink the window),
// then the internal slots still within it are ordered by box distance: the
// nearest is entered, the others pushed farthest first.  The pruning, the
// candidate bookkeeping and the tie rule are those of nearest(), so the answer
// is the same, bit for bit.  cnt->visits counts 4-wide records.
constexpr int kWideStack = 3 * kStackTotal / 2 + 2;   // up to 3 pushes per record, half the depth
constexpr int kWideEmpty = INT_MIN;

__device__ __forceinline__ void wide_swap(float &da, int &ca, float &db, int &cb) {
    if (db < da) {
        float t = da; da = db; db = t;
        int u = ca; ca = cb; cb = u;
    }
}

template <int kBlockT, int kSmem, bool kCount, bool kRange, bool kMmd>
__device__ __forceinline__ Hit nearest_wide_t(const Traversal &T, float3 q, float maxd2,
                                              int2 (*stk)[kBlockT], unsigned int *status, Counts *cnt,
                                              int hint_leaf) {
    Best B = make_best(T, q, maxd2);
    if (hint_leaf >= 0) test_leaf(T, B, hint_leaf, q, maxd2);
    if (T.n == 1) {
        if constexpr (kCount) cnt->tests++;
        test_leaf(T, B, 0, q, maxd2);
    } else if (T.n > 1) {
        const float4 *__restrict__ W = T.wide;
        int2 spill[kWideStack - kSmem];
        int sp = 0;
        int node = 0;
        const int tid = threadIdx.x % kBlockT;
        while (true) {
            const float4 *r = W + 8 * (size_t)node;
            if constexpr (kCount) cnt->visits++;
            const float4 lo0 = ldg4(r), hi0 = ldg4(r + 1), lo1 = ldg4(r + 2), hi1 = ldg4(r + 3), lo2 = ldg4(r + 4),
                         hi2 = ldg4(r + 5), lo3 = ldg4(r + 6), hi3 = ldg4(r + 7);
            float d0 = box_d2(q, lo0, hi0), d1 = box_d2(q, lo1, hi1), d2 = box_d2(q, lo2, hi2),
                  d3 = box_d2(q, lo3, hi3);
            int c0 = __float_as_int(lo0.w), c1 = __float_as_int(lo1.w), c2 = __float_as_int(lo2.w),
                c3 = __float_as_int(lo3.w);
            if constexpr (kMmd) {
                float u = INFINITY;
                if (c0 != kWideEmpty) u = fminf(u, box_minmax_d2(q, lo0, hi0));
                if (c1 != kWideEmpty) u = fminf(u, box_minmax_d2(q, lo1, hi1));
                if (c2 != kWideEmpty) u = fminf(u, box_minmax_d2(q, lo2, hi2));
                if (c3 != kWideEmpty) u = fminf(u, box_minmax_d2(q, lo3, hi3));
                B.thr = fminf(B.thr, bound_window2(u, T.tau, query_slack(T, q)));
            }
            // leaf slots (the face count of a leaf link is read only with leaf collapse)
            auto leaf = [&](int c, float d, float hw) {
                if (c < 0 && c != kWideEmpty && d <= B.thr) {
                    const int m = kRange ? __float_as_int(hw) : 1;
                    if constexpr (kCount) cnt->tests += m;
                    test_range<kRange>(T, B, -c - 1, m, q, maxd2);
                }
            };
            leaf(c0, d0, hi0.w);
            leaf(c1, d1, hi1.w);
            leaf(c2, d2, hi2.w);
            leaf(c3, d3, hi3.w);
            float k0 = (c0 >= 0 && d0 <= B.thr) ? d0 : INFINITY;
            float k1 = (c1 >= 0 && d1 <= B.thr) ? d1 : INFINITY;
            float k2 = (c2 >= 0 && d2 <= B.thr) ? d2 : INFINITY;
            float k3 = (c3 >= 0 && d3 <= B.thr) ? d3 : INFINITY;
            const int nin = (k0 < INFINITY) + (k1 < INFINITY) + (k2 < INFINITY) + (k3 < INFINITY);
            if (nin > 0) {
                wide_swap(k0, c0, k1, c1);
                wide_swap(k2, c2, k3, c3);
                wide_swap(k0, c0, k2, c2);
                wide_swap(k1, c1, k3, c3);
                wide_swap(k1, c1, k2, c2);
                auto push = [&](int c, float k) {
                    const int2 e = make_int2(c, __float_as_int(k));
                    if (sp < kSmem) stk[sp][tid] = e;
                    else if (sp < kWideStack) spill[sp - kSmem] = e;
                    else atomicOr(status, (unsigned)MESH_DEV_STACK_OVERFLOW);
                    if (sp < kWideStack) ++sp;
                };
                if (nin > 3) push(c3, k3);
                if (nin > 2) push(c2, k2);
                if (nin > 1) push(c1, k1);
                node = c0;
                continue;
            }
            bool found = false;
            while (sp > 0) {
                --sp;
                int2 e = sp < kSmem ? stk[sp][tid] : spill[sp - kSmem];
                if (__int_as_float(e.y) <= B.thr) { node = e.x; found = true; break; }
            }
            if (!found) break;
        }
    }
    return finish(T, B, q, status);
}

// (the MinMaxDist form, for unbounded queries, is a separate loop: the bounded
// one keeps the register budget of the search alone)
template <int kBlockT, int kSmem = 8, bool kCount = false, bool kRange = false>
__device__ __forceinline__ Hit nearest_wide(const Traversal &T, float3 q, float maxd2,
                                            int2 (*stk)[kBlockT], unsigned int *status,
                                            Counts *cnt = nullptr, int hint_leaf = -1) {
    if (T.mmd) return nearest_wide_t<kBlockT, kSmem, kCount, kRange, true>(T, q, maxd2, stk, status, cnt, hint_leaf);
    return nearest_wide_t<kBlockT, kSmem, kCount, kRange, false>(T, q, maxd2, stk, status, cnt, hint_leaf);
}

// The 4-wide records from the node records, one thread per (internal node,
// side): the record's half for that side is the child's own node record when the
// child is internal (its two children as two slots), else the node's slot for the
// leaf link and an empty slot -- a copy of 64 bytes.
__global__ void k_wide_update(const float4 *__restrict__ nodes, int nint, float4 *__restrict__ wide) {
    pdl_wait();
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int n = (int)(t >> 1), s = (int)(t & 1);
    if (n >= nint) return;
    const float4 a = __ldg(nodes + 4 * (size_t)n + 2 * s), b = __ldg(nodes + 4 * (size_t)n + 2 * s + 1);
    const int link = __float_as_int(a.w);
    float4 *w = wide + 8 * (size_t)n + 4 * s;
    if (link < 0) {
        w[0] = a;
        w[1] = b;
        w[2] = make_float4(INFINITY, INFINITY, INFINITY, __int_as_float(kWideEmpty));
        w[3] = make_float4(-INFINITY, -INFINITY, -INFINITY, __int_as_float(0));
    } else {
        const float4 *c = nodes + 4 * (size_t)link;
        w[0] = __ldg(c);
        w[1] = __ldg(c + 1);
        w[2] = __ldg(c + 2);
        w[3] = __ldg(c + 3);
    }
}

// One thread per query, "while-while" form: internal nodes are traversed
// while leaf children are only queued (up to kLeafQueue); the queued leaves
// are tested when every lane still traversing has one queued (or its queue is
// full, or it is done).  Leaf tests then run with the warp mostly converged
// instead of in almost every step.  Same answers as nearest().
constexpr int kLeafQueue = 4;

template <int kBlockT>
__device__ __forceinline__ Hit nearest_ww(const Traversal &T, float3 q, float maxd2,
                                          int2 (*stk)[kBlockT], unsigned int *status) {
    Best B = make_best(T, q, maxd2);
    if (T.n == 1) {
        test_leaf(T, B, 0, q, maxd2);
        return Hit{B.leaf, B.leaf >= 0 ? face_of(T, B.leaf) : 0x7fffffff, B.d2};
    }
    if (T.n < 1) return Hit{-1, 0x7fffffff, INFINITY};
    int2 spill[kStackTotal - kStackShared];
    const int tid = threadIdx.x;
    int sp = 0, node = 0;
    bool done = false;
    int2 lq[kLeafQueue];                         // (first face, count) of each queued leaf link
    int nq = 0;
    while (true) {
        while (!done && nq + 2 <= kLeafQueue) {
            if (nq > 0 && __all_sync(__activemask(), nq > 0)) break;
            const float4 *r = T.nodes + 4 * (size_t)node;
            float4 l0 = ldg4(r), l1 = ldg4(r + 1), r0 = ldg4(r + 2), r1 = ldg4(r + 3);
            float dl = box_d2(q, l0, l1), dr = box_d2(q, r0, r1);
            float ml = 0.0f, mr = 0.0f;
            if (T.mmd) {
                ml = box_minmax_d2(q, l0, l1);
                mr = box_minmax_d2(q, r0, r1);
                B.thr = fminf(B.thr, bound_window2(fminf(ml, mr), T.tau, query_slack(T, q)));
            }
            int cl = __float_as_int(l0.w), cr = __float_as_int(r0.w);
            if (cl < 0 && dl <= B.thr) lq[nq++] = make_int2(-cl - 1, link_count(l1));
            if (cr < 0 && dr <= B.thr) lq[nq++] = make_int2(-cr - 1, link_count(r1));
            bool gol = cl >= 0 && dl <= B.thr, gor = cr >= 0 && dr <= B.thr;
            if (gol && gor) {
                bool lfirst = dl < dr || (dl == dr && ml <= mr);
                int2 e = make_int2(lfirst ? cr : cl, __float_as_int(lfirst ? dr : dl));
                if (sp < kStackShared) stk[sp][tid] = e;
                else if (sp < kStackTotal) spill[sp - kStackShared] = e;
                else atomicOr(status, (unsigned)MESH_DEV_STACK_OVERFLOW);
                if (sp < kStackTotal) ++sp;
                node = lfirst ? cl : cr;
                continue;
            }
            if (gol) { node = cl; continue; }
            if (gor) { node = cr; continue; }
            done = true;
            while (sp > 0) {
                --sp;
                int2 e = sp < kStackShared ? stk[sp][tid] : spill[sp - kStackShared];
                if (__int_as_float(e.y) <= B.thr) { node = e.x; done = false; break; }
            }
        }
        for (int k = 0; k < nq; ++k) test_range<false>(T, B, lq[k].x, lq[k].y, q, maxd2);
        nq = 0;
        if (done) break;
    }
    return finish(T, B, q, status);
}

// The weights of the contact step, after its search (which writes face and
// distance only): one thread per query, so the recomputation of a hit's weights
// no longer holds a search warp until its last lane is done.  Same values as
// write_hit.
__global__ void __launch_bounds__(256)
k_hit_weights(Traversal T, const float *__restrict__ Q, int64_t nQ, const int *__restrict__ face,
              const float *__restrict__ dist2, const int *__restrict__ iperm, float *bary, float *point) {
    pdl_wait();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nQ) return;
    const int f = face[i];
    if (f < 0) {
        if (bary) { bary[3 * i] = 0.0f; bary[3 * i + 1] = 0.0f; bary[3 * i + 2] = 0.0f; }
        if (point) { point[3 * i] = 0.0f; point[3 * i + 1] = 0.0f; point[3 * i + 2] = 0.0f; }
        return;
    }
    const float3 q = make_float3(Q[3 * i], Q[3 * i + 1], Q[3 * i + 2]);
    write_weights(T, __ldg(iperm + f), dist2[i], q, i, bary, point);
}

// kMode: 0 depth-first, 1 while-while, 2 depth-first with one leaf-test site,
// 3 depth-first over the 4-wide records.
// kMinBlocks: resident blocks per SM the register budget must allow
// (8 -> 64 registers, 9 -> 56, 12 -> 40, 16 -> 32; fewer registers, more warps
// to hide latency, more spilling).
// Work class of a query from its node visits, heaviest first (the contact step
// orders the next step's queries by it): 0: 48 or more, 1: 24-47, 2: 12-23, 3: fewer.
__device__ __forceinline__ unsigned int work_class(int visits) {
    return visits >= 48 ? 0u : visits >= 24 ? 1u : visits >= 12 ? 2u : 3u;
}

// kRecord: also count the node visits of each query and store its work class
// in cls[i] (the contact step).
// kBlock: threads per block (128, or 64 / 32 with the same register budget: the
// same warps per SM in finer blocks, so a block whose warps finish early frees
// its slot sooner -- the searches of one block end at very different times).
template <int kSmem, int kMode, int kMinBlocks = kQueryMinBlocks, bool kRecord = false,
          int kBlock = kQueryBlock, bool kRange = false>
__global__ void __launch_bounds__(kBlock, kMinBlocks * kQueryBlock / kBlock)
k_closest_point(Traversal T, const Header *__restrict__ hdr, unsigned int *status,
                const float *__restrict__ Q, int64_t nQ, float maxd2, int *face, float *bary,
                float *point, float *dist2, const int *hint, const int *__restrict__ iperm,
                const int *__restrict__ order = nullptr, unsigned int *__restrict__ cls = nullptr) {
    __shared__ int2 stk[kSmem > 0 ? kSmem : 1][kBlock];
    pdl_wait();
    int64_t k = (int64_t)blockIdx.x * kBlock + threadIdx.x;
    if (k >= nQ) return;
    const int64_t i = order ? (int64_t)order[k] : k;       // order: a permutation of the queries
    set_scale(T, hdr);
    float3 q = make_float3(Q[3 * i], Q[3 * i + 1], Q[3 * i + 2]);
    int hint_leaf = -1;
    if (hint) {                                   // may alias face: read before the write below
        int hf = hint[i];
        if (hf >= 0 && hf < T.n) hint_leaf = __ldg(iperm + hf);
    }
    Hit h;
    if constexpr (kRecord) {
        static_assert(kMode != 1, "the recording form uses the depth-first traversal");
        Counts c{0, 0};
        if constexpr (kMode == 3) {          // a 4-wide record counts as two binary visits
            h = nearest_wide<kBlock, kSmem, true, kRange>(T, q, maxd2, stk, status, &c, hint_leaf);
            cls[i] = work_class(2 * c.visits);
        } else {
            h = nearest<kBlock, kSmem, kMode == 2, true, kRange>(T, q, maxd2, stk, status, &c, hint_leaf);
            cls[i] = work_class(c.visits);
        }
    } else if constexpr (kMode == 1) {
        static_assert(!kRange, "the while-while form has no leaf-range instantiation");
        h = nearest_ww<kBlock>(T, q, maxd2, stk, status);
    } else if constexpr (kMode == 3) {
        h = nearest_wide<kBlock, kSmem, false, kRange>(T, q, maxd2, stk, status, nullptr, hint_leaf);
    } else {
        h = nearest<kBlock, kSmem, kMode == 2, false, kRange>(T, q, maxd2, stk, status, nullptr, hint_leaf);
    }
    write_hit(T, h, q, i, face, bary, point, dist2);
}

// Warp-packet traversal: the 32 queries of a warp (consecutive, so nearby
// when the caller keeps them in Morton order) share one depth-first node
// sequence.  Each lane tests the node's two child boxes against its own query
// and bound; a child is entered when any lane needs it, nearer-first by a
// vote of the lanes, and the other child is deferred on a per-warp stack of
// (parent, side) entries.  A deferred child is re-tested against the lanes'
// bounds when it is popped (bounds only shrink), so a lane sees every leaf
// its own traversal would.  Node loads are warp-uniform (one broadcast per
// record) and all control flow outside the leaf tests is warp-uniform: the
// warp runs the union of its queries' traversals with every lane active,
// instead of each lane's traversal with most lanes idle.  Same answers as the
// depth-first kernels.
// hint_leaf >= 0 warm-starts the lane as in nearest(); visits (when not NULL)
// counts the nodes whose children this lane needed (its share of the work).
template <bool kRange>
__device__ __forceinline__ Hit nearest_packet(const Traversal &T, float3 q, float maxd2, bool valid,
                                              int *wstk, unsigned int *status, int hint_leaf = -1,
                                              int *visits = nullptr) {
    const unsigned int kFull = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    Best B = make_best(T, q, maxd2);
    if (!valid) B.thr = -1.0f;                   // a lane past the end prunes everything
    if (valid && hint_leaf >= 0) test_leaf(T, B, hint_leaf, q, maxd2);
    if (T.n == 1) {
        if (valid) test_leaf(T, B, 0, q, maxd2);
        return Hit{B.leaf, B.leaf >= 0 ? face_of(T, B.leaf) : 0x7fffffff, B.d2};
    }
    if (T.n < 1) return Hit{-1, 0x7fffffff, INFINITY};
    int sp = 0, node = 0;
    while (true) {
        const float4 *r = T.nodes + 4 * (size_t)node;
        float4 l0 = ldg4(r), l1 = ldg4(r + 1), r0 = ldg4(r + 2), r1 = ldg4(r + 3);
        float dl = box_d2(q, l0, l1), dr = box_d2(q, r0, r1);
        if (T.mmd && valid)
            B.thr = fminf(B.thr, bound_window2(fminf(box_minmax_d2(q, l0, l1), box_minmax_d2(q, r0, r1)),
                                               T.tau, query_slack(T, q)));
        int cl = __float_as_int(l0.w), cr = __float_as_int(r0.w);
        bool wl = dl <= B.thr, wr = dr <= B.thr;
        if (visits) *visits += (wl || wr);
        unsigned int bl = __ballot_sync(kFull, wl), br = __ballot_sync(kFull, wr);
        if (cl < 0 && wl) test_range<kRange>(T, B, -cl - 1, link_count(l1), q, maxd2);
        if (cr < 0 && wr) test_range<kRange>(T, B, -cr - 1, link_count(r1), q, maxd2);
        bool gl = cl >= 0 && bl != 0u, gr = cr >= 0 && br != 0u;
        if (gl && gr) {
            unsigned int pl = __ballot_sync(kFull, wl && (!wr || dl <= dr));
            bool lfirst = 2 * __popc(pl) >= __popc(bl | br);
            if (sp < kStackTotal) {
                if (lane == 0) wstk[sp] = 2 * node + (lfirst ? 1 : 0);
                ++sp;
            } else if (lane == 0) {
                atomicOr(status, (unsigned)MESH_DEV_STACK_OVERFLOW);
            }
            node = lfirst ? cl : cr;
            continue;
        }
        if (gl) { node = cl; continue; }
        if (gr) { node = cr; continue; }
        bool found = false;
        __syncwarp();
        while (sp > 0) {
            --sp;
            int e = wstk[sp];
            const float4 *pr = T.nodes + 4 * (size_t)(e >> 1) + 2 * (e & 1);
            float4 lo = ldg4(pr), hi = ldg4(pr + 1);
            if (__any_sync(kFull, box_d2(q, lo, hi) <= B.thr)) {
                node = __float_as_int(lo.w);
                found = true;
                break;
            }
        }
        __syncwarp();
        if (!found) break;
    }
    return finish(T, B, q, status);
}

// hint / iperm: warm start as k_closest_point.  order: the queries' order (a
// permutation; NULL = as stored).  kRecord: also store each query's work class
// in cls (the contact step).
template <bool kRecord = false, bool kRange = false>
__global__ void __launch_bounds__(kQueryBlock, kQueryMinBlocks)
k_closest_point_packet(Traversal T, const Header *__restrict__ hdr, unsigned int *status,
                       const float *__restrict__ Q, int64_t nQ, float maxd2, int *face, float *bary,
                       float *point, float *dist2, const int *hint, const int *__restrict__ iperm,
                       const int *__restrict__ order = nullptr, unsigned int *__restrict__ cls = nullptr) {
    __shared__ int wstk[kQueryBlock / 32][kStackTotal];
    pdl_wait();
    const int64_t w0 = (int64_t)blockIdx.x * kQueryBlock + (threadIdx.x & ~31);
    if (w0 >= nQ) return;                                  // whole warp past the end
    const int64_t k = w0 + (threadIdx.x & 31);
    const bool valid = k < nQ;
    const int64_t i = valid && order ? (int64_t)order[k] : k;
    set_scale(T, hdr);
    float3 q = valid ? make_float3(Q[3 * i], Q[3 * i + 1], Q[3 * i + 2]) : make_float3(0.0f, 0.0f, 0.0f);
    int hint_leaf = -1;
    if (valid && hint) {                          // may alias face: read before the write below
        int hf = hint[i];
        if (hf >= 0 && hf < T.n) hint_leaf = __ldg(iperm + hf);
    }
    int visits = 0;
    Hit h = nearest_packet<kRange>(T, q, maxd2, valid, wstk[threadIdx.x >> 5], status, hint_leaf,
                                   kRecord ? &visits : nullptr);
    if (valid) {
        write_hit(T, h, q, i, face, bary, point, dist2);
        if constexpr (kRecord) cls[i] = work_class(visits);
    }
}

// Persistent depth-first traversal with dynamic fetch (Aila & Laine 2009):
// a fixed grid of warps; each lane works through a stream of queries, one
// node visit per step, and when at least kRefill lanes of the warp are idle
// the warp takes that many new query indices from a global counter.  Lanes no
// longer wait for the slowest query of their warp (contact queries near the
// surface need ~6x the visits of those far from it).  Same answers as the
// depth-first kernels.
// The counter lives in the mesh header (zeroed before each launch), so
// concurrent calls on one handle must not overlap.
constexpr int kRefill = 8;

template <int kSmem>
__global__ void __launch_bounds__(kQueryBlock, kQueryMinBlocks)
k_closest_point_persistent(Traversal T, const Header *__restrict__ hdr, unsigned int *status,
                           const float *__restrict__ Q, int64_t nQ, float maxd2, int *face,
                           float *bary, float *point, float *dist2, unsigned int *work) {
    __shared__ int2 stk[kSmem > 0 ? kSmem : 1][kQueryBlock];
    int2 spill[kStackTotal - kSmem];
    const int lane = threadIdx.x & 31, tid = threadIdx.x;
    const unsigned lt = (1u << lane) - 1u;
    set_scale(T, hdr);
    int64_t qi = -1;
    float3 q = make_float3(0.f, 0.f, 0.f);
    Best B = make_best(T, q, maxd2);
    int node = 0, sp = 0;
    bool exhausted = false;
    while (true) {
        bool fin = false;
        unsigned idle = __ballot_sync(0xffffffffu, qi < 0);
        if (!exhausted && (__popc(idle) >= kRefill || idle == 0xffffffffu)) {
            unsigned int base = 0, want = __popc(idle);
            if (lane == 0) base = atomicAdd(work, want);
            base = __shfl_sync(0xffffffffu, base, 0);
            if ((int64_t)base + want >= nQ) exhausted = true;
            if (qi < 0) {
                int64_t cand = (int64_t)base + __popc(idle & lt);
                if (cand < nQ) {
                    qi = cand;
                    q = make_float3(Q[3 * qi], Q[3 * qi + 1], Q[3 * qi + 2]);
                    B = make_best(T, q, maxd2);
                    node = 0;
                    sp = 0;
                    if (T.n <= 1) {                      // no internal node to visit
                        if (T.n == 1) test_leaf(T, B, 0, q, maxd2);
                        fin = true;
                    }
                }
            }
        }
        // every lane reaches this vote each iteration (a full-warp collective
        // must never sit on a path only some lanes take)
        const bool all_idle = __all_sync(0xffffffffu, qi < 0);
        if (all_idle && exhausted) break;
        if (qi < 0) continue;
        if (!fin) {                                      // one node visit
            const float4 *r = T.nodes + 4 * (size_t)node;
            float4 l0 = ldg4(r), l1 = ldg4(r + 1), r0 = ldg4(r + 2), r1 = ldg4(r + 3);
            float dl = box_d2(q, l0, l1), dr = box_d2(q, r0, r1);
            float ml = 0.0f, mr = 0.0f;
            if (T.mmd) {
                ml = box_minmax_d2(q, l0, l1);
                mr = box_minmax_d2(q, r0, r1);
                B.thr = fminf(B.thr, bound_window2(fminf(ml, mr), T.tau, query_slack(T, q)));
            }
            int cl = __float_as_int(l0.w), cr = __float_as_int(r0.w);
            if (cl < 0 && dl <= B.thr) test_range<false>(T, B, -cl - 1, link_count(l1), q, maxd2);
            if (cr < 0 && dr <= B.thr) test_range<false>(T, B, -cr - 1, link_count(r1), q, maxd2);
            bool gol = cl >= 0 && dl <= B.thr, gor = cr >= 0 && dr <= B.thr;
            if (gol && gor) {
                bool lfirst = dl < dr || (dl == dr && ml <= mr);
                int2 e = make_int2(lfirst ? cr : cl, __float_as_int(lfirst ? dr : dl));
                if (sp < kSmem) stk[sp][tid] = e;
                else if (sp < kStackTotal) spill[sp - kSmem] = e;
                else atomicOr(status, (unsigned)MESH_DEV_STACK_OVERFLOW);
                if (sp < kStackTotal) ++sp;
                node = lfirst ? cl : cr;
            } else if (gol) {
                node = cl;
            } else if (gor) {
                node = cr;
            } else {
                fin = true;
                while (sp > 0) {
                    --sp;
                    int2 e = sp < kSmem ? stk[sp][tid] : spill[sp - kSmem];
                    if (__int_as_float(e.y) <= B.thr) { node = e.x; fin = false; break; }
                }
            }
        }
        if (fin) {
            write_hit(T, finish(T, B, q, status), q, qi, face, bary, point, dist2);
            qi = -1;
        }
    }
}

// Counting form of the one-thread depth-first traversal (the visiting order of
// variants 2 and 3; the pooled search of variant 0 visits a few per cent more): node visits, triangle tests and hits, summed over
// all queries.  Separate instantiation; the timed kernels carry no counters.
// kWide: the traversal over the 4-wide records (its visits count records).
template <bool kRange, bool kWide = false>
__global__ void __launch_bounds__(kQueryBlock, kQueryMinBlocks)
k_closest_point_count(Traversal T, const Header *__restrict__ hdr, unsigned int *status,
                      const float *__restrict__ Q, int64_t nQ, float maxd2,
                      unsigned long long *counts) {
    __shared__ int2 stk[kStackShared][kQueryBlock];
    int64_t i = (int64_t)blockIdx.x * kQueryBlock + threadIdx.x;
    Counts c{0, 0};
    int hit = 0;
    if (i < nQ) {
        set_scale(T, hdr);
        float3 q = make_float3(Q[3 * i], Q[3 * i + 1], Q[3 * i + 2]);
        Hit h;
        if constexpr (kWide)
            h = nearest_wide<kQueryBlock, kStackShared, true, kRange>(T, q, maxd2, stk, status, &c);
        else
            h = nearest<kQueryBlock, kStackShared, false, true, kRange>(T, q, maxd2, stk, status, &c);
        hit = h.leaf >= 0;
    }
    unsigned long long v = c.visits, t = c.tests, k = hit;
    for (int o = 16; o > 0; o >>= 1) {
        v += __shfl_xor_sync(0xffffffffu, v, o);
        t += __shfl_xor_sync(0xffffffffu, t, o);
        k += __shfl_xor_sync(0xffffffffu, k, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(counts, v);
        atomicAdd(counts + 1, t);
        atomicAdd(counts + 2, k);
    }
}

__global__ void k_interpolate(const int4 *__restrict__ faces, const float4 *__restrict__ verts,
                              int nF, const int *__restrict__ face, const float *__restrict__ bary,
                              int64_t n, float *__restrict__ out, unsigned int *status) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int f = face[i];
    if ((unsigned)f >= (unsigned)nF) {
        atomicOr(status, (unsigned)MESH_DEV_INDEX_RANGE);
        out[3 * i] = out[3 * i + 1] = out[3 * i + 2] = 0.0f;
        return;
    }
    int4 fv = faces[f];
    float4 a = verts[fv.x], b = verts[fv.y], c = verts[fv.z];
    float u = bary[3 * i], v = bary[3 * i + 1], w = bary[3 * i + 2];
    out[3 * i] = u * a.x + v * b.x + w * c.x;
    out[3 * i + 1] = u * a.y + v * b.y + w * c.y;
    out[3 * i + 2] = u * a.z + v * b.z + w * c.z;
}

static Traversal traversal_of(const mesh_bvh *b, bool mmd = true) {
    return Traversal{b->nodes(), b->tris(), (int)b->L.n_faces, 0.0f, 0.0f, mmd, b->wide()};
}

// The 4-wide records written from the node records: by every build or refit of a
// handle whose traversal is variant 13 (so a captured refit carries the update),
// and otherwise by the first variant-13 query after the records went stale
// (host-side flag; the update runs on that query's stream, ahead of it).
static void ensure_wide(const mesh_bvh *b, cudaStream_t s) {
    if (!b->wide_valid) wide_refresh(b, s, false);
}

}  // namespace meshgs

void meshgs::wide_refresh(const mesh_bvh *b, cudaStream_t s, bool pdl) {
    const int nint = (int)b->L.n_faces - 1;
    if (nint > 0) {
        launch_ex(pdl, k_wide_update, grid_for(2 * (int64_t)nint, 256), 256, 0, s, (const float4 *)b->nodes(), nint,
                  b->wide());
        count_launch();
    }
    b->wide_valid = true;
}

namespace meshgs {

static size_t chamfer_blocks(int64_t n, int G) {         // of 128 / G samples (G = 0: 128)
    return (size_t)((n * (G > 0 ? G : 1) + kQueryBlock - 1) / kQueryBlock);
}

// The one-thread searches' weights in their own launch after the search (k_hit_weights).
constexpr bool kContactSplitWeights = true;

static int g_group_override = 0;
static int g_traversal = 0;          // traversal variant, see mesh_set_traversal

bool wide_wanted(const mesh_bvh *b) {
    return (b->cfg_variant >= 0 ? b->cfg_variant : g_traversal) == 13 && b->cfg_lanes <= 1;
}

// Lanes per query that fill 2048 lanes per SM (twice what the search kernels hold at a
// time): 1 with enough queries, else a power of two up to 32.
static int fill_lanes(int64_t nQ) {
    static int sms = 0;
    if (sms == 0) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
            sms = 152;
    }
    const int64_t target = (int64_t)sms * 2048;
    int G = 1;
    while (nQ > 0 && G < 32 && nQ * G < target) G <<= 1;
    return G;
}

// Lanes per query of the pooled search when the caller names none: what fills
// the GPU, and at most 16 queries per warp.  More queries than that keep no more
// lanes busy and take stack from the L1 cache: 1M queries of the 200k-face torus
// took 289 / 267 / 349 us with 32 / 16 / 8 queries per warp under a cutoff and
// 6.3 / 4.5 / 4.3 ms without; 20k took 97 / 58 / 50 / 40 / 44 / 56 us with 32 ... 1
// (2 by this rule; 4, the best, would be a single fill), 5k 68 ... 27 us (1 by this rule: 27).
// Meshes of few faces do without (0): 12 faces, 300k queries 74 us with it, 35 without (one
// thread per query of the tree 87), 50k signed distances 54 and 22 (30), 100 queries 13 and
// 13; 20 faces, 50k queries 36 and 21 (52), 100 queries 11 and 17 (15); 40 faces, 300k
// queries 74 and 93 (162).
static int pool_lanes(int64_t nQ, int64_t n_faces) {
    const int G = fill_lanes(nQ);
    if (n_faces <= (G <= 8 ? kFewFaces : 16)) return 0;
    return G > 2 ? G : 2;
}

// Lanes per query of a call: the handle's setting, else the process-wide one, else
// (0) the library's choice; 1 asks for the one-thread variants.
static int lanes_of(const mesh_bvh *b) { return b && b->cfg_lanes > 0 ? b->cfg_lanes : g_group_override; }

mesh_status launch_signed_query(const mesh_bvh *bvh, const float *d_Q, int64_t nQ, float max_dist,
                                int32_t *d_face, float *d_bary, float *d_point, float *d_sdist,
                                cudaStream_t s) {
    const bool unbounded = isinf(max_dist);
    pool_signed(bvh, traversal_of(bvh, unbounded), d_Q, nQ, unbounded ? INFINITY : max_dist * max_dist,
                pool_lanes(nQ, bvh->L.n_faces), d_face, d_bary, d_point, d_sdist, s);
    return check_launch();
}

// The one-thread launch of mesh_closest_point_hinted (variants 1-13) for a tree
// with (R) or without leaf collapse; with it, variants 2, 3, 12 and 13 exist.
template <bool R>
static void launch_closest_point(Traversal T, Header *h, const float *d_Q, int64_t nQ, float maxd2, int32_t *d_face,
                                 float *d_bary, float *d_point, float *d_dist2, const int32_t *d_hint,
                                 const int *iperm, int variant, int blk, cudaStream_t s) {
    auto go = [&](auto kern, int block) {
        kern<<<grid_for(nQ, block), block, 0, s>>>(T, h, &h->status, d_Q, nQ, maxd2, d_face, d_bary, d_point, d_dist2,
                                                   d_hint, iperm, nullptr, nullptr);
    };
    constexpr int B = kQueryBlock, M = kQueryMinBlocks;
    switch (variant) {
        case 2:
            if (blk == 32) go(k_closest_point<8, 0, M, false, 32, R>, 32);
            else if (blk == 64) go(k_closest_point<8, 0, M, false, 64, R>, 64);
            else go(k_closest_point<8, 0, M, false, B, R>, B);
            return;
        case 3:
            if (blk == 32) go(k_closest_point<0, 0, M, false, 32, R>, 32);
            else if (blk == 64) go(k_closest_point<0, 0, M, false, 64, R>, 64);
            else go(k_closest_point<0, 0, M, false, B, R>, B);
            return;
        case 13:
            if (blk == 32) go(k_closest_point<8, 3, M, false, 32, R>, 32);
            else if (blk == 64) go(k_closest_point<8, 3, M, false, 64, R>, 64);
            else go(k_closest_point<8, 3, M, false, B, R>, B);
            return;
        case 12: go(k_closest_point_packet<false, R>, B); return;
        default: break;
    }
    if constexpr (!R) {
        switch (variant) {
            case 1: go(k_closest_point<kStackShared, 1>, B); return;
            case 4: go(k_closest_point<kStackShared, 2>, B); return;
            case 5: go(k_closest_point<0, 2>, B); return;
            case 6: go(k_closest_point<8, 0, 9>, B); return;
            case 7: go(k_closest_point<0, 0, 9>, B); return;
            case 8: go(k_closest_point<0, 0, 16>, B); return;
            case 9: go(k_closest_point<0, 2, 12>, B); return;
            default: break;
        }
        static int sms = 0;                              // 10, 11: persistent
        if (sms == 0) {
            int dv = 0;
            if (cudaGetDevice(&dv) != cudaSuccess ||
                cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dv) != cudaSuccess || sms <= 0)
                sms = 152;
        }
        unsigned int *work = &h->pad[0];
        cudaMemsetAsync(work, 0, sizeof(unsigned int), s);
        const int64_t grid = grid_for(nQ, B), most = (int64_t)sms * M;
        const unsigned int pg = (unsigned int)(most < grid ? most : grid);
        if (variant == 10)
            k_closest_point_persistent<8><<<pg, B, 0, s>>>(T, h, &h->status, d_Q, nQ, maxd2, d_face, d_bary, d_point,
                                                           d_dist2, work);
        else
            k_closest_point_persistent<0><<<pg, B, 0, s>>>(T, h, &h->status, d_Q, nQ, maxd2, d_face, d_bary, d_point,
                                                           d_dist2, work);
    }
}

// The ordered, recording launch of mesh_contact (variants 2-9, 12, 13) for a tree
// with (R) or without leaf collapse (with it, 2, 3, 12 and 13 exist).
template <bool R>
static void launch_contact(Traversal T, Header *h, const float *d_Q, int64_t nQ, float maxd2, int32_t *d_face,
                           float *d_bary, float *d_point, float *d_dist2, const int *iperm, const int *order,
                           unsigned int *cls, int variant, int blk, cudaStream_t s) {
    // every form runs right after the sort of the classes: launched as its dependent
    auto go = [&](auto kern, int block) {
        pdl_launch(kern, grid_for(nQ, block), block, 0, s, T, h, &h->status, d_Q, nQ, maxd2, d_face, d_bary, d_point,
                   d_dist2, d_face, iperm, order, cls);
    };
    constexpr int B = kQueryBlock, M = kQueryMinBlocks;
    switch (variant) {
        case 2:
            if (blk == 32) go(k_closest_point<8, 0, M, true, 32, R>, 32);
            else if (blk == 64) go(k_closest_point<8, 0, M, true, 64, R>, 64);
            else go(k_closest_point<8, 0, M, true, B, R>, B);
            return;
        case 3:
            if (blk == 32) go(k_closest_point<0, 0, M, true, 32, R>, 32);
            else if (blk == 64) go(k_closest_point<0, 0, M, true, 64, R>, 64);
            else go(k_closest_point<0, 0, M, true, B, R>, B);
            return;
        case 13:
            if (blk == 32) go(k_closest_point<8, 3, M, true, 32, R>, 32);
            else if (blk == 64) go(k_closest_point<8, 3, M, true, 64, R>, 64);
            else go(k_closest_point<8, 3, M, true, B, R>, B);
            return;
        case 12: go(k_closest_point_packet<true, R>, B); return;
        default: break;
    }
    if constexpr (!R) {
        switch (variant) {
            case 4: go(k_closest_point<kStackShared, 2, M, true>, B); return;
            case 5: go(k_closest_point<0, 2, M, true>, B); return;
            case 6: go(k_closest_point<8, 0, 9, true>, B); return;
            case 7: go(k_closest_point<0, 0, 9, true>, B); return;
            case 8: go(k_closest_point<0, 0, 16, true>, B); return;
            default: go(k_closest_point<0, 2, 12, true>, B); return;    // 9
        }
    }
}

// Lanes per sample of the Chamfer searches (unbounded), unless the process-wide
// setting names more than one.
static int chamfer_lanes(const mesh_bvh *A, const mesh_bvh *B, int64_t n) {
    const int64_t most = A->L.n_faces > B->L.n_faces ? A->L.n_faces : B->L.n_faces;
    return g_group_override > 1 ? g_group_override : pool_lanes(n, most);
}

static mesh_status run_chamfer(const mesh_bvh *A, const float *SA, int64_t nSA, const mesh_bvh *B, const float *SB,
                               int64_t nSB, int G, double *partial, unsigned int *ticket, double *out,
                               const int32_t *hintA, const int32_t *hintB, int32_t *faceA, float *baryA,
                               float *dist2A, int32_t *faceB, float *baryB, float *dist2B, cudaStream_t s) {
    const size_t nbA = chamfer_blocks(nSA, G), nbB = chamfer_blocks(nSB, G);
    if (nbA + nbB == 0) {
        cudaMemsetAsync(out, 0, 2 * sizeof(double), s);
        return check_launch();
    }
    cudaMemsetAsync(ticket, 0, sizeof(unsigned int), s);
    const ChamferSide a2b{traversal_of(B), B->hdr(), SA, nSA, faceA, baryA, dist2A, hintA, B->iperm()};
    const ChamferSide b2a{traversal_of(A), A->hdr(), SB, nSB, faceB, baryB, dist2B, hintB, A->iperm()};
    pool_chamfer(G, A->leaf_size > 1 || B->leaf_size > 1, a2b, b2a, (unsigned)nbA, (unsigned)(nbA + nbB),
                 &A->hdr()->status, partial, ticket, out, s);
    return check_launch();
}

// The workspace of mesh_chamfer_step: mesh_chamfer's, and room for the samples'
// order of an earlier form of the step, which callers' sizes may still count.
static size_t chamfer_step_bytes(int64_t nSA, int64_t nSB) {
    const int64_t m = nSA + nSB > 0 ? nSA + nSB : 1;
    return align_up(mesh_chamfer_workspace_bytes(nSA, nSB), 256) + 3 * align_up(4 * m, 256) +
           align_up(sort_pairs_ws_bytes(m), 256);
}

}  // namespace meshgs

using namespace meshgs;

extern "C" {

mesh_status mesh_closest_point(const mesh_bvh *bvh, const float *d_Q, int64_t nQ, float max_dist,
                               int32_t *d_face, float *d_bary, float *d_point, float *d_dist2,
                               void *stream) {
    return mesh_closest_point_hinted(bvh, d_Q, nQ, max_dist, nullptr, d_face, d_bary, d_point, d_dist2,
                                     stream);
}

mesh_status mesh_closest_point_hinted(const mesh_bvh *bvh, const float *d_Q, int64_t nQ, float max_dist,
                                      const int32_t *d_hint, int32_t *d_face, float *d_bary,
                                      float *d_point, float *d_dist2, void *stream) {
    if (!bvh || nQ < 0 || (nQ > 0 && !d_Q) || !(max_dist >= 0.0f)) return MESH_ERR_INVALID_ARG;
    if (nQ == 0) return MESH_OK;
    const int *iperm = bvh->iperm();
    float maxd2 = isinf(max_dist) ? INFINITY : max_dist * max_dist;
    cudaStream_t s = (cudaStream_t)stream;
    int variant = bvh->cfg_variant >= 0 ? bvh->cfg_variant : g_traversal;
    if (variant >= 10 && variant <= 12 && nQ >= ((int64_t)1 << 31)) variant = 0;   // 32-bit work counter
    if (bvh->leaf_size > 1 && !(variant == 2 || variant == 3 || variant == 12 || variant == 13)) variant = 0;
    // a one-thread variant runs when lanes is 1, or is the library's choice and the queries
    // fill the GPU; everything else is the pooled search
    const int lanes = lanes_of(bvh);
    const bool one = variant != 0 && (lanes == 1 || (lanes == 0 && fill_lanes(nQ) == 1));
    if (one && variant == 13) ensure_wide(bvh, s);
    Traversal T = traversal_of(bvh, isinf(max_dist));
    if (!one) {
        pool_closest_point(bvh, T, d_Q, nQ, maxd2, lanes > 1 ? lanes : pool_lanes(nQ, bvh->L.n_faces), d_face, d_bary,
                           d_point, d_dist2, d_hint, s);
        return check_launch();
    }
    // the one-thread depth-first searches write face and distance; the weights and
    // closest points follow in one thread per query (as in the contact step)
    const bool split = kContactSplitWeights && d_face && d_dist2 && (d_bary || d_point) &&
                       !(variant == 1 || (variant >= 10 && variant <= 12));
    float *sb = split ? nullptr : d_bary, *sp = split ? nullptr : d_point;
    if (bvh->leaf_size > 1)
        launch_closest_point<true>(T, bvh->hdr(), d_Q, nQ, maxd2, d_face, sb, sp, d_dist2, d_hint,
                                   iperm, variant, bvh->cfg_block, s);
    else
        launch_closest_point<false>(T, bvh->hdr(), d_Q, nQ, maxd2, d_face, sb, sp, d_dist2, d_hint,
                                    iperm, variant, bvh->cfg_block, s);
    count_launch();
    if (split) {
        pdl_launch(k_hit_weights, grid_for(nQ, 256), 256, 0, s, T, d_Q, nQ, (const int *)d_face,
                   (const float *)d_dist2, iperm, d_bary, d_point);
        count_launch();
    }
    return check_launch();
}

// Contact queries of a physics step: warm-started by the previous step's faces
// and run in the order of the previous step's work classes (heaviest first,
// each class in the given order), so that a warp holds queries of similar
// depth -- near the surface (deep searches), near misses, or far away (short
// ones) -- instead of a mix that runs as long as its slowest lane.  The
// classes (their low two bits) are ordered by a stable counting sort in two
// launches: each tile of queries counts its classes, then each tile scatters
// its query indices from the counts of the tiles before it.  Any class bits
// give a valid permutation, so a workspace whose classes are stale or garbage
// only gives a worse order.
constexpr int kClassTile = 2048, kClassThreads = 256;

__global__ void __launch_bounds__(kClassThreads)
k_class_count(const unsigned int *__restrict__ cls, int n, int4 *__restrict__ counts) {
    __shared__ int s_cnt[4];
    pdl_wait();
    pdl_trigger();
    if (threadIdx.x < 4) s_cnt[threadIdx.x] = 0;
    __syncthreads();
    const int base = blockIdx.x * kClassTile, lane = threadIdx.x & 31;
    int c[4] = {0, 0, 0, 0};
#pragma unroll
    for (int r = 0; r < kClassTile / kClassThreads; ++r) {
        int i = base + r * kClassThreads + threadIdx.x;
        unsigned int k = i < n ? (cls[i] & 3u) : 4u;
#pragma unroll
        for (int q = 0; q < 4; ++q) c[q] += __popc(__ballot_sync(0xffffffffu, k == (unsigned)q));
    }
    if (lane < 4) atomicAdd(&s_cnt[lane], c[lane]);
    __syncthreads();
    if (threadIdx.x == 0) counts[blockIdx.x] = make_int4(s_cnt[0], s_cnt[1], s_cnt[2], s_cnt[3]);
}

__global__ void __launch_bounds__(kClassThreads)
k_class_scatter(const unsigned int *__restrict__ cls, int n, const int4 *__restrict__ counts, int tiles,
                int *__restrict__ order) {
    constexpr int kWarps = kClassThreads / 32;
    __shared__ int s_red[kWarps][8];
    __shared__ int s_run[4];
    __shared__ int s_off[kWarps][4];
    pdl_wait();
    pdl_trigger();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // every class's total and this tile's prefix, from the tiles' counts
    int v[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (int t = threadIdx.x; t < tiles; t += kClassThreads) {
        int4 c = counts[t];
        v[0] += c.x; v[1] += c.y; v[2] += c.z; v[3] += c.w;
        if (t < (int)blockIdx.x) { v[4] += c.x; v[5] += c.y; v[6] += c.z; v[7] += c.w; }
    }
#pragma unroll
    for (int q = 0; q < 8; ++q)
        for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
    if (lane == 0)
        for (int q = 0; q < 8; ++q) s_red[wid][q] = v[q];
    __syncthreads();
    if (threadIdx.x == 0) {
        int tot[4] = {0, 0, 0, 0}, pre[4] = {0, 0, 0, 0};
        for (int w = 0; w < kWarps; ++w)
            for (int q = 0; q < 4; ++q) { tot[q] += s_red[w][q]; pre[q] += s_red[w][4 + q]; }
        int run = 0;
        for (int q = 0; q < 4; ++q) { s_run[q] = run + pre[q]; run += tot[q]; }
    }
    __syncthreads();
    const int base = blockIdx.x * kClassTile;
    const unsigned int lt = (1u << lane) - 1u;
    for (int r = 0; r < kClassTile / kClassThreads; ++r) {
        int i = base + r * kClassThreads + threadIdx.x;
        unsigned int k = i < n ? (cls[i] & 3u) : 4u;
        unsigned int mine = 0u;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            unsigned int b = __ballot_sync(0xffffffffu, k == (unsigned)q);
            if (lane == 0) s_off[wid][q] = __popc(b);
            if (k == (unsigned)q) mine = b;
        }
        __syncthreads();
        if (threadIdx.x < 4) {                         // warp offsets within the round, per class
            int q = threadIdx.x, run = s_run[q];
            for (int w = 0; w < kWarps; ++w) { int c = s_off[w][q]; s_off[w][q] = run; run += c; }
            s_run[q] = run;
        }
        __syncthreads();
        if (k < 4u) order[s_off[wid][k] + __popc(mine & lt)] = i;
        __syncthreads();
    }
}

struct ContactWs {
    unsigned int *cls;
    int *order;
    int4 *counts;
    float *d2;             // the distances, when the caller does not take them
    size_t bytes;
};

static ContactWs contact_ws(void *ws, int64_t n) {
    size_t off = 0;
    auto take = [&](size_t b) { size_t o = off; off = align_up(off + b, 256); return o; };
    int64_t m = n > 0 ? n : 1;
    size_t oC = take(4 * m), oO = take(4 * m), oT = take(16 * ((m + kClassTile - 1) / kClassTile)),
           oD = take(4 * m);
    char *b = (char *)ws;
    return ContactWs{(unsigned int *)(b + oC), (int *)(b + oO), (int4 *)(b + oT), (float *)(b + oD), off};
}


mesh_status mesh_knn_project(const mesh_bvh *bvh, const float *d_Q, int64_t nQ, int k,
                             const float *d_anchor, float anchor_weight, float *d_point,
                             int32_t *d_face, float *d_dist2, void *stream) {
    if (!bvh || nQ < 0 || k < 1 || k > kKnnMax || !(anchor_weight >= 0.0f && anchor_weight <= 1.0f))
        return MESH_ERR_INVALID_ARG;
    if (nQ == 0) return MESH_OK;
    if (!d_Q || !d_point) return MESH_ERR_INVALID_ARG;
    pool_knn(bvh, traversal_of(bvh, false), d_Q, nQ, k, pool_lanes(nQ, bvh->L.n_faces), d_anchor, anchor_weight, d_point,
             d_face, d_dist2, (cudaStream_t)stream);
    return check_launch();
}


size_t mesh_contact_workspace_bytes(int64_t nQ) {
    if (nQ < 0 || nQ > INT32_MAX) return 0;
    return contact_ws(nullptr, nQ).bytes;
}

mesh_status mesh_contact(const mesh_bvh *bvh, const float *d_Q, int64_t nQ, float max_dist, int32_t *d_face,
                         float *d_bary, float *d_point, float *d_dist2, void *d_ws, size_t ws_bytes,
                         void *stream) {
    if (!bvh || nQ < 0 || nQ > INT32_MAX || (nQ > 0 && (!d_Q || !d_face)) || !(max_dist >= 0.0f))
        return MESH_ERR_INVALID_ARG;
    if (nQ == 0) return MESH_OK;
    ContactWs w = contact_ws(d_ws, nQ);
    if (!d_ws || ws_bytes < w.bytes || ((uintptr_t)d_ws & 255u)) return MESH_ERR_WORKSPACE;
    int variant = bvh->cfg_variant >= 0 ? bvh->cfg_variant : g_traversal;
    if (bvh->leaf_size > 1 && !(variant == 2 || variant == 3 || variant == 12 || variant == 13)) variant = 0;
    if (variant <= 1 || (variant >= 10 && variant <= 11) || (bvh->cfg_lanes > 1))
        return mesh_closest_point_hinted(bvh, d_Q, nQ, max_dist, d_face, d_face, d_bary, d_point, d_dist2,
                                         stream);
    cudaStream_t s = (cudaStream_t)stream;
    const int n = (int)nQ;
    const int tiles = (n + kClassTile - 1) / kClassTile;
    if (variant == 13) ensure_wide(bvh, s);
    // the call's first kernel is a plain launch (ordered after whatever the caller
    // put on the stream); the two after it are its programmatic dependents
    k_class_count<<<tiles, kClassThreads, 0, s>>>(w.cls, n, w.counts);
    pdl_launch(k_class_scatter, tiles, kClassThreads, 0, s, w.cls, n, w.counts, tiles, w.order);
    count_launch(2);
    float maxd2 = isinf(max_dist) ? INFINITY : max_dist * max_dist;
    Traversal T = traversal_of(bvh, isinf(max_dist));
    Header *h = bvh->hdr();
    const int *iperm = bvh->iperm();
    // the search writes face and distance; the weights follow in one thread per query
    const bool split = kContactSplitWeights && variant != 12 && (d_bary || d_point);
    float *sb = split ? nullptr : d_bary, *sp = split ? nullptr : d_point;
    float *sd = split && !d_dist2 ? w.d2 : d_dist2;
    if (bvh->leaf_size > 1)
        launch_contact<true>(T, h, d_Q, nQ, maxd2, d_face, sb, sp, sd, iperm, w.order, w.cls, variant,
                             bvh->cfg_block, s);
    else
        launch_contact<false>(T, h, d_Q, nQ, maxd2, d_face, sb, sp, sd, iperm, w.order, w.cls, variant,
                              bvh->cfg_block, s);
    count_launch();
    if (split) {
        pdl_launch(k_hit_weights, grid_for(nQ, 256), 256, 0, s, T, d_Q, nQ, (const int *)d_face, (const float *)sd,
                   iperm, d_bary, d_point);
        count_launch();
    }
    return check_launch();
}


size_t mesh_chamfer_workspace_bytes(int64_t nSA, int64_t nSB) {
    if (nSA < 0 || nSB < 0) return 0;
    return align_up(8 * (chamfer_blocks(nSA, 32) + chamfer_blocks(nSB, 32) + 1), 256) + 256;
}

mesh_status mesh_chamfer(const mesh_bvh *A, const float *d_SA, int64_t nSA, const mesh_bvh *B,
                         const float *d_SB, int64_t nSB, void *d_ws, size_t ws_bytes,
                         double *d_out, int32_t *d_faceA, float *d_baryA, float *d_dist2A,
                         int32_t *d_faceB, float *d_baryB, float *d_dist2B, void *stream) {
    return mesh_chamfer_hinted(A, d_SA, nSA, B, d_SB, nSB, d_ws, ws_bytes, d_out, nullptr, nullptr,
                               d_faceA, d_baryA, d_dist2A, d_faceB, d_baryB, d_dist2B, stream);
}

mesh_status mesh_chamfer_hinted(const mesh_bvh *A, const float *d_SA, int64_t nSA, const mesh_bvh *B,
                                const float *d_SB, int64_t nSB, void *d_ws, size_t ws_bytes,
                                double *d_out, const int32_t *d_hintA, const int32_t *d_hintB,
                                int32_t *d_faceA, float *d_baryA, float *d_dist2A,
                                int32_t *d_faceB, float *d_baryB, float *d_dist2B, void *stream) {
    if (!A || !B || !d_out || nSA < 0 || nSB < 0 || (nSA > 0 && !d_SA) || (nSB > 0 && !d_SB))
        return MESH_ERR_INVALID_ARG;
    size_t need = mesh_chamfer_workspace_bytes(nSA, nSB);
    if (!d_ws || ws_bytes < need || ((uintptr_t)d_ws & 255u)) return MESH_ERR_WORKSPACE;
    double *partial = (double *)d_ws;
    unsigned int *ticket = (unsigned int *)((char *)d_ws + need - 256);
    return run_chamfer(A, d_SA, nSA, B, d_SB, nSB, chamfer_lanes(A, B, nSA + nSB), partial, ticket, d_out, d_hintA, d_hintB,
                       d_faceA, d_baryA, d_dist2A, d_faceB, d_baryB, d_dist2B, (cudaStream_t)stream);
}

size_t mesh_chamfer_step_workspace_bytes(int64_t nSA, int64_t nSB) {
    if (nSA < 0 || nSB < 0 || nSA + nSB > INT32_MAX) return 0;
    return chamfer_step_bytes(nSA, nSB);
}

mesh_status mesh_chamfer_step(const mesh_bvh *A, const float *d_SA, int64_t nSA, const mesh_bvh *B,
                              const float *d_SB, int64_t nSB, void *d_ws, size_t ws_bytes, double *d_out,
                              int32_t *d_faceA, float *d_baryA, float *d_dist2A, int32_t *d_faceB,
                              float *d_baryB, float *d_dist2B, void *stream) {
    if (!A || !B || !d_out || nSA < 0 || nSB < 0 || nSA + nSB > INT32_MAX || (nSA > 0 && (!d_SA || !d_faceA)) ||
        (nSB > 0 && (!d_SB || !d_faceB)))
        return MESH_ERR_INVALID_ARG;
    if (!d_ws || ws_bytes < chamfer_step_bytes(nSA, nSB) || ((uintptr_t)d_ws & 255u)) return MESH_ERR_WORKSPACE;
    return mesh_chamfer_hinted(A, d_SA, nSA, B, d_SB, nSB, d_ws, ws_bytes, d_out, d_faceA, d_faceB, d_faceA, d_baryA,
                               d_dist2A, d_faceB, d_baryB, d_dist2B, stream);
}

mesh_status mesh_batch_closest_point(mesh_batch *batch, const float *d_Q,
                                     const int32_t *d_query_off, int64_t nQ, float max_dist,
                                     int32_t *d_face, float *d_bary, float *d_point,
                                     float *d_dist2, void *stream) {
    if (!batch || nQ < 0 || nQ > 0xffff0000LL || (nQ > 0 && (!d_Q || !d_query_off)) ||
        !(max_dist >= 0.0f))
        return MESH_ERR_INVALID_ARG;
    if (nQ == 0) return MESH_OK;
    const bool unbounded = isinf(max_dist);
    pool_batch(batch, d_Q, d_query_off, nQ, unbounded ? INFINITY : max_dist * max_dist, unbounded,
               pool_lanes(nQ, batch->L.n_faces / (batch->L.n_scenes > 0 ? batch->L.n_scenes : 1)), d_face, d_bary,
               d_point, d_dist2, (cudaStream_t)stream);
    return check_launch();
}

mesh_status mesh_closest_point_stats(const mesh_bvh *bvh, const float *d_Q, int64_t nQ,
                                     float max_dist, unsigned long long *d_counts, void *stream) {
    if (!bvh || !d_counts || nQ < 0 || (nQ > 0 && !d_Q) || !(max_dist >= 0.0f))
        return MESH_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    cudaMemsetAsync(d_counts, 0, 3 * sizeof(unsigned long long), s);
    if (nQ == 0) return check_launch();
    float maxd2 = isinf(max_dist) ? INFINITY : max_dist * max_dist;
    const int variant = bvh->cfg_variant >= 0 ? bvh->cfg_variant : g_traversal;
    const bool wide = variant == 13 && bvh->cfg_lanes <= 1;   // the 4-wide records' visits
    if (wide) ensure_wide(bvh, s);
    (bvh->leaf_size > 1 ? (wide ? k_closest_point_count<true, true> : k_closest_point_count<true>)
                        : (wide ? k_closest_point_count<false, true> : k_closest_point_count<false>))
        <<<grid_for(nQ, kQueryBlock), kQueryBlock, 0, s>>>(
        traversal_of(bvh, isinf(max_dist)), bvh->hdr(), &bvh->hdr()->status, d_Q, nQ, maxd2,
        d_counts);
    count_launch();
    return check_launch();
}

mesh_status mesh_set_query_group(int lanes) {
    if (lanes != 0 && lanes != 1 && lanes != 2 && lanes != 4 && lanes != 8 && lanes != 16 &&
        lanes != 32)
        return MESH_ERR_INVALID_ARG;
    g_group_override = lanes;
    return MESH_OK;
}

mesh_status mesh_bvh_set_query_config(mesh_bvh *bvh, int lanes, int variant) {
    if (!bvh) return MESH_ERR_INVALID_ARG;
    if (lanes != -1 && lanes != 0 && lanes != 1 && lanes != 2 && lanes != 4 && lanes != 8 &&
        lanes != 16 && lanes != 32)
        return MESH_ERR_INVALID_ARG;
    if (variant < -1 || variant > 13) return MESH_ERR_INVALID_ARG;
    bvh->cfg_lanes = lanes;
    bvh->cfg_variant = variant;
    return MESH_OK;
}

mesh_status mesh_bvh_set_query_block(mesh_bvh *bvh, int threads) {
    if (!bvh || (threads != 0 && threads != 32 && threads != 64 && threads != 128))
        return MESH_ERR_INVALID_ARG;
    bvh->cfg_block = threads == 0 ? kQueryBlock : threads;
    return MESH_OK;
}

mesh_status mesh_set_traversal(int variant) {
    if (variant < 0 || variant > 13) return MESH_ERR_INVALID_ARG;
    g_traversal = variant;
    return MESH_OK;
}

mesh_status mesh_interpolate(const mesh_bvh *bvh, const int32_t *d_face, const float *d_bary,
                             int64_t n, float *d_out, void *stream) {
    if (!bvh || n < 0 || (n > 0 && (!d_face || !d_bary || !d_out))) return MESH_ERR_INVALID_ARG;
    if (n == 0) return MESH_OK;
    cudaStream_t s = (cudaStream_t)stream;
    k_interpolate<<<grid_for(n, 256), 256, 0, s>>>(bvh->faces(), bvh->verts(), (int)bvh->L.n_faces,
                                                   d_face, d_bary, n, d_out, &bvh->hdr()->status);
    count_launch();
    return check_launch();
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Chamfer without caller workspace.
//
// Some callers cannot allocate device memory at all -- a physics or renderer
// plugin whose host application owns every device allocation, or code that
// runs while another framework is capturing the stream into a CUDA graph and
// forbids allocation -- so they cannot hand mesh_chamfer a workspace.  This
// entry point runs the same Chamfer kernel, with the lanes per sample
// mesh_chamfer would pick (fewer when that many blocks would not fit), with its
// scratch (per-block float64 partial sums and the last-block ticket) in a fixed
// file-scope device array instead.  Every GPU that loads the library holds that
// array until exit.  The array's device address is looked up once per device
// and kept; a cudaDeviceReset invalidates it, so no call may follow a reset in
// the same process.
// ---------------------------------------------------------------------------
namespace meshgs {

constexpr int kNoAllocMaxBlocks = 16384;   // partial sums: 16384 x 8 B = 128 KB
static __device__ __align__(256) double g_chamfer_scratch[kNoAllocMaxBlocks + 32];

constexpr int kMaxDevices = 64;
static double *g_scratch_ptr[kMaxDevices];          // device address per device ordinal
static std::mutex g_scratch_mu;

// Device address of g_chamfer_scratch on the current device, looked up once per
// device (the host-side symbol is only a stand-in, never a device address).
static mesh_status scratch_address(double **out) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return MESH_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    if (!g_scratch_ptr[dev]) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_chamfer_scratch) != cudaSuccess || !p) return MESH_ERR_CUDA;
        g_scratch_ptr[dev] = (double *)p;
    }
    *out = g_scratch_ptr[dev];
    return MESH_OK;
}

}  // namespace meshgs

extern "C" mesh_status mesh_chamfer_noalloc(const mesh_bvh *A, const float *d_SA, int64_t nSA,
                                            const mesh_bvh *B, const float *d_SB, int64_t nSB,
                                            double *d_out, int32_t *d_faceA, float *d_baryA,
                                            float *d_dist2A, int32_t *d_faceB, float *d_baryB,
                                            float *d_dist2B, void *stream) {
    using namespace meshgs;
    if (!A || !B || !d_out || nSA < 0 || nSB < 0 || (nSA > 0 && !d_SA) || (nSB > 0 && !d_SB))
        return MESH_ERR_INVALID_ARG;
    // the lanes per sample mesh_chamfer would use, fewer if its blocks exceed the array
    int G = chamfer_lanes(A, B, nSA + nSB);
    while (G > 1 && chamfer_blocks(nSA, G) + chamfer_blocks(nSB, G) > (size_t)kNoAllocMaxBlocks) G >>= 1;
    size_t nbA = chamfer_blocks(nSA, G), nbB = chamfer_blocks(nSB, G);
    if (nbA + nbB > (size_t)kNoAllocMaxBlocks) return MESH_ERR_WORKSPACE;
    double *scratch = nullptr;
    mesh_status st = scratch_address(&scratch);
    if (st != MESH_OK) return st;
    unsigned int *ticket = (unsigned int *)(scratch + kNoAllocMaxBlocks);
    return run_chamfer(A, d_SA, nSA, B, d_SB, nSB, G, scratch, ticket, d_out, nullptr, nullptr, d_faceA, d_baryA,
                       d_dist2A, d_faceB, d_baryB, d_dist2B, (cudaStream_t)stream);
}
