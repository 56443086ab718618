// NearestSurface by warps that pool the work of several queries.
//
// A warp holds S queries (16 when there are many, fewer when the queries would
// not fill the GPU; 32 in the largest calls of mesh_chamfer_noalloc) and one stack of (node, query) entries for all of them.
// Each step its 32 lanes take the top 32 entries, whoever they belong to: a lane
// reads one node record (two child boxes), tests both against its entry's query
// and pruning radius, and the surviving children go back on the stack -- the
// farther ones of all lanes below the nearer ones, so the pool advances about
// depth first.  Surviving leaves wait in a second queue until 32 of them fill
// the warp, and are then tested together.  What a query has found -- the least
// distance, the pruning radius, the faces near the least distance -- lives in
// shared memory, where any lane updates it.
//
// Why: one thread per query runs as long as its warp's deepest search, and
// tests a face in nearly every step with three or four lanes on; 8 of 32 lanes
// did useful work.  Here a lane is idle only while the pool holds fewer entries
// than lanes, and the tail of one long search is shared by the whole warp: 26 of
// 32 lanes on, 172 warp instructions per warm-started contact query.  Bound by
// the mix of issue (60 % of the slots) and the reads of scattered 64-byte records
// (L1 throughput 65 %) at some 24 resident warps per SM.  1M contact queries of the
// 200k-face torus: 549 -> 309 us cold, 380 -> 255 us warm-started (the one-thread
// form with its work classes); unbounded 12.7 -> 4.5 ms; 20k queries 117 -> 44 us.
//
// The answer is the tie rule's (see nearest.cuh), as every search gives it: a
// node is skipped only when its box is farther than a radius never smaller than
// the final tie window's, and the nearest face is the lowest id among the
// recorded faces inside the final window.
#include <type_traits>

#include "nearest.cuh"

namespace meshgs {

constexpr int kQueryWarps = 1;         // warps per block of the query kernels: a block ends with its own warp (the
                                       // 64-scene batch 17.4 ms against 17.8 with four)
constexpr int kChamferWarps = 4;       // and of the Chamfer kernel (its partial sums are per 128 / G samples)
constexpr int kPoolLeaf = 96;         // waiting leaves: below 32 before a step, at most 64 more after it
// Faces recorded per query near its least distance; a query that meets more keeps
// those that can still be its answer (pool_absorb).
template <int S> constexpr int kPoolRing = S == 32 ? 8 : S == 16 ? 12 : S == 8 ? 16 : 32;
constexpr int kPoolLost = 1 << 20;    // a count from which on faces were not recorded

// An entry is a node or first leaf (30 bits), its query's slot (5 bits), a
// face count less one (3 bits, leaves) and the box distance, its low six bits
// rounded off: an entry's distance only ever rounds down, so it is never
// dropped too early.
template <int S> struct __align__(16) PoolWarp {
    // Node entries.  A depth-first search deep inside a mesh defers about 20 siblings; a warp whose
    // stack fills up goes on with fewer lanes, down to one.  What the stacks leave of an SM's memory
    // caches the tree, but a third less stack for searches under a cutoff gained nothing (1M contacts
    // 555 us, 539 with these) and made those under a loose one up to 5 times as long.
    static constexpr int kStack = S == 32 ? 448 : S == 16 ? 512 : S == 8 ? 384 : S == 4 ? 320 : 256;
    float4 q[S];                      // position, float32 error bound of a distance
    uint2 stack[kStack];
    uint2 leaf[kPoolLeaf];
    uint2 ring[S][kPoolRing<S>];         // (distance bits, leaf) of faces within the window when tested
    unsigned int dmin[S];             // least squared distance, as bits
    float thr[S];                     // pruning radius, squared
    int cnt[S];                       // faces in the ring; kPoolLost or more: some were not recorded
};

// What differs per query when the queries belong to several scenes.
template <int S> struct PoolScene {
    int base[S];                      // first node record and leaf
    float tau[S];
};

__device__ __forceinline__ uint2 pool_entry(int id, int slot, int cnt1, float d2) {
    return make_uint2((unsigned)id | ((unsigned)slot << 30),
                      (__float_as_uint(d2) & ~63u) | ((unsigned)slot >> 2 << 3) | (unsigned)cnt1);
}
__device__ __forceinline__ int pool_id(uint2 e) { return (int)(e.x & 0x3fffffffu); }
__device__ __forceinline__ int pool_slot(uint2 e) { return (int)((e.x >> 30) | (e.y >> 1 & 0x1cu)); }
__device__ __forceinline__ int pool_count(uint2 e) { return (int)(e.y & 7u) + 1; }
__device__ __forceinline__ float pool_dist(uint2 e) { return __uint_as_float(e.y & ~63u); }

// Makes room in the rings of the queries that have just met more faces than their
// rings hold; each such face waits in the lane that tested it (over: slot, d2, leaf,
// face).  Of two recorded faces the farther one with the higher id is never the
// answer, whatever the final window: what remains is a front of falling ids over
// rising distances, one face where many are exactly as far (the faces around a
// vertex).  A window is 2e-6 of a squared distance wide, some 17 to 34 float32
// values, and a front of ids in no order is the logarithm of that; one longer than
// the ring is left to resolve_ties.
//
// The search itself may not be left to resolve_ties: it is one lane's depth-first
// search while the warp waits.  On the axis through a vertex of 512 faces 100 queries
// took 181 us so and 20k 1211, now 46 and 279; 100 queries 1000 radii from a sphere
// of 82k faces (hundreds of faces tie in float32) 443 us, now 54.
template <int S, bool kScenes>
static __device__ __noinline__ void pool_absorb(const float4 *tris, float tau, PoolWarp<S> &W,
                                                const PoolScene<S> *sc, bool over, int slot, float d2, int leaf,
                                                int face) {
    const unsigned int kFull = 0xffffffffu, kNone = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    unsigned int todo = __ballot_sync(kFull, over);
    while (todo) {
        const int sl = __shfl_sync(kFull, slot, __ffs(todo) - 1);
        const bool mine = over && slot == sl;
        todo &= ~__ballot_sync(kFull, mine);
        if (W.cnt[sl] >= kPoolLost) continue;                // decided by resolve_ties already
        const float4 *t = kScenes ? tris + 3 * (size_t)sc->base[sl] : tris;
        float w2, p2;
        windows(__uint_as_float(W.dmin[sl]), kScenes ? sc->tau[sl] : tau, W.q[sl].w, w2, p2);
        // the candidates: a ring entry and a waiting face per lane (a full ring: every entry is set)
        const uint2 e = W.ring[sl][lane < kPoolRing<S> ? lane : 0];
        unsigned int ed = lane < kPoolRing<S> && __uint_as_float(e.x) <= w2 ? e.x : kNone;
        unsigned int nd = mine && d2 <= w2 ? __float_as_uint(d2) : kNone;
        const unsigned int ef = ed != kNone ? __float_as_uint(ldg4(t + 3 * (size_t)e.y).w) : kNone;
        const unsigned int nf = (unsigned)face;
        __syncwarp();                                        // read before the entries are written again
        int n = 0;
        while (true) {                                       // the nearest left, and of those the lowest id
            const unsigned int m = __reduce_min_sync(kFull, min(ed, nd));
            if (m == kNone) break;
            const unsigned int f = __reduce_min_sync(kFull, min(ed == m ? ef : kNone, nd == m ? nf : kNone));
            if (n < kPoolRing<S>) {
                if (ed == m && ef == f) W.ring[sl][n] = e;
                if (nd == m && nf == f) W.ring[sl][n] = make_uint2(m, (unsigned)leaf);
            }
            ++n;
            if (ef >= f) ed = kNone;
            if (nf >= f) nd = kNone;
        }
        if (lane == 0) W.cnt[sl] = n <= kPoolRing<S> ? n : kPoolLost;
        __syncwarp();
    }
}

// A cutoff is loose when the ball of that radius may hold more faces than a search
// should meet without a nearer radius: about n r^2 / diag^2 of a surface of n faces,
// some three times that for a closed one.  With lines at 50, 150 and 200: two contact
// steps of 943k particles, 80k faces, cutoff 0.1 (54 by this estimate) 696 us above the
// line, 675 below it; 50k queries near a 5k-face torus, cutoff 0.7 (160) 79 above, 99
// below.  With no line a loose cutoff cost 2 to 18 times one thread per query (1M
// queries near the 200k-face torus, cutoff 2.0: 19.9 ms against 1.2; 0.96 now).
constexpr float kLooseFaces = 150.0f;

// Meshes of at most kFewFaces faces: a thread per query tests every face.  A warp
// of the pool spends more on starting and ending its queries than such a search
// takes (300k queries of one face: 60 us in the Chamfer kernel's pool, 34 so; figures
// over sizes at pool_lanes).  Bound by the tests, some 100 instructions each.
constexpr int kFewThreads = 128;

__device__ __forceinline__ Hit few_search(const Traversal &T, float4 lo, float4 hi, float3 q, float maxd2,
                                          unsigned int *status) {
    Best B = make_best(T, q, maxd2);
    if (box_d2(q, lo, hi) > B.thr) return Hit{-1, 0x7fffffff, INFINITY};   // (lo, hi: the mesh's box)
    for (int leaf = 0; leaf < T.n; ++leaf) test_leaf(T, B, leaf, q, maxd2);
    return finish(T, B, q, status);
}

// The search of a warp's S queries; lane l < S brings query l (valid or not; T
// holds its mesh's scale and size) and takes its hit.  hint: a leaf tested first, or -1.  A query without a
// hint starts at the first node with two children inside the cutoff (descend: at the
// root), which ends most misses at once (from the root, timed over 792 calls: 2 % more in
// two contact steps or signed distances of 1M ordered particles, 10 to 15 % more where
// most miss; only 1M queries close to the surface and in no order were faster, 977
// against 1076 us); when the cutoff is loose or there is none
// (descend) it then goes down the nearer children to one leaf, so that the pool
// starts with a radius for it.
// sc: per-query offsets into T's arrays (queries of several scenes), or NULL.
template <int S, bool kRange, bool kScenes>
__device__ __forceinline__ Hit pool_search(const Traversal &T, PoolWarp<S> &W, PoolScene<S> *sc, float3 q, bool valid,
                                           float maxd2, int hint, bool descend, unsigned int *status) {
    constexpr int kStack = PoolWarp<S>::kStack;
    const unsigned int kFull = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned int lt = (1u << lane) - 1u;
    // Traversal of slot's scene
    auto scene_of = [&](int slot) {
        Traversal t = T;
        if constexpr (kScenes) {
            t.nodes += 4 * (size_t)sc->base[slot];
            t.tris += 3 * (size_t)sc->base[slot];
            t.tau = sc->tau[slot];
        }
        return t;
    };
    const bool mine = lane < S && valid && T.n > 0;
    if (lane < S) {
        const float slack = query_slack(T, q);
        W.q[lane] = make_float4(q.x, q.y, q.z, slack);
        W.dmin[lane] = 0x7f800000u;
        W.thr[lane] = cutoff_window2(maxd2, T.tau, slack);
        W.cnt[lane] = 0;
        if constexpr (kScenes) sc->tau[lane] = T.tau;        // base is set by the caller
    }
    __syncwarp();
    int first = -1, first_cnt = 1, root = -1;                // the leaf this query tests first, the node it starts from
    if (mine) {
        if (T.n == 1) {
            first = 0;
        } else if (hint >= 0) {
            first = hint;
            root = 0;
        } else {
            const Traversal t = scene_of(lane);
            const float thr = W.thr[lane];
            // down to the first node with two children inside the cutoff
            int node = 0;
            while (node >= 0 && !descend) {
                const float4 *r = t.nodes + 4 * (size_t)node;
                const float4 l0 = ldg4(r), l1 = ldg4(r + 1), r0 = ldg4(r + 2), r1 = ldg4(r + 3);
                const bool il = box_d2(q, l0, l1) <= thr, ir = box_d2(q, r0, r1) <= thr;
                if (il && ir) break;
                node = -1;
                if (il || ir) {
                    const int c = __float_as_int(il ? l0.w : r0.w);
                    if (c >= 0) {
                        node = c;
                    } else {
                        first = -c - 1;
                        if constexpr (kRange) first_cnt = __float_as_int(il ? l1.w : r1.w);
                    }
                }
            }
            root = node;
            // a radius, where the cutoff leaves many faces: down the nearer children to a leaf
            const float diag = T.tau * (1.0f / kTieAbs);
            if (node >= 0 && (descend || maxd2 * (float)T.n > kLooseFaces * diag * diag)) {
                while (true) {
                    const float4 *r = t.nodes + 4 * (size_t)node;
                    const float4 l0 = ldg4(r), l1 = ldg4(r + 1), r0 = ldg4(r + 2), r1 = ldg4(r + 3);
                    const float dl = box_d2(q, l0, l1), dr = box_d2(q, r0, r1);
                    bool left = dl < dr;
                    if (dl == dr) left = box_minmax_d2(q, l0, l1) <= box_minmax_d2(q, r0, r1);
                    const int c = __float_as_int(left ? l0.w : r0.w);
                    if (c >= 0) { node = c; continue; }
                    first = -c - 1;
                    if constexpr (kRange) first_cnt = __float_as_int(left ? l1.w : r1.w);
                    break;
                }
            }
        }
    }
    const unsigned int fm = __ballot_sync(kFull, first >= 0), rm = __ballot_sync(kFull, root >= 0);
    if (first >= 0) W.leaf[__popc(fm & lt)] = pool_entry(first, lane, first_cnt - 1, 0.0f);
    if (root >= 0) W.stack[__popc(rm & lt)] = pool_entry(root, lane, 0, 0.0f);
    int nleaf = __popc(fm), nstack = __popc(rm);
    bool start = nleaf > 0;                                  // the first leaves are tested before any node
    __syncwarp();
    while (true) {
        if (nleaf >= 32 || start || (nstack == 0 && nleaf > 0)) {
            // ---- test up to 32 waiting leaves, one per lane
            const int take = min(32, nleaf);
            start = start && nleaf > 32;
            uint2 e = make_uint2(0u, 0u);
            if (lane < take) e = W.leaf[nleaf - 1 - lane];
            nleaf -= take;
            const int slot = pool_slot(e);
            const bool act = lane < take && pool_dist(e) <= W.thr[slot];
            const float4 qs = W.q[slot];
            const float3 p = xyz(qs);
            const Traversal t = scene_of(slot);
            int most = 1, cnt = act ? 1 : 0;
            if constexpr (kRange) {
                cnt = act ? pool_count(e) : 0;
                most = (int)__reduce_max_sync(kFull, (unsigned)cnt);
            }
            for (int k = 0; k < most; ++k) {
                const int leaf = pool_id(e) + k;
                float d2 = INFINITY;
                int face = 0;
                const bool test = k < cnt;
                if (test) {
                    const float4 *tr = t.tris + 3 * (size_t)leaf;
                    const float4 a = ldg4(tr), b = ldg4(tr + 1), c = ldg4(tr + 2);
                    d2 = tri_distance2(p, xyz(a), xyz(b), xyz(c), b.w != 0.0f);
                    face = __float_as_int(a.w);
                    atomicMin(&W.dmin[slot], __float_as_uint(d2));
                }
                __syncwarp();
                bool over = false;                           // met, and the ring is full
                if (test) {
                    float w2, p2;
                    windows(__uint_as_float(W.dmin[slot]), t.tau, qs.w, w2, p2);
                    W.thr[slot] = fminf(W.thr[slot], p2);    // the same value from every lane of the slot
                    if (d2 <= w2) {
                        const int pos = atomicAdd(&W.cnt[slot], 1);
                        over = pos >= kPoolRing<S>;
                        if (!over) W.ring[slot][pos] = make_uint2(__float_as_uint(d2), (unsigned)leaf);
                    }
                }
                __syncwarp();
                if (__any_sync(kFull, over))
                    pool_absorb<S, kScenes>(T.tris, T.tau, W, sc, over, slot, d2, leaf, face);
            }
            continue;
        }
        if (nstack == 0) break;
        // ---- visit up to 32 nodes, one per lane; fewer when the stack is nearly full (its last
        // kMaxTreeDepth entries are room for one entry's subtree taken depth first)
        const int take = min(min(32, nstack), max(1, kStack - kMaxTreeDepth - nstack));
        uint2 e = make_uint2(0u, 0u);
        if (lane < take) e = W.stack[nstack - 1 - lane];
        nstack -= take;
        __syncwarp();
        const int slot = pool_slot(e);
        const float thr = W.thr[slot];
        const bool act = lane < take && pool_dist(e) <= thr;
        const float3 p = xyz(W.q[slot]);
        int cn = 0, cf = 0, leaves = 0;                      // nearer and farther child; 1: left leaf, 2: right leaf
        float dn = 0.0f, df = 0.0f, dl = 0.0f, dr = 0.0f;
        int ll = 0, lr = 0, nl = 0, nr = 0;
        bool pn = false, pf = false;
        if (act) {
            const Traversal t = scene_of(slot);
            const float4 *r = t.nodes + 4 * (size_t)pool_id(e);
            const float4 l0 = ldg4(r), l1 = ldg4(r + 1), r0 = ldg4(r + 2), r1 = ldg4(r + 3);
            dl = box_d2(p, l0, l1);
            dr = box_d2(p, r0, r1);
            const int cl = __float_as_int(l0.w), cr = __float_as_int(r0.w);
            const bool il = dl <= thr, ir = dr <= thr;
            const bool gl = il && cl >= 0, gr = ir && cr >= 0;
            leaves = (il && cl < 0 ? 1 : 0) | (ir && cr < 0 ? 2 : 0);
            ll = -cl - 1;
            lr = -cr - 1;
            if constexpr (kRange) { nl = __float_as_int(l1.w) - 1; nr = __float_as_int(r1.w) - 1; }
            const bool left = gl && (!gr || dl <= dr);
            pn = gl || gr;
            pf = gl && gr;
            cn = left ? cl : cr;
            dn = left ? dl : dr;
            cf = left ? cr : cl;
            df = left ? dr : dl;
        }
        const unsigned int bf = __ballot_sync(kFull, pf), bn = __ballot_sync(kFull, pn);
        const unsigned int bl = __ballot_sync(kFull, leaves & 1), br = __ballot_sync(kFull, leaves & 2);
        const int nf = __popc(bf), lf = __popc(bl);
        if (pf) W.stack[nstack + __popc(bf & lt)] = pool_entry(cf, slot, 0, df);
        if (pn) W.stack[nstack + nf + __popc(bn & lt)] = pool_entry(cn, slot, 0, dn);
        if (leaves & 1) W.leaf[nleaf + __popc(bl & lt)] = pool_entry(ll, slot, nl, dl);
        if (leaves & 2) W.leaf[nleaf + lf + __popc(br & lt)] = pool_entry(lr, slot, nr, dr);
        nstack += nf + __popc(bn);
        nleaf += lf + __popc(br);
        __syncwarp();
    }
    // ---- each query's answer: the lowest id inside the final window
    Hit h{-1, 0x7fffffff, INFINITY};
    if (mine) {
        const float m = __uint_as_float(W.dmin[lane]);
        if (m <= maxd2) {
            const Traversal t = scene_of(lane);
            const int cnt = W.cnt[lane];
            if (cnt >= kPoolLost) {
                Best B{-1, INFINITY, m, 0.0f, -1.0f};
                resolve_ties(t, B, q, status);
                h.leaf = B.leaf;
                h.d2 = B.d2;
            } else {
                float w2, p2;
                windows(m, t.tau, W.q[lane].w, w2, p2);
                for (int j = 0; j < cnt; ++j) {
                    const uint2 c = W.ring[lane][j];
                    if (!(__uint_as_float(c.x) <= w2)) continue;
                    const int f = face_of(t, (int)c.y);
                    if (f < h.face) { h.face = f; h.leaf = (int)c.y; h.d2 = __uint_as_float(c.x); }
                }
            }
            if (h.leaf >= 0 && cnt >= kPoolLost) h.face = face_of(t, h.leaf);
        }
    }
    return h;
}

// The queries of a warp: S consecutive ones.
template <int S, bool kRange>
__global__ void __launch_bounds__(32 * kQueryWarps, 32 / kQueryWarps)
k_pool_closest_point(Traversal T, const Header *__restrict__ hdr, unsigned int *status, const float *__restrict__ Q,
                     int64_t nQ, float maxd2, int *face, float *bary, float *point, float *dist2, const int *hint,
                     const int *__restrict__ iperm) {
    __shared__ PoolWarp<S> s_pool[kQueryWarps];
    pdl_wait();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t i0 = ((int64_t)blockIdx.x * kQueryWarps + wid) * S, i = i0 + lane;
    if (i0 >= nQ) return;                                    // whole warp past the end
    const bool valid = lane < S && i < nQ;
    set_scale(T, hdr);
    const float3 q = valid ? make_float3(Q[3 * i], Q[3 * i + 1], Q[3 * i + 2]) : make_float3(0.0f, 0.0f, 0.0f);
    int hl = -1;
    if (valid && hint) {                                     // may alias face: read before the write below
        const int hf = hint[i];
        if (hf >= 0 && hf < T.n) hl = __ldg(iperm + hf);
    }
    const Hit h = pool_search<S, kRange, false>(T, s_pool[wid], nullptr, q, valid, maxd2, hl, T.mmd, status);
    if (valid) write_hit(T, h, q, i, face, bary, point, dist2);
}

__global__ void __launch_bounds__(kFewThreads)
k_few_closest_point(Traversal T, const Header *__restrict__ hdr, unsigned int *status, const float *__restrict__ Q,
                    int64_t nQ, float maxd2, int *face, float *bary, float *point, float *dist2) {
    const int64_t i = (int64_t)blockIdx.x * kFewThreads + threadIdx.x;
    if (i >= nQ) return;
    set_scale(T, hdr);
    const float3 q = make_float3(Q[3 * i], Q[3 * i + 1], Q[3 * i + 2]);
    write_hit(T, few_search(T, hdr->root_lo, hdr->root_hi, q, maxd2, status), q, i, face, bary, point, dist2);
}

// Queries of many scenes (mesh_batch_closest_point): each lane finds its query's
// scene, and the pool's entries carry scene-local nodes.
template <int S>
__global__ void __launch_bounds__(32, 32)
k_pool_batch(const float4 *__restrict__ nodes, const float4 *__restrict__ tris, const float4 *__restrict__ scene_box,
             const int *__restrict__ face_off, const int *__restrict__ query_off, int nscenes,
             const float *__restrict__ Q, int64_t nQ, float maxd2, bool mmd, int *face, float *bary, float *point,
             float *dist2, unsigned int *status) {
    __shared__ PoolWarp<S> s_pool;
    __shared__ PoolScene<S> s_scene;
    const int lane = threadIdx.x;
    const int64_t i0 = (int64_t)blockIdx.x * S, i = i0 + lane;
    if (i0 >= nQ) return;
    const bool valid = lane < S && i < nQ;
    Traversal T{nodes, tris, 0, 0.0f, 0.0f, mmd, nullptr};
    float3 q = make_float3(0.0f, 0.0f, 0.0f);
    int fb = 0;
    if (valid) {
        const int sc = segment_of(query_off, nscenes, i);
        fb = __ldg(face_off + sc);
        T.n = __ldg(face_off + sc + 1) - fb;
        set_scale(T, scene_box[2 * sc], scene_box[2 * sc + 1]);
        q = make_float3(Q[3 * i], Q[3 * i + 1], Q[3 * i + 2]);
    }
    if (lane < S) s_scene.base[lane] = fb;
    Hit h = pool_search<S, false, true>(T, s_pool, &s_scene, q, valid, maxd2, -1, mmd, status);
    if (!valid) return;
    if (h.leaf >= 0) h.face -= fb;
    T.tris += 3 * (size_t)fb;
    write_hit(T, h, q, i, face, bary, point, dist2);
}

// The same for batches whose scenes have at most kFewFaces faces on average: a thread
// per query of such a scene; the queries of the others go to the pool, half a warp
// at a time.
__global__ void __launch_bounds__(32, 32)
k_few_batch(const float4 *__restrict__ nodes, const float4 *__restrict__ tris, const float4 *__restrict__ scene_box,
            const int *__restrict__ face_off, const int *__restrict__ query_off, int nscenes,
            const float *__restrict__ Q, int64_t nQ, float maxd2, bool mmd, int *face, float *bary, float *point,
            float *dist2, unsigned int *status) {
    constexpr int S = 16;
    __shared__ PoolWarp<S> s_pool;
    __shared__ PoolScene<S> s_scene;
    const unsigned int kFull = 0xffffffffu;
    const int lane = threadIdx.x;
    const int64_t i = (int64_t)blockIdx.x * 32 + lane;
    Traversal T{nodes, tris, 0, 0.0f, 0.0f, mmd, nullptr};
    float3 q = make_float3(0.0f, 0.0f, 0.0f);
    int fb = 0, sc = 0;
    if (i < nQ) {
        sc = segment_of(query_off, nscenes, i);
        fb = __ldg(face_off + sc);
        T.n = __ldg(face_off + sc + 1) - fb;
        set_scale(T, scene_box[2 * sc], scene_box[2 * sc + 1]);
        q = make_float3(Q[3 * i], Q[3 * i + 1], Q[3 * i + 2]);
    }
    Hit h{-1, 0x7fffffff, INFINITY};
    if (T.n > 0 && T.n <= kFewFaces) {
        Traversal own = T;
        own.tris += 3 * (size_t)fb;
        own.nodes += 4 * (size_t)fb;
        h = few_search(own, scene_box[2 * sc], scene_box[2 * sc + 1], q, maxd2, status);
    }
    for (int half = 0; half < 2; ++half) {
        const bool mine = T.n > kFewFaces && lane / S == half;
        if (!__any_sync(kFull, mine)) continue;
        const int src = half * S + lane % S;                 // lanes 0 to 15 take the half's queries
        const bool valid = __shfl_sync(kFull, (int)mine, src) && lane < S;
        const float3 qh = make_float3(__shfl_sync(kFull, q.x, src), __shfl_sync(kFull, q.y, src),
                                      __shfl_sync(kFull, q.z, src));
        Traversal Th = T;
        Th.n = __shfl_sync(kFull, T.n, src);
        Th.tau = __shfl_sync(kFull, T.tau, src);
        Th.vmax = __shfl_sync(kFull, T.vmax, src);
        const int fh = __shfl_sync(kFull, fb, src);
        if (lane < S) s_scene.base[lane] = fh;
        const Hit g = pool_search<S, false, true>(Th, s_pool, &s_scene, qh, valid, maxd2, -1, mmd, status);
        const int leaf = __shfl_sync(kFull, g.leaf, lane % S), f = __shfl_sync(kFull, g.face, lane % S);
        const float d2 = __shfl_sync(kFull, g.d2, lane % S);
        if (mine) h = Hit{leaf, f, d2};
        __syncwarp();
    }
    if (i >= nQ) return;
    if (h.leaf >= 0) h.face -= fb;
    T.tris += 3 * (size_t)fb;
    write_hit(T, h, q, i, face, bary, point, dist2);
}

// ---------------------------------------------------------------------------
// Chamfer (Sec. 4.2): both directions in one launch (blocks [0, nbA) query SA
// against B, the rest SB against A).  Each block sums its squared distances in
// float64 with a fixed reduction tree and stores the partial; the last block
// to finish (ticket counter) adds the partials in a fixed order, writes the
// two means and resets the counter, so the result is bit-reproducible.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double block_sum_d(double x, double *s) {
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) s[w] = x;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) t += s[k];
    __syncthreads();
    return t;
}

// S = 0: both meshes have few faces, a thread per sample.
template <int S, bool kRange>
__global__ void __launch_bounds__(32 * kChamferWarps, 32 / kChamferWarps)
k_pool_chamfer(ChamferSide A2B, ChamferSide B2A, unsigned int nbA, unsigned int *status, double *partial,
               unsigned int *ticket, double *out) {
    constexpr int kOwn = S == 0 ? 32 : S;                    // samples of a warp
    __shared__ double s_red[kChamferWarps];
    __shared__ bool s_last;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const bool first = blockIdx.x < nbA;
    const ChamferSide &C = first ? A2B : B2A;
    const int64_t i0 = ((int64_t)(first ? blockIdx.x : blockIdx.x - nbA) * kChamferWarps + wid) * kOwn, i = i0 + lane;
    const bool valid = lane < kOwn && i < C.n;
    double d2 = 0.0;
    if (i0 < C.n) {                                          // uniform in the warp
        Traversal T = C.T;
        set_scale(T, C.hdr);
        const float3 q = valid ? make_float3(C.S[3 * i], C.S[3 * i + 1], C.S[3 * i + 2]) : make_float3(0.0f, 0.0f, 0.0f);
        Hit h{-1, 0x7fffffff, INFINITY};
        if constexpr (S == 0) {
            if (valid) h = few_search(T, C.hdr->root_lo, C.hdr->root_hi, q, INFINITY, status);
        } else {
            __shared__ PoolWarp<S> s_pool[kChamferWarps];
            int hl = -1;
            if (valid && C.hint) {
                const int hf = C.hint[i];
                if (hf >= 0 && hf < T.n) hl = __ldg(C.iperm + hf);
            }
            h = pool_search<S, kRange, false>(T, s_pool[wid], nullptr, q, valid, INFINITY, hl, true, status);
        }
        if (valid) {
            write_hit(T, h, q, i, C.face, C.bary, nullptr, C.dist2);
            d2 = h.leaf >= 0 ? (double)h.d2 : 0.0;
        }
    }
    const double s = block_sum_d(d2, s_red);
    if (threadIdx.x == 0) {
        partial[blockIdx.x] = s;
        __threadfence();
        unsigned int t = atomicAdd(ticket, 1u);
        s_last = (t == gridDim.x - 1);
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // fixed-order final sums: thread k adds partials k, k + blockDim, ... of each side
    double a = 0.0, b = 0.0;
    for (unsigned int k = threadIdx.x; k < nbA; k += blockDim.x) a += __ldcg(partial + k);
    for (unsigned int k = nbA + threadIdx.x; k < gridDim.x; k += blockDim.x) b += __ldcg(partial + k);
    a = block_sum_d(a, s_red);
    b = block_sum_d(b, s_red);
    if (threadIdx.x == 0) {
        out[0] = A2B.n > 0 ? a / (double)A2B.n : 0.0;
        out[1] = B2A.n > 0 ? b / (double)B2A.n : 0.0;
        *ticket = 0u;
    }
}

// Angle-weighted pseudo-normal of vertex vid (Baerentzen & Aanaes 2005): the
// sum over the faces around it of the unit face normal times the face's angle
// at the vertex.  The ring is found from face f through the face adjacency
// (for a consistently oriented mesh, crossing the edge that follows the vertex
// in each face turns one way round it; an open ring is also walked the other
// way from f), up to kMaxRing faces, and summed in ascending face id, so the
// result is the same whichever face the walk starts from and run to run.  A
// ring larger than kMaxRing (or one the adjacency cannot close) sets
// MESH_DEV_NONMANIFOLD and sums the faces found.
constexpr int kMaxRing = 32;

__device__ __forceinline__ int slot_of(int4 fv, int vid) {
    return fv.x == vid ? 0 : (fv.y == vid ? 1 : (fv.z == vid ? 2 : -1));
}

__device__ __forceinline__ float4 vertex_pseudo_normal(const int4 *__restrict__ faces, const int *__restrict__ adj,
                                                    const float4 *__restrict__ verts,
                                                    const float4 *__restrict__ fnorm, int f, int vid,
                                                    unsigned int *status) {
    int ring[kMaxRing];
    int nr = 0;
    bool full = false;
    int g = f;
    while (true) {                                   // one way round
        ring[nr++] = g;
        int k = slot_of(faces[g], vid);
        int h = k < 0 ? -1 : adj[3 * g + (k + 2) % 3];
        if (h == f) break;
        if (h < 0) break;
        if (nr == kMaxRing) { full = true; break; }
        g = h;
    }
    if (!full && nr < kMaxRing) {                     // open ring: the other way from f
        int k0 = slot_of(faces[f], vid);
        int h = k0 < 0 ? -1 : adj[3 * f + (k0 + 1) % 3];
        bool closed = false;
        for (int i = 0; i < nr; ++i) closed |= ring[i] == h;
        while (h >= 0 && !closed) {
            if (nr == kMaxRing) { full = true; break; }
            ring[nr++] = h;
            int k = slot_of(faces[h], vid);
            int nh = k < 0 ? -1 : adj[3 * h + (k + 1) % 3];
            for (int i = 0; i < nr; ++i) closed |= ring[i] == nh;
            h = nh;
        }
    }
    if (full) atomicOr(status, (unsigned)MESH_DEV_NONMANIFOLD);
    float nx = 0.0f, ny = 0.0f, nz = 0.0f;
    int last = -1;
    for (int done = 0; done < nr; ++done) {          // ascending face id (distinct ids)
        int pick = 0x7fffffff;
        for (int i = 0; i < nr; ++i)
            if (ring[i] > last && ring[i] < pick) pick = ring[i];
        if (pick == 0x7fffffff) break;
        last = pick;
        int4 fv = faces[pick];
        int k = slot_of(fv, vid);
        if (k < 0) continue;
        int id[3] = {fv.x, fv.y, fv.z};
        float4 p = verts[id[k]], a = verts[id[(k + 1) % 3]], b = verts[id[(k + 2) % 3]];
        float ax = a.x - p.x, ay = a.y - p.y, az = a.z - p.z;
        float bx = b.x - p.x, by = b.y - p.y, bz = b.z - p.z;
        float la = sqrtf(ax * ax + ay * ay + az * az), lb = sqrtf(bx * bx + by * by + bz * bz);
        if (la == 0.0f || lb == 0.0f) continue;
        float cs = fminf(1.0f, fmaxf(-1.0f, (ax * bx + ay * by + az * bz) / (la * lb)));
        float ang = acosf(cs);
        float4 n = fnorm[pick];
        nx += ang * n.x; ny += ang * n.y; nz += ang * n.z;
    }
    return make_float4(nx, ny, nz, 0.0f);
}

// NearestSurface plus the sign of (q - c) . N, N the pseudo-normal of the
// feature the nearest point lies on: face interior (no zero weight), edge
// opposite vertex k (weight k zero), vertex (two zero weights).
static __device__ __noinline__ float signed_of_hit(const Traversal &T, Hit h, float3 q, const int4 *__restrict__ faces,
                                                   const int *__restrict__ adj, const float4 *__restrict__ fnorm,
                                                   const float4 *__restrict__ verts, unsigned int *status) {
    const float4 *t = T.tris + 3 * (size_t)h.leaf;
    float4 a = ldg4(t), b = ldg4(t + 1), c = ldg4(t + 2);
    float u, v, w;
    tri_closest(q, xyz(a), xyz(b), xyz(c), b.w != 0.0f, u, v, w);
    if (weights_need_f64(xyz(a), xyz(b), xyz(c), h.d2))
        tri_weights_f64(q, xyz(a), xyz(b), xyz(c), b.w != 0.0f, u, v, w);
    int f = h.face;
    int zeros = (u == 0.0f) + (v == 0.0f) + (w == 0.0f);
    float4 N;
    if (zeros == 0) {
        N = fnorm[f];
    } else if (zeros == 1) {
        int k = u == 0.0f ? 0 : (v == 0.0f ? 1 : 2);
        N = fnorm[f];
        int g = adj[3 * f + k];
        if (g >= 0) { float4 m = fnorm[g]; N.x += m.x; N.y += m.y; N.z += m.z; }
    } else {
        int4 fv = faces[f];
        int vid = u != 0.0f ? fv.x : (v != 0.0f ? fv.y : fv.z);
        N = vertex_pseudo_normal(faces, adj, verts, fnorm, f, vid, status);
    }
    float cx = u * a.x + v * b.x + w * c.x, cy = u * a.y + v * b.y + w * c.y, cz = u * a.z + v * b.z + w * c.z;
    float dn = (q.x - cx) * N.x + (q.y - cy) * N.y + (q.z - cz) * N.z;
    return (dn >= 0.0f ? 1.0f : -1.0f) * sqrtf(h.d2);
}

template <int S, bool kRange>
__global__ void __launch_bounds__(32 * kQueryWarps, 32 / kQueryWarps)
k_pool_signed(Traversal T, const Header *__restrict__ hdr, unsigned int *status, const float *__restrict__ Q,
              int64_t nQ, float maxd2, const int4 *__restrict__ faces, const int *__restrict__ adj,
              const float4 *__restrict__ fnorm, const float4 *__restrict__ verts, int *face, float *bary,
              float *point, float *sdist) {
    __shared__ PoolWarp<S> s_pool[kQueryWarps];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t i0 = ((int64_t)blockIdx.x * kQueryWarps + wid) * S, i = i0 + lane;
    if (i0 >= nQ) return;
    const bool valid = lane < S && i < nQ;
    set_scale(T, hdr);
    const float3 q = valid ? make_float3(Q[3 * i], Q[3 * i + 1], Q[3 * i + 2]) : make_float3(0.0f, 0.0f, 0.0f);
    const Hit h = pool_search<S, kRange, false>(T, s_pool[wid], nullptr, q, valid, maxd2, -1, T.mmd, status);
    if (!valid) return;
    write_hit(T, h, q, i, face, bary, point, nullptr);
    sdist[i] = h.leaf < 0 ? INFINITY : signed_of_hit(T, h, q, faces, adj, fnorm, verts, status);
}

__global__ void __launch_bounds__(kFewThreads)
k_few_signed(Traversal T, const Header *__restrict__ hdr, unsigned int *status, const float *__restrict__ Q,
             int64_t nQ, float maxd2, const int4 *__restrict__ faces, const int *__restrict__ adj,
             const float4 *__restrict__ fnorm, const float4 *__restrict__ verts, int *face, float *bary, float *point,
             float *sdist) {
    const int64_t i = (int64_t)blockIdx.x * kFewThreads + threadIdx.x;
    if (i >= nQ) return;
    set_scale(T, hdr);
    const float3 q = make_float3(Q[3 * i], Q[3 * i + 1], Q[3 * i + 2]);
    const Hit h = few_search(T, hdr->root_lo, hdr->root_hi, q, maxd2, status);
    write_hit(T, h, q, i, face, bary, point, nullptr);
    sdist[i] = h.leaf < 0 ? INFINITY : signed_of_hit(T, h, q, faces, adj, fnorm, verts, status);
}

// ---------------------------------------------------------------------------
// k-NN weighted surface projection: the NearestSurface of temporal tracking
// (Sec. 3.3, Strategy 1, Eq. 1).  The paper names the method without k or
// weights; here: the k faces nearest to the query (ties by the lower face
// id), each giving its closest point p_j at distance d_j, blended with
// weights 1 / max(d_j, 1e-6 x box diagonal); optionally mixed with an anchor
// point, (1 - a) v' + a anchor (the periodic re-anchoring to the template).
//
// The pooled search with a sorted list of the k best (distance, face) per query
// in shared memory; a face that enters is inserted by the whole warp, one lane per
// list entry, a query's nearest first, which rules out most of the others (14k
// template points' rebuild and projection 177 us in the order met, 163 so; 300k
// queries on the axis through a vertex of 512 faces, k = 4, 9.0 and 3.0 ms).  The pruning radius is the k-th distance, widened by the
// float32 bound, so the k faces are those of least (distance, id) whatever the
// order.  A query first goes down to one leaf and tests the leaves beside it in
// leaf order, which are near it, so the search starts with k faces.  A tracked
// template has some 10k vertices: one thread each left 108 blocks waiting on
// their longest search (367 us at 13.7k queries and 40k faces; rebuild and
// projection together 583 us, 231 us with the pool).
// ---------------------------------------------------------------------------
template <int S> struct __align__(16) PoolKnn {
    static constexpr int kStack = S == 8 ? 320 : 256;
    static constexpr int kSeeds = kPoolLeaf / 8;         // leaves a query tests first
    float4 q[S];
    uint2 stack[kStack];
    uint2 leaf[kPoolLeaf];
    float d2[S][kKnnMax];                                // sorted by (distance, face)
    int face[S][kKnnMax], pos[S][kKnnMax];               // face id and leaf
    float thr[S];
};

// Does a face come before the last of a query's list?
template <int S>
__device__ __forceinline__ bool knn_enters(const PoolKnn<S> &W, int slot, int k, float d2, int f) {
    const float last = W.d2[slot][k - 1];
    return d2 < last || (d2 == last && f < W.face[slot][k - 1]);
}

template <int S, bool kRange>
__global__ void __launch_bounds__(32, 32)
k_pool_knn(Traversal T, const Header *__restrict__ hdr, const float *Q, int64_t nQ, int k, const float *anchor,
           float anchor_w, float *point, int *face_out, float *d2_out) {
    __shared__ PoolKnn<S> W;
    constexpr int kStack = PoolKnn<S>::kStack, kSeeds = PoolKnn<S>::kSeeds;
    const unsigned int kFull = 0xffffffffu;
    const int lane = threadIdx.x;
    const unsigned int lt = (1u << lane) - 1u;
    const int64_t i0 = (int64_t)blockIdx.x * S;
    const int own = (int)(nQ - i0 < S ? nQ - i0 : S);    // this warp's queries
    set_scale(T, hdr);
    for (int j = lane; j < S * kKnnMax; j += 32) {
        W.d2[j / kKnnMax][j % kKnnMax] = INFINITY;
        W.face[j / kKnnMax][j % kKnnMax] = 0x7fffffff;
        W.pos[j / kKnnMax][j % kKnnMax] = -1;
    }
    float3 q = make_float3(0.0f, 0.0f, 0.0f);
    int seed = -1;                                       // the leaf this query comes down to
    if (lane < own) {
        const int64_t i = i0 + lane;
        q = make_float3(Q[3 * i], Q[3 * i + 1], Q[3 * i + 2]);   // may alias point
        W.q[lane] = make_float4(q.x, q.y, q.z, query_slack(T, q));
        W.thr[lane] = INFINITY;
        if (T.n == 1) {
            seed = 0;
        } else if (T.n > 1) {
            int node = 0;
            while (seed < 0) {
                const float4 *r = T.nodes + 4 * (size_t)node;
                const float4 l0 = ldg4(r), l1 = ldg4(r + 1), r0 = ldg4(r + 2), r1 = ldg4(r + 3);
                const float dl = box_d2(q, l0, l1), dr = box_d2(q, r0, r1);
                bool left = dl < dr;
                if (dl == dr) left = box_minmax_d2(q, l0, l1) <= box_minmax_d2(q, r0, r1);
                const int c = __float_as_int(left ? l0.w : r0.w);
                if (c >= 0) node = c;
                else seed = -c - 1;
            }
        }
    }
    // the leaves around each query's own, and its root
    int nleaf = 0, nstack = 0;
    {
        const int m = min(min(2 * k, kSeeds), T.n);      // seeds per query
        const int s0 = min(max(seed - m / 2, 0), T.n - m);
        if (seed >= 0)
            for (int j = 0; j < m; ++j) W.leaf[lane * m + j] = pool_entry(s0 + j, lane, 0, 0.0f);
        if (T.n > 0) nleaf = own * m;
        if (T.n > 1) {
            if (lane < own) W.stack[lane] = pool_entry(0, lane, 0, 0.0f);
            nstack = own;
        }
    }
    bool start = nleaf > 0;
    __syncwarp();
    while (true) {
        if (nleaf >= 32 || start || (nstack == 0 && nleaf > 0)) {
            const int take = min(32, nleaf);
            uint2 e = make_uint2(0u, 0u);
            if (lane < take) e = W.leaf[nleaf - 1 - lane];
            nleaf -= take;
            start = start && nleaf > 0;
            const int slot = pool_slot(e);
            const bool act = lane < take && pool_dist(e) <= W.thr[slot];
            const float3 p = xyz(W.q[slot]);
            int most = 1, cnt = act ? 1 : 0;
            if constexpr (kRange) {
                cnt = act ? pool_count(e) : 0;
                most = (int)__reduce_max_sync(kFull, (unsigned)cnt);
            }
            for (int j = 0; j < most; ++j) {
                const int leaf = pool_id(e) + j;
                float d2 = INFINITY;
                int f = 0;
                bool in = j < cnt;
                if (in) {
                    const float4 *tr = T.tris + 3 * (size_t)leaf;
                    const float4 a = ldg4(tr), b = ldg4(tr + 1), c = ldg4(tr + 2);
                    d2 = tri_distance2(p, xyz(a), xyz(b), xyz(c), b.w != 0.0f);
                    f = __float_as_int(a.w);
                    in = knn_enters(W, slot, k, d2, f);
                }
                unsigned int todo = __ballot_sync(kFull, in);
                while (todo) {                           // insert one face: lane l < k has entry l
                    const int sl = __shfl_sync(kFull, slot, __ffs(todo) - 1);
                    const unsigned int db = in && slot == sl ? __float_as_uint(d2) : 0xffffffffu;
                    const unsigned int dm = __reduce_min_sync(kFull, db);
                    const unsigned int fm = __reduce_min_sync(kFull, db == dm ? (unsigned)f : 0xffffffffu);
                    const int src = __ffs(__ballot_sync(kFull, db == dm && (unsigned)f == fm)) - 1;
                    const int fc = (int)fm, lf = __shfl_sync(kFull, leaf, src);
                    const float d = __uint_as_float(dm);
                    const bool entry = lane < k;
                    const float ed = entry ? W.d2[sl][lane] : INFINITY;
                    const int ef = entry ? W.face[sl][lane] : 0x7fffffff, ep = entry ? W.pos[sl][lane] : -1;
                    const bool listed = __any_sync(kFull, entry && ef == fc);
                    const int at = __popc(__ballot_sync(kFull, entry && (ed < d || (ed == d && ef < fc))));
                    const float ud = __shfl_up_sync(kFull, ed, 1);
                    const int uf = __shfl_up_sync(kFull, ef, 1), up = __shfl_up_sync(kFull, ep, 1);
                    if (!listed && entry && lane >= at) {
                        const float nd = lane == at ? d : ud;
                        W.d2[sl][lane] = nd;
                        W.face[sl][lane] = lane == at ? fc : uf;
                        W.pos[sl][lane] = lane == at ? lf : up;
                        if (lane == k - 1) {
                            const float r = sqrtf(nd) + W.q[sl].w;
                            W.thr[sl] = r * r;
                        }
                    }
                    __syncwarp();
                    in = in && lane != src && knn_enters(W, slot, k, d2, f);
                    todo = __ballot_sync(kFull, in);
                }
            }
            continue;
        }
        if (nstack == 0) break;
        // (as pool_search)
        const int take = min(min(32, nstack), max(1, kStack - kMaxTreeDepth - nstack));
        uint2 e = make_uint2(0u, 0u);
        if (lane < take) e = W.stack[nstack - 1 - lane];
        nstack -= take;
        __syncwarp();
        const int slot = pool_slot(e);
        const float thr = W.thr[slot];
        const bool act = lane < take && pool_dist(e) <= thr;
        const float3 p = xyz(W.q[slot]);
        int cn = 0, cf = 0, ll = 0, lr = 0, nl = 0, nr = 0;
        float dn = 0.0f, df = 0.0f, dl = 0.0f, dr = 0.0f;
        bool pn = false, pf = false, tl = false, tr = false;
        if (act) {
            const float4 *r = T.nodes + 4 * (size_t)pool_id(e);
            const float4 l0 = ldg4(r), l1 = ldg4(r + 1), r0 = ldg4(r + 2), r1 = ldg4(r + 3);
            dl = box_d2(p, l0, l1);
            dr = box_d2(p, r0, r1);
            const int cl = __float_as_int(l0.w), cr = __float_as_int(r0.w);
            const bool il = dl <= thr, ir = dr <= thr, gl = il && cl >= 0, gr = ir && cr >= 0;
            tl = il && cl < 0;
            tr = ir && cr < 0;
            ll = -cl - 1;
            lr = -cr - 1;
            if constexpr (kRange) { nl = __float_as_int(l1.w) - 1; nr = __float_as_int(r1.w) - 1; }
            const bool left = gl && (!gr || dl <= dr);
            pn = gl || gr;
            pf = gl && gr;
            cn = left ? cl : cr;
            dn = left ? dl : dr;
            cf = left ? cr : cl;
            df = left ? dr : dl;
        }
        const unsigned int bf = __ballot_sync(kFull, pf), bn = __ballot_sync(kFull, pn);
        const unsigned int bl = __ballot_sync(kFull, tl), br = __ballot_sync(kFull, tr);
        const int nf = __popc(bf), lf = __popc(bl);
        if (pf) W.stack[nstack + __popc(bf & lt)] = pool_entry(cf, slot, 0, df);
        if (pn) W.stack[nstack + nf + __popc(bn & lt)] = pool_entry(cn, slot, 0, dn);
        if (tl) W.leaf[nleaf + __popc(bl & lt)] = pool_entry(ll, slot, nl, dl);
        if (tr) W.leaf[nleaf + lf + __popc(br & lt)] = pool_entry(lr, slot, nr, dr);
        nstack += nf + __popc(bn);
        nleaf += lf + __popc(br);
        __syncwarp();
    }
    // the blend: lane 8 s + j takes face j of query s, and lane 8 s sums them nearest first
    const float4 rlo = hdr->root_lo, rhi = hdr->root_hi;
    const float dx = rhi.x - rlo.x, dy = rhi.y - rlo.y, dz = rhi.z - rlo.z;
    const float delta = 1e-6f * sqrtf(dx * dx + dy * dy + dz * dz);
    for (int b0 = 0; b0 < S; b0 += 4) {
        const int sl = b0 + lane / 8, j = lane % 8;
        const bool on = sl < own && j < k;
        float wt = 0.0f, px = 0.0f, py = 0.0f, pz = 0.0f;
        if (on) {
            const int64_t i = i0 + sl;
            const int leaf = W.pos[sl][j];
            const float d2 = W.d2[sl][j];
            if (leaf >= 0) {
                const float4 *t = T.tris + 3 * (size_t)leaf;
                const float4 a = ldg4(t), b = ldg4(t + 1), c = ldg4(t + 2);
                float u, v, w;
                tri_closest(xyz(W.q[sl]), xyz(a), xyz(b), xyz(c), b.w != 0.0f, u, v, w);
                wt = 1.0f / fmaxf(sqrtf(d2), delta);
                px = u * a.x + v * b.x + w * c.x;
                py = u * a.y + v * b.y + w * c.y;
                pz = u * a.z + v * b.z + w * c.z;
            }
            if (face_out) face_out[i * k + j] = leaf >= 0 ? W.face[sl][j] : -1;
            if (d2_out) d2_out[i * k + j] = leaf >= 0 ? d2 : INFINITY;
        }
        float sw = 0.0f, ax = 0.0f, ay = 0.0f, az = 0.0f;
#pragma unroll
        for (int m = 0; m < kKnnMax; ++m) {
            const int src = (lane & ~7) + m;
            const float wm = __shfl_sync(kFull, wt, src), xm = __shfl_sync(kFull, px, src),
                        ym = __shfl_sync(kFull, py, src), zm = __shfl_sync(kFull, pz, src);
            sw += wm;
            ax += wm * xm;
            ay += wm * ym;
            az += wm * zm;
        }
        if (sl < own && j == 0) {
            const int64_t i = i0 + sl;
            const float4 qs = W.q[sl];
            float ox = qs.x, oy = qs.y, oz = qs.z;
            if (W.pos[sl][0] >= 0) { ox = ax / sw; oy = ay / sw; oz = az / sw; }
            if (anchor) {
                ox = (1.0f - anchor_w) * ox + anchor_w * anchor[3 * i];
                oy = (1.0f - anchor_w) * oy + anchor_w * anchor[3 * i + 1];
                oz = (1.0f - anchor_w) * oz + anchor_w * anchor[3 * i + 2];
            }
            point[3 * i] = ox;
            point[3 * i + 1] = oy;
            point[3 * i + 2] = oz;
        }
    }
}

// Meshes of few faces (see few_search): a thread per query tests every face, its
// sorted list in shared memory, and blends as above.
__global__ void __launch_bounds__(kFewThreads)
k_few_knn(Traversal T, const Header *__restrict__ hdr, const float *Q, int64_t nQ, int k, const float *anchor,
          float anchor_w, float *point, int *face_out, float *d2_out) {
    __shared__ float s_d2[kKnnMax][kFewThreads];
    __shared__ int s_face[kKnnMax][kFewThreads], s_pos[kKnnMax][kFewThreads];
    const int t = threadIdx.x;
    const int64_t i = (int64_t)blockIdx.x * kFewThreads + t;
    if (i >= nQ) return;
    const float3 q = make_float3(Q[3 * i], Q[3 * i + 1], Q[3 * i + 2]);   // may alias point
    int n = 0;                                           // listed
    for (int leaf = 0; leaf < T.n; ++leaf) {
        const float4 *tr = T.tris + 3 * (size_t)leaf;
        const float4 a = ldg4(tr), b = ldg4(tr + 1), c = ldg4(tr + 2);
        const float d2 = tri_distance2(q, xyz(a), xyz(b), xyz(c), b.w != 0.0f);
        const int f = __float_as_int(a.w);
        auto before = [&](int j) { return d2 < s_d2[j][t] || (d2 == s_d2[j][t] && f < s_face[j][t]); };
        if (!(n < k ? d2 <= INFINITY : before(k - 1))) continue;
        int j = n < k ? n++ : k - 1;
        for (; j > 0 && before(j - 1); --j) {
            s_d2[j][t] = s_d2[j - 1][t];
            s_face[j][t] = s_face[j - 1][t];
            s_pos[j][t] = s_pos[j - 1][t];
        }
        s_d2[j][t] = d2;
        s_face[j][t] = f;
        s_pos[j][t] = leaf;
    }
    const float4 rlo = hdr->root_lo, rhi = hdr->root_hi;
    const float dx = rhi.x - rlo.x, dy = rhi.y - rlo.y, dz = rhi.z - rlo.z;
    const float delta = 1e-6f * sqrtf(dx * dx + dy * dy + dz * dz);
    float sw = 0.0f, ax = 0.0f, ay = 0.0f, az = 0.0f;
    for (int j = 0; j < k; ++j) {
        const bool on = j < n;
        if (on) {
            const float4 *tr = T.tris + 3 * (size_t)s_pos[j][t];
            const float4 a = ldg4(tr), b = ldg4(tr + 1), c = ldg4(tr + 2);
            float u, v, w;
            tri_closest(q, xyz(a), xyz(b), xyz(c), b.w != 0.0f, u, v, w);
            const float wt = 1.0f / fmaxf(sqrtf(s_d2[j][t]), delta);
            sw += wt;
            ax += wt * (u * a.x + v * b.x + w * c.x);
            ay += wt * (u * a.y + v * b.y + w * c.y);
            az += wt * (u * a.z + v * b.z + w * c.z);
        }
        if (face_out) face_out[i * k + j] = on ? s_face[j][t] : -1;
        if (d2_out) d2_out[i * k + j] = on ? s_d2[j][t] : INFINITY;
    }
    float ox = q.x, oy = q.y, oz = q.z;
    if (n > 0) { ox = ax / sw; oy = ay / sw; oz = az / sw; }
    if (anchor) {
        ox = (1.0f - anchor_w) * ox + anchor_w * anchor[3 * i];
        oy = (1.0f - anchor_w) * oy + anchor_w * anchor[3 * i + 1];
        oz = (1.0f - anchor_w) * oz + anchor_w * anchor[3 * i + 2];
    }
    point[3 * i] = ox;
    point[3 * i + 1] = oy;
    point[3 * i + 2] = oz;
}

// Calls f with S = 32 / G as a compile-time constant (G of 2 or more).
template <typename F> static void pool_dispatch(int G, F f) {
    switch (G) {
        case 2: f(std::integral_constant<int, 16>()); break;
        case 4: f(std::integral_constant<int, 8>()); break;
        case 8: f(std::integral_constant<int, 4>()); break;
        case 16: f(std::integral_constant<int, 2>()); break;
        default: f(std::integral_constant<int, 1>()); break;
    }
}

void pool_closest_point(const mesh_bvh *b, Traversal T, const float *Q, int64_t nQ, float maxd2, int G, int *face,
                        float *bary, float *point, float *dist2, const int *hint, cudaStream_t s) {
    Header *h = b->hdr();
    count_launch();
    if (G == 0) {
        k_few_closest_point<<<grid_for(nQ, kFewThreads), kFewThreads, 0, s>>>(T, h, &h->status, Q, nQ, maxd2, face, bary,
                                                                              point, dist2);
        return;
    }
    pool_dispatch(G, [&](auto S) {
        auto kern = b->leaf_size > 1 ? k_pool_closest_point<S.value, true> : k_pool_closest_point<S.value, false>;
        kern<<<grid_for(nQ, kQueryWarps * S.value), 32 * kQueryWarps, 0, s>>>(T, h, &h->status, Q, nQ, maxd2, face, bary,
                                                                       point, dist2, hint, b->iperm());
    });
}

void pool_signed(const mesh_bvh *b, Traversal T, const float *Q, int64_t nQ, float maxd2, int G, int *face, float *bary,
                 float *point, float *sdist, cudaStream_t s) {
    Header *h = b->hdr();
    count_launch();
    if (G == 0) {
        k_few_signed<<<grid_for(nQ, kFewThreads), kFewThreads, 0, s>>>(T, h, &h->status, Q, nQ, maxd2, b->faces(), b->adj(),
                                                                       b->fnorm(), b->verts(), face, bary, point, sdist);
        return;
    }
    pool_dispatch(G, [&](auto S) {
        auto kern = b->leaf_size > 1 ? k_pool_signed<S.value, true> : k_pool_signed<S.value, false>;
        kern<<<grid_for(nQ, kQueryWarps * S.value), 32 * kQueryWarps, 0, s>>>(T, h, &h->status, Q, nQ, maxd2, b->faces(),
                                                                       b->adj(), b->fnorm(), b->verts(), face, bary,
                                                                       point, sdist);
    });
}

void pool_knn(const mesh_bvh *b, Traversal T, const float *Q, int64_t nQ, int k, int G, const float *anchor,
              float anchor_w, float *point, int *face, float *d2, cudaStream_t s) {
    auto go = [&](auto S) {
        auto kern = b->leaf_size > 1 ? k_pool_knn<S.value, true> : k_pool_knn<S.value, false>;
        kern<<<grid_for(nQ, S.value), 32, 0, s>>>(T, b->hdr(), Q, nQ, k, anchor, anchor_w, point, face, d2);
    };
    if (G == 0)
        k_few_knn<<<grid_for(nQ, kFewThreads), kFewThreads, 0, s>>>(T, b->hdr(), Q, nQ, k, anchor, anchor_w, point, face, d2);
    else if (G <= 4) go(std::integral_constant<int, 8>());
    else if (G == 8) go(std::integral_constant<int, 4>());
    else if (G == 16) go(std::integral_constant<int, 2>());
    else go(std::integral_constant<int, 1>());
    count_launch();
}

void pool_chamfer(int G, bool range, const ChamferSide &a2b, const ChamferSide &b2a, unsigned nbA, unsigned grid,
                  unsigned *status, double *partial, unsigned *ticket, double *out, cudaStream_t s) {
    auto go = [&](auto S) {
        auto kern = range ? k_pool_chamfer<S.value, true> : k_pool_chamfer<S.value, false>;
        kern<<<grid, 32 * kChamferWarps, 0, s>>>(a2b, b2a, nbA, status, partial, ticket, out);
    };
    count_launch();
    if (G == 0) k_pool_chamfer<0, false><<<grid, 32 * kChamferWarps, 0, s>>>(a2b, b2a, nbA, status, partial, ticket, out);
    else if (G == 1) go(std::integral_constant<int, 32>());   // mesh_chamfer_noalloc's largest calls
    else pool_dispatch(G, go);
}

void pool_batch(const mesh_batch *b, const float *Q, const int *query_off, int64_t nQ, float maxd2, bool mmd, int G,
                int *face, float *bary, float *point, float *dist2, cudaStream_t s) {
    count_launch();
    auto go = [&](auto kern, int queries) {
        kern<<<grid_for(nQ, queries), 32, 0, s>>>(b->nodes(), b->tris(), b->scene_box(), b->face_off(), query_off,
                                                  (int)b->L.n_scenes, Q, nQ, maxd2, mmd, face, bary, point, dist2,
                                                  &b->st()->status);
    };
    if (G == 0) go(k_few_batch, 32);
    else pool_dispatch(G, [&](auto S) { go(k_pool_batch<S.value>, S.value); });
}

}  // namespace meshgs
