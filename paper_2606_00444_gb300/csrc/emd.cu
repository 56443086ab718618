// Earth Mover's Distance between two equal-size point sets (the EMD of
// Sec. 4.2, on 10K points sampled from each mesh): the minimum over bijections
// of the mean Euclidean distance, by Bertsekas's auction algorithm with
// epsilon scaling (Jacobi form: every unassigned point bids at once).  Each
// phase ends with every point assigned and prices epsilon-complementary, so
// the final assignment costs at most n * eps_final more than the optimum: the
// mean is within eps_final of the exact EMD.
//
// Bid kernel without lists (more than kTailMaxN points): one warp per unassigned point of A; the points of B and their
// prices are streamed through shared memory in tiles; each lane keeps the best
// and second-best value (-distance - price) and the warp merges them; the bid
// (price + best - second + eps) goes to the object with a 64-bit atomic max of
// (bid bits, bidder) -- bids are positive floats, so their bits order like
// the values, and equal bids resolve to the higher bidder id.  Resolve kernel:
// one thread per object with a bid moves the object to the winner and frees
// its previous owner.  The host runs the iterations, reading the count of
// unassigned points every 16 iterations; the call returns when done.
#include <math.h>

#include <cstring>
#include <type_traits>

#include "common.cuh"

namespace meshgs {

constexpr int kEmdBlock = 256;
constexpr int kEmdWarps = kEmdBlock / 32;
constexpr int kEmdTile = 1024;
constexpr int kEmdCheck = 16;

__device__ __forceinline__ unsigned f2ord_emd(float f) {
    unsigned u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float ord2f_emd(unsigned u) {
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

__global__ void k_emd_init(const float *__restrict__ A, const float *__restrict__ B, int n, float4 *A4,
                           float4 *B4, float *price, int *owner, int *assign, unsigned long long *bids,
                           unsigned *box) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float4 a = make_float4(A[3 * i], A[3 * i + 1], A[3 * i + 2], 0.0f);
    float4 b = make_float4(B[3 * i], B[3 * i + 1], B[3 * i + 2], 0.0f);
    A4[i] = a;
    B4[i] = b;
    price[i] = 0.0f;
    owner[i] = -1;
    assign[i] = -1;
    bids[i] = 0ull;
    atomicMin(&box[0], f2ord_emd(fminf(a.x, b.x)));
    atomicMin(&box[1], f2ord_emd(fminf(a.y, b.y)));
    atomicMin(&box[2], f2ord_emd(fminf(a.z, b.z)));
    atomicMax(&box[3], f2ord_emd(fmaxf(a.x, b.x)));
    atomicMax(&box[4], f2ord_emd(fmaxf(a.y, b.y)));
    atomicMax(&box[5], f2ord_emd(fmaxf(a.z, b.z)));
}

__global__ void k_emd_unassign(int n, int *owner, int *assign) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    owner[i] = -1;
    assign[i] = -1;
}

// Squared distance of a point and an object: the one expression every path values with,
// its roundings written out -- a list's entry and a scan's value of the same object are
// compiled in different kernels and must be the same float.
__device__ __forceinline__ float emd_d2(float4 a, float bx, float by, float bz) {
    const float dx = a.x - bx, dy = a.y - by, dz = a.z - bz;
    return __fmaf_rn(dz, dz, __fmaf_rn(dx, dx, __fmul_rn(dy, dy)));
}

// (best, second best) of a lane merged with another lane's
__device__ __forceinline__ void merge2(float &b1, int &j1, float &b2, float o1, int oj, float o2) {
    if (o1 > b1 || (o1 == b1 && oj < j1)) {
        b2 = fmaxf(b1, o2);
        b1 = o1;
        j1 = oj;
    } else {
        b2 = fmaxf(b2, o1);
    }
}

__global__ void __launch_bounds__(kEmdBlock)
k_emd_bid(int n, const float4 *__restrict__ A4, const float4 *__restrict__ B4, const float *__restrict__ price,
          const int *__restrict__ assign, unsigned long long *bids, float eps, unsigned *active) {
    __shared__ float4 sb[kEmdTile];
    __shared__ float sp[kEmdTile];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int i = blockIdx.x * kEmdWarps + wid;
    const bool mine = i < n && assign[i] < 0;
    if (!__syncthreads_or(mine)) return;
    float4 a = mine ? A4[i] : make_float4(0.f, 0.f, 0.f, 0.f);
    float b1 = -INFINITY, b2 = -INFINITY;
    int j1 = 0x7fffffff;
    for (int t0 = 0; t0 < n; t0 += kEmdTile) {
        int m = min(kEmdTile, n - t0);
        for (int t = threadIdx.x; t < m; t += kEmdBlock) {
            sb[t] = B4[t0 + t];
            sp[t] = price[t0 + t];
        }
        __syncthreads();
        if (mine) {
            for (int t = lane; t < m; t += 32) {
                const float4 b = sb[t];
                merge2(b1, j1, b2, -sqrtf(emd_d2(a, b.x, b.y, b.z)) - sp[t], t0 + t, -INFINITY);
            }
        }
        __syncthreads();
    }
    if (!mine) return;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        float o1 = __shfl_xor_sync(0xffffffffu, b1, o), o2 = __shfl_xor_sync(0xffffffffu, b2, o);
        int oj = __shfl_xor_sync(0xffffffffu, j1, o);
        merge2(b1, j1, b2, o1, oj, o2);
    }
    if (lane == 0) {
        atomicAdd(active, 1u);
        if ((unsigned)j1 >= (unsigned)n) return;     // no comparable value (NaN input): no bid
        float inc = (b2 == -INFINITY ? 0.0f : b1 - b2) + eps;
        float bid = price[j1] + inc;
        atomicMax(&bids[j1], ((unsigned long long)__float_as_uint(bid) << 32) | (unsigned)i);
    }
}

__global__ void k_emd_resolve(int n, float *price, int *owner, int *assign, unsigned long long *bids) {
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    unsigned long long b = bids[j];
    if (b == 0ull) return;
    bids[j] = 0ull;
    int winner = (int)(b & 0xffffffffull);
    int old = owner[j];
    if (old >= 0) assign[old] = -1;
    owner[j] = winner;
    assign[winner] = j;
    price[j] = __uint_as_float((unsigned)(b >> 32));
}

// ---------------------------------------------------------------------------
// Candidate lists.  A point's bid needs its best and second-best value over
// all n objects, but prices only rise within a call, so values only fall: a
// list of the objects whose value exceeded a threshold T when it was made, with
// their distances, still holds the best two as long as the best listed value
// is above T and the second is not below it (everything outside is at most T).
// Such a bid reads kListMax entries instead of n objects.  The threshold is the
// second-best value at that time less a margin, scaled per point by the count it
// gave so that about 160 objects qualify.  A list that no longer decides is made
// again by a scan of all objects, which also gives the bid.
//
// A list pays when it outlives a few bids -- fewer the more objects a scan reads --
// and every bid raises a price by at least eps: where the margin that holds 160 objects
// is below list_margin (the coarse phases; many points in one place, of which no
// margin is small enough), a point makes none and bids by one exact scan.  Lists everywhere, with the margin changed by a quarter
// at a time, cost up to 6 times the scans alone (10k points in one place 17.9 s against
// 3.1, 2.6 so; 10k points of a plane and of a cube, eps 1e-2, 106 ms against 60, 53 so).
// Either way the bid is the one a full scan gives, bit for bit: the same
// distances, the same subtraction, ties to the lowest object id.
// ---------------------------------------------------------------------------
constexpr int kListMax = 256;                        // entries; eight per lane
constexpr int kListLow = 120, kListHigh = 208;       // entries aimed for
constexpr float kListAim = 160.0f;

// Least margin of a list at a phase's eps.  Multiples of 2, 3, 4 and 6 eps were timed at 1000
// to 10000 points on surfaces, volumes and clusters: 10000 points in a cube, eps 1e-2, take
// 75, 120, 123 and 123 ms (scans 115); 5000 of a 3-D normal and its image 1.25 apart 58,
// 56, 55, 56 (scans 50); 5000 in a cube 40, 40, 59, 64 (56); 3000 in a cube 19, 19, 19, 28
// (24).  Below 3333 points 4, at 10000 2.
inline float list_margin(int n, double eps) { return (float)(eps * fmin(4.0, 1.0 + 1e4 / (double)n)); }

struct EmdLists {
    int4 *entry;       // [n][kListMax / 2], two (object, distance bits) pairs each
    float2 *hdr;       // [n] (threshold, margin); threshold +inf: no list yet
};

__device__ __forceinline__ float warp_max(float v) { return ord2f_emd(__reduce_max_sync(0xffffffffu, f2ord_emd(v))); }

// Best (lowest object on ties) and second-best value of a warp from its lanes'.
__device__ __forceinline__ void warp_best2(float &b1, int &j1, float &b2) {
    const unsigned full = 0xffffffffu;
    const float m = warp_max(b1);
    const int j = (int)__reduce_min_sync(full, b1 == m ? (unsigned)j1 : 0x7fffffffu);
    const bool owner = b1 == m && j1 == j;
    b2 = warp_max(owner ? b2 : b1);
    b1 = m;
    j1 = j;
}

// The best two of a point from its list (e: this lane's eight entries) at the
// current prices.
template <typename Price>
__device__ __forceinline__ void list_best2(const int4 (&e)[4], Price price, float &b1, int &j1, float &b2) {
    b1 = b2 = -INFINITY;
    j1 = 0x7fffffff;
    auto take = [&](int j, int dbits) {
        const float v = -__int_as_float(dbits) - price(j);
        const bool better = v > b1 || (v == b1 && j < j1);
        b2 = fmaxf(b2, better ? b1 : v);
        if (better) { b1 = v; j1 = j; }
    };
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        take(e[m].x, e[m].y);
        take(e[m].z, e[m].w);
    }
    warp_best2(b1, j1, b2);
}

__device__ __forceinline__ void list_load(const EmdLists &L, int i, int lane, int4 (&e)[4]) {
    const int4 *p = L.entry + (size_t)i * (kListMax / 2) + lane;
#pragma unroll
    for (int m = 0; m < 4; ++m) e[m] = p[32 * m];
}

// An object belongs on the list of threshold T when its value exceeds T; tested
// on the squared distance (no square root) and widened for rounding, so none
// is missed -- an extra entry does no harm.
__device__ __forceinline__ bool list_qualifies(float d2, float price, float T) {
    const float r = (-T - price) + 2e-6f * (fabsf(T) + fabsf(price));
    return r > 0.0f && d2 <= r * r * 1.000002f;
}

// Lists an object and takes it into the (best, second best) values met.  The two best of
// all objects qualify, so a list's scan gives the bid.
__device__ __forceinline__ void list_append(const EmdLists &L, int i, int *cnt, int j, float d2, float price, float &b1,
                                            int &j1, float &b2) {
    const int pos = atomicAdd(cnt, 1);
    const float d = sqrtf(d2);
    if (pos < kListMax) reinterpret_cast<int2 *>(L.entry)[(size_t)i * kListMax + pos] = make_int2(j, __float_as_int(d));
    merge2(b1, j1, b2, -d - price, j, -INFINITY);
}

// Closes a list of cnt entries: the rest padded with entries of value -inf
// (thread t of nt), threshold and next margin by thread 0.
__device__ __forceinline__ void list_close(const EmdLists &L, int i, int cnt, int n, float T, float margin, int t,
                                           int nt) {
    for (int k = cnt + t; k < kListMax; k += nt)
        reinterpret_cast<int2 *>(L.entry)[(size_t)i * kListMax + k] = make_int2(0, 0x7f800000);
    if (t != 0) return;
    if (cnt < n && (cnt < kListLow || cnt > kListHigh))              // about r^2 objects within r
        margin *= fminf(4.0f, fmaxf(0.25f, sqrtf(kListAim / fmaxf((float)cnt, 1.0f))));
    else if (cnt > kListMax)                                         // (and every object)
        margin *= 0.25f;
    if (cnt > kListMax) T = INFINITY;                                // too many: no list
    else if (cnt == n) T = -INFINITY;                                // every object is listed
    L.hdr[i] = make_float2(T, margin);
}

// Value of an object to within about 1e-6 of its distance, for choosing a
// threshold: one reciprocal-root instruction instead of a rounded square root.
__device__ __forceinline__ float value_approx(float d2, float price) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(fmaxf(d2, 1e-30f)));
    return -(d2 * r) - price;
}

__global__ void k_emd_lists_init(int n, EmdLists L, float margin) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) L.hdr[i] = make_float2(INFINITY, margin);
}

// One round of bids with lists (n <= kTailMaxN): one warp per unassigned point
// reads its list; the block then scans the objects for the points whose lists
// did not decide: two at a time those that get a new list, up to four at a time
// those that make none.  B4 holds the prices in w.
__global__ void __launch_bounds__(kEmdBlock)
k_emd_bid_lists(int n, const float4 *__restrict__ A4, const float4 *__restrict__ B4, const int *__restrict__ assign,
                unsigned long long *bids, EmdLists L, float eps, float least, unsigned *active) {
    __shared__ int s_list[kEmdWarps], s_lists, s_scan[kEmdWarps], s_scans;
    __shared__ float s_b1[4][kEmdWarps], s_b2[4][kEmdWarps];
    __shared__ int s_j[4][kEmdWarps], s_cnt[2];
    pdl_wait();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (threadIdx.x == 0) { s_lists = 0; s_scans = 0; }
    __syncthreads();
    auto price = [&](int j) { return __ldcg(&B4[j].w); };
    auto place = [&](int i, float b1, int j1, float b2) {
        if (lane != 0) return;
        atomicAdd(active, 1u);
        if ((unsigned)j1 >= (unsigned)n) return;      // no comparable value (NaN input): unassigned, no bid
        const float inc = (b2 == -INFINITY ? 0.0f : b1 - b2) + eps;
        const float bid = price(j1) + inc;
        atomicMax(&bids[j1], ((unsigned long long)__float_as_uint(bid) << 32) | (unsigned)i);
    };
    // true when point i bid from its list
    auto bid_from_list = [&](int i) {
        const float T = L.hdr[i].x;
        if (T == INFINITY) return false;
        int4 e[4];
        list_load(L, i, lane, e);
        float b1, b2;
        int j1;
        list_best2(e, price, b1, j1, b2);
        if (!(b1 > T && b2 >= T)) return false;
        place(i, b1, j1, b2);
        return true;
    };
    {
        const int i = blockIdx.x * kEmdWarps + wid;
        if (i < n && assign[i] < 0 && !bid_from_list(i) && lane == 0) {
            if (L.hdr[i].y >= least) s_list[atomicAdd(&s_lists, 1)] = i;
            else s_scan[atomicAdd(&s_scans, 1)] = i;
        }
    }
    __syncthreads();
    const int lists = s_lists, scans = s_scans;
    // the block's best two values of K points, from its threads'
    auto block_best2 = [&](auto K, float *b1, int *j1, float *b2) {
#pragma unroll
        for (int k = 0; k < K.value; ++k) {
            warp_best2(b1[k], j1[k], b2[k]);
            if (lane == 0) { s_b1[k][wid] = b1[k]; s_b2[k][wid] = b2[k]; s_j[k][wid] = j1[k]; }
        }
        __syncthreads();
    };
    auto of_block = [&](int k, float &b1, int &j1, float &b2) {
        b1 = lane < kEmdWarps ? s_b1[k][lane] : -INFINITY;
        b2 = lane < kEmdWarps ? s_b2[k][lane] : -INFINITY;
        j1 = lane < kEmdWarps ? s_j[k][lane] : 0x7fffffff;
        warp_best2(b1, j1, b2);
    };
    // exact scans for K points of s_scan
    auto scan = [&](auto K, int m0) {
        float4 a[K.value];
        float b1[K.value], b2[K.value];
        int j1[K.value];
#pragma unroll
        for (int k = 0; k < K.value; ++k) {
            a[k] = A4[s_scan[min(m0 + k, scans - 1)]];
            b1[k] = b2[k] = -INFINITY;
            j1[k] = 0x7fffffff;
        }
        for (int j = threadIdx.x; j < n; j += kEmdBlock) {
            const float4 b = __ldcg(&B4[j]);
#pragma unroll
            for (int k = 0; k < K.value; ++k)
                merge2(b1[k], j1[k], b2[k], -sqrtf(emd_d2(a[k], b.x, b.y, b.z)) - b.w, j, -INFINITY);
        }
        block_best2(K, b1, j1, b2);
        if (wid < K.value && m0 + wid < scans) {
            of_block(wid, b1[0], j1[0], b2[0]);
            place(s_scan[m0 + wid], b1[0], j1[0], b2[0]);
        }
        __syncthreads();
    };
    for (int m0 = 0; m0 < scans; m0 += 4) {
        if (scans - m0 > 2) scan(std::integral_constant<int, 4>(), m0);
        else if (scans - m0 == 2) scan(std::integral_constant<int, 2>(), m0);
        else scan(std::integral_constant<int, 1>(), m0);
    }
    for (int m0 = 0; m0 < lists; m0 += 2) {
        const std::integral_constant<int, 2> two;
        const int cnt = min(2, lists - m0);
        const int pt[2] = {s_list[m0], s_list[m0 + cnt - 1]};
        const float4 a[2] = {A4[pt[0]], A4[pt[1]]};
        const float margin[2] = {L.hdr[pt[0]].y, L.hdr[pt[1]].y};
        float b1[2] = {-INFINITY, -INFINITY}, b2[2] = {-INFINITY, -INFINITY};
        int j1[2] = {lane, lane};                     // (which object does not matter here)
        for (int j = threadIdx.x; j < n; j += kEmdBlock) {
            const float4 b = __ldcg(&B4[j]);
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const float v = value_approx(emd_d2(a[k], b.x, b.y, b.z), b.w);
                b2[k] = fmaxf(b2[k], fminf(b1[k], v));
                b1[k] = fmaxf(b1[k], v);
            }
        }
        if (threadIdx.x < 2) s_cnt[threadIdx.x] = 0;
        block_best2(two, b1, j1, b2);
        float T[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            float c1 = lane < kEmdWarps ? s_b1[k][lane] : -INFINITY, c2 = lane < kEmdWarps ? s_b2[k][lane] : -INFINITY;
            int dummy = lane;
            warp_best2(c1, dummy, c2);
            T[k] = c2 - margin[k];
            b1[k] = b2[k] = -INFINITY;
            j1[k] = 0x7fffffff;
        }
        for (int j = threadIdx.x; j < n; j += kEmdBlock) {
            const float4 b = __ldcg(&B4[j]);
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                if (k >= cnt) break;
                const float d2 = emd_d2(a[k], b.x, b.y, b.z);
                if (list_qualifies(d2, b.w, T[k])) list_append(L, pt[k], &s_cnt[k], j, d2, b.w, b1[k], j1[k], b2[k]);
            }
        }
        __syncthreads();                              // the counts, and the thresholds' values are read
#pragma unroll
        for (int k = 0; k < 2; ++k)
            if (k < cnt) list_close(L, pt[k], s_cnt[k], n, T[k], margin[k], threadIdx.x, kEmdBlock);
        block_best2(two, b1, j1, b2);
        if (wid < cnt) {
            const int i = pt[wid];
            float c1, c2;
            int jb;
            of_block(wid, c1, jb, c2);
            if (!(c1 > T[wid] && c2 >= T[wid])) {     // (rounding of the threshold) exact scan by the warp
                c1 = c2 = -INFINITY;
                jb = 0x7fffffff;
                for (int j = lane; j < n; j += 32) {
                    const float4 b = __ldcg(&B4[j]);
                    merge2(c1, jb, c2, -sqrtf(emd_d2(a[wid], b.x, b.y, b.z)) - b.w, j, -INFINITY);
                }
                warp_best2(c1, jb, c2);
            }
            place(i, c1, jb, c2);
        }
        __syncthreads();
    }
}

__global__ void k_emd_resolve_lists(int n, float4 *__restrict__ B4, int *owner, int *assign,
                                    unsigned long long *bids) {
    pdl_wait();
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    unsigned long long b = bids[j];
    if (b == 0ull) return;
    bids[j] = 0ull;
    int winner = (int)(b & 0xffffffffull);
    int old = owner[j];
    if (old >= 0) assign[old] = -1;
    owner[j] = winner;
    assign[winner] = j;
    B4[j].w = __uint_as_float((unsigned)(b >> 32));
}

// Gauss-Seidel tail: once few points are unassigned, one block finishes the
// phase, one bid at a time: the unassigned points are queued in index order and
// an evicted owner joins the back of the queue.  At most max_bids bids;
// *active gets the points still queued.
//
// A call is a chain of ~270k dependent bids at 10k points, so the latency of one
// bid is the time.  A list's trip from L2 is most of a bid's (a block-wide scan
// of all objects for each bid took 2.0 us, a bid from its list 0.8), so the
// lists of the next kTailAhead queued points are read together, each by a warp,
// which leaves the lane-wise best 32 entries in shared memory with the value
// that everything left out stays below.  Warp 0 then commits those bids in
// queue order, each from its 32 entries at the prices of that moment (in shared
// memory, as are the owners), as long as they decide it: prices only rise, so
// what was left out stays below.  The head of the queue, with no bid since its
// list was read, bids from the whole list.  A point whose list no longer decides
// bids from a scan by all other warps, which hold the objects' coordinates in
// registers: one that makes a new list, for it and for the next point that needs
// one, or an exact scan for a point that makes none.
// 10k points, eps 1e-4: 259 ms with one list at a time, 178 ms so (531 with scans).
constexpr int kTailThreads = 768;                    // 80 registers each: 48 of coordinates
constexpr int kTailQueue = 256;
constexpr int kTailAhead = 16;
constexpr int kScanThreads = kTailThreads - 32;      // all but warp 0
constexpr int kScanPer = 16;                         // objects a scanning thread holds
constexpr int kTailMaxN = 11417;                     // largest n taken: every object in a scanning thread's registers
static_assert(kScanThreads * kScanPer >= kTailMaxN, "every object is held by a thread");
static_assert(kTailAhead < kTailThreads / 32, "a warp per list, beside warp 0");

enum { kTailDone = 0, kTailRead = 1, kTailList = 2, kTailExact = 3 };

__device__ __forceinline__ void bar_sync(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// What a warp leaves of a queued point's list: per lane its least cost (distance
// plus price; the value negated) entry, and the least cost not among them.
struct TailAhead {
    float d[kTailAhead][32];
    int j[kTailAhead][32];
    float rest[kTailAhead];            // -inf: the list does not decide; NaN: to be read again
    bool wants[kTailAhead];            // a new list pays (list_margin)
    float b1, b2;                      // the head's bid from its whole list
    int j1;
};

// Least and second-least cost of a warp's lanes (one entry each) and the lowest
// object at the least.  Costs are not negative, so their bits order like them.
__device__ __forceinline__ void least2(float c, int j, float &c1, int &j1, float &c2) {
    const unsigned full = 0xffffffffu, u = __float_as_uint(c);
    const unsigned m = __reduce_min_sync(full, u);
    j1 = (int)__reduce_min_sync(full, u == m ? (unsigned)j : 0x7fffffffu);
    c2 = __uint_as_float(__reduce_min_sync(full, u == m && j == j1 ? 0x7f800000u : u));
    c1 = __uint_as_float(m);
}

__global__ void __launch_bounds__(kTailThreads, 1)
k_emd_tail(int n, const float4 *__restrict__ A4, float4 *B4, float *price, int *owner, int *assign, EmdLists L,
           float eps, float least, int max_bids, unsigned *active) {
    extern __shared__ float sp[];                    // prices, then owners
    int *s_own = reinterpret_cast<int *>(sp + n);
    __shared__ TailAhead s_ahead;
    __shared__ int queue[kTailQueue];
    __shared__ float r1[2][32], r2[2][32];
    __shared__ int rj[32], s_wcnt[32];
    __shared__ int s_len, s_mode, s_head, s_point[2], s_cnt[2];
    __shared__ float s_T;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const bool lists = L.entry != nullptr;
    for (int j = tid; j < n; j += kTailThreads) { sp[j] = price ? price[j] : B4[j].w; s_own[j] = owner[j]; }
    if (tid == 0) s_len = 0;
    __syncthreads();
    // unassigned points in index order (up to the queue's size)
    for (int c0 = 0; c0 < n; c0 += kTailThreads) {
        int i = c0 + tid;
        bool un = i < n && assign[i] < 0;
        unsigned ball = __ballot_sync(0xffffffffu, un);
        if (lane == 0) s_wcnt[wid] = __popc(ball);
        __syncthreads();
        int before = s_len;
        for (int w = 0; w < wid; ++w) before += s_wcnt[w];
        int pos = before + __popc(ball & ((1u << lane) - 1u));
        if (un && pos < kTailQueue) queue[pos] = i;
        __syncthreads();
        if (tid == 0) {
            int tot = s_len;
            for (int w = 0; w < (kTailThreads >> 5); ++w) tot += s_wcnt[w];
            s_len = min(tot, kTailQueue);
        }
        __syncthreads();
    }
    if (wid == 0) {
        int head = 0, len = s_len, bids = 0;
        auto commit = [&](int i, float gap, int j1) {    // gap: best less second-best value
            const int old = s_own[j1];
            __syncwarp();
            if (lane == 0) {
                sp[j1] += gap + eps;
                s_own[j1] = i;
                assign[i] = j1;
                if (old >= 0) {
                    assign[old] = -1;
                    queue[(head + len) % kTailQueue] = old;
                }
            }
            ++head;
            ++bids;
            if (old < 0) --len;
            __syncwarp();
        };
        // hand a step to the other warps and wait for it
        auto step = [&](int mode) {
            if (lane == 0) { s_mode = mode; s_head = head; s_len = len; }
            bar_sync(1, kTailThreads);
            if (mode != kTailDone) bar_sync(1, kTailThreads);
        };
        // a scan's best two, from the other warps'
        auto scanned = [&](float &b1, int &j1, float &b2) {
            const bool in = lane > 0 && lane < kTailThreads / 32;
            b1 = in ? r1[0][lane] : -INFINITY;
            b2 = in ? r2[0][lane] : -INFINITY;
            j1 = in ? rj[lane] : 0x7fffffff;
            warp_best2(b1, j1, b2);
        };
        int ahead = 0, done = 0;                     // bids read ahead, and used
        while (bids < max_bids && len > 0) {
            bool list = false;
            if (lists) {
                if (done == ahead) {
                    step(kTailRead);
                    ahead = min(len, kTailAhead);
                    done = 0;
                    if (s_ahead.rest[0] >= 0.0f) {   // the head, from its whole list
                        const float b1 = s_ahead.b1, b2 = s_ahead.b2;
                        commit(queue[head % kTailQueue], b2 == -INFINITY ? 0.0f : b1 - b2, s_ahead.j1);
                        done = 1;
                        continue;
                    }
                }
                const int before = done;
                bool again = false;                  // an entry whose 32 costs do not decide
                float rest = s_ahead.rest[done];
                float d = s_ahead.d[done][lane];     // the next entries, one bid ahead of their use
                int j = s_ahead.j[done][lane];
                while (rest >= 0.0f && bids < max_bids) {
                    const float nd = d + sp[j];
                    const int i = queue[head % kTailQueue], nj = j;
                    const float limit = rest;
                    if (done + 1 < ahead) {
                        d = s_ahead.d[done + 1][lane];
                        j = s_ahead.j[done + 1][lane];
                        rest = s_ahead.rest[done + 1];
                    }
                    float c1, c2;
                    int j1;
                    least2(nd, nj, c1, j1, c2);
                    again = !(c1 < limit && c2 <= limit);
                    if (again) break;
                    commit(i, c2 == INFINITY ? 0.0f : c2 - c1, j1);
                    if (++done == ahead) break;
                }
                if (again || (done == before && done > 0 && !(rest < 0.0f))) {
                    ahead = done;                    // read its whole list, as the head's
                    continue;
                }
                if (done > before) continue;
                list = s_ahead.wants[done];
                const int q = lane < kTailAhead ? lane : 0;
                const unsigned need = __ballot_sync(0xffffffffu, list && lane > done && lane < ahead &&
                                                                     s_ahead.rest[q] < 0.0f && s_ahead.wants[q]);
                if (lane == 0) {
                    s_point[1] = -1;
                    if (need) {                      // the next that needs one: its list is read again
                        const int next = __ffs(need) - 1;
                        s_point[1] = queue[(head + next - done) % kTailQueue];
                        s_ahead.rest[next] = NAN;
                    }
                }
            }
            if (lane == 0) s_point[0] = queue[head % kTailQueue];
            float b1, b2;
            int j1;
            if (list) {
                step(kTailList);
                scanned(b1, j1, b2);
                list = b1 > s_T && b2 >= s_T;
            }
            if (!list) {
                step(kTailExact);
                scanned(b1, j1, b2);
            }
            if ((unsigned)j1 >= (unsigned)n) break;  // no comparable value (NaN input): leave the point queued
            commit(s_point[0], b2 == -INFINITY ? 0.0f : b1 - b2, j1);
            if (lists) ++done;
        }
        step(kTailDone);
        if (lane == 0) *active = (unsigned)len;
    } else {
        const int t = tid - 32;
        float bx[kScanPer], by[kScanPer], bz[kScanPer];
#pragma unroll
        for (int k = 0; k < kScanPer; ++k) {
            const int j = t + k * kScanThreads;
            const float4 b = j < n ? B4[j] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            bx[k] = b.x; by[k] = b.y; bz[k] = b.z;
        }
        // calls f for each object this thread holds; few slots for few objects (1000 points' call
        // from scans 15.7 ms with all 16, 11.2 so)
        auto objects = [&](auto f) {
            auto run = [&](auto slots) {
#pragma unroll
                for (int k = 0; k < slots.value; ++k) {
                    const int j = t + k * kScanThreads;
                    if (j < n) f(j, bx[k], by[k], bz[k]);
                }
            };
            if (n <= 2 * kScanThreads) run(std::integral_constant<int, 2>());
            else if (n <= 7 * kScanThreads) run(std::integral_constant<int, 7>());
            else run(std::integral_constant<int, kScanPer>());
        };
        while (true) {
            bar_sync(1, kTailThreads);
            const int mode = s_mode;
            if (mode == kTailDone) break;
            if (mode == kTailRead) {
                const int q = wid - 1;
                if (q < min(s_len, kTailAhead)) {
                    const int i = queue[(s_head + q) % kTailQueue];
                    const float2 hdr = L.hdr[i];
                    const float T = hdr.x;
                    if (lane == 0) s_ahead.wants[q] = hdr.y >= least;
                    int4 e[4];
                    list_load(L, i, lane, e);
                    if (T == INFINITY) {             // no list (its entries are not read)
                        s_ahead.d[q][lane] = INFINITY;
                        s_ahead.j[q][lane] = 0;
                        if (lane == 0) s_ahead.rest[q] = -INFINITY;
                    } else {
                        // this lane's least cost, its object, and its second-least
                        float c1 = INFINITY, c2 = INFINITY, d1 = INFINITY;
                        int j1 = 0;
                        auto take = [&](int j, int dbits) {
                            const float d = __int_as_float(dbits), c = d + sp[j];
                            const bool better = c < c1 || (c == c1 && j < j1);
                            c2 = fminf(c2, better ? c1 : c);
                            if (better) { c1 = c; d1 = d; j1 = j; }
                        };
#pragma unroll
                        for (int m = 0; m < 4; ++m) {
                            take(e[m].x, e[m].y);
                            take(e[m].z, e[m].w);
                        }
                        s_ahead.d[q][lane] = d1;
                        s_ahead.j[q][lane] = j1;
                        const float second = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(c2)));
                        float l1, l2;
                        int lj;
                        least2(c1, j1, l1, lj, l2);
                        l2 = fminf(l2, second);      // the list's second-least: another lane's best or some lane's second
                        if (lane == 0) {
                            const bool decides = l1 < -T && l2 <= -T;
                            s_ahead.rest[q] = decides ? fminf(second, -T) : -INFINITY;
                            if (q == 0) { s_ahead.b1 = -l1; s_ahead.b2 = -l2; s_ahead.j1 = lj; }
                        }
                    }
                }
                bar_sync(1, kTailThreads);
                continue;
            }
            if (mode == kTailExact) {
                const float4 a = A4[s_point[0]];
                float b1 = -INFINITY, b2 = -INFINITY;
                int j1 = 0x7fffffff;
                objects([&](int j, float x, float y, float z) {
                    merge2(b1, j1, b2, -sqrtf(emd_d2(a, x, y, z)) - sp[j], j, -INFINITY);
                });
                warp_best2(b1, j1, b2);
                if (lane == 0) { r1[0][wid] = b1; r2[0][wid] = b2; rj[wid] = j1; }
                bar_sync(1, kTailThreads);
                continue;
            }
            // new lists of one or two points
            const int i0 = s_point[0], i1 = s_point[1];
            const float4 a0 = A4[i0], a1 = A4[i1 >= 0 ? i1 : i0];
            const float margin0 = L.hdr[i0].y, margin1 = L.hdr[i1 >= 0 ? i1 : i0].y;
            if (t < 2) s_cnt[t] = 0;
            float b1 = -INFINITY, b2 = -INFINITY, e1 = -INFINITY, e2 = -INFINITY;
            objects([&](int j, float x, float y, float z) {
                const float p = sp[j];
                float v = value_approx(emd_d2(a0, x, y, z), p);
                b2 = fmaxf(b2, fminf(b1, v));
                b1 = fmaxf(b1, v);
                v = value_approx(emd_d2(a1, x, y, z), p);
                e2 = fmaxf(e2, fminf(e1, v));
                e1 = fmaxf(e1, v);
            });
            int dummy = lane;
            warp_best2(b1, dummy, b2);
            dummy = lane;
            warp_best2(e1, dummy, e2);
            if (lane == 0) { r1[0][wid] = b1; r2[0][wid] = b2; r1[1][wid] = e1; r2[1][wid] = e2; }
            bar_sync(2, kScanThreads);
            const bool in = lane > 0 && lane < kTailThreads / 32;
            b1 = in ? r1[0][lane] : -INFINITY;
            b2 = in ? r2[0][lane] : -INFINITY;
            e1 = in ? r1[1][lane] : -INFINITY;
            e2 = in ? r2[1][lane] : -INFINITY;
            dummy = lane;
            warp_best2(b1, dummy, b2);
            dummy = lane;
            warp_best2(e1, dummy, e2);
            const float T0 = b2 - margin0, T1 = e2 - margin1;
            b1 = b2 = e1 = e2 = -INFINITY;               // now of the objects listed
            int j1 = 0x7fffffff, e1j = 0x7fffffff;
            objects([&](int j, float x, float y, float z) {
                const float p = sp[j], d0 = emd_d2(a0, x, y, z);
                if (list_qualifies(d0, p, T0)) list_append(L, i0, &s_cnt[0], j, d0, p, b1, j1, b2);
                if (i1 >= 0) {
                    const float d1 = emd_d2(a1, x, y, z);
                    if (list_qualifies(d1, p, T1)) list_append(L, i1, &s_cnt[1], j, d1, p, e1, e1j, e2);
                }
            });
            bar_sync(2, kScanThreads);
            list_close(L, i0, s_cnt[0], n, T0, margin0, t, kScanThreads);
            if (i1 >= 0) list_close(L, i1, s_cnt[1], n, T1, margin1, t, kScanThreads);
            warp_best2(b1, j1, b2);
            if (lane == 0) { r1[0][wid] = b1; r2[0][wid] = b2; rj[wid] = j1; }
            if (t == 0) s_T = T0;
            bar_sync(1, kTailThreads);
        }
    }
    __syncthreads();
    for (int j = tid; j < n; j += kTailThreads) {
        if (price) price[j] = sp[j];
        else B4[j].w = sp[j];
        owner[j] = s_own[j];
    }
}

// Mean cost of the assignment in float64, summed in a fixed order.
__global__ void __launch_bounds__(kEmdBlock)
k_emd_cost(int n, const float4 *__restrict__ A4, const float4 *__restrict__ B4, const int *__restrict__ assign,
           int *out_assign, double *partial, unsigned *ticket, double *out) {
    __shared__ double red[kEmdWarps];
    __shared__ bool last;
    int i = blockIdx.x * kEmdBlock + threadIdx.x;
    double c = 0.0;
    if (i < n) {
        int j = assign[i];
        if (out_assign) out_assign[i] = j;
        float4 a = A4[i], b = B4[j];
        double dx = (double)a.x - b.x, dy = (double)a.y - b.y, dz = (double)a.z - b.z;
        c = sqrt(dx * dx + dy * dy + dz * dz);
    }
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < kEmdWarps; ++w) s += red[w];
        partial[blockIdx.x] = s;
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last || threadIdx.x != 0) return;
    __threadfence();
    double s = 0.0;
    for (unsigned k = 0; k < gridDim.x; ++k) s += __ldcg(partial + k);
    out[0] = s / (double)n;
    *ticket = 0u;
}

struct EmdWs {
    EmdLists L;
    size_t base_bytes;             // without the lists
    float4 *A4, *B4;
    float *price;
    int *owner, *assign;
    unsigned long long *bids;
    unsigned *box, *active, *ticket;
    double *partial;
    size_t bytes;
};

static EmdWs emd_ws(void *ws, int64_t n) {
    size_t off = 0;
    auto take = [&](size_t b) { size_t o = off; off = align_up(off + b, 256); return o; };
    int64_t m = n > 0 ? n : 1;
    size_t oA = take(16 * m), oB = take(16 * m), oP = take(4 * m), oO = take(4 * m), oS = take(4 * m),
           oBid = take(8 * m), oBox = take(64), oPart = take(8 * (size_t)((m + kEmdBlock - 1) / kEmdBlock));
    char *b = (char *)ws;
    EmdWs w;
    w.A4 = (float4 *)(b + oA);
    w.B4 = (float4 *)(b + oB);
    w.price = (float *)(b + oP);
    w.owner = (int *)(b + oO);
    w.assign = (int *)(b + oS);
    w.bids = (unsigned long long *)(b + oBid);
    w.box = (unsigned *)(b + oBox);
    w.active = w.box + 8;
    w.ticket = w.box + 9;
    w.partial = (double *)(b + oPart);
    w.base_bytes = off;
    w.L = EmdLists{nullptr, nullptr};
    if (n <= kTailMaxN) {
        size_t oE = take(8 * (size_t)kListMax * m), oH = take(8 * m);
        w.L = EmdLists{(int4 *)(b + oE), (float2 *)(b + oH)};
    }
    w.bytes = off;
    return w;
}

}  // namespace meshgs

using namespace meshgs;

extern "C" {

size_t mesh_emd_workspace_bytes(int64_t n) {
    if (n < 0 || n > ((int64_t)1 << 26)) return 0;
    // never less than for fewer points: past kTailMaxN a call takes no lists, but the same
    // workspace then serves smaller calls, with theirs
    const size_t own = emd_ws(nullptr, n).bytes, lists = n > kTailMaxN ? emd_ws(nullptr, kTailMaxN).bytes : 0;
    return own > lists ? own : lists;
}

mesh_status mesh_emd(const float *d_A, const float *d_B, int64_t n, float eps_rel, int64_t max_iters,
                     void *d_ws, size_t ws_bytes, double *d_out, int32_t *d_assign, int64_t *iters_out,
                     void *stream) {
    if (n < 0 || n > ((int64_t)1 << 26) || !d_out || (n > 0 && (!d_A || !d_B)) || !(eps_rel > 0.0f) ||
        max_iters < 1)
        return MESH_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    if (n == 0) {
        cudaMemsetAsync(d_out, 0, sizeof(double), s);
        if (iters_out) *iters_out = 0;
        return check_launch();
    }
    EmdWs w = emd_ws(d_ws, n);
    if (!d_ws || ws_bytes < w.base_bytes || ((uintptr_t)d_ws & 255u)) return MESH_ERR_WORKSPACE;
    // Lists where they fit: to kTailMaxN points (2 KB each; beyond that the tail, which
    // makes most bids, does not run), and not in a workspace without room for them.
    const bool lists = n <= kTailMaxN && ws_bytes >= w.bytes;
    if (!lists) w.L = EmdLists{nullptr, nullptr};
    const int N = (int)n;
    unsigned init_box[10] = {0xffffffffu, 0xffffffffu, 0xffffffffu, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
    if (cudaMemcpyAsync(w.box, init_box, sizeof(init_box), cudaMemcpyHostToDevice, s) != cudaSuccess)
        return MESH_ERR_CUDA;
    k_emd_init<<<grid_for(N, 256), 256, 0, s>>>(d_A, d_B, N, w.A4, w.B4, w.price, w.owner, w.assign, w.bids,
                                               w.box);
    count_launch();
    unsigned hb[6];
    if (cudaMemcpyAsync(hb, w.box, sizeof(hb), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return MESH_ERR_CUDA;
    auto dec = [](unsigned u) {
        unsigned b = (u & 0x80000000u) ? (u & 0x7fffffffu) : ~u;
        float f;
        memcpy(&f, &b, 4);
        return (double)f;
    };
    double dx = dec(hb[3]) - dec(hb[0]), dy = dec(hb[4]) - dec(hb[1]), dz = dec(hb[5]) - dec(hb[2]);
    double C = sqrt(dx * dx + dy * dy + dz * dz);
    if (!(C > 0.0)) C = 1.0;
    const double eps_final = eps_rel * C;
    const unsigned bid_grid = grid_for(N, kEmdWarps);
    static std::atomic<unsigned long long> tail_smem{0};
    if (!allow_smem(k_emd_tail, 8 * (size_t)kTailMaxN, tail_smem)) return MESH_ERR_CUDA;
    if (lists) {
        // a first guess of the margin: about 1 % of the box diagonal's objects at 10k points;
        // every object where a list holds them all (such a list decides every bid)
        const float margin = N <= kListMax ? 1e30f : (float)(0.25 * C * sqrt((double)kListAim / (double)N));
        k_emd_lists_init<<<grid_for(N, 256), 256, 0, s>>>(N, w.L, margin);
        count_launch();
    }
    int64_t iters = 0;
    for (double eps = C / 10.0;; eps /= 8.0) {
        if (eps < eps_final) eps = eps_final;
        k_emd_unassign<<<grid_for(N, 256), 256, 0, s>>>(N, w.owner, w.assign);
        count_launch();
        bool done = false;
        while (!done) {
            for (int k = 0; k < kEmdCheck; ++k) {
                // the count wanted is the last round's
                if (k == 0 || k == kEmdCheck - 1 || !lists) cudaMemsetAsync(w.active, 0, sizeof(unsigned), s);
                if (lists) {
                    const bool after_kernel = k != 0 && k != kEmdCheck - 1;
                    launch_ex(after_kernel, k_emd_bid_lists, bid_grid, kEmdBlock, 0, s, N, (const float4 *)w.A4,
                              (const float4 *)w.B4, (const int *)w.assign, w.bids, w.L, (float)eps,
                              list_margin(N, eps), w.active);
                    pdl_launch(k_emd_resolve_lists, grid_for(N, 256), 256, 0, s, N, w.B4, w.owner, w.assign, w.bids);
                } else {
                    k_emd_bid<<<bid_grid, kEmdBlock, 0, s>>>(N, w.A4, w.B4, w.price, w.assign, w.bids, (float)eps,
                                                             w.active);
                    k_emd_resolve<<<grid_for(N, 256), 256, 0, s>>>(N, w.price, w.owner, w.assign, w.bids);
                }
                count_launch(2);
                ++iters;
            }
            unsigned act = 0;
            if (cudaMemcpyAsync(&act, w.active, sizeof(unsigned), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
                cudaStreamSynchronize(s) != cudaSuccess)
                return MESH_ERR_CUDA;
            done = act == 0;
            if (!done && act <= (unsigned)kTailQueue && n <= kTailMaxN) {
                int64_t left = max_iters > iters ? max_iters - iters : 1;
                int cap = (int)(left < (int64_t)(1 << 24) ? left : (int64_t)(1 << 24));
                k_emd_tail<<<1, kTailThreads, 8 * (size_t)N, s>>>(N, w.A4, w.B4, lists ? nullptr : w.price, w.owner,
                                                                  w.assign, w.L, (float)eps, list_margin(N, eps), cap, w.active);
                count_launch();
                if (cudaMemcpyAsync(&act, w.active, sizeof(unsigned), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
                    cudaStreamSynchronize(s) != cudaSuccess)
                    return MESH_ERR_CUDA;
                done = act == 0;
                iters += 1;
            }
            if (!done && iters >= max_iters) {
                if (iters_out) *iters_out = iters;
                return MESH_ERR_DEVICE;
            }
        }
        if (eps <= eps_final) break;
    }
    cudaMemsetAsync(w.ticket, 0, sizeof(unsigned), s);
    k_emd_cost<<<grid_for(N, kEmdBlock), kEmdBlock, 0, s>>>(N, w.A4, w.B4, w.assign, d_assign, w.partial,
                                                           w.ticket, d_out);
    count_launch();
    if (iters_out) *iters_out = iters;
    return check_launch();
}

}  // extern "C"
