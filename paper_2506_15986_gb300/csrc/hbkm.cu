// hbkm.cu -- hierarchical balanced k-means, HBKM (Sec. 4.1, Def. 2 and
// Algorithm 2), and the hub of every final cluster (Def. 3).
//
// Each of `levels` levels splits every cluster of the level above (level 0:
// the whole data set) into k children.  A split runs T iterations; each
// iteration empties the children, visits the cluster's members in
// increasing id and puts member x into
//     j = argmin_j ||x - mu_j||^2 + lam * (2 (c_j - m) + 1)
// (ties to the smaller j), c_j the child's current size and m = |C| / k.  The
// penalty is the increase of Def. 2's size-variance objective that adding x
// to child j causes; lam = lambda * sigma^2 / m, sigma^2 the members' mean
// squared distance to the cluster's centroid.  Every non-empty child then
// moves to its members' mean; an empty child keeps its centroid.  A split
// starts from its members with the min(k, |C|) smallest (key, id); children
// past |C| stay at the cluster's own centroid, empty.
//
// The assignment is an integer decided by float32 sums, so every float
// operation here is rounded on its own (no contraction) and summed in a fixed
// order: distances over coordinates 0..dim-1, sigma^2 and centroid sums over
// members in increasing id, division last.  What is sequential by definition
// is kept so and made short: the visit in id order decides 32 members at a
// time where their choices provably cannot depend on one another (hb_visit),
// the ordered sums stream rows through shared memory ahead of one chain of
// additions (hb_means).  The distances, the partition and the hub search are
// parallel.
//
// Layout: perm[] holds the row ids grouped by current cluster, increasing id
// inside a cluster; seg[] the clusters' first positions; own[] the cluster of
// each position.  D holds the distances child-major (D[j n + i]), so that the
// lanes of a warp, one member each, read a child's distances coalesced.  The
// visit leaves each member's child and its rank in the child; together with
// the children's sizes they give the stable partition of every cluster by
// child, both the next level's order and the children's member lists.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <utility>

#include "internal.h"

namespace ann {
namespace {

constexpr int kMaxBranch = 32;
constexpr int64_t kMaxClusters = int64_t{1} << 20;
constexpr int kVisitWarps = 16;              // warps of a large cluster's visit ...
constexpr int64_t kVisitMinMembers = 8192;  // ... of a level whose clusters have this many members on average

// squared L2 over coordinates 0..dim-1, each step rounded on its own
__device__ __forceinline__ float dist_seq(const float *x, const float *mu, int dim)
{
    float acc = 0.f;
    for (int t = 0; t < dim; t += 4) {
        const float4 a = *reinterpret_cast<const float4 *>(x + t);
        const float4 b = *reinterpret_cast<const float4 *>(mu + t);
        float d = __fsub_rn(a.x, b.x);
        acc = __fadd_rn(acc, __fmul_rn(d, d));
        d = __fsub_rn(a.y, b.y);
        acc = __fadd_rn(acc, __fmul_rn(d, d));
        d = __fsub_rn(a.z, b.z);
        acc = __fadd_rn(acc, __fmul_rn(d, d));
        d = __fsub_rn(a.w, b.w);
        acc = __fadd_rn(acc, __fmul_rn(d, d));
    }
    return acc;
}

// order-preserving map of a float (finite or +inf) to unsigned bits
__device__ __forceinline__ uint32_t ord_bits(float v)
{
    const uint32_t u = __float_as_uint(v);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ void hb_hub_one(int64_t c, int lane, const float *x, int dim, const int64_t *seg, const int32_t *perm,
                           const float *cent, int32_t *hubs);

__global__ void hb_iota(int64_t n, int32_t *perm, int32_t *own)
{
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        perm[i] = static_cast<int32_t>(i);
        own[i] = 0;
    }
}

// distance of every position's row to its cluster's centroid
__global__ void hb_dist_parent(const float *x, int dim, int64_t n, const int32_t *perm, const int32_t *own,
                               const float *cent, float *dp)
{
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x)
        dp[i] = dist_seq(x + static_cast<int64_t>(perm[i]) * dim, cent + static_cast<int64_t>(own[i]) * dim, dim);
}

// Per cluster, one warp: sigma^2 (its members' distances added in order; the
// warp reads 32 at a time and every lane runs the same chain of additions), m,
// lam, and the starting members, the kk smallest (key, id), kept sorted one
// per lane (a member below the largest kept enters by its rank; few do).
// One thread per cluster, each value loaded when it was needed, took 5.5 ms a
// launch at 60,000 rows.
__global__ void hb_setup(int64_t P, int k, float lambda, const int64_t *seg, const int32_t *perm, const float *dp,
                         const uint32_t *keys, float *lamv, float *mv, int32_t *kkv, int32_t *init)
{
    constexpr unsigned kAll = 0xffffffffu;
    constexpr int U = 8;  // groups of 32 members loaded together
    const int lane = threadIdx.x & 31;
    const int64_t wpb = blockDim.x >> 5;
    for (int64_t c = blockIdx.x * wpb + (threadIdx.x >> 5); c < P; c += gridDim.x * wpb) {
        const int64_t b = seg[c], e = seg[c + 1], s = e - b;
        const int kk = s < k ? static_cast<int>(s) : k;
        float sig = 0.f;
        uint64_t top = ~0ull;    // lane j: the j-th smallest (key, id) so far
        uint64_t worst = ~0ull;  // the kk-th
        for (int64_t i0 = b; i0 < e; i0 += 32 * U) {
            float d[U];
            int32_t id[U];
            uint64_t v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t i = i0 + 32 * u + lane;
                d[u] = i < e ? dp[i] : 0.f;
                id[u] = i < e ? perm[i] : -1;
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
                v[u] = id[u] >= 0 ? (static_cast<uint64_t>(keys[id[u]]) << 32) | static_cast<uint32_t>(id[u]) : ~0ull;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t left = e - i0 - 32 * u;
                if (left <= 0)
                    break;
                const int cnt = left < 32 ? static_cast<int>(left) : 32;
                if (cnt == 32) {
#pragma unroll
                    for (int q = 0; q < 32; ++q)
                        sig = __fadd_rn(sig, __shfl_sync(kAll, d[u], q));
                } else {
                    for (int q = 0; q < cnt; ++q)
                        sig = __fadd_rn(sig, __shfl_sync(kAll, d[u], q));
                }
                unsigned in = __ballot_sync(kAll, v[u] < worst);
                while (in) {
                    const uint64_t x = __shfl_sync(kAll, v[u], __ffs(in) - 1);
                    in &= in - 1;
                    const int rank = __popc(__ballot_sync(kAll, top < x));
                    const uint64_t up = __shfl_up_sync(kAll, top, 1);
                    if (rank >= kk)
                        continue;
                    top = lane == rank ? x : (lane > rank ? up : top);
                    worst = __shfl_sync(kAll, top, kk - 1);
                }
            }
        }
        if (lane == 0) {
            float lam = 0.f, m = 0.f;
            if (s > 0) {
                sig = __fdiv_rn(sig, static_cast<float>(s));
                m = __fdiv_rn(static_cast<float>(s), static_cast<float>(k));
                lam = __fdiv_rn(__fmul_rn(lambda, sig), m);
            }
            lamv[c] = lam;
            mv[c] = m;
            kkv[c] = kk;
        }
        if (lane < k)
            init[c * k + lane] = lane < kk ? static_cast<int32_t>(top & 0xffffffffu) : -1;
    }
}

// children's starting centroids: a starting member's row, else the parent's
__global__ void hb_init_children(const float *x, int dim, int k, const int32_t *init, const float *cent_p,
                                 float *cent_c)
{
    const int64_t cj = blockIdx.x;  // child c * k + j
    const int32_t id = init[cj];
    const float *src = id >= 0 ? x + static_cast<int64_t>(id) * dim : cent_p + (cj / k) * dim;
    for (int t = threadIdx.x; t < dim; t += blockDim.x)
        cent_c[cj * dim + t] = src[t];
}

// Distance of every position's row to its cluster's k children (+inf past
// kk), one thread per pair: for levels of many small clusters.
__global__ void hb_dist_children(const float *x, int dim, int64_t n, int k, const int32_t *perm,
                                 const int32_t *own, const int32_t *kkv, const float *cent_c, float *D)
{
    const int64_t total = n * k;
    for (int64_t q = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; q < total;
         q += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t i = q / k;
        const int j = static_cast<int>(q - i * k);
        const int32_t c = own[i];
        D[j * n + i] = j < kkv[c] ? dist_seq(x + static_cast<int64_t>(perm[i]) * dim,
                                             cent_c + (static_cast<int64_t>(c) * k + j) * dim, dim)
                                  : __int_as_float(0x7f800000);
    }
}

// The same for levels of large clusters: a CTA takes 64 positions x all
// children; rows and centroids are staged in shared memory 32 coordinates at
// a time, a thread keeps 4 positions x 2 children in registers, so each
// staged value is read once per 4 or 2 pairs instead of once per pair from
// L1.  Every pair's sum runs over the coordinates in order.  A tile that
// spans clusters is worked once per cluster.  60,000 x 128, k = 32: 227 us a
// launch by pairs, 44 us here (three rounded operations per
// coordinate: 20 us of issue).
constexpr int kDistTile = 64;   // positions per CTA
constexpr int kDistStep = 32;   // coordinates per stage
constexpr int kDistPad = kDistStep + 4;

__global__ void __launch_bounds__(256)
    hb_dist_tiles(const float *__restrict__ x, int dim, int64_t n, int k, const int32_t *__restrict__ perm,
                  const int32_t *__restrict__ own, const int32_t *__restrict__ kkv, const float *__restrict__ cent_c,
                  float *__restrict__ D)
{
    __shared__ __align__(16) float xs[kDistTile * kDistPad];
    __shared__ __align__(16) float cs[kMaxBranch * kDistPad];
    __shared__ int32_t rows[kDistTile];
    __shared__ int32_t owner[kDistTile];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int64_t i0 = blockIdx.x * static_cast<int64_t>(kDistTile);
    const int cnt = static_cast<int>(min(static_cast<int64_t>(kDistTile), n - i0));
    if (tid < kDistTile) {
        rows[tid] = tid < cnt ? perm[i0 + tid] : -1;
        owner[tid] = tid < cnt ? own[i0 + tid] : -1;
    }
    __syncthreads();
    for (int first = 0; first < cnt;) {  // the clusters of the tile, in position order
        const int32_t c = owner[first];
        const int kk = kkv[c];
        float acc[4][2];
#pragma unroll
        for (int a = 0; a < 4; ++a)
            acc[a][0] = acc[a][1] = 0.f;
        for (int t0 = 0; t0 < dim; t0 += kDistStep) {
            const int w4 = min(kDistStep, dim - t0) / 4;  // dim % 4 == 0
            for (int q = tid; q < kDistTile * (kDistStep / 4); q += 256) {
                const int r = q / (kDistStep / 4), o = q % (kDistStep / 4);
                if (o < w4 && rows[r] >= 0)
                    *reinterpret_cast<float4 *>(xs + r * kDistPad + 4 * o) =
                        *reinterpret_cast<const float4 *>(x + static_cast<int64_t>(rows[r]) * dim + t0 + 4 * o);
            }
            for (int q = tid; q < kMaxBranch * (kDistStep / 4); q += 256) {
                const int j = q / (kDistStep / 4), o = q % (kDistStep / 4);
                if (o < w4 && j < kk)
                    *reinterpret_cast<float4 *>(cs + j * kDistPad + 4 * o) = *reinterpret_cast<const float4 *>(
                        cent_c + (static_cast<int64_t>(c) * k + j) * dim + t0 + 4 * o);
            }
            __syncthreads();
            for (int o = 0; o < w4; ++o) {
                float4 xv[4], cv[2];
#pragma unroll
                for (int a = 0; a < 4; ++a)
                    xv[a] = *reinterpret_cast<const float4 *>(xs + (tx + 16 * a) * kDistPad + 4 * o);
#pragma unroll
                for (int g = 0; g < 2; ++g)
                    cv[g] = *reinterpret_cast<const float4 *>(cs + (ty + 16 * g) * kDistPad + 4 * o);
#pragma unroll
                for (int a = 0; a < 4; ++a)
#pragma unroll
                    for (int g = 0; g < 2; ++g) {
                        float d = __fsub_rn(xv[a].x, cv[g].x);
                        acc[a][g] = __fadd_rn(acc[a][g], __fmul_rn(d, d));
                        d = __fsub_rn(xv[a].y, cv[g].y);
                        acc[a][g] = __fadd_rn(acc[a][g], __fmul_rn(d, d));
                        d = __fsub_rn(xv[a].z, cv[g].z);
                        acc[a][g] = __fadd_rn(acc[a][g], __fmul_rn(d, d));
                        d = __fsub_rn(xv[a].w, cv[g].w);
                        acc[a][g] = __fadd_rn(acc[a][g], __fmul_rn(d, d));
                    }
            }
            __syncthreads();
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int r = tx + 16 * a;
            if (r < cnt && owner[r] == c) {
#pragma unroll
                for (int g = 0; g < 2; ++g) {
                    const int j = ty + 16 * g;
                    if (j < k)
                        D[j * n + i0 + r] = j < kk ? acc[a][g] : __int_as_float(0x7f800000);
                }
            }
        }
        while (first < cnt && owner[first] == c)
            ++first;
    }
}

// the size penalty of a child that holds cj members
__device__ __forceinline__ float hb_penalty(float lam, float m, int cj)
{
    return __fmul_rn(lam, __fadd_rn(__fmul_rn(2.f, __fsub_rn(static_cast<float>(cj), m)), 1.f));
}

// The visit in id order.  One member: the child with the smallest
// (distance + penalty, index), whose size then grows.  A child's penalty never
// falls during a visit, so a cost taken at earlier sizes is a lower bound.
// A cluster's members go in rounds of 32 W, one per thread:
//   - every thread finds its member's best and second-best child at the sizes
//     when the round starts, and assumes the best;
//   - from the assumptions of the members before it follow the exact sizes a
//     member meets.  A member whose assumed child still costs less at its
//     exact size than the second-best lower bound is certain; the few others
//     are decided over all children at their exact sizes (lane = child);
//   - until no assumption changes.  Then every member has the child that the
//     visit one by one gives it: by induction each assumption is the choice at
//     the sizes that the earlier choices lead to.  Two or three passes do, unless
//     the penalties outweigh the distances or rows lie in the order of their
//     clusters, so that most choices hang on the ones before: after kVisitPasses
//     passes, or one that changes an eighth of the members, the rest of the
//     round goes one by one, from the first warp with a member that changed (all
//     before it are final).
// For large clusters, whose sizes move slowly against their members'
// preferences (about one member in thirty is uncertain); small ones go to
// hb_visit_warp.  60,000 rows, k = 32: 11 ms a visit at level 1 one by one with a
// 64-bit shuffle argmin per member, 5.2 ms one by one as hb_visit_warp, 790 us
// here (990 us with W = 8, 910 us with 32).  Two levels of ten visits each, random
// rows 12.5 ms; lambda = 1e9, rows along a line, and tight clusters stored one
// after another 2,937, 2,728 and 1,240 ms with passes alone (one member at a time
// with a 64-bit argmin: 175), 51, 52 and 45 ms here.
constexpr int kVisitPasses = 4;
constexpr int kVisitSmem = kVisitWarps * kMaxBranch * 33 * 4;

template <int W>
__global__ void __launch_bounds__(32 * W)
    hb_visit(int64_t n, int k, const int64_t *__restrict__ seg, const float *__restrict__ D,
             const float *__restrict__ lamv, const float *__restrict__ mv, const int32_t *__restrict__ kkv,
             int32_t *__restrict__ lab, int32_t *__restrict__ rank, int32_t *__restrict__ cnt)
{
    constexpr unsigned kAll = 0xffffffffu;
    extern __shared__ float tile_mem[];
    auto tile = reinterpret_cast<float(*)[kMaxBranch][33]>(tile_mem);  // [W]: the round's distances, 32 members per warp
    __shared__ float pen[kMaxBranch];
    __shared__ int size[kMaxBranch];
    __shared__ unsigned mask[W][kMaxBranch];   // the warp's lanes that assume a child
    __shared__ int first_open;                 // the first warp with a member that changed
    __shared__ int2 won[32 * W];               // members decided one by one: child and rank
    const int64_t c = blockIdx.x;
    const int64_t b = seg[c], e = seg[c + 1];
    const float lam = lamv[c], m = mv[c];
    const int kk = kkv[c];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    // an infinite penalty is no ordered one (inf - inf): then every member is
    // decided over all children
    const bool ordered = isfinite(hb_penalty(lam, m, 0)) && isfinite(hb_penalty(lam, m, static_cast<int>(e - b)));
    if (tid < kMaxBranch) {
        size[tid] = 0;
        pen[tid] = hb_penalty(lam, m, 0);
    }
    float d[kMaxBranch];
    auto load = [&](int64_t i) {
#pragma unroll
        for (int j = 0; j < kMaxBranch; ++j)
            d[j] = (j < kk && i < e) ? D[j * n + i] : __int_as_float(0x7f800000);
    };
    load(b + tid);
    __syncthreads();
    for (int64_t i0 = b; i0 < e; i0 += 32 * W) {
        const bool live = i0 + tid < e;
        uint32_t o1 = 0xffffffffu, o2 = 0xffffffffu;
        int j1 = 0, j2 = 0;
        float d1 = 0.f;
#pragma unroll
        for (int j = 0; j < kMaxBranch; ++j) {
            tile[w][j][lane] = d[j];
            if (j < kk) {
                const uint32_t o = ord_bits(__fadd_rn(d[j], pen[j]));
                if (o < o1 || j == 0) {
                    o2 = o1;
                    j2 = j1;
                    o1 = o;
                    j1 = j;
                    d1 = d[j];
                } else if (o < o2 || j == 1) {
                    o2 = o;
                    j2 = j;
                }
            }
        }
        load(i0 + 32 * W + tid);  // in flight during the passes
        int my = j1, at = 0;
        bool alone = false;  // the round ends one by one
        for (int pass = 0;; ++pass) {
            mask[w][lane] = 0u;
            __syncwarp();
            if (live)
                atomicOr(&mask[w][my], 1u << lane);
            __syncthreads();
            int fl = size[lane];  // lane = child: its size when the warp's members come
#pragma unroll
            for (int v = 0; v < W - 1; ++v)
                fl += v < w ? __popc(mask[v][lane]) : 0;
            const unsigned ml = mask[w][lane];
            at = __shfl_sync(kAll, fl, my) + __popc(mask[w][my] & ((1u << lane) - 1u));
            const uint32_t o = ord_bits(__fadd_rn(d1, hb_penalty(lam, m, at)));
            const bool sure = kk < 2 || (ordered && my == j1 && (o < o2 || (o == o2 && j1 < j2)));
            unsigned open = __ballot_sync(kAll, live && !sure);
            bool changed = false;
            while (open) {  // lane = child, for one uncertain member after another
                const int f = __ffs(open) - 1;
                open &= open - 1;
                const int sz = fl + __popc(ml & ((1u << f) - 1u));
                const uint32_t key =
                    lane < kk ? ord_bits(__fadd_rn(tile[w][lane][f], hb_penalty(lam, m, sz))) : 0xffffffffu;
                const uint32_t mn = __reduce_min_sync(kAll, key);
                const int win = __ffs(__ballot_sync(kAll, lane < kk && key == mn)) - 1;
                if (lane == f) {
                    changed = win != my;
                    my = win;
                }
            }
            const int moves = __syncthreads_count(changed);
            if (moves == 0)
                break;
            if (pass + 1 < kVisitPasses && moves < 4 * W)
                continue;
            alone = true;
            if (tid == 0)
                first_open = W;
            __syncthreads();
            if (changed)
                atomicMin(&first_open, w);
            __syncthreads();
            const int w0 = first_open;
            if (w == 0) {  // lane = child, as hb_visit_warp
                int cj = size[lane];
                for (int v = 0; v < w0; ++v)
                    cj += __popc(mask[v][lane]);
                float now = hb_penalty(lam, m, cj), next = hb_penalty(lam, m, cj + 1);
                const int count = static_cast<int>(min(static_cast<int64_t>(32 * W), e - i0));
                for (int v = w0; 32 * v < count; ++v) {
                    const int left = min(32, count - 32 * v);
#pragma unroll 4
                    for (int u = 0; u < left; ++u) {
                        const uint32_t key = lane < kk ? ord_bits(__fadd_rn(tile[v][lane][u], now)) : 0xffffffffu;
                        const uint32_t mn = __reduce_min_sync(kAll, key);
                        const unsigned eq = __ballot_sync(kAll, key == mn);
                        const bool win = key == mn && (eq & ((1u << lane) - 1u)) == 0;
                        if (win)
                            won[32 * v + u] = make_int2(lane, cj);
                        cj += win ? 1 : 0;
                        now = win ? next : now;
                        next = hb_penalty(lam, m, cj + 1);
                    }
                }
                size[lane] = cj;
                pen[lane] = now;
            }
            __syncthreads();
            if (live && w >= w0) {
                my = won[tid].x;
                at = won[tid].y;
            }
            break;
        }
        if (live) {
            lab[i0 + tid] = my;
            rank[i0 + tid] = at;
        }
        if (w == 0 && !alone) {
            int sz = size[lane];
            for (int v = 0; v < W; ++v)
                sz += __popc(mask[v][lane]);
            size[lane] = sz;
            pen[lane] = hb_penalty(lam, m, sz);
        }
        __syncthreads();
    }
    if (tid < k)
        cnt[c * k + tid] = size[tid];
}

// The visit of small clusters: one warp per cluster, lane j = child j, one
// member after another.  Per member one chain of an addition, a 32-bit minimum
// over the warp, a ballot for its first holder and a choice between two
// penalties kept ready; distances come 32 members at a time through shared
// memory.  32 clusters of 1,875 members, k = 32: 164 us
// (hb_visit: 380 us; a 64-bit shuffle argmin per member: 400 us).
constexpr int kSmallVisitWarps = 4;

__global__ void __launch_bounds__(32 * kSmallVisitWarps)
    hb_visit_warp(int64_t P, int64_t n, int k, const int64_t *__restrict__ seg, const float *__restrict__ D,
                  const float *__restrict__ lamv, const float *__restrict__ mv, const int32_t *__restrict__ kkv,
                  int32_t *__restrict__ lab, int32_t *__restrict__ rank, int32_t *__restrict__ cnt)
{
    constexpr unsigned kAll = 0xffffffffu;
    __shared__ float sh[kSmallVisitWarps][kMaxBranch][33];
    __shared__ int2 won[kSmallVisitWarps][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned below = (1u << lane) - 1u;
    for (int64_t c = blockIdx.x * static_cast<int64_t>(kSmallVisitWarps) + w; c < P;
         c += static_cast<int64_t>(gridDim.x) * kSmallVisitWarps) {
        const int64_t b = seg[c], e = seg[c + 1];
        const float lam = lamv[c], m = mv[c];
        const int kk = kkv[c];
        int cj = 0;
        float pen = hb_penalty(lam, m, 0), next = hb_penalty(lam, m, 1);
        float d[kMaxBranch];
        auto load = [&](int64_t i) {
#pragma unroll
            for (int j = 0; j < kMaxBranch; ++j)
                d[j] = (j < kk && i < e) ? D[j * n + i] : 0.f;
        };
        load(b + lane);
        for (int64_t i0 = b; i0 < e; i0 += 32) {
            const int left = static_cast<int>(min(static_cast<int64_t>(32), e - i0));
#pragma unroll
            for (int j = 0; j < kMaxBranch; ++j)
                sh[w][j][lane] = d[j];
            load(i0 + 32 + lane);  // in flight during these members
            __syncwarp();
#pragma unroll 4
            for (int u = 0; u < left; ++u) {
                // past the children: a key above every cost; ties go to the
                // smaller lane, so a NaN cost (the same key) of a child wins
                const uint32_t key = lane < kk ? ord_bits(__fadd_rn(sh[w][lane][u], pen)) : 0xffffffffu;
                const uint32_t mn = __reduce_min_sync(kAll, key);
                const unsigned eq = __ballot_sync(kAll, key == mn);
                const bool win = key == mn && (eq & below) == 0;
                if (win)
                    won[w][u] = make_int2(lane, cj);
                cj += win ? 1 : 0;
                pen = win ? next : pen;
                next = hb_penalty(lam, m, cj + 1);
            }
            __syncwarp();
            if (lane < left) {
                const int2 r = won[w][lane];
                lab[i0 + lane] = r.x;
                rank[i0 + lane] = r.y;
            }
            __syncwarp();
        }
        if (lane < k)
            cnt[c * k + lane] = cj;
    }
}

// the children's first positions: their cluster's, plus the sizes before them
__global__ void hb_offsets(int64_t P, int k, const int64_t *seg, const int32_t *cnt, int64_t *seg2)
{
    for (int64_t c = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; c < P;
         c += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        int64_t o = seg[c];
        for (int j = 0; j < k; ++j) {
            seg2[c * k + j] = o;
            o += cnt[c * k + j];
        }
        if (c == P - 1)
            seg2[P * k] = o;
    }
}

// the stable partition by child: a member's place is its child's first plus
// its rank
__global__ void hb_scatter(int64_t n, int k, const int32_t *perm, const int32_t *own, const int32_t *lab,
                           const int32_t *rank, const int64_t *seg2, int32_t *perm2, int32_t *own2)
{
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t child = static_cast<int64_t>(own[i]) * k + lab[i];
        const int64_t d = seg2[child] + rank[i];
        perm2[d] = perm[i];
        own2[d] = static_cast<int32_t>(child);
    }
}

// Means of lists of rows, each coordinate added in list order (an empty list
// leaves its mean as it was).  One warp per (list, 32 coordinates): a ring of
// stages of 32 rows in shared memory, filled by 16-byte asynchronous copies
// well ahead of the additions, so that what bounds a list is its chain of
// dependent additions and not a load's latency.  60,000 x 128,
// k = 32, two levels of 10 iterations: 38.7 ms with one CTA per cluster and the
// children's sums in shared memory, and 1.1 ms for the mean of all rows; 1.1 ms
// here, the mean of all rows among them.
constexpr int kMeanStages = 8;

template <typename I>
__global__ void __launch_bounds__(32)
    hb_means(const float *__restrict__ x, int dim, int64_t lists, const int64_t *__restrict__ seg,
             const I *__restrict__ perm, float *__restrict__ out)
{
    __shared__ __align__(16) float ring[kMeanStages][32][32];
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x;
    const int t0 = blockIdx.y * 32;
    const int w4 = min(32, dim - t0) / 4;  // 16-byte pieces of a row's slice
    const int piece = lane & 7, sub = lane >> 3;  // this lane copies piece `piece` of rows sub, sub + 4, ...
    for (int64_t c = blockIdx.x; c < lists; c += gridDim.x) {
        const int64_t b = seg[c], e = seg[c + 1];
        if (b == e)
            continue;
        const int64_t stages = (e - b + 31) / 32;
        I ids = b + lane < e ? perm[b + lane] : -1;  // the next stage's rows
        auto fill = [&](int64_t s) {
            if (s < stages) {
                const I cur = ids;
                const int64_t nx = b + (s + 1) * 32 + lane;
                ids = nx < e ? perm[nx] : -1;
                float *dst = &ring[s % kMeanStages][0][0];
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    const I row = __shfl_sync(kAll, cur, 4 * r + sub);
                    if (row >= 0 && piece < w4) {
                        const unsigned to = static_cast<unsigned>(
                            __cvta_generic_to_shared(dst + (4 * r + sub) * 32 + 4 * piece));
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to),
                                     "l"(x + static_cast<int64_t>(row) * dim + t0 + 4 * piece)
                                     : "memory");
                    }
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        for (int s = 0; s < kMeanStages - 1; ++s)
            fill(s);
        float sum = 0.f;
        for (int64_t s = 0; s < stages; ++s) {
            asm volatile("cp.async.wait_group %0;" ::"n"(kMeanStages - 2) : "memory");
            __syncwarp();  // stage s has landed for every lane, and stage s - 1 is read
            fill(s + kMeanStages - 1);
            const float *src = &ring[s % kMeanStages][0][lane];
            const int64_t left = e - b - s * 32;
            if (left >= 32) {
#pragma unroll
                for (int r = 0; r < 32; ++r)
                    sum = __fadd_rn(sum, src[r * 32]);
            } else {
                for (int r = 0; r < left; ++r)
                    sum = __fadd_rn(sum, src[r * 32]);
            }
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncwarp();
        if (lane < 4 * w4)
            out[c * dim + t0 + lane] = __fdiv_rn(sum, static_cast<float>(e - b));
    }
}

// hub of every final cluster: its member nearest the centroid (smaller id on
// ties), one warp per cluster; labels back in row order
__global__ void hb_hubs(const float *x, int dim, int64_t nc, const int64_t *seg, const int32_t *perm,
                        const float *cent, int32_t *hubs)
{
    const int lane = threadIdx.x & 31;
    const int64_t wpb = blockDim.x >> 5;
    for (int64_t c = blockIdx.x * wpb + (threadIdx.x >> 5); c < nc; c += gridDim.x * wpb)
        hb_hub_one(c, lane, x, dim, seg, perm, cent, hubs);
}

__device__ void hb_hub_one(int64_t c, int lane, const float *x, int dim, const int64_t *seg, const int32_t *perm,
                           const float *cent, int32_t *hubs)
{
    uint64_t best = ~0ull;
    for (int64_t i = seg[c] + lane; i < seg[c + 1]; i += 32) {
        const int32_t id = perm[i];
        const float d = dist_seq(x + static_cast<int64_t>(id) * dim, cent + c * dim, dim);
        const uint64_t key = (static_cast<uint64_t>(ord_bits(d)) << 32) | static_cast<uint32_t>(id);
        best = key < best ? key : best;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const uint64_t other = __shfl_xor_sync(0xffffffffu, best, o);
        best = other < best ? other : best;
    }
    if (lane == 0)
        hubs[c] = best == ~0ull ? -1 : static_cast<int32_t>(best & 0xffffffffu);
}

__global__ void hb_labels(int64_t n, const int32_t *perm, const int32_t *own, int32_t *label)
{
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x)
        label[perm[i]] = own[i];
}

struct Buf {
    void *p = nullptr;
    cudaStream_t s;
    explicit Buf(cudaStream_t st) : s(st) {}
    cudaError_t alloc(size_t bytes) { return builder_alloc(&p, bytes, s); }
    template <typename T>
    T *as() const
    {
        return static_cast<T *>(p);
    }
    ~Buf()
    {
        if (p)
            cudaFreeAsync(p, s);
    }
};

#define HB_CK(x)                         \
    do {                                 \
        cudaError_t e_ = (x);            \
        if (e_ != cudaSuccess)           \
            return cuda_status(e_);      \
    } while (0)

dim3 means_grid(int64_t lists, int dim)
{
    return dim3(static_cast<unsigned>(std::min<int64_t>(lists, 152 * 64)), (dim + 31) / 32);
}

unsigned grid_for(int64_t items, int per_block)
{
    return static_cast<unsigned>(std::min<int64_t>((items + per_block - 1) / per_block, 152 * 64));
}

}  // namespace

void list_means(const float *x, int dim, int64_t lists, const int64_t *seg, const int64_t *list, float *out,
                cudaStream_t s)
{
    hb_means<int64_t><<<means_grid(lists, dim), 32, 0, s>>>(x, dim, lists, seg, list, out);
}

}  // namespace ann

using namespace ann;

extern "C" {

ann_status ann_hbkm(const float *d_x, int64_t n, int32_t dim, int32_t k, int32_t levels, double lambda, int32_t T,
                    const uint32_t *d_keys, int32_t *d_hubs, float *d_centroids, int32_t *d_label, void *stream)
{
    if (!d_x || !d_keys || !d_hubs || n < 1 || n > INT32_MAX || dim < 4 || dim % 4 != 0 || dim > 4096 || k < 2 ||
        k > kMaxBranch || levels < 1 || T < 1 || !(lambda >= 0.0) ||
        (reinterpret_cast<uintptr_t>(d_x) & 15) || (reinterpret_cast<uintptr_t>(d_centroids) & 15))
        return ANN_ERR_INVALID_ARG;
    int64_t nc = 1;
    for (int l = 0; l < levels; ++l) {
        nc *= k;
        if (nc > kMaxClusters)
            return ANN_ERR_INVALID_ARG;
    }
    if (static_cast<size_t>(k) * dim * 4 > 227 * 1024)  // the interface's bound, no kernel's here
        return ANN_ERR_UNSUPPORTED;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    HB_CK(cudaFuncSetAttribute(hb_visit<kVisitWarps>, cudaFuncAttributeMaxDynamicSharedMemorySize, kVisitSmem));
    Buf perm(s), perm2(s), own(s), own2(s), seg(s), seg2(s), cent(s), cent2(s), dp(s), D(s), lab(s), rank(s), cnt(s),
        lamv(s), mv(s), kkv(s), init(s);
    const int64_t cl_max = nc;  // clusters of the last level; earlier levels have fewer
    HB_CK(perm.alloc(n * 4));
    HB_CK(perm2.alloc(n * 4));
    HB_CK(own.alloc(n * 4));
    HB_CK(own2.alloc(n * 4));
    HB_CK(seg.alloc((cl_max + 1) * 8));
    HB_CK(seg2.alloc((cl_max + 1) * 8));
    HB_CK(cent.alloc(cl_max * dim * 4));
    HB_CK(cent2.alloc(cl_max * dim * 4));
    HB_CK(dp.alloc(n * 4));
    HB_CK(D.alloc(n * k * 4));
    HB_CK(lab.alloc(n * 4));
    HB_CK(rank.alloc(n * 4));
    HB_CK(cnt.alloc(cl_max * 4));
    HB_CK(lamv.alloc(cl_max / k * 4));
    HB_CK(mv.alloc(cl_max / k * 4));
    HB_CK(kkv.alloc(cl_max / k * 4));
    HB_CK(init.alloc(cl_max * 4));

    hb_iota<<<grid_for(n, 256), 256, 0, s>>>(n, perm.as<int32_t>(), own.as<int32_t>());
    const int64_t seg0[2] = {0, n};
    HB_CK(cudaMemcpyAsync(seg.p, seg0, sizeof(seg0), cudaMemcpyHostToDevice, s));
    auto means = [&](int64_t lists, const Buf &sg, const Buf &list, const Buf &out) {
        hb_means<int32_t><<<means_grid(lists, dim), 32, 0, s>>>(d_x, dim, lists, sg.as<int64_t>(), list.as<int32_t>(),
                                                                out.as<float>());
    };
    means(1, seg, perm, cent);  // level 0: the mean of all rows
    int64_t P = 1;
    for (int l = 1; l <= levels; ++l) {
        hb_dist_parent<<<grid_for(n, 256), 256, 0, s>>>(d_x, dim, n, perm.as<int32_t>(), own.as<int32_t>(),
                                                        cent.as<float>(), dp.as<float>());
        hb_setup<<<grid_for(P * 32, 128), 128, 0, s>>>(P, k, static_cast<float>(lambda), seg.as<int64_t>(),
                                                       perm.as<int32_t>(), dp.as<float>(), d_keys, lamv.as<float>(),
                                                       mv.as<float>(), kkv.as<int32_t>(), init.as<int32_t>());
        hb_init_children<<<static_cast<unsigned>(P * k), 128, 0, s>>>(d_x, dim, k, init.as<int32_t>(),
                                                                       cent.as<float>(), cent2.as<float>());
        // large clusters: position tiles (a tile spans one or two clusters)
        // and the visit by rounds of 512 members; below, pairs and warps.
        // A visit by rounds assumes sizes up to 512 members old: its uncertain
        // members grow as the round's share of a cluster.  One cluster, k = 32, ten
        // iterations (ms, by rounds | one by one): 32,768 members 6.1 | 28.7, 8,192
        // 4.0 | 7.5, 4,096 3.3 | 4.0, 1,024 1.2 | 1.3; with lambda = 10, where rounds
        // end one by one, 6.9 | 7.5 at 8,192.  Below the line a level has many
        // clusters, of which a warp each fills the chip with fewer registers.
        const bool tiles = n / P >= kDistTile;
        const bool rounds = n / P >= kVisitMinMembers;
        for (int it = 0; it < T; ++it) {
            if (tiles)
                hb_dist_tiles<<<static_cast<unsigned>((n + kDistTile - 1) / kDistTile), 256, 0, s>>>(
                    d_x, dim, n, k, perm.as<int32_t>(), own.as<int32_t>(), kkv.as<int32_t>(), cent2.as<float>(),
                    D.as<float>());
            else
                hb_dist_children<<<grid_for(n * k, 256), 256, 0, s>>>(d_x, dim, n, k, perm.as<int32_t>(),
                                                                      own.as<int32_t>(), kkv.as<int32_t>(),
                                                                      cent2.as<float>(), D.as<float>());
            if (rounds)
                hb_visit<kVisitWarps><<<static_cast<unsigned>(P), 32 * kVisitWarps, kVisitSmem, s>>>(
                    n, k, seg.as<int64_t>(), D.as<float>(), lamv.as<float>(), mv.as<float>(), kkv.as<int32_t>(),
                    lab.as<int32_t>(), rank.as<int32_t>(), cnt.as<int32_t>());
            else
                hb_visit_warp<<<grid_for(P, kSmallVisitWarps), 32 * kSmallVisitWarps, 0, s>>>(
                    P, n, k, seg.as<int64_t>(), D.as<float>(), lamv.as<float>(), mv.as<float>(), kkv.as<int32_t>(),
                    lab.as<int32_t>(), rank.as<int32_t>(), cnt.as<int32_t>());
            hb_offsets<<<grid_for(P, 128), 128, 0, s>>>(P, k, seg.as<int64_t>(), cnt.as<int32_t>(),
                                                        seg2.as<int64_t>());
            hb_scatter<<<grid_for(n, 256), 256, 0, s>>>(n, k, perm.as<int32_t>(), own.as<int32_t>(),
                                                        lab.as<int32_t>(), rank.as<int32_t>(), seg2.as<int64_t>(),
                                                        perm2.as<int32_t>(), own2.as<int32_t>());
            means(P * k, seg2, perm2, cent2);
        }
        P *= k;
        std::swap(perm.p, perm2.p);
        std::swap(own.p, own2.p);
        std::swap(seg.p, seg2.p);
        std::swap(cent.p, cent2.p);
        HB_CK(cudaGetLastError());
    }
    hb_hubs<<<grid_for(nc * 32, 128), 128, 0, s>>>(d_x, dim, nc, seg.as<int64_t>(), perm.as<int32_t>(),
                                                   cent.as<float>(), d_hubs);
    if (d_label)
        hb_labels<<<grid_for(n, 256), 256, 0, s>>>(n, perm.as<int32_t>(), own.as<int32_t>(), d_label);
    if (d_centroids)
        HB_CK(cudaMemcpyAsync(d_centroids, cent.p, nc * dim * 4, cudaMemcpyDeviceToDevice, s));
    HB_CK(cudaGetLastError());
    HB_CK(cudaStreamSynchronize(s));
    return ANN_OK;
}

}  // extern "C"
