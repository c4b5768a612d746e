// build.cu -- offline index construction on the GPU: the proximity graph of
// Sec. 2.1 Def. 1 (exact K-NN candidates from knn.cu, relative-neighbourhood
// pruning, reachability repair from the navigating node) and the navigating
// node (medoid).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "device_util.cuh"
#include "internal.h"

namespace ann {
namespace {

// squared distance between two FP32 rows, as order-preserving key bits
__device__ __forceinline__ uint32_t exact_dist_bits(const uint8_t *x, const uint8_t *q, int dim)
{
    const float4 *x4 = reinterpret_cast<const float4 *>(x);
    const float4 *q4 = reinterpret_cast<const float4 *>(q);
    float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
    for (int c = 0; c < dim / 4; ++c) {
        const float4 u = x4[c], v = q4[c];
        const float d0 = u.x - v.x, d1 = u.y - v.y, d2 = u.z - v.z, d3 = u.w - v.w;
        a0 = fmaf(d0, d0, a0);
        a1 = fmaf(d1, d1, a1);
        a2 = fmaf(d2, d2, a2);
        a3 = fmaf(d3, d3, a3);
    }
    return f32_to_ord((a0 + a1) + (a2 + a3));
}

// Squared distances of row x to the rows q0 and q1 at once, each as
// exact_dist_bits adds it, as floats.
template <int DT>
__device__ __forceinline__ void two_dists(const uint8_t *x, const uint8_t *q0, const uint8_t *q1, int dim, float *d)
{
    if constexpr (DT == ANN_U8) {
        uint32_t a0 = 0, a1 = 0;
        for (int c = 0; c < dim / 4; ++c) {
            const uint32_t u = reinterpret_cast<const uint32_t *>(x)[c];
            const uint32_t e0 = __vabsdiffu4(u, reinterpret_cast<const uint32_t *>(q0)[c]);
            const uint32_t e1 = __vabsdiffu4(u, reinterpret_cast<const uint32_t *>(q1)[c]);
            a0 = __dp4a(e0, e0, a0);
            a1 = __dp4a(e1, e1, a1);
        }
        d[0] = static_cast<float>(a0);
        d[1] = static_cast<float>(a1);
    } else {
        // four FP32 accumulators a row in two packed pairs: each f32x2 operation
        // rounds both halves as two scalar ones would
        uint64_t acc[2][2] = {};
        auto add = [](uint64_t (&a)[2], float4 u, float4 v) {
            asm("{\n\t.reg .b64 x, y, d;\n\t"
                "mov.b64 x, {%2, %3};\n\tmov.b64 y, {%6, %7};\n\t"
                "sub.rn.f32x2 d, x, y;\n\tfma.rn.f32x2 %0, d, d, %0;\n\t"
                "mov.b64 x, {%4, %5};\n\tmov.b64 y, {%8, %9};\n\t"
                "sub.rn.f32x2 d, x, y;\n\tfma.rn.f32x2 %1, d, d, %1;\n\t}"
                : "+l"(a[0]), "+l"(a[1])
                : "f"(u.x), "f"(u.y), "f"(u.z), "f"(u.w), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w));
        };
#pragma unroll 4
        for (int c = 0; c < dim / 4; ++c) {
            const float4 u = reinterpret_cast<const float4 *>(x)[c];
            add(acc[0], u, reinterpret_cast<const float4 *>(q0)[c]);
            add(acc[1], u, reinterpret_cast<const float4 *>(q1)[c]);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i)
            d[i] = (__uint_as_float(static_cast<uint32_t>(acc[i][0])) +
                    __uint_as_float(static_cast<uint32_t>(acc[i][0] >> 32))) +
                   (__uint_as_float(static_cast<uint32_t>(acc[i][1])) +
                    __uint_as_float(static_cast<uint32_t>(acc[i][1] >> 32)));
    }
}

// Relative-neighbourhood pruning of node p's K candidates (sorted by exact
// (dist, id)): c is kept unless a node s kept before it has
// alpha * delta(s, c) <= delta(p, c); at most R are kept; -1 pads the row.
// One CTA per node takes eight candidates at a time, two to a warp: its lanes
// measure both against the nodes kept so far and against the earlier ones of the
// eight, and the eight are then decided in order.  So the chain of decisions is
// an eighth as long as one candidate at a time, the staged rows are shared by
// four warps, and a kept row read from shared memory, whose bandwidth bounds the
// kernel, serves two candidates (50,000 x 128, K = 64, R = 32: one warp a node
// 4.26 ms, four with a candidate each 2.34 ms, 1.73 ms here).
// STAGED: the K candidate rows are copied into shared memory first (when they
// fit); otherwise they are read from global memory (L1/L2-cached) in place.
constexpr int kPruneWarps = 4, kPruneGroup = 2 * kPruneWarps;

template <int DT, bool STAGED>
__global__ void __launch_bounds__(32 * kPruneWarps)
    rng_prune(const uint8_t *base, int rowbytes, int dim, int64_t n, const int32_t *cand, const void *cand_d, int K,
              int R, float alpha, int stride, int32_t *graph)
{
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ unsigned pruned[kPruneGroup];  // bit v < w: by the v-th of the eight if kept; bit 31: by a kept node
    __shared__ int32_t ids[128];
    __shared__ int32_t kept[64 + kPruneGroup];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int64_t p = blockIdx.x;
    if (p >= n)
        return;
    for (int c = tid; c < K; c += 32 * kPruneWarps)
        ids[c] = cand[p * K + c];
    __syncthreads();
    if constexpr (STAGED) {
        const int pieces = rowbytes / 16;
        for (int i = tid; i < K * pieces; i += 32 * kPruneWarps) {
            const int c = i / pieces, o = i - c * pieces;
            if (ids[c] >= 0)
                reinterpret_cast<uint4 *>(smem + c * stride)[o] =
                    reinterpret_cast<const uint4 *>(base + static_cast<int64_t>(ids[c]) * rowbytes)[o];
        }
        __syncthreads();
    }
    auto row = [&](int c) -> const uint8_t * {
        if constexpr (STAGED)
            return smem + c * stride;
        else
            return base + static_cast<int64_t>(ids[c]) * rowbytes;
    };
    int nk = 0;
    for (int c0 = 0; c0 < K && nk < R; c0 += kPruneGroup) {
        const int ca = c0 + w, cb = ca + kPruneWarps;
        const bool live_a = ca < K && ids[ca] >= 0, live_b = cb < K && ids[cb] >= 0;
        auto limit = [&](int c) {
            if constexpr (DT == ANN_U8)
                return static_cast<float>(reinterpret_cast<const int32_t *>(cand_d)[p * K + c]);
            else
                return reinterpret_cast<const float *>(cand_d)[p * K + c];
        };
        unsigned by_a = 0, by_b = 0;
        if (live_a) {  // pads come last: cb is live only if ca is
            const float la = limit(ca), lb = live_b ? limit(cb) : 0.f;
            const uint8_t *xa = row(ca), *xb = live_b ? row(cb) : xa;
            for (int j = lane; j < nk + w + (live_b ? kPruneWarps : 0); j += 32) {
                const int s = j < nk ? kept[j] : c0 + (j - nk);
                const unsigned bit = j < nk ? 0x80000000u : 1u << (j - nk);
                float d[2];
                two_dists<DT>(row(s), xa, xb, dim, d);
                if (j < nk + w && alpha * d[0] <= la)
                    by_a |= bit;
                if (alpha * d[1] <= lb)
                    by_b |= bit;
            }
        }
        by_a = __reduce_or_sync(kFull, by_a);
        by_b = __reduce_or_sync(kFull, by_b);
        if (lane == 0) {
            pruned[w] = by_a;
            pruned[w + kPruneWarps] = by_b;
        }
        __syncthreads();
        // the eight in order, by every thread alike
        unsigned in = 0;
        bool end = false;
        for (int v = 0; v < kPruneGroup && !end; ++v) {
            if (c0 + v >= K || ids[c0 + v] < 0 || nk >= R) {
                end = true;
            } else if (!((pruned[v] & 0x80000000u) || (pruned[v] & in))) {
                in |= 1u << v;
                if (tid == 0)
                    kept[nk] = c0 + v;
                ++nk;
            }
        }
        __syncthreads();
        if (end)
            break;
    }
    for (int j = tid; j < R; j += 32 * kPruneWarps)
        graph[p * R + j] = j < nk ? ids[kept[j]] : -1;
}

// ---- medoid ---------------------------------------------------------------

template <typename T, typename Acc>
__global__ void col_partial_sums(const T *x, int64_t n, int dim, int64_t rows_per, Acc *partial)
{
    const int64_t r0 = blockIdx.x * rows_per;
    const int64_t r1 = min(n, r0 + rows_per);
    for (int c = threadIdx.x; c < dim; c += blockDim.x) {
        Acc s = 0;
        for (int64_t r = r0; r < r1; ++r)
            s += static_cast<Acc>(x[r * dim + c]);
        partial[blockIdx.x * static_cast<int64_t>(dim) + c] = s;
    }
}

template <typename Acc>
__global__ void col_total(const Acc *partial, int blocks, int dim, Acc *total)
{
    for (int c = threadIdx.x; c < dim; c += blockDim.x) {
        Acc s = 0;
        for (int b = 0; b < blocks; ++b)
            s += partial[static_cast<int64_t>(b) * dim + c];
        total[c] = s;
    }
}

// fp32: key = (ord(|x - mean|^2), id), atomicMin gives the (dist, id) argmin
__global__ void medoid_f32(const float *x, int64_t n, int dim, const float *sum, unsigned long long *best)
{
    const int lane = threadIdx.x & 31;
    const int64_t row = (blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) >> 5;
    if (row >= n)
        return;
    const float inv = 1.0f / static_cast<float>(n);
    float s = 0.f;
    for (int c = lane; c < dim; c += 32) {
        const float d = x[row * dim + c] - sum[c] * inv;
        s = fmaf(d, d, s);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        s += __shfl_xor_sync(kFull, s, o);
    if (lane == 0)
        atomicMin(best, static_cast<unsigned long long>(make_key(f32_to_ord(s), static_cast<int32_t>(row)) >> 1));
}

// uint8: exact ||n x - sum||^2 in 64-bit integers; first pass the minimum
// value, second pass the smallest id attaining it
__global__ void medoid_u8_value(const uint8_t *x, int64_t n, int dim, const unsigned long long *sum,
                                unsigned long long *vals, unsigned long long *best)
{
    const int lane = threadIdx.x & 31;
    const int64_t row = (blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) >> 5;
    if (row >= n)
        return;
    unsigned long long s = 0;
    for (int c = lane; c < dim; c += 32) {
        const long long v = n * static_cast<long long>(x[row * dim + c]) - static_cast<long long>(sum[c]);
        s += static_cast<unsigned long long>(v * v);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        s += __shfl_xor_sync(kFull, s, o);
    if (lane == 0) {
        vals[row] = s;
        atomicMin(best, s);
    }
}

__global__ void medoid_u8_id(const unsigned long long *vals, int64_t n, const unsigned long long *best,
                             unsigned long long *best_id)
{
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x)
        if (vals[i] == *best)
            atomicMin(best_id, static_cast<unsigned long long>(i));
}

// ---- reachability repair ----------------------------------------------------

// What the repair keeps on the device from launch to launch.
struct Repair {
    unsigned long long best;  // (distance, id) of the nearest node with a free slot to u
    int64_t added;            // edges added
    int32_t u;                // the unreachable node in turn
    int32_t done, failed;     // no node left; a node found no reachable free slot
    int32_t lo, hi, tail;     // breadth-first search: the frontier and the queue's end
    unsigned blocks;          // CTAs of the level that are through
};

__global__ void repair_init(const int32_t *graph, int64_t n, int R, int32_t root, int32_t *deg, int32_t *reached,
                            int32_t *queue, Repair *st)
{
    for (int64_t v = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; v < n;
         v += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        int c = 0;
        while (c < R && graph[v * R + c] >= 0)
            ++c;
        deg[v] = c;
        reached[v] = v == root;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        queue[0] = root;
        *st = Repair{~0ull, 0, -1, 0, 0, 0, 1, 1, 0u};
    }
}

// the unreached neighbours of node v join the queue; the whole warp calls it
__device__ __forceinline__ void reach_neighbours(const int32_t *graph, int R, int32_t v, int32_t *reached,
                                                 int32_t *queue, int32_t *tail, int lane)
{
    for (int j = lane; j < R; j += 32) {
        const int32_t x = graph[static_cast<int64_t>(v) * R + j];
        if (x >= 0 && __ldcg(reached + x) == 0 && atomicExch(reached + x, 1) == 0)
            queue[atomicAdd(tail, 1)] = x;
    }
}

// Levels of the search by one CTA, while they have at most `most` nodes: queue
// [lo, hi) is the frontier, and is what is left at the end.  A level of a few
// nodes is a chain of round trips (adjacency rows, then flags), so their ids
// stay in shared memory, and where most of what they point to is new (NEW) the
// flags take one trip instead of a look and an exchange: the 10,000 levels of
// 20,000 rows along a line take 156 ms at a launch a level, 7.8 here.
constexpr int kNarrow = 64;

struct Frontier {
    int32_t ids[2][kNarrow];  // the first of this level, and of the next
    int32_t tail;
};

template <bool NEW>
__device__ void reach_in_block(const int32_t *graph, int R, int32_t *reached, int32_t *queue, int32_t &lo, int32_t &hi,
                               int32_t most, Frontier &f)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, warps = blockDim.x >> 5;
    if (threadIdx.x < kNarrow && lo + static_cast<int>(threadIdx.x) < hi)
        f.ids[0][threadIdx.x] = __ldcg(queue + lo + threadIdx.x);
    if (threadIdx.x == 0)
        f.tail = hi;
    __syncthreads();
    for (int side = 0; lo < hi && hi - lo <= most; side ^= 1) {
        for (int i = w; i < hi - lo; i += warps) {
            if (hi - lo > kNarrow) {
                reach_neighbours(graph, R, __ldcg(queue + lo + i), reached, queue, &f.tail, lane);
                continue;
            }
            const int32_t v = f.ids[side][i];
            for (int j = lane; j < R; j += 32) {
                const int32_t x = graph[static_cast<int64_t>(v) * R + j];
                if (x >= 0 && (NEW || __ldcg(reached + x) == 0) && atomicExch(reached + x, 1) == 0) {
                    const int32_t at = atomicAdd(&f.tail, 1);
                    queue[at] = x;
                    if (at - hi < kNarrow)
                        f.ids[side ^ 1][at - hi] = x;
                }
            }
        }
        __syncthreads();
        const bool was_wide = hi - lo > kNarrow;
        lo = hi;
        hi = f.tail;
        if (was_wide && static_cast<int>(threadIdx.x) < min(kNarrow, hi - lo))
            f.ids[side ^ 1][threadIdx.x] = __ldcg(queue + lo + threadIdx.x);
        __syncthreads();
    }
}

// one level of the breadth-first search from the root, a warp per frontier
// node; the last CTA through moves the frontier on, and over the narrow levels
// that follow
__global__ void __launch_bounds__(256)
    reach_level(const int32_t *graph, int R, int32_t *reached, int32_t *queue, Repair *st)
{
    __shared__ int last;
    __shared__ Frontier frontier;
    const int32_t lo = __ldcg(&st->lo), hi = __ldcg(&st->hi);
    if (lo < hi) {
        const int lane = threadIdx.x & 31;
        for (int64_t i = lo + (blockIdx.x * 256ll + threadIdx.x) / 32; i < hi; i += gridDim.x * 8ll)
            reach_neighbours(graph, R, __ldcg(queue + i), reached, queue, &st->tail, lane);
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0)
        last = atomicAdd(&st->blocks, 1u) == gridDim.x - 1;
    __syncthreads();
    if (last) {
        int32_t next_lo = hi, next_hi = __ldcg(&st->tail);
        reach_in_block<true>(graph, R, reached, queue, next_lo, next_hi, kNarrow, frontier);
        if (threadIdx.x == 0) {
            st->lo = next_lo;
            st->hi = st->tail = next_hi;
            st->blocks = 0;
        }
    }
}

// nearest reachable node with a free slot to u: key (ord distance, id); one
// atomic per CTA
template <int DT>
__global__ void __launch_bounds__(256)
    nearest_eligible(const uint8_t *base, int rowbytes, int dim, int64_t n, int R, const int32_t *deg,
                     const int32_t *reached, Repair *st)
{
    __shared__ unsigned long long warp_best[8];
    if (st->done)
        return;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint8_t *xu = base + static_cast<int64_t>(st->u) * rowbytes;
    unsigned long long best = ~0ull;
    for (int64_t w = blockIdx.x * 8ll + wid; w < n; w += gridDim.x * 8ll) {
        if (!reached[w] || deg[w] >= R)
            continue;
        const uint8_t *xw = base + w * rowbytes;
        uint32_t bits;
        if constexpr (DT == ANN_U8) {
            uint32_t acc = 0;
            for (int c = lane; c < dim / 4; c += 32) {
                const uint32_t d = __vabsdiffu4(reinterpret_cast<const uint32_t *>(xu)[c],
                                                reinterpret_cast<const uint32_t *>(xw)[c]);
                acc = __dp4a(d, d, acc);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                acc += __shfl_xor_sync(kFull, acc, o);
            bits = acc;
        } else {
            float s = 0.f;
            for (int c = lane; c < dim; c += 32) {
                const float d = reinterpret_cast<const float *>(xu)[c] - reinterpret_cast<const float *>(xw)[c];
                s = fmaf(d, d, s);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                s += __shfl_xor_sync(kFull, s, o);
            bits = f32_to_ord(s);
        }
        const unsigned long long key = make_key(bits, static_cast<int32_t>(w)) >> 1;
        best = key < best ? key : best;
    }
    if (lane == 0)
        warp_best[wid] = best;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < 8; ++i)
            best = warp_best[i] < best ? warp_best[i] : best;
        if (best != ~0ull)
            atomicMin(&st->best, best);
    }
}

// One CTA: the edge from the nearest node found to u, all that u reaches, and
// the next unreachable node in id order (the first launch, u = -1, only that).
__global__ void __launch_bounds__(1024)
    repair_step(int32_t *graph, int64_t n, int R, int32_t *deg, int32_t *reached, int32_t *queue, Repair *st)
{
    __shared__ int32_t first;
    __shared__ Frontier frontier;
    const int tid = threadIdx.x;
    if (st->done)
        return;
    const int32_t u = st->u;
    if (u >= 0) {
        const unsigned long long key = st->best;
        __syncthreads();
        if (key == ~0ull) {
            if (tid == 0)
                st->failed = st->done = 1;
            return;
        }
        if (tid == 0) {
            const int32_t w = static_cast<int32_t>(key & 0x7fffffffu);
            graph[static_cast<int64_t>(w) * R + deg[w]] = u;
            deg[w] += 1;
            st->added += 1;
            st->best = ~0ull;
            reached[u] = 1;
            queue[0] = u;
        }
        __syncthreads();
        int32_t lo = 0, hi = 1;
        reach_in_block<false>(graph, R, reached, queue, lo, hi, INT32_MAX, frontier);
    }
    // the nodes before u are all reached
    if (tid == 0)
        first = INT32_MAX;
    __syncthreads();
    for (int64_t v0 = u + 1; v0 < n; v0 += 4096) {
        int32_t mine = INT32_MAX;
#pragma unroll
        for (int i = 3; i >= 0; --i) {
            const int64_t v = v0 + i * 1024 + tid;
            if (v < n && __ldcg(reached + v) == 0)
                mine = static_cast<int32_t>(v);
        }
        if (mine != INT32_MAX)
            atomicMin(&first, mine);
        __syncthreads();
        const bool found = first != INT32_MAX;
        __syncthreads();  // read by all before the next group may set it
        if (found)
            break;
    }
    if (tid == 0) {
        st->u = first;
        st->done = first == INT32_MAX;
    }
}

template <typename T>
struct DevBuf {
    T *p = nullptr;
    cudaStream_t s = nullptr;
    cudaError_t alloc(size_t count, cudaStream_t st)
    {
        s = st;
        return builder_alloc(reinterpret_cast<void **>(&p), count * sizeof(T), st);
    }
    ~DevBuf()
    {
        if (p)
            cudaFreeAsync(p, s);
    }
};

#define CK(x)                                \
    do {                                     \
        cudaError_t e_ = (x);                \
        if (e_ != cudaSuccess)               \
            return cuda_status(e_);          \
    } while (0)

}  // namespace

ann_status medoid_gpu(const void *d_base, int64_t n, int dim, int dtype, cudaStream_t s, int32_t *out)
{
    const int blocks = static_cast<int>(std::min<int64_t>(1024, n));
    const int64_t rows_per = (n + blocks - 1) / blocks;
    const unsigned rgrid = static_cast<unsigned>((n * 32 + 255) / 256);
    if (dtype == ANN_U8) {
        if (n > (1 << 20) || dim > 128)
            return ANN_ERR_UNSUPPORTED;  // keeps ||n x - sum||^2 within 64 bits
        DevBuf<unsigned long long> part, tot, vals, best;
        CK(part.alloc(static_cast<size_t>(blocks) * dim, s));
        CK(tot.alloc(dim, s));
        CK(vals.alloc(n, s));
        CK(best.alloc(2, s));
        CK(cudaMemsetAsync(best.p, 0xff, 16, s));
        col_partial_sums<uint8_t, unsigned long long><<<blocks, 128, 0, s>>>(
            static_cast<const uint8_t *>(d_base), n, dim, rows_per, part.p);
        col_total<unsigned long long><<<1, 128, 0, s>>>(part.p, blocks, dim, tot.p);
        medoid_u8_value<<<rgrid, 256, 0, s>>>(static_cast<const uint8_t *>(d_base), n, dim, tot.p, vals.p, best.p);
        medoid_u8_id<<<1024, 256, 0, s>>>(vals.p, n, best.p, best.p + 1);
        unsigned long long id = 0;
        CK(cudaMemcpyAsync(&id, best.p + 1, 8, cudaMemcpyDeviceToHost, s));
        CK(cudaStreamSynchronize(s));
        *out = static_cast<int32_t>(id);
        return ANN_OK;
    }
    if (dtype != ANN_F32)
        return ANN_ERR_UNSUPPORTED;
    DevBuf<float> part, tot;
    DevBuf<unsigned long long> best;
    CK(part.alloc(static_cast<size_t>(blocks) * dim, s));
    CK(tot.alloc(dim, s));
    CK(best.alloc(1, s));
    CK(cudaMemsetAsync(best.p, 0xff, 8, s));
    col_partial_sums<float, float><<<blocks, 128, 0, s>>>(static_cast<const float *>(d_base), n, dim,
                                                          rows_per, part.p);
    col_total<float><<<1, 128, 0, s>>>(part.p, blocks, dim, tot.p);
    medoid_f32<<<rgrid, 256, 0, s>>>(static_cast<const float *>(d_base), n, dim, tot.p, best.p);
    unsigned long long key = 0;
    CK(cudaMemcpyAsync(&key, best.p, 8, cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    *out = static_cast<int32_t>(key & 0x7fffffffu);
    return ANN_OK;
}

ann_status prune_rows(const void *d_base, int64_t n, int dim, int dtype, int K, int R, float alpha,
                      const int32_t *cand, const void *cand_d, int32_t *d_graph, cudaStream_t s);
ann_status repair_reachability(const void *d_base, int64_t n, int dim, int dtype, int R, int32_t *d_graph,
                               int32_t medoid_id, int64_t *repairs, cudaStream_t s);

ann_status build_graph_gpu(const void *d_base, int64_t n, int dim, int dtype, int K, int R, float alpha,
                           int32_t *d_graph, int32_t *medoid, int64_t *repairs, cudaStream_t s)
{
    // 1. exact K-NN candidates of every node (itself excluded)
    DevBuf<int32_t> cids;
    DevBuf<float> cd;
    CK(cids.alloc(static_cast<size_t>(n) * K, s));
    CK(cd.alloc(static_cast<size_t>(n) * K, s));
    ann_status st = knn_exact(d_base, n, dim, dtype, ANN_L2, d_base, n, K, true, cids.p, cd.p, s);
    if (st != ANN_OK)
        return st;
    // 2. relative-neighbourhood pruning
    if ((st = prune_rows(d_base, n, dim, dtype, K, R, alpha, cids.p, cd.p, d_graph, s)) != ANN_OK)
        return st;
    // 3. navigating node
    if (*medoid < 0 && (st = medoid_gpu(d_base, n, dim, dtype, s, medoid)) != ANN_OK)
        return st;
    // 4. reachability repair
    return repair_reachability(d_base, n, dim, dtype, R, d_graph, *medoid, repairs, s);
}

// Relative-neighbourhood pruning of n candidate rows (K per row, ascending
// (distance, id), -1 pads at the end) into the n adjacency rows at d_graph.
ann_status prune_rows(const void *d_base, int64_t n, int dim, int dtype, int K, int R, float alpha,
                      const int32_t *cand, const void *cand_d, int32_t *d_graph, cudaStream_t s)
{
    const int es = elem_size(dtype);
    const int rowbytes = dim * es;
    int s16 = rowbytes / 16;
    if ((s16 & 1) == 0)
        s16 += 1;
    const int stride = s16 * 16;
    // staged up to two CTAs an SM
    constexpr int kStaged = 108 * 1024;  // also the kernel's limit whatever K is: a builder of another thread never lowers it
    const bool staged = static_cast<size_t>(K) * stride <= kStaged;
    const size_t smem = staged ? static_cast<size_t>(K) * stride : 0;
    const uint8_t *bb = static_cast<const uint8_t *>(d_base);
    const unsigned grid = static_cast<unsigned>(n);
#define PRUNE(DT, ST)                                                                                          \
    do {                                                                                                       \
        CK(cudaFuncSetAttribute(rng_prune<DT, ST>, cudaFuncAttributeMaxDynamicSharedMemorySize, kStaged));     \
        rng_prune<DT, ST><<<grid, 32 * kPruneWarps, smem, s>>>(bb, rowbytes, dim, n, cand, cand_d, K, R,       \
                                                               alpha, stride, d_graph);                        \
    } while (0)
    if (dtype == ANN_U8 && staged)
        PRUNE(ANN_U8, true);
    else if (dtype == ANN_U8)
        PRUNE(ANN_U8, false);
    else if (staged)
        PRUNE(ANN_F32, true);
    else
        PRUNE(ANN_F32, false);
#undef PRUNE
    return cuda_status(cudaGetLastError());
}

// Reachability repair: nodes in id order; an unreachable node u gets the edge
// w -> u from the nearest reachable node w with a free slot; all that u
// reaches becomes reachable before the next node is taken.  The whole state
// stays on the device: levels of the first search and repairs are queued in
// batches, with one look at the state after each (launches past the end
// return at once).  With the graph, the search and the flags on the host,
// which waited for every nearest node, 83 repairs of 50,000 rows took about
// 24 ms; 1.4 ms here.
ann_status repair_reachability(const void *d_base, int64_t n, int dim, int dtype, int R, int32_t *d_graph,
                               int32_t medoid_id, int64_t *repairs, cudaStream_t s)
{
    constexpr int kBatch = 16;
    const int rowbytes = dim * elem_size(dtype);
    DevBuf<int32_t> deg, reached, queue;
    DevBuf<Repair> st;
    CK(deg.alloc(n, s));
    CK(reached.alloc(n, s));
    CK(queue.alloc(n, s));
    CK(st.alloc(1, s));
    const unsigned wide = static_cast<unsigned>(std::min<int64_t>((n + 7) / 8, 152 * 8));
    const uint8_t *bb = static_cast<const uint8_t *>(d_base);
    Repair h{};
    repair_init<<<wide, 256, 0, s>>>(d_graph, n, R, medoid_id, deg.p, reached.p, queue.p, st.p);
    do {
        for (int i = 0; i < kBatch; ++i)
            reach_level<<<wide, 256, 0, s>>>(d_graph, R, reached.p, queue.p, st.p);
        CK(cudaMemcpyAsync(&h, st.p, sizeof(h), cudaMemcpyDeviceToHost, s));
        CK(cudaStreamSynchronize(s));
    } while (h.lo < h.hi);
    if (h.tail < n) {
        repair_step<<<1, 1024, 0, s>>>(d_graph, n, R, deg.p, reached.p, queue.p, st.p);
        do {
            for (int i = 0; i < kBatch; ++i) {
                if (dtype == ANN_U8)
                    nearest_eligible<ANN_U8><<<wide, 256, 0, s>>>(bb, rowbytes, dim, n, R, deg.p, reached.p, st.p);
                else
                    nearest_eligible<ANN_F32><<<wide, 256, 0, s>>>(bb, rowbytes, dim, n, R, deg.p, reached.p, st.p);
                repair_step<<<1, 1024, 0, s>>>(d_graph, n, R, deg.p, reached.p, queue.p, st.p);
            }
            CK(cudaMemcpyAsync(&h, st.p, sizeof(h), cudaMemcpyDeviceToHost, s));
            CK(cudaStreamSynchronize(s));
        } while (!h.done);
    }
    if (h.failed)
        return ANN_ERR_CAPACITY;  // no reachable node has a free slot
    if (repairs)
        *repairs = h.added;
    return ANN_OK;
}

namespace {

constexpr int kInbox = 32;  // reverse-edge requests kept per node and batch

// every new node's out-edges become requests in their targets' inboxes
__global__ void reverse_collect(const int32_t *rows, int64_t b0, int64_t nb, int R, int32_t *inbox, int32_t *cnt,
                                int32_t *touched, int32_t *ntouched)
{
    const int64_t t = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
    if (t >= nb * R)
        return;
    const int32_t q = rows[t];
    if (q < 0)
        return;
    const int slot = atomicAdd(&cnt[q], 1);
    if (slot == 0)
        touched[atomicAdd(ntouched, 1)] = q;
    if (slot < kInbox)
        inbox[static_cast<int64_t>(q) * kInbox + slot] = static_cast<int32_t>(b0 + t / R);
}

// A touched node's row: its neighbours plus its inbox; appended while they
// fit, else all of them sorted by (squared L2, id) and pruned to R as
// rng_prune does.  One warp per node (R <= 32: lane j holds slot j of the
// row and inbox entry j).
__global__ void reverse_prune(const float *x, int dim, const int32_t *touched, const int32_t *ntouched,
                              const int32_t *inbox, int32_t *cnt, int R, float alpha, int32_t *graph)
{
    __shared__ uint64_t keys[64];
    __shared__ int32_t kept[32];
    const int lane = threadIdx.x;
    const int nt = *ntouched;
    const uint8_t *xb = reinterpret_cast<const uint8_t *>(x);
    const int rowbytes = dim * 4;
    for (int w = blockIdx.x; w < nt; w += gridDim.x) {
        const int32_t q = touched[w];
        const int nin = min(cnt[q], kInbox);
        const int32_t c0 = lane < R ? graph[static_cast<int64_t>(q) * R + lane] : -1;
        const int32_t c1 = lane < nin ? inbox[static_cast<int64_t>(q) * kInbox + lane] : -1;
        const int deg = __popc(__ballot_sync(kFull, c0 >= 0));
        if (deg + nin <= R) {
            if (lane < nin)
                graph[static_cast<int64_t>(q) * R + deg + lane] = c1;
        } else {
            const uint8_t *xq = xb + static_cast<int64_t>(q) * rowbytes;
            uint64_t k0 = c0 >= 0 ? make_key(exact_dist_bits(xb + static_cast<int64_t>(c0) * rowbytes,
                                                                               xq, dim), c0)
                                  : kKeyMax;
            uint64_t k1 = c1 >= 0 ? make_key(exact_dist_bits(xb + static_cast<int64_t>(c1) * rowbytes,
                                                                               xq, dim), c1)
                                  : kKeyMax;
            warp_sort64(k0, k1, lane);
            keys[lane] = k0;
            keys[lane + 32] = k1;
            __syncwarp();
            int nk = 0;
            for (int c = 0; c < 64 && nk < R; ++c) {
                const uint64_t kc = keys[c];
                if (kc == kKeyMax)
                    break;
                const int32_t id = key_id(kc);
                const float dqc = ord_to_f32(static_cast<uint32_t>(kc >> 32));
                bool pruned = false;
                for (int j = lane; j < nk; j += 32)
                    pruned |= alpha * ord_to_f32(exact_dist_bits(
                                          xb + static_cast<int64_t>(kept[j]) * rowbytes,
                                          xb + static_cast<int64_t>(id) * rowbytes, dim)) <= dqc;
                if (!__any_sync(kFull, pruned)) {
                    if (lane == 0)
                        kept[nk] = id;
                    ++nk;
                }
                __syncwarp();
            }
            if (lane < R)
                graph[static_cast<int64_t>(q) * R + lane] = lane < nk ? kept[lane] : -1;
        }
        __syncwarp();
        if (lane == 0)
            cnt[q] = 0;
    }
}

}  // namespace

// Insertion by search: the exact graph of the first n0 rows, then batches of
// rows each searched on the graph built so far (their k nearest found become
// their candidates, pruned to R), with the reverse edges added or re-pruned;
// then the navigating node of all rows and the reachability repair.
ann_status build_graph_insert(const float *x, int64_t n, int dim, int K, int R, float alpha, int64_t n0,
                              int64_t batch, int32_t *d_graph, int32_t *medoid, int64_t *repairs, cudaStream_t s)
{
    int device = 0;
    CK(cudaGetDevice(&device));
    int32_t m0 = -1;
    ann_status st = build_graph_gpu(x, n0, dim, ANN_F32, K, R, alpha, d_graph, &m0, nullptr, s);
    if (st != ANN_OK)
        return st;
    CK(cudaMemsetAsync(d_graph + n0 * R, 0xff, static_cast<size_t>(n - n0) * R * 4, s));
    DevBuf<int32_t> inbox, cnt, touched, ntouched, ids;
    DevBuf<float> dd;
    CK(inbox.alloc(static_cast<size_t>(n) * kInbox, s));
    CK(cnt.alloc(n, s));
    CK(touched.alloc(n, s));
    CK(ntouched.alloc(1, s));
    CK(ids.alloc(static_cast<size_t>(batch) * K, s));
    CK(dd.alloc(static_cast<size_t>(batch) * K, s));
    CK(cudaMemsetAsync(cnt.p, 0, n * 4, s));
    ann_search_params p{};
    p.k = K;
    p.L = std::max(K, 128);
    p.W = R <= 32 ? 4 : 2;
    for (int64_t b0 = n0, nb = 0; b0 < n; b0 += nb) {
        // a batch holds at most a quarter of the rows inserted so far: rows of
        // one batch do not see each other
        nb = std::min({batch, n - b0, std::max<int64_t>(1, b0 / 4)});
        // the graph so far (rows past b0 are empty, so unreachable)
        ann_index_desc desc{};
        desc.n = n;
        desc.dim = dim;
        desc.degree = R;
        desc.dtype = ANN_F32;
        desc.metric = ANN_L2;
        desc.base = x;
        desc.graph = d_graph;
        desc.medoid = m0;
        CK(cudaStreamSynchronize(s));
        ann_index *idx = nullptr;
        if ((st = ann_index_create(&desc, device, &idx)) != ANN_OK)
            return st;
        st = ann_search_batch(idx, x + b0 * dim, nb, nullptr, &p, ids.p, dd.p, nullptr, s);
        if (st == ANN_OK)
            st = ann_sync_status(idx, s);
        ann_free_index(idx);
        if (st != ANN_OK)
            return st;
        if ((st = prune_rows(x, nb, dim, ANN_F32, K, R, alpha, ids.p, dd.p, d_graph + b0 * R, s)) != ANN_OK)
            return st;
        CK(cudaMemsetAsync(ntouched.p, 0, 4, s));
        reverse_collect<<<static_cast<unsigned>((nb * R + 255) / 256), 256, 0, s>>>(
            d_graph + b0 * R, b0, nb, R, inbox.p, cnt.p, touched.p, ntouched.p);
        reverse_prune<<<152 * 8, 32, 0, s>>>(x, dim, touched.p, ntouched.p, inbox.p, cnt.p, R, alpha, d_graph);
        CK(cudaGetLastError());
    }
    if (*medoid < 0 && (st = medoid_gpu(x, n, dim, ANN_F32, s, medoid)) != ANN_OK)
        return st;
    return repair_reachability(x, n, dim, ANN_F32, R, d_graph, *medoid, repairs, s);
}

}  // namespace ann

using namespace ann;

extern "C" {

ann_status ann_knn(const void *d_base, int64_t n, int32_t dim, int32_t dtype, int32_t metric,
                   const void *d_queries, int64_t nq, int32_t k, int32_t exclude_self, int32_t *d_ids,
                   void *d_dists, void *stream)
{
    const int es = elem_size(dtype);
    if (!d_base || !d_queries || !d_ids || !d_dists || n < 1 || n > INT32_MAX || dim < 1 || nq < 0 ||
        k < 1 || k > 128 || k > n || es == 0 || (metric != ANN_L2 && metric != ANN_IP))
        return ANN_ERR_INVALID_ARG;
    if ((dtype != ANN_U8 && dtype != ANN_F32) || (dtype == ANN_U8 && metric != ANN_L2))
        return ANN_ERR_UNSUPPORTED;
    if ((static_cast<int64_t>(dim) * es) % 16 != 0 || (exclude_self && d_queries != d_base) ||
        (reinterpret_cast<uintptr_t>(d_base) & 15) || (reinterpret_cast<uintptr_t>(d_queries) & 15))
        return ANN_ERR_INVALID_ARG;
    if (nq == 0)
        return ANN_OK;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    ann_status st = knn_exact(d_base, n, dim, dtype, metric, d_queries, nq, k, exclude_self != 0, d_ids, d_dists, s);
    if (st == ANN_OK)
        st = cuda_status(cudaStreamSynchronize(s));
    return st;
}

ann_status ann_medoid(const void *d_base, int64_t n, int32_t dim, int32_t dtype, int32_t *medoid, void *stream)
{
    if (!d_base || !medoid || n < 1 || n > INT32_MAX || dim < 1)
        return ANN_ERR_INVALID_ARG;
    return medoid_gpu(d_base, n, dim, dtype, static_cast<cudaStream_t>(stream), medoid);
}

ann_status ann_build_graph_insert(const void *d_base, int64_t n, int32_t dim, int32_t dtype, int32_t K, int32_t R,
                                  float alpha, int64_t n_seed, int64_t batch, int32_t *d_graph, int32_t *medoid,
                                  int64_t *repairs, void *stream)
{
    if (!d_base || !d_graph || !medoid || n < 2 || n > INT32_MAX || dim < 4 || K < 1 || K > 128 || R < 1 ||
        R > K || R > 32 || !(alpha > 0.f) || n_seed < K + 1 || n_seed > n || batch < 1 || *medoid >= n)
        return ANN_ERR_INVALID_ARG;
    if (dtype != ANN_F32)
        return ANN_ERR_UNSUPPORTED;
    if ((static_cast<int64_t>(dim) * 4) % 16 != 0 || (reinterpret_cast<uintptr_t>(d_base) & 15))
        return ANN_ERR_INVALID_ARG;
    return build_graph_insert(static_cast<const float *>(d_base), n, dim, K, R, alpha, n_seed,
                              std::min<int64_t>(batch, n), d_graph, medoid, repairs,
                              static_cast<cudaStream_t>(stream));
}

ann_status ann_build_graph(const void *d_base, int64_t n, int32_t dim, int32_t dtype, int32_t K, int32_t R,
                           float alpha, int32_t *d_graph, int32_t *medoid, int64_t *repairs, void *stream)
{
    const int es = elem_size(dtype);
    if (!d_base || !d_graph || !medoid || n < 2 || n > INT32_MAX || dim < 1 || K < 1 || K > 128 ||
        K > n - 1 || R < 1 || R > K || R > 64 || !(alpha > 0.f) || es == 0)
        return ANN_ERR_INVALID_ARG;
    if (dtype != ANN_U8 && dtype != ANN_F32)
        return ANN_ERR_UNSUPPORTED;
    if ((static_cast<int64_t>(dim) * es) % 16 != 0 ||
        (reinterpret_cast<uintptr_t>(d_base) & 15) || *medoid >= n)
        return ANN_ERR_INVALID_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    return build_graph_gpu(d_base, n, dim, dtype, K, R, alpha, d_graph, medoid, repairs, s);
}

}  // extern "C"
