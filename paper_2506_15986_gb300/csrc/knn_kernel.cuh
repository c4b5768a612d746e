// knn_kernel.cuh -- exact k-NN on the GPU: ground truth of recall@k, the graph
// builder's candidates, k-means assignment.
//
// Scores |y|^2 - 2 x.y (or -x.y) of every (query, base) pair come from
// tcgen05 tensor cores and never reach memory: a CTA keeps 128 queries as the
// A operand, streams the base through in tiles of 128 rows, and its epilogue
// warps keep each query's best KP candidates (64 up to k = 32, else 128).  Of
// those, the ones that the scores' errors leave in question are then re-scored
// exactly (direct differences: int32 for uint8, fp32 otherwise) and sorted by
// (distance, id).
//
// Precision of the scores.  An fp32 value is the exact sum of three BF16 values
// (8 + 8 + 8 significant bits: high, middle, low), so x.y is six BF16 products
// plus three dropped ones below 2^-24 relative.  The tensor cores truncate each
// accumulation step, so sums are kept short: the high-high products of every
// 64 coordinates have an accumulator of their own, the five small products of
// 128 coordinates share one (its steps are 2^-8 as large), and the accumulators
// are added in registers, rounded.  Against 64 bits, rms error over |x||y| on
// anisotropic rows: 7.4e-8 at 128 coordinates (fp32 SGEMM 1.5e-7), 1.1e-7 at
// 256 (3.0e-7), 1.2e-7 at 960 (5.8e-7); on centred rows 6.7e-9, 5.1e-9 and
// 3.4e-9 (1.8e-8).  One accumulator for all six products would be worse than
// SGEMM (5.1e-7 at 128).  uint8 values are BF16 values: one product, exact in
// each 128 coordinates.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <float.h>
#include <stdint.h>

#include <algorithm>
#include <numeric>

#include "device_util.cuh"
#include "internal.h"
#include "tc.cuh"

namespace ann {
namespace {

constexpr int kEpiWarps = 8;          // epilogue warps of a CTA
constexpr int kTile = 128;            // queries, and base rows, of one MMA tile
constexpr int kImage = kTile * 128;   // bytes of a tile's 64-wide K chunk of one plane
constexpr int kSlotsA = 6, kSlotsB = 8;  // images in the operands' rings

struct KnnBars {
    uint64_t full_a[kSlotsA], empty_a[kSlotsA], full_b[kSlotsB], empty_b[kSlotsB], acc_full[2], acc_empty[2];
};

constexpr int kOffB = kSlotsA * kImage;
constexpr int kOffNy = kOffB + kSlotsB * kImage;
constexpr int kOffThr = kOffNy + 2 * kTile * 4;
constexpr int kOffBars = kOffThr + 2 * kTile * 4;
constexpr int kKnnSmem = kOffBars + sizeof(KnnBars) + 16;

struct KnnArgs {
    const uint8_t *A, *B;  // packed images [tile][chunk][plane]
    int chunks;            // 64-wide K chunks
    const float *ny;       // |y|^2 of the block's base rows
    const float *nx;       // |x|^2 of the block's queries
    const unsigned *nmax;  // bits of the largest |y|^2 of all base rows
    int64_t n;             // base rows of the block
    int64_t col0;          // id of its first row
    int64_t rows;          // queries of the block
    int64_t row0;          // index of its first query (self exclusion)
    int64_t tiles_m, tiles_n;
    int64_t stride;        // the j-th base tile a query tile meets is j * stride mod tiles_n
    int64_t unit;          // CTAs take ranges of this many (query tile, base tile) pairs: 1 or tiles_n
    int ip, self;          // inner product; skip the query's own index
    int dim, k;
    uint64_t *lists;       // [rows rounded up to kTile][slots][list_keys(KPL, KR)] candidate keys
    uint2 *ends;           // [rows rounded up to kTile][slots] a list's length and last threshold
    int slots;             // lists per query
    int *status;
};

// A (query tile, base tile) pair in the order that CTAs take them: query tile tm's
// j-th pair has base tile j * stride mod tiles_n.  (Tiles, and a CTA's pairs, are
// counted in 32 bits: the epilogue's registers are few.)
struct TileWalk {
    int tm, j;
    unsigned tn;
    __device__ TileWalk(const KnnArgs &a, int64_t t)
        : tm(static_cast<int>(t / a.tiles_n)), j(static_cast<int>(t - static_cast<int64_t>(tm) * a.tiles_n)),
          tn(static_cast<unsigned>(j * a.stride % a.tiles_n))
    {
    }
    __device__ void next(const KnnArgs &a)
    {
        const unsigned n = static_cast<unsigned>(a.tiles_n);
        tn += static_cast<unsigned>(a.stride);
        tn -= tn >= n ? n : 0;
        if (++j == static_cast<int>(n)) {
            j = 0;
            tn = 0;
            ++tm;
        }
    }
};

// The score of a certain candidate: keys are (order-preserving score, id).
__device__ __forceinline__ uint64_t score_key(float s, int64_t id)
{
    return (static_cast<uint64_t>(f32_to_ord(s)) << 32) | static_cast<uint32_t>(id);
}

// More than what two scores' errors and two exact distances' rounding can hide
// for a query with squared norm nx: any sum of dim products or squares in fp32,
// in whatever order, is within (16 + dim) 2^-24 of the sum of their
// magnitudes, |x| |y| at most (twice that for -2 x.y), |x|^2 or |y|^2.  (A norm
// that is no float leaves its products' size open.)
__device__ __forceinline__ float score_slack(float nx, float nmax, int dim, int ip)
{
    if (!(nx < FLT_MAX && nmax < FLT_MAX))
        return INFINITY;
    const float u = static_cast<float>(16 + dim) * 1.1920929e-7f;  // 2 * 2^-24
    const float xy = sqrtf(nx) * sqrtf(nmax);
    return 2.f * u * (ip ? xy : 2.f * xy + nmax + nx);
}

// CTA of a grid of G over T units (CTA b: units [b T / G, (b + 1) T / G)) whose
// range holds unit t
__host__ __device__ __forceinline__ int64_t cta_of_tile(int64_t t, int64_t T, int64_t G)
{
    return ((t + 1) * G - 1) / T;
}

__device__ __forceinline__ uint64_t bitonic_merge32(uint64_t v, int lane)
{
#pragma unroll
    for (int j = 16; j > 0; j >>= 1) {
        const uint64_t o = __shfl_xor_sync(kFull, v, j);
        v = (lane & j) == 0 ? kmin(v, o) : kmax(v, o);
    }
    return v;
}

// The KP = 32 KPL smallest of the sorted list T (element 32 r + lane in T[r])
// and 32 sorted keys v: the top block keeps its 32 smallest with v, and the
// blocks below are merged with it one after another.
template <int KPL>
__device__ __forceinline__ void merge_sorted(uint64_t (&T)[KPL], uint64_t v, int lane)
{
    T[KPL - 1] = bitonic_merge32(kmin(T[KPL - 1], __shfl_sync(kFull, v, 31 - lane)), lane);
#pragma unroll
    for (int b = KPL - 2; b >= 0; --b) {
        const uint64_t o = __shfl_sync(kFull, T[b + 1], 31 - lane);
        const uint64_t lo = kmin(T[b], o), hi = kmax(T[b], o);
        T[b] = bitonic_merge32(lo, lane);
        T[b + 1] = bitonic_merge32(hi, lane);
    }
}

// A list that is full keeps its KP smallest keys (at most half of it).  The lists
// of the lanes in `rows`, cnt keys each, at most 32 J; returns the lane's new
// count and its list's last key.  From then on only a key below that can enter,
// which bounds what a list takes in when the slack hides every
// difference between the scores (rows far from the origin, or one row farther
// than the rest): 10,000 queries among 300,000 rows of 128 coordinates, k = 10,
// one row of 1e20: 148 ms without the cut, 8.6 ms with it; 4.6 ms without that
// row.  The KP-th smallest score is found bit by bit over the keys in
// registers, and where it cuts equal scores their ids'; sorting the list 32 keys
// at a time instead took 12.8 ms, its warp's chain of shuffles holding up the
// others at the next tile.
struct ListEnd {
    int cnt;
    float score;
    uint32_t id;
};

template <int J, int KP>
__device__ __noinline__ ListEnd compact_rows(unsigned rows, int cnt, uint64_t *mine, float score, uint32_t id)
{
    static_assert(32 * J >= 2 * KP, "room for what comes between two compactions");
    const int lane = threadIdx.x & 31;
    __syncwarp();
    while (rows) {
        const int r = __ffs(rows) - 1;
        rows &= rows - 1;
        const int nb = __shfl_sync(kFull, cnt, r);  // more than 32 J - 32 >= KP
        uint64_t *L = reinterpret_cast<uint64_t *>(__shfl_sync(kFull, reinterpret_cast<unsigned long long>(mine), r));
        // (the scores only: with whole keys in registers the call would cost the
        // epilogue more spills)
        uint32_t o[J];
#pragma unroll
        for (int j = 0; j < J; ++j)
            o[j] = 32 * j + lane < nb ? static_cast<uint32_t>(L[32 * j + lane] >> 32) : 0xffffffffu;
        uint32_t v = 0;   // the leading bits of the KP-th smallest score
        int left = KP;    // its rank among the keys with those bits
#pragma unroll 1
        for (uint32_t bit = 0x80000000u; bit; bit >>= 1) {
            int below = 0;  // keys with the bits found so far and a zero here
#pragma unroll
            for (int j = 0; j < J; ++j)
                below += __popc(__ballot_sync(kFull, (o[j] ^ v) < bit));
            if (below < left) {
                left -= below;
                v |= bit;
            }
        }
        unsigned keep = 0, equal = 0;  // bit j: of the lane's j-th key
        int same = 0;
#pragma unroll
        for (int j = 0; j < J; ++j) {
            keep |= (o[j] < v ? 1u : 0u) << j;
            equal |= (o[j] == v ? 1u : 0u) << j;
            same += __popc(__ballot_sync(kFull, o[j] == v));
        }
        uint32_t cut = 0xffffffffu;  // the last id kept of that score
        if (same > left) {
            cut = 0;
#pragma unroll
            for (int j = 0; j < J; ++j)
                o[j] = equal >> j & 1 ? static_cast<uint32_t>(L[32 * j + lane]) : 0xffffffffu;  // ids are 31 bits
#pragma unroll 1
            for (uint32_t bit = 0x40000000u; bit; bit >>= 1) {
                int below = 0;
#pragma unroll
                for (int j = 0; j < J; ++j)
                    below += __popc(__ballot_sync(kFull, (o[j] ^ cut) < bit));
                if (below < left) {
                    left -= below;
                    cut |= bit;
                }
            }
#pragma unroll
            for (int j = 0; j < J; ++j)
                equal &= ~((o[j] > cut ? 1u : 0u) << j);
        }
        keep |= equal;
        int at = 0;
        constexpr int B = J % 8 ? J : 8;  // keys read before any place up to theirs is written
#pragma unroll 1
        for (int j0 = 0; j0 < J; j0 += B) {
            uint64_t x[B];
#pragma unroll
            for (int j = 0; j < B; ++j)
                x[j] = keep >> (j0 + j) & 1 ? L[32 * (j0 + j) + lane] : 0;
#pragma unroll
            for (int j = 0; j < B; ++j) {
                const bool in = keep >> (j0 + j) & 1;
                const unsigned m = __ballot_sync(kFull, in);
                if (in)
                    L[at + __popc(m & lanemask_lt())] = x[j];
                at += __popc(m);
            }
        }
        if (lane == r) {
            cnt = KP;
            score = ord_to_f32(v);
            id = cut;
        }
        __syncwarp();
    }
    return {cnt, score, id};
}

// 32 columns of several accumulators with one wait
__device__ __forceinline__ void tmem_load_start(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
          "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
          "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
          "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}

__device__ __forceinline__ void tmem_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// orders uses of the registers after the wait before it
__device__ __forceinline__ void tmem_landed(uint32_t (&r)[32])
{
    asm volatile(""
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                   "+r"(r[15])::"memory");
    asm volatile(""
                 : "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]),
                   "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]),
                   "+r"(r[30]), "+r"(r[31])::"memory");
}

// Keys that a list holds: about what a search of a million rows in random order
// appends, and well above what a compaction leaves.
constexpr int list_keys(int KPL, int KR) { return KR == 1 ? 160 : 128 * KPL; }

// P planes (1: BF16 values, 3: fp32 split), 32 KPL candidates kept of a list that
// fills, KR scores in registers (SPLIT: half as many as k), MULTI: more than
// one phase (128 coordinates) a tile.
// A persistent CTA per SM takes a contiguous range of the (query tile, base
// tile) pairs in row-major order, so the ranges differ by at most one tile
// whatever the shape, and a query tile is shared by two or three CTAs at most
// ranges' ends, each with a list of its own.  From eight query tiles a CTA on
// the ranges are whole query tiles instead: an eighth longer at worst, with half
// as many lists.
//   warp 0      copies operand images (16 KB bulk copies, one barrier each);
//   warp 1      issues the MMAs, M = N = 128, in phases of two K chunks.  A
//               phase of P = 3 fills three of TMEM's four accumulators (small,
//               high of either chunk) in rotation: the next phase's small
//               products go to the fourth while the epilogue reads these.  P =
//               1 fills one, of two in turn;
//   warps 2..9  one query and half of a tile's columns per thread: score,
//               compare with the query's threshold.  The few that pass are
//               appended to the thread's list in memory and their scores enter
//               its k best, kept sorted in registers (KR of them), so that the
//               threshold is always the current one and nothing is sorted
//               across lanes.  (Candidates collected in shared memory and
//               merged into sorted lists by the warp: 20 ms for 50,000 queries
//               among themselves, k = 64, and 6.9 ms for 10,000 among 300,000,
//               k = 10, most of it waiting for merges; the warp stopping at
//               every column that passes in some lane: 9.4 and 4.6 ms; the k
//               smallest minima of groups of eight columns: 28.8 and 5.0 ms.)
//               The two threads of a query share their thresholds once a tile.
//               SPLIT, for k > 32: each keeps the k / 2 best (rounded up) of its
//               own columns, and the larger of their last ones stands for the
//               k-th of all: half the registers and insertions (10,000 queries
//               among 30,000 rows of 64 coordinates: k = 64 1,179 us with all 64
//               scores in either thread's registers, 687 us; k = 100 3,711 us with
//               128 in those of four warps, 956 us).
// The A images of a query tile stay in shared memory when they fit (K x P <=
// six images: 128 fp32 or 384 uint8 coordinates), else they stream with the
// base's.  The threshold is the k-th best score plus what the scores' errors
// could hide, and no more than the last key that a compaction kept.
// 10,000 queries among 300,000 rows of 128 coordinates, k = 10: an SGEMM, its 12 GB
// of scores and a pass that selects from them 23.3 ms; 4.5 ms here, six products
// at 1,030 TFLOP/s, 55 % of the measured BF16 rate (bounded by shared-memory
// reads of the N = 128 MMAs and the epilogue's hand-over).  960 coordinates:
// 790 TFLOP/s, the operands streaming from L2 and the epilogue's sums of several
// phases spilling (MULTI: 324 to 536 bytes a thread).
template <int P, int KPL, int KR, bool SPLIT, bool MULTI>
__global__ void __launch_bounds__(64 + 32 * kEpiWarps, 1) knn_tile_kernel(const KnnArgs a)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    float *sny = reinterpret_cast<float *>(smem + kOffNy);
    uint32_t *sthr = reinterpret_cast<uint32_t *>(smem + kOffThr);  // the queries' thresholds, order-preserving bits
    KnnBars *bars = reinterpret_cast<KnnBars *>(smem + kOffBars);
    uint32_t *slot = reinterpret_cast<uint32_t *>(smem + kOffBars + sizeof(KnnBars));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int i = 0; i < kSlotsA; ++i) {
            mbar_init(&bars->full_a[i], 1);
            mbar_init(&bars->empty_a[i], 1);
        }
        for (int i = 0; i < kSlotsB; ++i) {
            mbar_init(&bars->full_b[i], 1);
            mbar_init(&bars->empty_b[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&bars->acc_full[i], 1);
            mbar_init(&bars->acc_empty[i], kEpiWarps);
        }
        fence_mbar_init();
    }
    if (warp == 1)
        tmem_alloc(slot, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *slot;
    const int64_t T = a.tiles_m * a.tiles_n / a.unit, G = gridDim.x;
    const int64_t t0 = blockIdx.x * T / G * a.unit;
    const int pairs = static_cast<int>((blockIdx.x + 1) * T / G * a.unit - t0);
    const int chunks = a.chunks;
    const bool resident = chunks * P <= kSlotsA;

    if (warp == 0) {
        if (lane == 0) {
            // ---- operand copies; the i-th use of a ring slot waits for the
            // MMAs of the use before it
            int64_t ia = 0, ib = 0;  // images issued into the A and B rings
            bool ok = true;
            auto copy = [&](uint8_t *ring, int slots, uint64_t *full, uint64_t *empty, int64_t &i, const uint8_t *src) {
                const int s = static_cast<int>(i % slots);
                const int64_t use = i / slots;
                if (use > 0 && !mbar_wait_bounded(empty + s, static_cast<uint32_t>((use - 1) & 1), kTcWaitIters)) {
                    ok = false;
                    return;
                }
                mbar_arrive_expect_tx(full + s, kImage);
                bulk_g2s(ring + s * kImage, src, kImage, full + s);
                ++i;
            };
            // resident A images: use u of slot s is the u-th query tile's
            auto copy_resident = [&](int64_t tm, int64_t use) {
                for (int s = 0; s < chunks * P && ok; ++s) {
                    if (use > 0 && !mbar_wait_bounded(&bars->empty_a[s], static_cast<uint32_t>((use - 1) & 1), kTcWaitIters)) {
                        ok = false;
                        return;
                    }
                    mbar_arrive_expect_tx(&bars->full_a[s], kImage);
                    bulk_g2s(smem + s * kImage, a.A + (tm * chunks * P + s) * kImage, kImage, &bars->full_a[s]);
                }
            };
            int64_t uses = 0;
            TileWalk at(a, t0);
            for (int t = 0; t < pairs && ok; ++t, at.next(a)) {
                const int64_t tm = at.tm, tn = at.tn;
                if (resident && (t == 0 || at.j == 0))
                    copy_resident(tm, uses++);
                for (int c = 0; c < chunks && ok; ++c) {
                    const uint8_t *sa = a.A + (tm * chunks + c) * P * kImage, *sb = a.B + (tn * chunks + c) * P * kImage;
                    for (int p = 0; p < P && ok; ++p) {  // base planes low to high, query planes high to low
                        copy(smem + kOffB, kSlotsB, bars->full_b, bars->empty_b, ib, sb + (P - 1 - p) * kImage);
                        if (!resident && ok)
                            copy(smem, kSlotsA, bars->full_a, bars->empty_a, ia, sa + p * kImage);
                    }
                }
            }
            if (!ok)
                atomicOr(a.status, kStatusTimeoutBit);
            // every copy lands before the CTA ends
            auto drain = [&](uint64_t *full, int slots, int64_t issued) {
                for (int64_t i = issued > slots ? issued - slots : 0; i < issued; ++i)
                    mbar_wait_bounded(full + i % slots, static_cast<uint32_t>((i / slots) & 1), kTcWaitIters);
            };
            drain(bars->full_b, kSlotsB, ib);
            if (!resident) {
                drain(bars->full_a, kSlotsA, ia);
            } else if (uses > 0) {
                for (int s = 0; s < chunks * P; ++s)
                    mbar_wait_bounded(&bars->full_a[s], static_cast<uint32_t>((uses - 1) & 1), kTcWaitIters);
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            // ---- MMAs
            constexpr uint32_t ID = idesc_bf16_f32(kTile, kTile);
            int64_t ia = 0, ib = 0, uses = 0, ph = 0;
            bool ok = true;
            auto landed = [&](uint64_t *bar, int64_t use) {
                if (ok && !mbar_wait_bounded(bar, static_cast<uint32_t>(use & 1), kTcWaitIters))
                    ok = false;
                tc_fence_after();
            };
            auto product = [&](uint32_t d, int sa, int sb, bool first) {
                if (!ok)
                    return;
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                    tc_mma(d, smem_desc(smem + sa * kImage + kk * 256, 128, 1024),
                           smem_desc(smem + kOffB + sb * kImage + kk * 256, 128, 1024), ID,
                           (first && kk == 0) ? 0u : 1u);
            };
            TileWalk at(a, t0);
            for (int t = 0; t < pairs && ok; ++t, at.next(a)) {
                const bool fresh = t == 0 || at.j == 0;
                if (fresh)
                    ++uses;
                for (int c = 0; c < chunks && ok; ++c) {
                    const bool begins = (c & 1) == 0;
                    const int r = static_cast<int>(3 * ph & 3);  // P == 3: the phase's first accumulator
                    const uint32_t small = tmem + r * 128;
                    const uint32_t main = P == 1 ? tmem + static_cast<int>(ph & 1) * 128
                                                 : tmem + ((r + 1 + (c & 1)) & 3) * 128;
                    if (P == 1 && begins && ph >= 2)
                        landed(&bars->acc_empty[ph & 1], (ph >> 1) - 1);  // the accumulator's last epilogue
                    int sa[P], sb[P];  // ring slots of the query planes (high first) and base planes (low first)
#pragma unroll
                    for (int p = 0; p < P; ++p) {
                        sb[p] = static_cast<int>((ib + p) % kSlotsB);
                        sa[p] = resident ? c * P + p : static_cast<int>((ia + p) % kSlotsA);
                    }
                    auto need_a = [&](int p) {
                        if (!resident)
                            landed(&bars->full_a[sa[p]], (ia + p) / kSlotsA);
                        else if (fresh)
                            landed(&bars->full_a[sa[p]], uses - 1);
                    };
                    auto need_b = [&](int p) { landed(&bars->full_b[sb[p]], (ib + p) / kSlotsB); };
                    if constexpr (P == 1) {
                        need_b(0);
                        need_a(0);
                        product(main, sa[0], sb[0], begins);
                        tc_commit(&bars->empty_b[sb[0]]);
                    } else {
                        need_b(0);  // base low
                        need_a(0);  // query high
                        product(small, sa[0], sb[0], begins);
                        tc_commit(&bars->empty_b[sb[0]]);
                        need_b(1);  // base middle
                        product(small, sa[0], sb[1], false);
                        need_a(1);  // query middle
                        product(small, sa[1], sb[1], false);
                        tc_commit(&bars->empty_b[sb[1]]);
                        need_b(2);  // base high
                        product(small, sa[1], sb[2], false);
                        need_a(2);  // query low
                        product(small, sa[2], sb[2], false);
                        // the high accumulators were the previous phase's (the
                        // small one its predecessor's: waited for a phase ago)
                        if (begins && ph >= 1)
                            landed(&bars->acc_empty[(ph - 1) & 1], (ph - 1) >> 1);
                        product(main, sa[0], sb[2], true);
                        tc_commit(&bars->empty_b[sb[2]]);
                    }
                    ib += P;
                    if (!resident) {
#pragma unroll
                        for (int p = 0; p < P; ++p)
                            tc_commit(&bars->empty_a[sa[p]]);
                        ia += P;
                    }
                    if (!begins || c == chunks - 1) {
                        tc_commit(&bars->acc_full[ph & 1]);
                        ++ph;
                    }
                }
                if (resident && (at.j == a.tiles_n - 1 || t == pairs - 1))
                    for (int s = 0; s < chunks * P; ++s)
                        tc_commit(&bars->empty_a[s]);
            }
            if (!ok)
                atomicOr(a.status, kStatusTimeoutBit);
        }
    } else {
        // ---- epilogue: thread = query row of the tile and its columns, or half of them
        constexpr int kHalves = kEpiWarps / 4, kCap = list_keys(KPL, KR);
        constexpr int kCols = kTile / kHalves;
        const int quad = warp & 3;         // a warp reads its own quarter of the TMEM lanes
        const int half = (warp - 2) >> 2;  // warps 2..5 the first half of the columns, 6..9 the second
        const int m = quad * 32 + lane;
        const uint32_t my_lane = tmem + (static_cast<uint32_t>(quad * 32) << 16) + half * kCols;
        const float nmax = __uint_as_float(*a.nmax);
        float coef = 0.f;
        // the `keep` best scores in best[KR - keep .. KR), ascending; the places
        // below never take one
        const int keep = SPLIT ? (a.k + 1) / 2 : a.k;
        float best[KR];
        float other = INFINITY;  // SPLIT: the other half's last one
        // scores up to thr pass (all, when it is NaN), but of those equal to cut, the
        // list's last score at its last compaction, only in groups of columns that
        // begin below cut_id (a few more than could enter)
        float thr = 0.f, slack = 0.f, cut = 0.f;
        uint32_t cut_id = 0;
        int cnt = 0;
        uint32_t self = 0xffffffffu;
        int64_t list = -1;
        int seg = 0;
        uint64_t *mine = nullptr;
        unsigned ph = 0;
        bool ok = true, pad = false;
        if (half == 0)
            sthr[m] = sthr[kTile + m] = 0xffffffffu;
        auto end_list = [&]() {
            if (list >= 0)
                a.ends[list] = make_uint2(static_cast<uint32_t>(cnt), __float_as_uint(thr));
        };
        TileWalk at(a, t0);
        for (int t = 0; t < pairs && ok; ++t, at.next(a)) {
            const bool fresh = t == 0 || at.j == 0;
            if (fresh) {
                end_list();
                if (t != 0)
                    ++seg;
                const int64_t tm = at.tm, row = tm * kTile + m;
                list = row * a.slots + kHalves * (blockIdx.x - cta_of_tile(tm * a.tiles_n / a.unit, T, G)) + half;
                mine = a.lists + list * kCap;
                // what the block of base rows before this one left (none: -1, NaN).
                // Its k best scores are not kept: the threshold stays at
                // theirs until k better ones have come
                const uint2 end = a.ends[list];
                cnt = max(static_cast<int>(end.x), 0);
#pragma unroll
                for (int i = 0; i < KR; ++i)
                    best[i] = i < KR - keep ? -INFINITY : INFINITY;
                // an infinite query's products, whatever their size, stand for
                // infinities of their sign; a NaN's scores are all NaN, so that
                // the ids decide
                const float nx = row < a.rows ? a.nx[row] : 0.f;
                coef = nx == nx ? (isinf(nx) ? -FLT_MAX : a.ip ? -1.f : -2.f) : nx;
                slack = score_slack(nx, nmax, a.dim, a.ip);
                self = a.self ? static_cast<uint32_t>(a.row0 + row) : 0xffffffffu;
                if constexpr (SPLIT) {  // read after the meeting below
                    other = INFINITY;
                    sthr[half * kTile + m] = __float_as_uint(INFINITY);
                }
                pad = row >= a.rows;  // a padding row: no score is below its threshold
                thr = pad ? -INFINITY : __uint_as_float(end.y);
                cut = __int_as_float(0x7fffffff);
                cut_id = 0;
            }
            uint32_t *shared_thr = sthr + (seg & 1) * kTile;
            const int b = t & 1;
            const int64_t c0 = static_cast<int64_t>(at.tn) * kTile;
            if (half == 0) {
                // (a NaN distance is ordered as -0: so is the score)
                const float ny = c0 + m < a.n ? a.ny[c0 + m] : INFINITY;
                sny[b * kTile + m] = c0 + m < a.n && (a.ip || ny != ny) ? 0.f : ny < FLT_MAX ? ny : INFINITY;
            }
            const int width = static_cast<int>(min(static_cast<int64_t>(kTile), a.n - c0)) - half * kCols;
            // a phase's sums for 32 columns
            auto sums = [&](int cc, bool two, float (&v)[32]) {
                uint32_t x[32];
                if constexpr (P == 1) {
                    tmem_load_start(my_lane + static_cast<int>(ph & 1) * 128 + cc, x);
                    tmem_wait();
                    tmem_landed(x);
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        v[j] = __uint_as_float(x[j]);
                } else {
                    const int r = static_cast<int>(3 * ph & 3);
                    if constexpr (KR >= 64) {  // few registers left: one after another
                        tmem_ld32(my_lane + ((r + 1) & 3) * 128 + cc, v);
                        float w[32];
                        if (two) {
                            tmem_ld32(my_lane + ((r + 2) & 3) * 128 + cc, w);
#pragma unroll
                            for (int j = 0; j < 32; ++j)
                                v[j] += w[j];
                        }
                        tmem_ld32(my_lane + r * 128 + cc, w);
#pragma unroll
                        for (int j = 0; j < 32; ++j)
                            v[j] += w[j];
                        return;
                    }
                    uint32_t y[32], z[32];
                    tmem_load_start(my_lane + ((r + 1) & 3) * 128 + cc, x);
                    if (two)
                        tmem_load_start(my_lane + ((r + 2) & 3) * 128 + cc, y);
                    tmem_load_start(my_lane + r * 128 + cc, z);
                    tmem_wait();
                    tmem_landed(x);
                    tmem_landed(z);
                    if (two) {
                        tmem_landed(y);
#pragma unroll
                        for (int j = 0; j < 32; ++j)
                            v[j] = (__uint_as_float(x[j]) + __uint_as_float(y[j])) + __uint_as_float(z[j]);
                    } else {
#pragma unroll
                        for (int j = 0; j < 32; ++j)
                            v[j] = __uint_as_float(x[j]) + __uint_as_float(z[j]);
                    }
                }
            };
            auto phase_ready = [&]() {
                // the epilogue warps go on, or give up, together; their meeting
                // also orders sny's and sthr's writes before their reads
                const int dead =
                    mbar_wait_bounded(&bars->acc_full[ph & 1], static_cast<uint32_t>((ph >> 1) & 1), kTcWaitIters) ? 0 : 1;
                int any;
                asm volatile(
                    "{\n\t.reg .pred p, q;\n\tsetp.ne.s32 p, %1, 0;\n\t"
                    "bar.red.or.pred q, 1, %2, p;\n\tselp.s32 %0, 1, 0, q;\n\t}"
                    : "=r"(any)
                    : "r"(dead), "n"(32 * kEpiWarps)
                    : "memory");
                ok = any == 0;
                tc_fence_after();
                return ok;
            };
            auto phase_read = [&]() {
                tc_fence_before();
                __syncwarp();
                if (lane == 0)
                    mbar_arrive(&bars->acc_empty[ph & 1]);
                ++ph;
            };
            // short of k scores, everything passes still
            auto lower_thr = [&]() {
                const float kth = SPLIT ? fmaxf(best[KR - 1], other) : best[KR - 1];
                thr = kth < INFINITY ? fminf(thr, kth + slack) : thr;
            };
            // SPLIT, any time after the tile's first meeting: the halves' last scores.
            // A half sets its word back before the next query tile's first meeting,
            // at which this one must be too.
            auto exchange = [&]() {
                volatile uint32_t *word = sthr;
                word[half * kTile + m] = __float_as_uint(best[KR - 1]);
                other = fminf(other, __uint_as_float(word[(half ^ 1) * kTile + m]));
                lower_thr();
            };
            auto score = [&](int cc, float (&s)[32]) {
                const float4 *ny4 = reinterpret_cast<const float4 *>(sny + b * kTile + half * kCols + cc);
                float lo = INFINITY;
#pragma unroll
                for (int g = 0; g < 8; ++g) {
                    const float4 y = ny4[g];
                    s[4 * g] = fmaf(coef, s[4 * g], y.x);
                    s[4 * g + 1] = fmaf(coef, s[4 * g + 1], y.y);
                    s[4 * g + 2] = fmaf(coef, s[4 * g + 2], y.z);
                    s[4 * g + 3] = fmaf(coef, s[4 * g + 3], y.w);
                    lo = fminf(lo, fminf(fminf(s[4 * g], s[4 * g + 1]), fminf(s[4 * g + 2], s[4 * g + 3])));
                }
                if (!__any_sync(kFull, !(lo > thr)))
                    return;
                if constexpr (SPLIT)
                    exchange();
                // the columns that pass, then every lane its own one after
                // another: a few turns, not one for every column that passes
                // in some lane
                const uint32_t id0 = static_cast<uint32_t>(a.col0 + c0) + half * kCols + cc;
                // past cut_id, scores below the cut: up to the float before it
                const float most = thr == cut && id0 >= cut_id && thr > -INFINITY ? ord_to_f32(f32_to_ord(thr) - 1) : thr;
                unsigned todo = 0;
#pragma unroll
                for (int j = 0; j < 32; ++j)
                    todo |= (s[j] > most ? 0u : 1u) << j;
                if (width - cc < 32)
                    todo &= width > cc ? (1u << (width - cc)) - 1u : 0u;
                if (self - id0 < 32)
                    todo &= ~(1u << (self - id0));
                const unsigned full = __ballot_sync(kFull, cnt + __popc(todo) > kCap);
                if (full) {
                    const ListEnd end = compact_rows<kCap / 32, 32 * KPL>(full, cnt, mine, cut, cut_id);
                    cnt = end.cnt;
                    cut = end.score;
                    cut_id = end.id;
                    thr = fminf(thr, cut);  // a NaN gives way
                }
                while (__any_sync(kFull, todo != 0)) {
                    const int j = __ffs(todo) - 1;
                    float h[16];
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        h[i] = j & 16 ? s[16 + i] : s[i];
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        h[i] = j & 8 ? h[8 + i] : h[i];
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        h[i] = j & 4 ? h[4 + i] : h[i];
#pragma unroll
                    for (int i = 0; i < 2; ++i)
                        h[i] = j & 2 ? h[2 + i] : h[i];
                    float x = j & 1 ? h[1] : h[0];
                    if (todo != 0 && !(x > thr)) {
                        mine[cnt++] = score_key(x, id0 + j);
                        x = x == x ? x : INFINITY;
#pragma unroll
                        for (int i = 0; i < KR; ++i) {
                            const float lower = fminf(best[i], x);
                            x = fmaxf(best[i], x);
                            best[i] = lower;
                        }
                        lower_thr();
                    }
                    todo &= todo - 1;
                }
            };
            // After the tile's first meeting: nobody reads the other copy of the
            // shared thresholds any more, the next query tile's.
            auto begin = [&]() {
                if constexpr (SPLIT) {
                    exchange();
                } else {
                    if (fresh && half == 0)
                        sthr[((seg & 1) ^ 1) * kTile + m] = 0xffffffffu;
                    if (thr == thr && !pad)
                        atomicMin(shared_thr + m, f32_to_ord(thr));
                    const uint32_t o = shared_thr[m];
                    if (o != 0xffffffffu)
                        thr = fminf(thr, ord_to_f32(o));  // a NaN gives way
                }
            };
            if constexpr (!MULTI) {
                if (!phase_ready())
                    break;
                begin();
#pragma unroll 1
                for (int cc = 0; cc < kCols; cc += 32) {
                    float v[32];
                    sums(cc, chunks > 1, v);
                    if (cc == kCols - 32)
                        phase_read();
                    score(cc, v);
                }
            } else {
                float tot[kCols / 32][32];
                for (int c = 0; c < chunks && ok; c += 2) {
                    if (!phase_ready())
                        break;
                    if (c == 0)
                        begin();
#pragma unroll
                    for (int q = 0; q < kCols / 32; ++q) {
                        float v[32];
                        sums(32 * q, c + 1 < chunks, v);
#pragma unroll
                        for (int j = 0; j < 32; ++j)
                            tot[q][j] = c == 0 ? v[j] : tot[q][j] + v[j];
                    }
                    phase_read();
                }
                if (!ok)
                    break;
#pragma unroll
                for (int q = 0; q < kCols / 32; ++q)
                    score(32 * q, tot[q]);
            }
        }
        end_list();
        if (!ok && lane == 0)
            atomicOr(a.status, kStatusTimeoutBit);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// rows [r0, r0 + rows) of src, whose norms (norms_kernel) are norm[0, rows), as
// packed images [tile][chunk][plane], one 16-byte piece (8 coordinates of a row)
// of all planes per thread.  Infinite coordinates are packed as +-2^100, which
// decides a score's sign as they do (an infinity itself times another row's zero
// planes is NaN), in a query with the others as zero; a row with a NaN as zero.
template <typename S, int P>
__global__ void __launch_bounds__(256)
    pack_kernel(const S *src, const float *norm, bool query, int64_t r0, int64_t rows, int dim, int chunks, uint8_t *out)
{
    const int64_t total = (rows + kTile - 1) / kTile * chunks * (kTile * 8);
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < total;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t img = i / (kTile * 8);
        const int c = static_cast<int>(i % (kTile * 8));
        const int64_t r = img / chunks * kTile + (c >> 6) * 8 + (c & 7);
        const int k = static_cast<int>(img % chunks) * 64 + ((c >> 3) & 7) * 8;
        float x[8];
#pragma unroll
        for (int j = 0; j < 8; ++j)
            x[j] = 0.f;
        if (r < rows && k < dim) {
            const S *p = src + (r0 + r) * dim + k;  // dim % 4 == 0: whole 4-coordinate pieces
            if constexpr (sizeof(S) == 4) {
                const float4 u = *reinterpret_cast<const float4 *>(p);
                x[0] = u.x, x[1] = u.y, x[2] = u.z, x[3] = u.w;
                if (k + 4 < dim) {
                    const float4 w = *reinterpret_cast<const float4 *>(p + 4);
                    x[4] = w.x, x[5] = w.y, x[6] = w.z, x[7] = w.w;
                }
            } else {
                const uint2 u = *reinterpret_cast<const uint2 *>(p);  // dim % 16 == 0
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    x[j] = static_cast<float>(((j < 4 ? u.x : u.y) >> (8 * (j & 3))) & 0xffu);
            }
            if (sizeof(S) == 4 && !isfinite(norm[r])) {
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    x[j] = !isinf(norm[r]) ? 0.f : isinf(x[j]) ? copysignf(0x1p100f, x[j]) : query ? 0.f : x[j];
            }
        }
        __nv_bfloat16 h[P][8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            // high + middle + low == x exactly (a value that would round to
            // infinity is cut instead)
            __nv_bfloat16 hi = __float2bfloat16_rn(x[j]);
            if (isinf(__bfloat162float(hi)))
                hi = __float2bfloat16_rz(x[j]);
            h[0][j] = hi;
            if constexpr (P == 3) {
                const float r1 = x[j] - __bfloat162float(hi);
                h[1][j] = __float2bfloat16_rn(r1);
                h[2][j] = __float2bfloat16_rn(r1 - __bfloat162float(h[1][j]));
            }
        }
#pragma unroll
        for (int p = 0; p < P; ++p)
            *reinterpret_cast<uint4 *>(out + (img * P + p) * kImage + c * 16) = *reinterpret_cast<const uint4 *>(h[p]);
    }
}

// squared norms of rows (exact whole numbers for uint8 rows): NaN where a
// coordinate is NaN, else infinity where one is infinite, else finite (the
// largest float where the sum passes it); and the bits of the finite ones'
// maximum (norms are never negative, so the bits order them)
template <typename S>
__global__ void __launch_bounds__(256) norms_kernel(const S *x, int64_t rows, int dim, float *out, unsigned *nmax)
{
    __shared__ float best[8];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    float mx = 0.f;
    for (int64_t r = blockIdx.x * 8ll + w; r < rows; r += gridDim.x * 8ll) {
        float s = 0.f;
        for (int c = lane; c < dim; c += 32) {
            const float v = static_cast<float>(x[r * dim + c]);
            s = fmaf(v, v, s);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            s += __shfl_xor_sync(kFull, s, o);
        if constexpr (sizeof(S) == 4) {
            if (isinf(s)) {  // every lane has the sum
                bool inf = false;
                for (int c = lane; c < dim; c += 32)
                    inf |= isinf(x[r * dim + c]);
                if (!__any_sync(kFull, inf))
                    s = FLT_MAX;
            }
        }
        if (lane == 0)
            out[r] = s;
        mx = fmaxf(mx, isfinite(s) ? s : 0.f);
    }
    if (lane == 0)
        best[w] = mx;
    __syncthreads();
    if (threadIdx.x == 0 && nmax) {
        for (int i = 1; i < 8; ++i)
            mx = fmaxf(mx, best[i]);
        atomicMax(nmax, __float_as_uint(mx));
    }
}

// Exact distance of uint8 base row x to query q by four lanes (u = 0..3: words
// 4c + u); the whole warp must call it.
__device__ __forceinline__ uint32_t quad_dist_u8(const uint8_t *x, const uint8_t *q, int dim, int u)
{
    const uint32_t *x4 = reinterpret_cast<const uint32_t *>(x), *q4 = reinterpret_cast<const uint32_t *>(q);
    uint32_t acc = 0;
    for (int c = u; c < dim / 4; c += 4) {
        const uint32_t d = __vabsdiffu4(x4[c], q4[c]);
        acc = __dp4a(d, d, acc);
    }
    acc += __shfl_xor_sync(kFull, acc, 1);
    acc += __shfl_xor_sync(kFull, acc, 2);
    return acc;
}

// Exact distances of eight FP32 base rows (ids in the low words of cand[0, 8),
// the last of `have` standing for those past it) to query q, four lanes a row:
// lane 4 j + u sums row j's coordinates 4c + u in order, as one thread with four
// accumulators would, and the four sums are added as (0 + 1) + (2 + 3).  The
// rows come through shared memory, 128 coordinates at a time: read in place, a
// warp's load takes 16 bytes from each of eight rows, and L1's lines bound the
// kernel (77 % of its throughput; 50,000 queries, k = 64, d = 128: 1,717 -> 1,644
// us).  Rows are 132 floats apart, so that the reads meet 32 banks.  The whole
// warp must call it.
template <int MT>
__device__ __forceinline__ uint32_t eight_dists(const float *base, int dim, const float *q, const uint64_t *cand,
                                                int have, float (*tile)[132], int lane)
{
    const int j = lane >> 2, u = lane & 3;
    float s = 0.f;
    for (int t = 0; t < dim; t += 128) {
        const int at = t + 4 * lane;
        __syncwarp();
        if (at < dim) {
            float4 v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i)
                v[i] = *reinterpret_cast<const float4 *>(
                    base + static_cast<int64_t>(static_cast<int32_t>(static_cast<uint32_t>(cand[min(i, have - 1)]))) * dim +
                    at);
#pragma unroll
            for (int i = 0; i < 8; ++i)
                *reinterpret_cast<float4 *>(&tile[i][4 * lane]) = v[i];
            *reinterpret_cast<float4 *>(&tile[8][4 * lane]) = *reinterpret_cast<const float4 *>(q + at);
        }
        __syncwarp();
        const int len = min(128, dim - t);
#pragma unroll 8
        for (int c = u; c < len; c += 4) {
            if constexpr (MT == ANN_L2) {
                const float d = tile[j][c] - tile[8][c];
                s = fmaf(d, d, s);
            } else {
                s = fmaf(tile[j][c], tile[8][c], s);
            }
        }
    }
    s += __shfl_xor_sync(kFull, s, 1);
    s += __shfl_xor_sync(kFull, s, 2);
    if constexpr (MT == ANN_IP)
        s = -s;
    return f32_to_ord(s);
}

// One warp per query: the 32 KPL best candidates of its lists (those above the
// smallest of their thresholds cannot be among the k nearest and are passed
// over, the rest sorted and merged 32 at a time), of which those that the
// scores' errors leave in question (the first ones: all below the k-th best
// score plus the slack) are re-scored exactly and sorted by (distance, id).
// Few queries have many lists, one or two of every CTA of the chip: then WARPS of
// a CTA share a query's lists, and the first merges what the others kept (one
// query, k = 64, 200,000 x 960: whole call 3,610 us by one warp, 1,650 us by sixteen).
template <int DT, int MT, int KPL, int WARPS>
__global__ void __launch_bounds__(WARPS == 1 ? 128 : 32 * WARPS)
    rescore_kernel(const uint8_t *base, int rowbytes, const uint8_t *queries, int qbytes, int dim, int64_t rows,
                   const uint64_t *lists, const uint2 *ends, int slots, int cap, const float *nx, const unsigned *nmax,
                   int k, int32_t *out_ids, void *out_dists)
{
    constexpr int KP = 32 * KPL;
    constexpr int kQueries = WARPS == 1 ? 4 : 1;
    __shared__ uint64_t sh[kQueries * WARPS][KP];  // first the candidates not yet merged, fewer than 64
    __shared__ __align__(16) float tile[DT == ANN_U8 ? 1 : kQueries][9][132];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t r = WARPS == 1 ? blockIdx.x * 4ll + w : blockIdx.x;
    if (r >= rows)
        return;
    float low = __int_as_float(0x7fffffff);
    for (int s = lane; s < slots; s += 32)
        low = fminf(low, __uint_as_float(ends[r * slots + s].y));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        low = fminf(low, __shfl_xor_sync(kFull, low, o));
    uint64_t T[KPL];
#pragma unroll
    for (int i = 0; i < KPL; ++i)
        T[i] = kKeyMax;
    int nq = 0;
    auto merge = [&]() {
        __syncwarp();
        const uint64_t v = warp_sort32(lane < nq ? sh[w][lane] : kKeyMax, lane);
        const uint64_t rest = lane + 32 < nq ? sh[w][32 + lane] : kKeyMax;
        __syncwarp();
        sh[w][lane] = rest;
        nq = nq > 32 ? nq - 32 : 0;
        merge_sorted<KPL>(T, v, lane);
        __syncwarp();
    };
    for (int s = WARPS == 1 ? 0 : w; s < slots; s += WARPS) {
        const uint2 end = ends[r * slots + s];
        const int len = static_cast<int>(end.x) < 0 ? 0 : static_cast<int>(end.x);  // -1: no list
        const uint64_t *L = lists + (r * slots + s) * cap;
        for (int i = 0; i < len; i += 32) {
            const uint64_t v = i + lane < len ? L[i + lane] : kKeyMax;
            const bool in = v != kKeyMax && !(ord_to_f32(static_cast<uint32_t>(v >> 32)) > low);
            const unsigned b = __ballot_sync(kFull, in);
            if (in)
                sh[w][nq + __popc(b & lanemask_lt())] = v;
            nq += __popc(b);
            if (nq >= 32)
                merge();
        }
    }
    if (nq > 0)
        merge();
    __syncwarp();
    if constexpr (WARPS > 1) {
#pragma unroll
        for (int i = 0; i < KPL; ++i)
            sh[w][32 * i + lane] = T[i];
        __syncthreads();
        if (w > 0)
            return;
        for (int v = 1; v < WARPS; ++v) {
#pragma unroll 1
            for (int i = 0; i < KP && sh[v][i] != kKeyMax; i += 32)
                merge_sorted<KPL>(T, sh[v][i + lane], lane);
        }
    }
    uint64_t kth = kKeyMax;
#pragma unroll
    for (int i = 0; i < KPL; ++i) {
        const uint64_t x = __shfl_sync(kFull, T[i], (k - 1) & 31);
        if (i == (k - 1) >> 5)
            kth = x;
    }
    const float edge = ord_to_f32(static_cast<uint32_t>(kth >> 32)) +
                       score_slack(nx[r], __uint_as_float(*nmax), dim, MT == ANN_IP);
    int ns = 0;
#pragma unroll
    for (int i = 0; i < KPL; ++i) {
        const bool in = T[i] != kKeyMax && (kth == kKeyMax || T[i] <= kth ||
                                            !(ord_to_f32(static_cast<uint32_t>(T[i] >> 32)) > edge));
        ns += __popc(__ballot_sync(kFull, in));
        sh[w][32 * i + lane] = T[i];
    }
    __syncwarp();
    const uint8_t *q = queries + r * qbytes;
    for (int c0 = 0; c0 < ns; c0 += 8) {
        const int c = c0 + (lane >> 2);
        const int32_t id = static_cast<int32_t>(static_cast<uint32_t>(sh[w][min(c, ns - 1)]));
        uint32_t bits;
        if constexpr (DT == ANN_U8)
            bits = quad_dist_u8(base + static_cast<int64_t>(id) * rowbytes, q, dim, lane & 3);
        else
            bits = eight_dists<MT>(reinterpret_cast<const float *>(base), dim, reinterpret_cast<const float *>(q),
                                   sh[w] + c0, ns - c0, tile[w], lane);
        __syncwarp();
        if (c < ns && (lane & 3) == 0)
            sh[w][c] = make_key(bits, id);
        __syncwarp();
    }
    uint64_t key[KPL];
#pragma unroll
    for (int i = 0; i < KPL; ++i)
        key[i] = 32 * i + lane < ns ? sh[w][32 * i + lane] : kKeyMax;
    if (ns <= 32)
        key[0] = warp_sort32(key[0], lane);
    else
        warp_sort_rolled<KPL>(key, lane);
#pragma unroll
    for (int i = 0; i < KPL; ++i) {
        const int e = 32 * i + lane;
        if (e < k) {
            const uint64_t v = key[i];
            const bool ok = v != kKeyMax;
            out_ids[r * k + e] = ok ? key_id(v) : -1;
            const uint32_t db = static_cast<uint32_t>(v >> 32);
            if constexpr (DT == ANN_U8)
                reinterpret_cast<int32_t *>(out_dists)[r * k + e] = ok ? static_cast<int32_t>(db) : INT32_MAX;
            else
                reinterpret_cast<float *>(out_dists)[r * k + e] = ok ? ord_to_f32(db) : __int_as_float(0x7f800000);
        }
    }
}

struct Scratch {
    void *p = nullptr;
    cudaStream_t s;
    explicit Scratch(cudaStream_t st) : s(st) {}
    cudaError_t alloc(size_t bytes) { return builder_alloc(&p, bytes, s); }
    template <typename T>
    T *as() const
    {
        return static_cast<T *>(p);
    }
    ~Scratch()
    {
        if (p)
            cudaFreeAsync(p, s);
    }
};

#define KNN_CK(x)                        \
    do {                                 \
        cudaError_t e_ = (x);            \
        if (e_ != cudaSuccess)           \
            return cuda_status(e_);      \
    } while (0)

unsigned pack_grid(int64_t rows, int chunks)
{
    return static_cast<unsigned>(
        std::min<int64_t>(((rows + kTile - 1) / kTile * chunks * (kTile * 8) + 255) / 256, 152 * 32));
}

template <typename S, int P, int KPL, int KR, bool SPLIT>
ann_status knn_typed(const S *base, int64_t n, int dim, int metric, const S *queries, int64_t nq, int k,
                     bool exclude_self, int32_t *d_ids, void *d_dists, cudaStream_t s)
{
    constexpr int kCap = list_keys(KPL, KR), kShare = 16;
    const int chunks = (dim + 63) / 64;
    const size_t tile_bytes = static_cast<size_t>(chunks) * P * kImage;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    auto kern = chunks > 2 ? knn_tile_kernel<P, KPL, KR, SPLIT, true> : knn_tile_kernel<P, KPL, KR, SPLIT, false>;
    KNN_CK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kKnnSmem));
    // blocks of base rows and of queries whose packed images stay within 1 GB
    // and 256 MB, and of queries whose lists stay within 512 MB
    auto whole_tiles = [](int64_t rows) { return std::max<int64_t>(1, rows / kTile) * kTile; };
    const int64_t nb = std::min(whole_tiles((int64_t{1} << 30) / static_cast<int64_t>(tile_bytes) * kTile),
                                (n + kTile - 1) / kTile * kTile);
    const int64_t nblocks = (n + nb - 1) / nb;
    int64_t qb = std::min(whole_tiles((int64_t{256} << 20) / static_cast<int64_t>(tile_bytes) * kTile),
                          (nq + kTile - 1) / kTile * kTile);
    // lists a query has: one for each of a tile's column halves and each CTA that
    // shares its query tile
    auto unit_of = [&](int64_t tm, int64_t tn) { return tm >= 8 * int64_t{sms} ? tn : int64_t{1}; };
    auto grid_of = [&](int64_t tm, int64_t tn) { return std::min<int64_t>(sms, tm * tn / unit_of(tm, tn)); };
    auto slots_of = [&](int64_t tm, int64_t tn) {
        const int64_t T = tm * tn, G = grid_of(tm, tn);
        int64_t most = 1;
        if (unit_of(tm, tn) == 1)
            for (int64_t i = 0; i < tm; ++i)
                most = std::max(most, cta_of_tile((i + 1) * tn - 1, T, G) - cta_of_tile(i * tn, T, G) + 1);
        return most * (kEpiWarps / 4);
    };
    // Base tiles are met by the golden section of their number, all CTAs alike (they
    // share them in L2).  In their own order, rows that lie along a path would
    // come nearer and nearer to a query until its own place, each of them among
    // the best so far (among themselves, 100,000 steps of a random walk, d = 96, k =
    // 64: 273 ms so, 22 here; along a line, k = 100: 412, 19).
    auto scattered = [](int64_t tn) {
        int64_t stride = std::max<int64_t>(1, static_cast<int64_t>(0.6180339887 * static_cast<double>(tn)));
        while (std::gcd(stride, tn) != 1)
            ++stride;
        return stride;
    };
    const int64_t tn_max = nb / kTile;
    for (;;) {
        const int64_t tm = qb / kTile;
        if (tm == 1 || qb * slots_of(tm, tn_max) * kCap * 8 <= (int64_t{512} << 20))
            break;
        qb = whole_tiles(qb / 2);
    }
    Scratch pa(s), pb(s), ny(s), nx(s), lists(s), ends(s), word(s);
    KNN_CK(pa.alloc(qb / kTile * tile_bytes));
    KNN_CK(pb.alloc(nb / kTile * tile_bytes));
    KNN_CK(ny.alloc(n * 4));
    KNN_CK(nx.alloc(qb * 4));
    KNN_CK(word.alloc(8));
    KNN_CK(cudaMemsetAsync(word.p, 0, 8, s));
    unsigned *nmax = word.as<unsigned>();
    int *status = word.as<int>() + 1;
    norms_kernel<S><<<static_cast<unsigned>(std::min<int64_t>((n + 7) / 8, 152 * 8)), 256, 0, s>>>(base, n, dim,
                                                                                                 ny.as<float>(), nmax);
    int64_t packed = -1;  // the block of base rows in pb
    int64_t list_count = 0;
    for (int64_t q0 = 0; q0 < nq; q0 += qb) {
        const int64_t rows = std::min(qb, nq - q0), tm = (rows + kTile - 1) / kTile;
        norms_kernel<S><<<static_cast<unsigned>(std::min<int64_t>((rows + 7) / 8, 152 * 8)), 256, 0, s>>>(
            queries + q0 * dim, rows, dim, nx.as<float>(), nullptr);
        pack_kernel<S, P><<<pack_grid(rows, chunks), 256, 0, s>>>(queries, nx.as<float>(), true, q0, rows, dim, chunks,
                                                                 pa.as<uint8_t>());
        // a query's lists go on from block to block of the base rows (a list of each block's own took memory by their number, which
        // left query blocks of 128 rows that each packed the whole base again:
        // 10,000 queries among 1,000,000 x 960, k = 64, 1,140 ms; 172 ms)
        const int64_t last = n - (nblocks - 1) * nb;
        const int64_t slots = std::max(nblocks > 1 ? slots_of(tm, tn_max) : 1, slots_of(tm, (last + kTile - 1) / kTile));
        const int64_t count = tm * kTile * slots;
        if (count > list_count) {
            for (Scratch *b : {&lists, &ends}) {
                if (b->p)
                    cudaFreeAsync(b->p, s);
                b->p = nullptr;
            }
            KNN_CK(lists.alloc(count * kCap * 8));
            KNN_CK(ends.alloc(count * 8));
            list_count = count;
        }
        KNN_CK(cudaMemsetAsync(ends.p, 0xff, count * 8, s));  // no list: length -1, threshold NaN
        for (int64_t b = 0; b < nblocks; ++b) {
            const int64_t cols = std::min(nb, n - b * nb), tn = (cols + kTile - 1) / kTile;
            if (packed != b) {
                pack_kernel<S, P><<<pack_grid(cols, chunks), 256, 0, s>>>(base, ny.as<float>() + b * nb, false, b * nb,
                                                                         cols, dim, chunks, pb.as<uint8_t>());
                packed = b;
            }
            KnnArgs a{};
            a.A = pa.as<uint8_t>();
            a.B = pb.as<uint8_t>();
            a.chunks = chunks;
            a.ny = ny.as<float>() + b * nb;
            a.nx = nx.as<float>();
            a.nmax = nmax;
            a.n = cols;
            a.col0 = b * nb;
            a.rows = rows;
            a.row0 = q0;
            a.tiles_m = tm;
            a.tiles_n = tn;
            a.unit = unit_of(tm, tn);
            a.stride = scattered(tn);
            a.ip = metric == ANN_IP;
            a.self = exclude_self;
            a.dim = dim;
            a.k = k;
            a.lists = lists.as<uint64_t>();
            a.ends = ends.as<uint2>();
            a.slots = static_cast<int>(slots);
            a.status = status;
            kern<<<static_cast<unsigned>(grid_of(tm, tn)), 64 + 32 * kEpiWarps, kKnnSmem, s>>>(a);
            KNN_CK(cudaGetLastError());
        }
        const int rowbytes = dim * static_cast<int>(sizeof(S));
        const uint8_t *bb = reinterpret_cast<const uint8_t *>(base);
        const uint8_t *qq = reinterpret_cast<const uint8_t *>(queries + q0 * dim);
        int32_t *oi = d_ids + q0 * k;
        void *od = static_cast<uint8_t *>(d_dists) + q0 * k * 4;
        // up to a query an SM, where one warp a query leaves the chip idle (500
        // queries, k = 100: 118 us by one warp each, 150 by sixteen)
        const bool few = rows <= sms;
        auto rescore = [&](auto one, auto shared) {
            (few ? shared : one)<<<static_cast<unsigned>(few ? rows : (rows + 3) / 4), few ? 32 * kShare : 128, 0, s>>>(
                bb, rowbytes, qq, rowbytes, dim, rows, lists.as<uint64_t>(), ends.as<uint2>(), static_cast<int>(slots),
                kCap, nx.as<float>(), nmax, k, oi, od);
        };
        if constexpr (sizeof(S) == 1)
            rescore(rescore_kernel<ANN_U8, ANN_L2, KPL, 1>, rescore_kernel<ANN_U8, ANN_L2, KPL, kShare>);
        else if (metric == ANN_L2)
            rescore(rescore_kernel<ANN_F32, ANN_L2, KPL, 1>, rescore_kernel<ANN_F32, ANN_L2, KPL, kShare>);
        else
            rescore(rescore_kernel<ANN_F32, ANN_IP, KPL, 1>, rescore_kernel<ANN_F32, ANN_IP, KPL, kShare>);
        KNN_CK(cudaGetLastError());
    }
    int failed = 0;
    KNN_CK(cudaMemcpyAsync(&failed, status, 4, cudaMemcpyDeviceToHost, s));
    KNN_CK(cudaStreamSynchronize(s));
    return failed ? ANN_ERR_TIMEOUT : ANN_OK;
}

// k nearest by the kernel with as many scores in registers as k needs, past 32 as
// half of it needs.
template <typename S, int P>
ann_status knn_by_k(const S *base, int64_t n, int dim, int metric, const S *queries, int64_t nq, int k,
                    bool exclude_self, int32_t *d_ids, void *d_dists, cudaStream_t s)
{
    auto run = [&](auto fn) { return fn(base, n, dim, metric, queries, nq, k, exclude_self, d_ids, d_dists, s); };
    if (k == 1)
        return run(knn_typed<S, P, 2, 1, false>);
    if (k <= 16)
        return run(knn_typed<S, P, 2, 16, false>);
    if (k <= 32)
        return run(knn_typed<S, P, 2, 32, false>);
    if (k <= 64)
        return run(knn_typed<S, P, 4, 32, true>);
    return run(knn_typed<S, P, 4, 64, true>);
}

}  // namespace
}  // namespace ann
