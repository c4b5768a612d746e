// search_kernel.cuh -- batched best-first beam search (Sec. 2.1, Algorithm 1) on
// sm_103a: the search kernel, its launch and the count of teams that fit, as
// templates on the storage type and metric.  search_<type>.cu hold the instances;
// search.cu chooses among them and has what surrounds the kernel.
//
// One warp (a "team") serves one query at a time; a persistent grid sized to
// the SM count pulls queries from a device work queue (one atomic counter), so
// queries of uneven cost and per-query (k, L) share one launch.  Optionally
// the queue hands the queries out grouped by their first seed (a counting sort
// by a hash of the seed), so that queries that start at the same node run at
// the same time and share the rows of their first steps in L2.  Per team the
// shared memory holds:
//   - the query row;
//   - a staging area the neighbour rows are gathered into by bulk copies
//     (cp.async.bulk, one 16-byte-aligned row per copy) or tensor gathers (four
//     rows each), completion counted on an mbarrier;
//   - the candidate pool: L 64-bit (distance, id, expanded) keys kept sorted;
//     new candidates are sorted (by counting, or a warp-shuffle bitonic
//     network) and merged in by rank;
//   - optionally, the first level of the visited set (hash_bits > 0).
// The visited set is an exact open-addressing hash (linear probing, key id+1,
// 0 = empty) with up to three levels: the optional shared-memory table, a
// per-team table in global scratch (2^spill_bits slots), and one four times
// larger.  A level that would pass 3/4 load hands its keys to the next one,
// which takes every later insert; only past the last does the query fail
// with a capacity status.  Without a shared table (hash_bits = -1, what the
// tuned configurations use) the set starts in the first global table.
// Semantics follow the sorted-pool reading of Algorithm 1: a seed set (one
// entry by default), a node is visited when its distance is computed, a step
// expands the first W unexpanded pool entries, the pool is truncated to L,
// the search stops when no unexpanded entry is left.  Results are
// independent of the order in which the lanes of a step insert, because the
// pool is the L smallest keys of the union under a total order.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "device_util.cuh"
#include "internal.h"

namespace ann {

constexpr int kFullTeams = 32;      // teams an SM holds at 64 registers a thread
constexpr int kMaxSearchWarps = 2;  // warps (teams) per CTA: 1 or 2, whichever fits more teams
constexpr int kTimeoutIters = 1 << 22;
constexpr int kSlots = ANN_MAX_STEP_CAND / 32;  // most neighbour slots per lane in one step

struct SearchArgs {
    CUtensorMap row_map;  // four-row TMA gathers of base rows (gather4 only)
    int gather4;          // 1: a round's rows come in TMA tensor gathers of four
    int nteams;           // teams of the launch (the first-level tables come first in the scratch)
    const uint8_t *base;
    const int32_t *graph;
    int64_t n;
    int dim, R, rowbytes;
    int R_inv;  // ceil(2^16 / R): (t * R_inv) >> 16 == t / R for all t < 128, 1 <= R <= 128
    const uint8_t *queries;
    int qbytes;
    int qpad;  // zero bytes after the query row in shared memory
    int64_t nq;
    int64_t qdiv;          // work item i reads query row and target i / qdiv
    const int32_t *order;  // optional: the w-th item taken from the queue is order[w]
    const int32_t *entries;
    int32_t medoid;
    int L, k, W;
    int n_entries;   // seeds per query in entries[] (1 when entries is null: the medoid)
    int fault_wait;  // fault injection: every bulk-copy wait gives up at once
    const int32_t *dk, *dL, *dtarget;
    int32_t *out_ids;
    void *out_dists;
    int32_t *out_stats;
    int32_t *pool_out;  // optional: the whole final pool (nq x L ids, -1 padded)
    int *status;
    unsigned long long *counter;
    uint32_t *spill;
    int hash_bits, spill_bits;
    int spill_by_query;  // 1: a query's first global table is sized by its own L (within spill_bits)
    // per-warp shared-memory layout (byte offsets)
    int off_sel, off_q, off_stage, off_pool, off_ptop, off_cbuf, off_hash, per_warp;
    int stage_rows, stage_stride;
    int team_lg;  // log2 of the lanes computing one distance
};

// log2 slots of a first global visited table that holds 40 evaluations per
// pool slot below 3/4 load (about 3x the typical count), 12..15: small enough
// to stay mostly L2-resident and cheap to clear
__host__ __device__ inline int spill_bits_for(int L)
{
    int sb = 12;
    while ((1 << sb) * 3 / 4 < 40 * L && sb < 15)
        ++sb;
    return sb;
}

__device__ __forceinline__ uint32_t hash_slot(uint32_t key, int bits)
{
    return (key * 0x9E3779B1u) >> (32 - bits);
}

// Visited test-and-insert.  Returns 1 when `id` was not yet visited (and is
// now), 0 when it was, -1 when the table is full (cannot happen below the
// load limits the caller enforces).
__device__ __forceinline__ int visit(uint32_t *htab, int hbits, bool global_mode, uint32_t *gtab,
                                     int gbits, int32_t id)
{
    const uint32_t key = static_cast<uint32_t>(id) + 1u;
    if (!global_mode) {
        const uint32_t hmask = (1u << hbits) - 1u;
        uint32_t h = hash_slot(key, hbits);
        for (uint32_t p = 0; p <= hmask; ++p) {
            uint32_t old = atomicCAS(&htab[h], 0u, key);
            if (old == 0u)
                return 1;
            if (old == key)
                return 0;
            h = (h + 1u) & hmask;
        }
        return -1;
    }
    // global mode: the set lives in a global table (after a spill, or from
    // the start when there is no shared table)
    const uint32_t gmask = (1u << gbits) - 1u;
    uint32_t g = hash_slot(key, gbits);
    for (uint32_t p = 0; p <= gmask; ++p) {
        uint32_t old = atomicCAS(&gtab[g], 0u, key);
        if (old == 0u)
            return 1;
        if (old == key)
            return 0;
        g = (g + 1u) & gmask;
    }
    return -1;
}

// Visited test-and-insert for NS ids per lane (-1 = none) in one table.
// res[s] = 1 when ids[s] was not yet visited (and is now), 0 when it was, -1
// when the table is full.  All first probes go out before any result is
// used, and the collision chains of all slots advance together, so their
// latencies overlap.  Concurrent inserts of the same id (from any lane or
// slot) give exactly one 1: every insert of a key walks the same probe
// sequence and the compare-and-swap decides each slot once.
template <int NS>
__device__ __forceinline__ void visit_slots(uint32_t *tab, int bits, const int32_t (&ids)[NS], int (&res)[NS])
{
    const uint32_t mask = (1u << bits) - 1u;
    uint32_t h[NS], key[NS], old[NS];
    // issue every compare-and-swap before looking at any result
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        key[s] = static_cast<uint32_t>(ids[s]) + 1u;
        h[s] = hash_slot(key[s], bits);
        old[s] = ids[s] >= 0 ? atomicCAS(&tab[h[s]], 0u, key[s]) : 0u;
    }
    bool more = false;
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        res[s] = ids[s] < 0 ? 0 : (old[s] == 0u ? 1 : (old[s] == key[s] ? 0 : 2));
        more |= res[s] == 2;
    }
    for (uint32_t p = 1; p <= mask && more; ++p) {
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            if (res[s] == 2) {
                h[s] = (h[s] + 1u) & mask;
                old[s] = atomicCAS(&tab[h[s]], 0u, key[s]);
            }
        }
        more = false;
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            if (res[s] == 2)
                res[s] = old[s] == 0u ? 1 : (old[s] == key[s] ? 0 : 2);
            more |= res[s] == 2;
        }
    }
#pragma unroll
    for (int s = 0; s < NS; ++s)
        if (res[s] == 2)
            res[s] = -1;  // every slot probed: the table is full
}

// Moves every key of the table src (2^sbits slots; in global memory when
// src_global) into the global table dst (2^dbits slots), which is cleared
// first.  The whole warp calls it.
__device__ __forceinline__ void migrate_keys(const uint32_t *src, int sbits, bool src_global, uint32_t *dst,
                                             int dbits, int lane)
{
    for (int o = lane; o < (1 << dbits) / 4; o += 32)
        reinterpret_cast<uint4 *>(dst)[o] = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
    const uint32_t dmask = (1u << dbits) - 1u;
    for (int o = lane; o < (1 << sbits); o += 32) {
        const uint32_t key = src_global ? __ldcg(src + o) : src[o];
        if (key == 0u)
            continue;
        uint32_t g = hash_slot(key, dbits);
        for (uint32_t pr = 0; pr <= dmask; ++pr) {
            if (atomicCAS(&dst[g], 0u, key) == 0u)
                break;
            g = (g + 1u) & dmask;
        }
    }
    __syncwarp();
}

// A running sum over 16-byte chunks of a row against the query's coordinates of
// the same chunk, as every distance form adds them.  int8 rows: chunks of codes
// (from byte 16 on), x_j = scale * code_j.  L2: the sum of (q_j - scale *
// code_j)^2, each difference from one fused multiply-add; IP: the sum of q_j
// code_j, to be scaled.  (The query buffer is zero beyond dim, where the codes
// are zero too.)
template <int DT, int MT>
struct RowSum {
    // four FP32 accumulators (coordinates 4c+0..3) held as two packed pairs:
    // each f32x2 operation rounds both halves exactly as the scalar operations
    // would, at half the instruction count, and the two pairs are independent
    // dependency chains
    uint64_t a = 0, b = 0;  // (0.f, 0.f)
    float scale, c0 = 0.f, c1 = 0.f;  // int8 rows: their scale, and two accumulators

    __device__ __forceinline__ void add4(float x0, float x1, float x2, float x3, float4 y)
    {
        if constexpr (MT == ANN_L2)
            asm("{\n\t.reg .b64 x, y, d;\n\t"
                "mov.b64 x, {%2, %3};\n\tmov.b64 y, {%6, %7};\n\t"
                "sub.rn.f32x2 d, x, y;\n\tfma.rn.f32x2 %0, d, d, %0;\n\t"
                "mov.b64 x, {%4, %5};\n\tmov.b64 y, {%8, %9};\n\t"
                "sub.rn.f32x2 d, x, y;\n\tfma.rn.f32x2 %1, d, d, %1;\n\t}"
                : "+l"(a), "+l"(b)
                : "f"(x0), "f"(x1), "f"(x2), "f"(x3), "f"(y.x), "f"(y.y), "f"(y.z), "f"(y.w));
        else
            asm("{\n\t.reg .b64 x, y;\n\t"
                "mov.b64 x, {%2, %3};\n\tmov.b64 y, {%6, %7};\n\t"
                "fma.rn.f32x2 %0, x, y, %0;\n\t"
                "mov.b64 x, {%4, %5};\n\tmov.b64 y, {%8, %9};\n\t"
                "fma.rn.f32x2 %1, x, y, %1;\n\t}"
                : "+l"(a), "+l"(b)
                : "f"(x0), "f"(x1), "f"(x2), "f"(x3), "f"(y.x), "f"(y.y), "f"(y.z), "f"(y.w));
    }
    __device__ __forceinline__ void add(uint4 x, const uint8_t *q, int c)
    {
        if constexpr (DT == ANN_U8) {
            const uint4 y = reinterpret_cast<const uint4 *>(q)[c];
            uint32_t acc = static_cast<uint32_t>(a), d;  // exact integers in one word
            d = __vabsdiffu4(x.x, y.x);
            acc = __dp4a(d, d, acc);
            d = __vabsdiffu4(x.y, y.y);
            acc = __dp4a(d, d, acc);
            d = __vabsdiffu4(x.z, y.z);
            acc = __dp4a(d, d, acc);
            d = __vabsdiffu4(x.w, y.w);
            a = __dp4a(d, d, acc);
        } else if constexpr (DT == ANN_I8S) {
            const float4 *q4 = reinterpret_cast<const float4 *>(q);
            const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float4 y = q4[4 * c + k];
                const float e0 = static_cast<float>(static_cast<int8_t>(w[k] & 0xffu));
                const float e1 = static_cast<float>(static_cast<int8_t>((w[k] >> 8) & 0xffu));
                const float e2 = static_cast<float>(static_cast<int8_t>((w[k] >> 16) & 0xffu));
                const float e3 = static_cast<float>(static_cast<int8_t>(w[k] >> 24));
                if constexpr (MT == ANN_L2) {
                    const float d0 = fmaf(-scale, e0, y.x), d1 = fmaf(-scale, e1, y.y);
                    const float d2 = fmaf(-scale, e2, y.z), d3 = fmaf(-scale, e3, y.w);
                    c0 = fmaf(d0, d0, c0);
                    c1 = fmaf(d1, d1, c1);
                    c0 = fmaf(d2, d2, c0);
                    c1 = fmaf(d3, d3, c1);
                } else {
                    c0 = fmaf(e0, y.x, c0);
                    c1 = fmaf(e1, y.y, c1);
                    c0 = fmaf(e2, y.z, c0);
                    c1 = fmaf(e3, y.w, c1);
                }
            }
        } else if constexpr (DT == ANN_F32) {
            add4(__uint_as_float(x.x), __uint_as_float(x.y), __uint_as_float(x.z), __uint_as_float(x.w),
                 reinterpret_cast<const float4 *>(q)[c]);
        } else {
            float2 f[4];
            const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if constexpr (DT == ANN_F16)
                    f[i] = __half22float2(*reinterpret_cast<const __half2 *>(&w[i]));
                else
                    f[i] = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&w[i]));
            }
            const float4 *q4 = reinterpret_cast<const float4 *>(q);
            add4(f[0].x, f[0].y, f[1].x, f[1].y, q4[2 * c]);
            add4(f[2].x, f[2].y, f[3].x, f[3].y, q4[2 * c + 1]);
        }
    }
    __device__ __forceinline__ auto sum() const
    {
        if constexpr (DT == ANN_U8)
            return static_cast<uint32_t>(a);
        else if constexpr (DT == ANN_I8S)
            return c0 + c1;
        else
            return (__uint_as_float(static_cast<uint32_t>(a)) + __uint_as_float(static_cast<uint32_t>(a >> 32))) +
                   (__uint_as_float(static_cast<uint32_t>(b)) + __uint_as_float(static_cast<uint32_t>(b >> 32)));
    }
};

// A staged row's chunks: where they start and how many there are.
template <int DT>
__device__ __forceinline__ const uint4 *row_chunks(const uint8_t *row)
{
    return reinterpret_cast<const uint4 *>(row) + (DT == ANN_I8S ? 1 : 0);
}

// One team lane's part of the distance of a staged row to the query: chunks
// first, first + G, ...  CPL > 0: exactly CPL chunks, unrolled so that their
// shared-memory loads issue back to back; CPL = 0: any count.
template <int DT, int MT, int CPL>
__device__ __forceinline__ auto lane_sum(const uint8_t *row, const uint8_t *q, int chunks, int first, int G)
{
    const uint4 *x4 = row_chunks<DT>(row);
    RowSum<DT, MT> acc;
    if constexpr (DT == ANN_I8S)
        acc.scale = *reinterpret_cast<const float *>(row);
    if constexpr (CPL > 0) {
#pragma unroll
        for (int i = 0; i < CPL; ++i)
            acc.add(x4[first + i * G], q, first + i * G);
    } else {
        for (int c = first; c < chunks; c += G)
            acc.add(x4[c], q, c);
    }
    return acc.sum();
}

// How the lanes of a row's distance share the work of its team; each is a
// kernel of its own, so that a launch's kernel holds one form's code (the search
// kernel lives by its instruction cache: with every form in one kernel, a
// launch lost 5 to 10 % to instruction fetches and spills).
enum Form {
    kOne,    // a lane is a team lane
    kOne8,   // the same, exactly 8 chunks each
    kPair4,  // two team lanes, one after the other, exactly 4 chunks each
    kRows2,  // a team lane of two rows at once
    kRows4,  // of four rows at once
};

// Distances of the ch staged rows of the candidates in cbuf[0, ch) by teams of
// G = 2^team_lg >= V lanes that take V rows at once: the query's chunks are read
// once for V rows, the sums are V independent chains, and the lanes halve the
// rows among themselves as the xor-shuffles go (G/2 apart first), so that V rows
// take V + log2(G / V) - 1 of them.  Bit for bit one row at a time.
template <int DT, int MT, int V>
__device__ __forceinline__ void rows_distances(const uint8_t *stage, int stride, const uint8_t *q, int chunks,
                                               uint64_t *cbuf, int ch, int team_lg, int lane)
{
    static_assert((V == 2 || V == 4) && DT != ANN_U8, "float rows, two or four at once");
    const int G = 1 << team_lg, sub = lane & (G - 1), teams = 32 >> team_lg;
    for (int r0 = 0; r0 < ch; r0 += V * teams) {
        int row = r0 + (lane >> team_lg);  // and every teams-th: neighbouring teams read neighbouring rows
        const uint4 *x[V];
#pragma unroll
        for (int v = 0; v < V; ++v)
            x[v] = row_chunks<DT>(stage + min(row + v * teams, ch - 1) * stride);
        RowSum<DT, MT> acc[V];
        if constexpr (DT == ANN_I8S) {
#pragma unroll
            for (int v = 0; v < V; ++v)
                acc[v].scale = *reinterpret_cast<const float *>(x[v] - 1);
        }
        for (int c = sub; c < chunks; c += G) {
#pragma unroll
            for (int v = 0; v < V; ++v)
                acc[v].add(x[v][c], q, c);
        }
        int o = G >> 1;
        const bool odd = lane & o;
        auto half = [&](auto even_sum, auto odd_sum, bool mine) {
            const auto give = mine ? even_sum : odd_sum;
            return (mine ? odd_sum : even_sum) + __shfl_xor_sync(kFull, give, o);
        };
        auto s = half(acc[0].sum(), acc[1].sum(), odd);
        row += odd ? teams : 0;
        if constexpr (V == 4) {
            const auto s2 = half(acc[2].sum(), acc[3].sum(), odd);
            o >>= 1;
            const bool high = lane & o;
            s = half(s, s2, high);
            row += high ? 2 * teams : 0;
        }
        while (o >>= 1)
            s += __shfl_xor_sync(kFull, s, o);
        if constexpr (DT == ANN_I8S && MT == ANN_IP)
            s *= *reinterpret_cast<const float *>(stage + min(row, ch - 1) * stride);
        const uint32_t bits = f32_to_ord(MT == ANN_IP ? -s : s);
        if (row < ch && (sub & (G / V - 1)) == 0)
            cbuf[row] = make_key(bits, key_id(cbuf[row]));
    }
}

// Distance of one staged row to the query by P lanes (a power of two; sub =
// lane % P) that stand for a team of P lanes, or of 2 P (kPair4): bit for bit the
// distance the whole team computes, with fewer shuffles and more rows at once.
// Every lane returns the order-preserving key bits; the whole warp must call it.
template <int DT, int MT, int FORM>
__device__ __forceinline__ uint32_t row_distance(const uint8_t *row, const uint8_t *q, int chunks, int sub, int P)
{
    auto team = [&](auto s) {
        for (int o = P >> 1; o > 0; o >>= 1)
            s += __shfl_xor_sync(kFull, s, o);
        return s;
    };
    if constexpr (DT == ANN_U8) {
        // exact non-negative int32 in any order, ordered as unsigned
        return team(lane_sum<DT, MT, 0>(row, q, chunks, sub, P));
    } else {
        float s;
        if constexpr (FORM == kPair4)
            s = lane_sum<DT, MT, 4>(row, q, chunks, sub, 2 * P) + lane_sum<DT, MT, 4>(row, q, chunks, sub + P, 2 * P);
        else
            s = lane_sum<DT, MT, FORM == kOne8 ? 8 : 0>(row, q, chunks, sub, P);
        s = team(s);
        if constexpr (DT == ANN_I8S && MT == ANN_IP)
            s *= *reinterpret_cast<const float *>(row);
        return f32_to_ord(MT == ANN_IP ? -s : s);
    }
}

// One TMA tensor gather of four whole base rows (row ids r0..r3) into four
// consecutive staging rows at dst, counted on bar.
__device__ __forceinline__ void gather4_rows(void *dst, const CUtensorMap *map, int32_t r0, int32_t r1, int32_t r2,
                                             int32_t r3, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile::gather4.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%2, %3, %4, %5, %6}], [%7];" ::"r"(smem_addr(dst)),
        "l"(map), "r"(0), "r"(r0), "r"(r1), "r"(r2), "r"(r3), "r"(smem_addr(bar))
        : "memory");
}

// NS: neighbour slots per lane in one step, the smallest of 1, 2, 4 that
// holds W * R candidates
template <int DT, int MT, int NS, int FORM>
__global__ void __launch_bounds__(32 * kMaxSearchWarps, 16) beam_search_kernel(const __grid_constant__ SearchArgs a)
{
    extern __shared__ __align__(128) uint8_t smem[];
    const int lane = threadIdx.x & 31;
    const int wid = threadIdx.x >> 5;
    uint8_t *my = smem + wid * a.per_warp;
    uint64_t *bar = reinterpret_cast<uint64_t *>(my);
    int32_t *sel = reinterpret_cast<int32_t *>(my + a.off_sel);
    uint8_t *qbuf = my + a.off_q;
    uint8_t *stage = my + a.off_stage;
    uint64_t *pool = reinterpret_cast<uint64_t *>(my + a.off_pool);
    uint64_t *ptop = reinterpret_cast<uint64_t *>(my + a.off_ptop);  // W keys for the prediction
    uint64_t *cbuf = reinterpret_cast<uint64_t *>(my + a.off_cbuf);
    uint32_t *htab = reinterpret_cast<uint32_t *>(my + a.off_hash);
    const int team = blockIdx.x * (blockDim.x >> 5) + wid;
    // two global spill tables per team: 2^spill_bits slots, then one four
    // times larger for the rare query that outgrows the first; the first
    // tables of all teams lie together at the front of the scratch (one
    // range for an L2 access-policy window), the larger ones after them
    uint32_t *gtab1 = a.spill + static_cast<size_t>(team) * (static_cast<size_t>(1) << a.spill_bits);
    uint32_t *gtab2 = a.spill + static_cast<size_t>(a.nteams) * (static_cast<size_t>(1) << a.spill_bits) +
                      static_cast<size_t>(team) * (static_cast<size_t>(4) << a.spill_bits);

    if (lane == 0) {
        mbar_init(bar, 1);
        fence_mbar_init();
    }
    __syncwarp();
    uint32_t phase = 0;
    // hash_bits < 0: no shared table, the visited set starts in the global one
    const bool shared_tab = a.hash_bits > 0;
    const int hcap = shared_tab ? 1 << a.hash_bits : 0;
    const int hlimit = hcap * 3 / 4;

    for (;;) {
        long long qi = 0;
        if (lane == 0)
            qi = static_cast<long long>(atomicAdd(a.counter, 1ull));
        qi = __shfl_sync(kFull, qi, 0);
        if (qi >= a.nq)
            break;
        if (a.order)
            qi = a.order[qi];

        const int Lq = a.dL ? a.dL[qi] : a.L;
        const int kq = a.dk ? a.dk[qi] : a.k;
        const int64_t qrow = qi / a.qdiv;
        const int32_t target = a.dtarget ? a.dtarget[qrow] : -1;
        // seed set: lane e < n_entries holds seed e (-1 = unused slot)
        const int32_t seed = a.entries ? (lane < a.n_entries ? a.entries[qi * a.n_entries + lane] : -1)
                                       : (lane == 0 ? a.medoid : -1);
        const bool seeds_ok = !__any_sync(kFull, seed < -1 || seed >= a.n) && __any_sync(kFull, seed >= 0);
        bool failed = false;
        bool timed_out = false, lost = false;
        if (Lq < 1 || Lq > a.L || kq < 1 || kq > a.k || kq > Lq || !seeds_ok) {
            failed = true;
            if (lane == 0)
                atomicOr(a.status, kStatusBadInputBit);
        }

        int cnt = 0, cursor = 0, evals = 0, hops = 0;
        // visited set: level 0 = the shared table, 1 and 2 = the global ones;
        // used = keys in the current table, limit = its 3/4 load
        // the first global table's size: the launch's, or the query's own L's,
        // so that a small query of a mixed batch clears and touches a small
        // table (the second one keeps the launch's size, so no query's
        // capacity shrinks), never smaller than the shared one, whose keys it takes
        const int qbits =
            a.spill_by_query ? min(max(spill_bits_for(max(Lq, 1)), a.hash_bits), a.spill_bits) : a.spill_bits;
        int level = shared_tab ? 0 : 1, used = 0, gbits = qbits;
        int limit = shared_tab ? hlimit : (1 << qbits) * 3 / 4;
        uint32_t *gtab = gtab1;
        int32_t *pred = sel + ANN_MAX_W;     // ids of the next selection
        int32_t *src = sel + 2 * ANN_MAX_W;  // where they come from
        int npred = 0;
        int32_t nxt[NS];  // their adjacency rows, lane-distributed like cur[]
#pragma unroll
        for (int r = 0; r < NS; ++r)
            nxt[r] = -1;
        bool found = false;
        if (!failed) {
            // query row -> shared memory; clear the visited table
            const uint8_t *qsrc = a.queries + qrow * a.qbytes;
            for (int o = lane * 16; o < a.qbytes; o += 32 * 16)
                *reinterpret_cast<uint4 *>(qbuf + o) = *reinterpret_cast<const uint4 *>(qsrc + o);
            for (int o = a.qbytes + lane * 4; o < a.qbytes + a.qpad; o += 32 * 4)
                *reinterpret_cast<float *>(qbuf + o) = 0.f;
            for (int o = lane; o < hcap / 4; o += 32)
                reinterpret_cast<uint4 *>(htab)[o] = make_uint4(0u, 0u, 0u, 0u);
            if (!shared_tab)
                for (int o = lane; o < (1 << qbits) / 4; o += 32)
                    reinterpret_cast<uint4 *>(gtab1)[o] = make_uint4(0u, 0u, 0u, 0u);
            __syncwarp();
            // the initial pool: every distinct seed, evaluated in the first step
            const int r = seed >= 0 ? visit(htab, a.hash_bits, !shared_tab, gtab1, qbits, seed) : 0;
            const unsigned nm = __ballot_sync(kFull, r == 1);
            if (r == 1)
                cbuf[__popc(nm & lanemask_lt())] = static_cast<uint64_t>(seed) << 1;
            used = evals = __popc(nm);
            found = __any_sync(kFull, r == 1 && seed == target);
        }
        int nc = failed ? 0 : evals;
        __syncwarp();

        while (!failed) {
            // ---- evaluate the nc candidates in cbuf[] (their ids in the key
            // layout, distance bits 0); the survivors end sorted
            // in cbuf[0, m)
            int m = 0;
            if (nc > 0) {
                for (int c0 = 0; c0 < nc; c0 += a.stage_rows) {
                    const int ch = min(a.stage_rows, nc - c0);
                    if (a.gather4) {
                        // groups of four rows, the last group padded by
                        // repeating its last row
                        const int ng = (ch + 3) >> 2;
                        if (lane == 0)
                            mbar_arrive_expect_tx(bar, static_cast<uint32_t>(ng) * 4 * a.rowbytes);
                        __syncwarp();
                        for (int g = lane; g < ng; g += 32) {
                            const int j = c0 + 4 * g, last = c0 + ch - 1;
                            gather4_rows(stage + 4 * g * a.stage_stride, &a.row_map, key_id(cbuf[j]),
                                         key_id(cbuf[min(j + 1, last)]), key_id(cbuf[min(j + 2, last)]),
                                         key_id(cbuf[min(j + 3, last)]), bar);
                        }
                    } else {
                        if (lane == 0)
                            mbar_arrive_expect_tx(bar, static_cast<uint32_t>(ch) * a.rowbytes);
                        __syncwarp();
                        for (int j = lane; j < ch; j += 32)
                            bulk_g2s(stage + j * a.stage_stride,
                                     a.base + static_cast<size_t>(key_id(cbuf[c0 + j])) * a.rowbytes, a.rowbytes,
                                     bar);
                    }
                    const bool ok = !a.fault_wait && mbar_wait_bounded(bar, phase, kTimeoutIters);
                    if (!__all_sync(kFull, ok)) {
                        // the query fails with a timeout; give the copies one
                        // more bounded wait: if they land, the barrier is in a
                        // known state and the team goes on with the next
                        // query, else it retires
                        const bool landed = __all_sync(kFull, mbar_wait_bounded(bar, phase, kTimeoutIters));
                        if (landed)
                            phase ^= 1u;
                        lost = !landed;
                        timed_out = true;
                        failed = true;
                        break;
                    }
                    phase ^= 1u;
                    // a team of G lanes per staged row, 32 / G rows per pass
                    const int chunks = a.rowbytes / 16 - (DT == ANN_I8S ? 1 : 0);
                    if constexpr (FORM == kRows2 || FORM == kRows4)
                        rows_distances<DT, MT, FORM == kRows2 ? 2 : 4>(stage, a.stage_stride, qbuf, chunks, cbuf + c0,
                                                                       ch, a.team_lg, lane);
                    else for (int r0 = 0; r0 < ch; r0 += 32 >> a.team_lg) {
                        const int r = r0 + (lane >> a.team_lg);
                        const int sub = lane & ((1 << a.team_lg) - 1);
                        const uint32_t bits = row_distance<DT, MT, FORM>(stage + min(r, ch - 1) * a.stage_stride,
                                                                         qbuf, chunks, sub, 1 << a.team_lg);
                        if (r < ch && sub == 0)
                            cbuf[c0 + r] = make_key(bits, key_id(cbuf[c0 + r]));
                    }
                    __syncwarp();
                    fence_proxy_async_smem();  // stage reads done before the next bulk writes
                }
                if (failed)
                    break;
                // candidates no better than a full pool's last entry cannot
                // enter it; only the survivors are sorted
                const uint64_t worst = (cnt == Lq) ? pool[Lq - 1] : kKeyMax;
                uint64_t kk[NS];
                unsigned bm[NS];
#pragma unroll
                for (int s = 0; s < NS; ++s) {
                    uint64_t v = lane + 32 * s < nc ? cbuf[lane + 32 * s] : kKeyMax;
                    if (v >= worst)
                        v = kKeyMax;
                    kk[s] = v;
                    bm[s] = __ballot_sync(kFull, v != kKeyMax);
                    m += __popc(bm[s]);
                }
                __syncwarp();
                if (m > 0) {
                    // up to 32 survivors: a survivor's place is the number of
                    // smaller ones, counted over broadcasts that do not wait
                    // for one another (a bitonic network's stages do)
                    if (NS == 1) {
                        int place = 0;
                        for (unsigned todo = bm[0]; todo; todo &= todo - 1)
                            place += __shfl_sync(kFull, kk[0], __ffs(todo) - 1) < kk[0];
                        if (kk[0] != kKeyMax)
                            cbuf[place] = kk[0];
                    } else {
                        if (m <= 32 || (m <= 64 && nc > 64)) {
                            // compact the survivors into cbuf[0, m) (a 64-key
                            // sort of candidates that all sit in slots 0-1 needs
                            // none: the dropped ones sort to the end)
                            int base = 0;
#pragma unroll
                            for (int s = 0; s < NS; ++s) {
                                if (kk[s] != kKeyMax)
                                    cbuf[base + __popc(bm[s] & lanemask_lt())] = kk[s];
                                base += __popc(bm[s]);
                            }
                            __syncwarp();
                            kk[0] = lane < m ? cbuf[lane] : kKeyMax;
                            if constexpr (NS > 1)
                                kk[1] = lane + 32 < m ? cbuf[lane + 32] : kKeyMax;
                            __syncwarp();
                        }
                        if (m <= 32) {
                            int place = 0;
                            for (int s = 0; s < m; s += 4) {
#pragma unroll
                                for (int u = 0; u < 4; ++u)
                                    place += __shfl_sync(kFull, kk[0], s + u) < kk[0];
                            }
                            if (lane < m)
                                cbuf[place] = kk[0];
                        } else if constexpr (NS > 1) {
                            if (NS == 2 || m <= 64) {
                                uint64_t k2[2] = {kk[0], kk[1]};
                                warp_sort_rolled<2>(k2, lane);
                                cbuf[lane] = k2[0];
                                cbuf[lane + 32] = k2[1];
                            } else if constexpr (NS == 4) {
                                warp_sort_rolled<4>(kk, lane);
#pragma unroll
                                for (int s = 0; s < NS; ++s)
                                    cbuf[lane + 32 * s] = kk[s];
                            }
                        }
                    }
                    __syncwarp();
                }
            }

            // ---- the next selection: the W smallest unexpanded keys among the
            // pool and the survivors, in order.  Their adjacency rows are
            // loaded now, so the loads overlap the merge.
            int from = 0;  // lane r < npred: the r-th one's pool index, or ~j for survivor j
            {
                int nf = 0;
                for (int i0 = cursor; i0 < cnt && nf < a.W; i0 += 32) {
                    const int i = i0 + lane;
                    const uint64_t v = i < cnt ? pool[i] : 1ull;
                    const bool un = !(v & 1ull);
                    const unsigned um = __ballot_sync(kFull, un);
                    const int g = nf + __popc(um & lanemask_lt());
                    if (un && g < a.W) {
                        ptop[g] = v;
                        sel[g] = i;
                    }
                    nf = min(a.W, nf + __popc(um));
                }
                __syncwarp();
                // lane l < nf places the pool's l-th, lane ANN_MAX_W + j the
                // survivors' j-th: its own index plus the other side's smaller ones
                const int mw = min(m, a.W), np = min(a.W, nf + mw);
                const bool mine = lane < ANN_MAX_W;
                const int own = mine ? lane : lane - ANN_MAX_W, other = mine ? mw : nf;
                if (own < (mine ? nf : mw)) {
                    const uint64_t *theirs = mine ? cbuf : ptop;
                    const uint64_t v = mine ? ptop[own] : cbuf[own];
                    int r = own;
#pragma unroll
                    for (int j = 0; j < ANN_MAX_W; ++j)
                        r += j < other && theirs[j] < v;
                    if (r < a.W) {
                        pred[r] = key_id(v);
                        src[r] = mine ? sel[own] : ~own;
                    }
                }
                npred = np;
                __syncwarp();
                from = lane < np ? src[lane] : 0;
                const int tp = npred * a.R;
#pragma unroll
                for (int r = 0; r < NS; ++r) {
                    const int t = lane + 32 * r;
                    const int e = (t * a.R_inv) >> 16;  // t / R
                    nxt[r] = t < tp ? __ldg(a.graph + static_cast<int64_t>(pred[e]) * a.R + (t - e * a.R)) : -1;
                }
            }

            // ---- merge the survivors into the pool by rank, in place: a
            // survivor's place is its index plus the number of pool entries
            // below it.  The places of a block of 32 as a bit mask tell each of
            // its slots where its key comes from: survivors and pool entries
            // both keep their order.  Blocks go from the back, so that no entry
            // is overwritten before it is read; a block costs about a dozen
            // instructions, where a search in the survivors for every pool
            // entry was a chain of loads (100 queries of 10,000 x 128 uint8: 343 us
            // so, 323 us here; 100,000 of 96 fp32 with L up to 512: 30.3, 29.0 ms).
            // (The expanded bit never decides a comparison: keys of different
            // nodes differ above it.)
            int dst0 = Lq;  // lane j < 32: survivor j's place in the pool
            if (m > 0) {
                const int T = min(Lq, cnt + m);
                int dst[NS];
                int left = 0;  // survivors placed below the block's end
#pragma unroll
                for (int r = 0; r < NS; ++r)
                    dst[r] = INT32_MAX;
#pragma unroll 1
                for (int j0 = 0; j0 < m; j0 += 32) {  // one copy of the search in the instruction cache
                    const int j = j0 + lane;
                    const int d = j < m ? j + count_less4(pool, cnt, cbuf[j]) : INT32_MAX;
                    left += __popc(__ballot_sync(kFull, d < T));
#pragma unroll
                    for (int r = 0; r < NS; ++r)
                        if (j0 == 32 * r && d < T)
                            dst[r] = d;
                }
                dst0 = dst[0];
                const int p0 = __shfl_sync(kFull, dst0, 0);  // place of the best survivor
                for (int b = p0 + (T - 1 - p0) / 64 * 64; b >= p0; b -= 64) {
                    unsigned w0 = 0, w1 = 0;
#pragma unroll
                    for (int r = 0; r < NS; ++r) {
                        if (r == 1 && m <= 32)
                            break;
                        const unsigned d = dst[r] - b;
                        w0 |= d < 32 ? 1u << d : 0u;
                        w1 |= d - 32 < 32 ? 1u << (d - 32) : 0u;
                    }
                    w0 = __reduce_or_sync(kFull, w0);
                    w1 = __reduce_or_sync(kFull, w1);
                    const int s1 = left - __popc(w1), s0 = s1 - __popc(w0);  // survivors below each half
                    const int c0 = s0 + __popc(w0 & lanemask_lt()), c1 = s1 + __popc(w1 & lanemask_lt());
                    const int i0 = b + lane, i1 = i0 + 32;
                    uint64_t v0 = 0, v1 = 0;
                    if (i0 < T)
                        v0 = w0 >> lane & 1 ? cbuf[c0] : pool[i0 - c0];
                    if (i1 < T)
                        v1 = w1 >> lane & 1 ? cbuf[c1] : pool[i1 - c1];
                    __syncwarp();
                    if (i0 < T)
                        pool[i0] = v0;
                    if (i1 < T)
                        pool[i1] = v1;
                    __syncwarp();
                    left = s0;
                }
                cnt = T;
            }
            if (found)
                break;

            // ---- mark the selected entries expanded where they are now: a pool
            // entry moved right by the survivors before it, all of them selected
            // too; one that the pool's end cut off takes the later ones with it
            const unsigned late = __ballot_sync(kFull, lane < npred && from < 0);
            const int at_dst = __shfl_sync(kFull, dst0, from < 0 ? ~from : 0);
            const int pos = from < 0 ? at_dst : from + __popc(late & lanemask_lt());
            const bool take = lane < npred && pos < Lq;
            if (take)
                pool[pos] |= 1ull;
            const int ns = __popc(__ballot_sync(kFull, take));
            if (ns == 0)
                break;
            cursor = __shfl_sync(kFull, pos, 0);
            hops += ns;

            const int total = ns * a.R;
            int32_t cur[NS];
#pragma unroll
            for (int r = 0; r < NS; ++r)
                cur[r] = nxt[r];
            __syncwarp();

            // ---- neighbours of the selected entries: visited test, compaction
            // A table that would pass 3/4 load hands its keys to the next,
            // larger one (shared -> global -> 4x larger global), which takes
            // every later insert, so a lookup probes one table only and the
            // set stays exact.
            while (used + total > limit && level < 2) {
                uint32_t *dst = level == 0 ? gtab1 : gtab2;
                const int dbits = level == 0 ? qbits : a.spill_bits + 2;
                if (level == 0)
                    migrate_keys(htab, a.hash_bits, false, dst, dbits, lane);
                else
                    migrate_keys(gtab, gbits, true, dst, dbits, lane);
                gtab = dst;
                gbits = dbits;
                limit = (1 << dbits) * 3 / 4;
                ++level;
            }
            if (used + total > limit) {
                failed = true;
                if (lane == 0)
                    atomicOr(a.status, kStatusCapacityBit);
                break;
            }
            // every slot's first probe is issued before any result is used, so
            // their latencies overlap (global atomics in spill mode)
            int32_t vid[NS];
            int res[NS];
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                const int32_t id = lane + 32 * s < total ? cur[s] : -1;
                vid[s] = (id >= 0 && id < a.n) ? id : -1;
            }
            if (level > 0)
                visit_slots<NS>(gtab, gbits, vid, res);
            else
                visit_slots<NS>(htab, a.hash_bits, vid, res);
            nc = 0;
            bool bad = false;
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                if (32 * s >= total)
                    break;
                bad |= (res[s] < 0);
                const unsigned nm = __ballot_sync(kFull, res[s] == 1);
                if (res[s] == 1) {
                    cbuf[nc + __popc(nm & lanemask_lt())] = static_cast<uint64_t>(static_cast<uint32_t>(vid[s])) << 1;
                    if (vid[s] == target)
                        found = true;
                }
                nc += __popc(nm);
            }
            found = __any_sync(kFull, found);
            if (__any_sync(kFull, bad)) {
                failed = true;
                if (lane == 0)
                    atomicOr(a.status, kStatusCapacityBit);
                break;
            }
            evals += nc;
            used += nc;
            __syncwarp();
        }

        if (timed_out && lane == 0)
            atomicOr(a.status, kStatusTimeoutBit);

        // ---- outputs
        for (int j = lane; j < a.k; j += 32) {
            int32_t id = -1;
            uint32_t db = 0;
            if (!failed && j < kq && j < cnt) {
                const uint64_t v = pool[j];
                id = key_id(v);
                db = static_cast<uint32_t>(v >> 32);
            }
            a.out_ids[qi * a.k + j] = id;
            if constexpr (DT == ANN_U8)
                reinterpret_cast<int32_t *>(a.out_dists)[qi * a.k + j] =
                    id >= 0 ? static_cast<int32_t>(db) : INT32_MAX;
            else
                reinterpret_cast<float *>(a.out_dists)[qi * a.k + j] =
                    id >= 0 ? ord_to_f32(db) : __int_as_float(0x7f800000);
        }
        if (a.pool_out) {
            for (int j = lane; j < a.L; j += 32)
                a.pool_out[qi * a.L + j] = (!failed && j < cnt) ? key_id(pool[j]) : -1;
        }
        if (a.out_stats && lane == 0) {
            const bool miss = failed || (target >= 0 && !found);
            a.out_stats[2 * qi] = miss && target >= 0 ? INT32_MAX : evals;
            a.out_stats[2 * qi + 1] = miss && target >= 0 ? INT32_MAX : hops;
        }
        __syncwarp();
        if (lost)
            return;  // this team's barrier state is unknown: retire it
    }
}

template <int DT, int MT, int FORM>
auto kernel_of_form(int maxc)
{
    return maxc <= 32 ? beam_search_kernel<DT, MT, 1, FORM>
                      : maxc <= 64 ? beam_search_kernel<DT, MT, 2, FORM> : beam_search_kernel<DT, MT, kSlots, FORM>;
}

// The search kernel for steps of up to maxc candidates and a distance form
// (one that search_form gives for the type).
template <int DT, int MT>
auto kernel_for(int maxc, int form)
{
    if constexpr (DT != ANN_U8) {
        if (form == kRows2)
            return kernel_of_form<DT, MT, kRows2>(maxc);
    }
    if constexpr (DT == ANN_F32) {
        if (form == kRows4)
            return kernel_of_form<DT, MT, kRows4>(maxc);
    }
    if constexpr (DT != ANN_U8 && DT != ANN_I8S) {
        if (form == kPair4)
            return kernel_of_form<DT, MT, kPair4>(maxc);
        if (form == kOne8)
            return kernel_of_form<DT, MT, kOne8>(maxc);
    }
    return kernel_of_form<DT, MT, kOne>(maxc);
}

// Resident teams for `per_warp` bytes of shared memory per team, with one or
// two teams per CTA, whichever fits more (each CTA also costs the SM a fixed
// reserve of shared memory, which two teams share).  When one team per CTA
// already holds all nq queries, it is taken: the queries then spread over
// twice as many SMs.
template <int DT, int MT>
ann_status teams_for(ann_index *idx, size_t per_warp, int maxc, int form, int64_t nq, int *teams, int *wpc)
{
    auto kern = kernel_for<DT, MT>(maxc, form);
    // The kernel's limit belongs to the device and not to a launch: always the
    // most a CTA may have, so that a search of another thread never lowers it
    // between this one's look at it and its launch.
    int cta_smem = 0;
    cudaError_t e = cudaDeviceGetAttribute(&cta_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, idx->device);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, cta_smem);
    if (e != cudaSuccess)
        return cuda_status(e);
    int best = 0, best_w = 1;
    for (int w = 1; w <= kMaxSearchWarps; ++w) {
        if (static_cast<int64_t>(best) * idx->num_sms >= nq)
            break;
        const size_t smem = per_warp * w;
        if (smem > static_cast<size_t>(cta_smem))
            break;  // too large for one CTA: not a candidate
        int per_sm = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * w, smem);
        if (e != cudaSuccess)
            return cuda_status(e);
        if (per_sm * w > best) {
            best = per_sm * w;
            best_w = w;
        }
    }
    if (best < 1)
        return ANN_ERR_UNSUPPORTED;  // the per-query state does not fit in shared memory
    *teams = best * idx->num_sms;
    *wpc = best_w;
    return ANN_OK;
}

// window: bytes of the first-level visited tables to keep resident in L2
// (0 = launch without an access-policy window), at the given hit ratio
template <int DT, int MT>
ann_status launch_typed(const SearchArgs &a, int maxc, int form, size_t smem, int teams, int wpc, cudaStream_t s, size_t window,
                        float hit_ratio)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(teams / wpc);
    cfg.blockDim = dim3(32 * wpc);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeAccessPolicyWindow;
    at[0].val.accessPolicyWindow.base_ptr = a.spill;
    at[0].val.accessPolicyWindow.num_bytes = window;
    at[0].val.accessPolicyWindow.hitRatio = hit_ratio;
    at[0].val.accessPolicyWindow.hitProp = cudaAccessPropertyPersisting;
    at[0].val.accessPolicyWindow.missProp = cudaAccessPropertyStreaming;
    cfg.attrs = at;
    cfg.numAttrs = window > 0 ? 1 : 0;
    return cuda_status(cudaLaunchKernelEx(&cfg, kernel_for<DT, MT>(maxc, form), a));
}

// What search.cu calls, per storage type and metric.
#define ANN_SEARCH_INSTANCE(LINKAGE, DT, MT)                                                                    \
    LINKAGE template ann_status teams_for<DT, MT>(ann_index *, size_t, int, int, int64_t, int *, int *);        \
    LINKAGE template ann_status launch_typed<DT, MT>(const SearchArgs &, int, int, size_t, int, int, cudaStream_t, \
                                                     size_t, float);

}  // namespace ann
