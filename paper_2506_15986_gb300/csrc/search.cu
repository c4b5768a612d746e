// search.cu -- batched best-first beam search: what surrounds the search kernel
// (search_kernel.cuh): the work order grouped by seed, the exact rerank of
// reduced-precision storage, and the launch with its choice of sizes.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "search_kernel.cuh"

namespace ann {

ANN_SEARCH_INSTANCE(extern, ANN_U8, ANN_L2)
ANN_SEARCH_INSTANCE(extern, ANN_F32, ANN_L2)
ANN_SEARCH_INSTANCE(extern, ANN_F32, ANN_IP)
ANN_SEARCH_INSTANCE(extern, ANN_F16, ANN_L2)
ANN_SEARCH_INSTANCE(extern, ANN_F16, ANN_IP)
ANN_SEARCH_INSTANCE(extern, ANN_BF16, ANN_L2)
ANN_SEARCH_INSTANCE(extern, ANN_BF16, ANN_IP)
ANN_SEARCH_INSTANCE(extern, ANN_I8S, ANN_L2)
ANN_SEARCH_INSTANCE(extern, ANN_I8S, ANN_IP)

namespace {

// Work order grouped by first seed: a counting sort of the work items by a
// 12-bit hash of their first seed, in one CTA (the histogram and the scatter
// use shared-memory atomics, so items of one bucket come out in no fixed
// order; the search's results do not depend on the order).  Each thread
// reads its items' seeds eight at a time, so their loads are in flight
// together, and keeps the buckets of the first kGroupCache items in shared
// memory for the scatter pass.
constexpr int kGroupThreads = 1024;
constexpr int kGroupBits = 12;
constexpr int kGroupPer = (1 << kGroupBits) / kGroupThreads;  // buckets per thread
constexpr int kGroupBatch = 8;                                 // seeds loaded together per thread
constexpr int kGroupCache = 12288;                             // items whose bucket is kept

__device__ __forceinline__ uint32_t seed_bucket(int32_t e)
{
    return (static_cast<uint32_t>(e) * 0x9E3779B1u) >> (32 - kGroupBits);
}

__global__ void __launch_bounds__(kGroupThreads)
    group_by_seed_kernel(const int32_t *__restrict__ entries, int n_entries, int64_t nitems,
                         int32_t *__restrict__ order)
{
    __shared__ int cnt[1 << kGroupBits];
    __shared__ int wsum[kGroupThreads / 32];
    __shared__ uint16_t bucket_of[kGroupCache];
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    for (int i = t; i < (1 << kGroupBits); i += kGroupThreads)
        cnt[i] = 0;
    __syncthreads();
    // item w = base + j * kGroupThreads + t for j < kGroupBatch
    constexpr int64_t kStride = static_cast<int64_t>(kGroupThreads) * kGroupBatch;
    for (int64_t base = 0; base < nitems; base += kStride) {
        int32_t e[kGroupBatch];
#pragma unroll
        for (int j = 0; j < kGroupBatch; ++j) {
            const int64_t w = base + j * kGroupThreads + t;
            e[j] = w < nitems ? __ldg(entries + w * n_entries) : 0;
        }
#pragma unroll
        for (int j = 0; j < kGroupBatch; ++j) {
            const int64_t w = base + j * kGroupThreads + t;
            if (w < nitems) {
                const uint32_t bk = seed_bucket(e[j]);
                atomicAdd(&cnt[bk], 1);
                if (w < kGroupCache)
                    bucket_of[w] = static_cast<uint16_t>(bk);
            }
        }
    }
    __syncthreads();
    // exclusive scan: thread t owns buckets [kGroupPer t, kGroupPer (t + 1))
    int v[kGroupPer], tot = 0;
#pragma unroll
    for (int j = 0; j < kGroupPer; ++j) {
        v[j] = cnt[kGroupPer * t + j];
        tot += v[j];
    }
    int inc = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o)
            inc += u;
    }
    if (lane == 31)
        wsum[wid] = inc;
    __syncthreads();
    if (wid == 0) {
        int x = wsum[lane], xi = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, xi, o);
            if (lane >= o)
                xi += u;
        }
        wsum[lane] = xi - x;
    }
    __syncthreads();
    int run = wsum[wid] + inc - tot;
#pragma unroll
    for (int j = 0; j < kGroupPer; ++j) {
        cnt[kGroupPer * t + j] = run;
        run += v[j];
    }
    __syncthreads();
    for (int64_t base = 0; base < nitems; base += kStride) {
        uint32_t bk[kGroupBatch];
#pragma unroll
        for (int j = 0; j < kGroupBatch; ++j) {
            const int64_t w = base + j * kGroupThreads + t;
            bk[j] = w >= nitems ? 0u : w < kGroupCache ? bucket_of[w] : seed_bucket(__ldg(entries + w * n_entries));
        }
#pragma unroll
        for (int j = 0; j < kGroupBatch; ++j) {
            const int64_t w = base + j * kGroupThreads + t;
            if (w < nitems)
                order[atomicAdd(&cnt[bk[j]], 1)] = static_cast<int32_t>(w);
        }
    }
}

// Exact rerank of the final pool (reduced-precision storage): one CTA per
// query re-scores every pool id against the fp32 copy of its row (a warp per
// row, lanes over the row, FP32 accumulation), sorts the (distance, id) keys in
// shared memory with a bitonic network and writes the best k.  Bounded by the
// gathered rows: each warp keeps four rows' loads in flight.  (One warp per
// query, one row after another: 663 us for 1,000 pools of 256 rows of 960
// coordinates, 983 MB; 223 us here.)
constexpr int kRerankWarps = 8;
constexpr int kRerankRows = 4;  // rows a warp re-scores together

template <int MT>
__global__ void __launch_bounds__(32 * kRerankWarps)
    rerank_kernel(const float *base_f32, int dim, const float *queries, int64_t nq, int64_t qdiv,
                  const int32_t *pool, int L, int P, int k, const int32_t *dk, int32_t *out_ids,
                  float *out_dists)
{
    extern __shared__ __align__(16) uint64_t keys[];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    for (int64_t qi = blockIdx.x; qi < nq; qi += gridDim.x) {
        const float *q = queries + (qi / qdiv) * dim;
        for (int c0 = w * kRerankRows; c0 < P; c0 += kRerankWarps * kRerankRows) {
            int32_t id[kRerankRows];
            const float *x[kRerankRows];
            float s[kRerankRows];
#pragma unroll
            for (int u = 0; u < kRerankRows; ++u) {
                id[u] = c0 + u < L ? pool[qi * L + c0 + u] : -1;
                x[u] = base_f32 + static_cast<int64_t>(max(id[u], 0)) * dim;
                s[u] = 0.f;
            }
            if (id[0] >= 0 || id[1] >= 0 || id[2] >= 0 || id[3] >= 0) {
#pragma unroll 4
                for (int j = lane; j < dim; j += 32) {
                    const float y = q[j];
#pragma unroll
                    for (int u = 0; u < kRerankRows; ++u) {
                        if constexpr (MT == ANN_L2) {
                            const float t = x[u][j] - y;
                            s[u] = fmaf(t, t, s[u]);
                        } else {
                            s[u] = fmaf(x[u][j], y, s[u]);
                        }
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < kRerankRows; ++u) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
                    s[u] += __shfl_xor_sync(kFull, s[u], o);
                if (lane == 0)
                    keys[c0 + u] = id[u] >= 0 ? make_key(f32_to_ord(MT == ANN_IP ? -s[u] : s[u]), id[u]) : kKeyMax;
            }
        }
        __syncthreads();
        for (int kk = 2; kk <= P; kk <<= 1) {
            for (int j = kk >> 1; j > 0; j >>= 1) {
                for (int i = tid; i < P; i += 32 * kRerankWarps) {
                    const int p = i ^ j;
                    if (p > i) {
                        const uint64_t a = keys[i], b = keys[p];
                        const bool asc = (i & kk) == 0;
                        if ((a > b) == asc) {
                            keys[i] = b;
                            keys[p] = a;
                        }
                    }
                }
                __syncthreads();
            }
        }
        const int kq = dk ? dk[qi] : k;
        for (int j = tid; j < k; j += 32 * kRerankWarps) {
            const uint64_t v = j < kq ? keys[j] : kKeyMax;
            const bool ok = v != kKeyMax;
            out_ids[qi * k + j] = ok ? key_id(v) : -1;
            out_dists[qi * k + j] = ok ? ord_to_f32(static_cast<uint32_t>(v >> 32)) : __int_as_float(0x7f800000);
        }
        __syncthreads();
    }
}

size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// The distance form of a launch: `chunks` 16-byte chunks of a row, a team of G
// lanes.  One lane a team lane and a row at a time, against here (us, queries):
// 4 G chunks of G = 8 as two lanes in turn: 1,835 -> 1,700 (10,000, d = 128 fp32);
// the other rows of eight lanes or more several at once, so that their chains of
// shared-memory loads and sums overlap: fp32 by twos up to G = 8 (10,000, d = 96:
// 824 -> 784; by fours 100,000 of them lose 7 %), by fours above (10,000, d = 384:
// 2,030 -> 1,389, by twos 1,529; 1,000, d = 960: 1,051 by twos, 978); 16-bit and int8
// rows by twos (3,000, d = 960 fp16: 1,738 -> 1,383; by fours registers spill:
// 1,397, and 1,209 -> 1,412 at d = 200).  Teams of four gain nothing (d = 128
// fp16: 1,040, 1,034; uint8: 792, 795).  A round (`rows`, 0: left open) that the
// teams take at once, one row each, leaves half of them idle by twos (one query, d
// = 960 int8, teams of eight, rounds of four: 447 us by twos, 311 by one).
int search_form(int dtype, int chunks, int G, bool gather4, int rows)
{
    if (dtype == ANN_U8)
        return kOne;
    if (!gather4 && G >= 8) {
        if (G == 8 && chunks == 4 * G && dtype != ANN_I8S)
            return kPair4;
        if (rows == 0 || rows * G > 32)
            return dtype == ANN_F32 && G > 8 ? kRows4 : kRows2;
    }
    return dtype != ANN_I8S && chunks == 8 * G ? kOne8 : kOne;
}

// Bytes of L2 the first-level visited tables may keep resident on the
// current device: the device's persisting-L2 maximum, to which the context's
// set-aside is raised (outside stream capture) when it is lower, for
// ANN_SEARCH_VISITED_L2; ann_release_l2 lowers it again.
size_t persisting_l2_bytes(int dev, cudaStream_t s)
{
    int maxp = 0;
    if (cudaDeviceGetAttribute(&maxp, cudaDevAttrMaxPersistingL2CacheSize, dev) != cudaSuccess || maxp <= 0)
        return 0;
    size_t cur = 0;
    if (cudaDeviceGetLimit(&cur, cudaLimitPersistingL2CacheSize) != cudaSuccess)
        return 0;
    if (cur < static_cast<size_t>(maxp)) {
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(s, &cs) == cudaSuccess && cs == cudaStreamCaptureStatusNone &&
            cudaDeviceSetLimit(cudaLimitPersistingL2CacheSize, static_cast<size_t>(maxp)) == cudaSuccess)
            cur = static_cast<size_t>(maxp);
        cudaGetLastError();
    }
    return cur;
}

#define ANN_DISPATCH(FN, ...)                                                        \
    switch (idx->dtype * 2 + idx->metric) {                                          \
    case ANN_U8 * 2 + ANN_L2: st = FN<ANN_U8, ANN_L2>(__VA_ARGS__); break;           \
    case ANN_F32 * 2 + ANN_L2: st = FN<ANN_F32, ANN_L2>(__VA_ARGS__); break;         \
    case ANN_F32 * 2 + ANN_IP: st = FN<ANN_F32, ANN_IP>(__VA_ARGS__); break;         \
    case ANN_F16 * 2 + ANN_L2: st = FN<ANN_F16, ANN_L2>(__VA_ARGS__); break;         \
    case ANN_F16 * 2 + ANN_IP: st = FN<ANN_F16, ANN_IP>(__VA_ARGS__); break;         \
    case ANN_BF16 * 2 + ANN_L2: st = FN<ANN_BF16, ANN_L2>(__VA_ARGS__); break;       \
    case ANN_BF16 * 2 + ANN_IP: st = FN<ANN_BF16, ANN_IP>(__VA_ARGS__); break;       \
    case ANN_I8S * 2 + ANN_L2: st = FN<ANN_I8S, ANN_L2>(__VA_ARGS__); break;         \
    case ANN_I8S * 2 + ANN_IP: st = FN<ANN_I8S, ANN_IP>(__VA_ARGS__); break;         \
    default: st = ANN_ERR_UNSUPPORTED; break;                                        \
    }

}  // namespace

int default_team(int rowbytes)
{
    const int chunks = rowbytes / 16;
    int G = 4;
    while (G < 32 && chunks > 4 * G)
        G <<= 1;
    return G;
}

int default_spill_bits(int L) { return spill_bits_for(L); }

bool opens_to_gathers(const ann_index *idx) { return idx->has_row_map && idx->rowbytes <= 256; }

size_t search_scratch_bytes(int teams, int spill_bits, int64_t order_items)
{
    return 256 + static_cast<size_t>(teams) * (static_cast<size_t>(20) << spill_bits) +
           4 * static_cast<size_t>(order_items);
}

ann_status launch_search(ann_index *idx, const SearchLaunch &L, cudaStream_t s)
{
    const ann_search_params *p = L.p;
    SearchArgs a{};
    a.base = static_cast<const uint8_t *>(idx->d_base);
    a.graph = idx->d_graph;
    a.n = idx->n;
    a.dim = idx->dim;
    a.R = idx->degree;
    a.R_inv = ((1 << 16) + a.R - 1) / a.R;
    a.rowbytes = idx->rowbytes;
    a.queries = static_cast<const uint8_t *>(L.queries);
    a.qbytes = L.qbytes;
    // int8 rows are read in whole 16-code chunks: the query is zero-extended
    // to the padded code count
    a.qpad = idx->dtype == ANN_I8S ? 4 * ((idx->dim + 15) / 16 * 16 - idx->dim) : 0;
    a.nq = L.nq;
    a.qdiv = L.qdiv > 0 ? L.qdiv : 1;
    a.entries = L.entries;
    a.medoid = idx->medoid;
    a.L = p->L;
    a.k = p->k;
    a.W = p->W;
    a.n_entries = L.n_entries > 0 ? L.n_entries : 1;
    a.fault_wait = (p->flags & ANN_SEARCH_FAULT_WAIT) != 0;
    a.dk = p->d_k;
    a.dL = p->d_L;
    a.dtarget = p->d_target;
    a.out_ids = L.ids;
    a.out_dists = L.dists;
    a.out_stats = L.stats;
    a.status = idx->status_sink ? idx->status_sink : idx->d_status;

    int sb = default_spill_bits(p->L);
    if (p->spill_bits > 0)
        sb = p->spill_bits;
    a.spill_bits = sb;
    a.spill_by_query = p->d_L && p->spill_bits == 0;

    const int maxc = p->W * idx->degree;
    // distance team: the smallest power of two >= 4 that leaves at most four
    // 16-byte chunks of a row to each lane, unless the caller fixed it
    const int chunks = idx->rowbytes / 16;
    const int G = p->team > 0 ? p->team : default_team(idx->rowbytes);
    // gather mode, when the index has a row map: one TMA tensor gather per four
    // rows when the caller asks for it or, left open, for rows of up to 256
    // bytes, where issuing a copy per row costs more than the row; else a bulk
    // copy per row (us, copies against gathers: 100 queries of 128-byte rows 283,
    // 268, 10,000 914, 823; 100 of 256-byte rows 376, 347; 10,000 of 512-byte rows
    // 1,179, 1,225; 1,000 of 1,024-byte rows 814, 918)
    a.gather4 = p->gather == 0 ? opens_to_gathers(idx) : p->gather == 4 && idx->has_row_map;
    if (a.gather4)
        a.row_map = idx->row_map;
    // Lanes per distance: where it pays, four lanes stand for a team of eight, or a
    // team takes several rows at once, so that a round's rows take fewer passes
    // and shuffles; the distances are bit for bit those of G lanes a row.  Tensor
    // gathers write rows back to back, where few lanes a row or neighbouring
    // rows at once would meet bank conflicts: they keep G lanes a row.
    const int form = search_form(idx->dtype, chunks, G, a.gather4, p->stage_rows);
    const int P = idx->dtype == ANN_U8 && !a.gather4 ? std::min(G, 4) : form == kPair4 ? G / 2 : G;
    a.team_lg = 0;
    while ((1 << a.team_lg) < P)
        ++a.team_lg;
    // staging stride in 16-byte units.  A quarter-warp phase of 16-byte loads
    // covers 8 lanes; with P < 8 they read 8 / P rows, whose P-chunk runs hit
    // distinct banks when the stride is P times an odd number.  Tensor
    // gathers write four rows back to back, so their stride is the row size.
    int s16 = chunks;
    if (P < 8 && !a.gather4)
        while (s16 % P != 0 || ((s16 / P) & 1) == 0)
            ++s16;
    a.stage_stride = s16 * 16;
    // shared memory of one team with 2^hb visited slots (hb < 1: no table) and
    // `rows` staged rows (at most 48 KB of them, which also keeps one mbarrier
    // phase's byte count far below its 2^20 limit); fills in the layout
    auto layout = [&](int hb, int rows) {
        a.hash_bits = hb;
        a.stage_rows = std::max(1, std::min({maxc, rows, 49152 / a.stage_stride}));
        if (a.gather4)
            a.stage_rows = (a.stage_rows + 3) / 4 * 4;  // whole groups of four
        size_t off = 16;  // mbarrier
        a.off_sel = static_cast<int>(off);
        off = align_up(off + 4 * 3 * ANN_MAX_W, 16);  // the selection: pool indices, ids, sources
        a.off_q = static_cast<int>(off);
        off = align_up(off + L.qbytes + a.qpad, 16);
        if (a.gather4)
            off = align_up(off, 128);  // tensor gathers land on 128-byte boundaries
        a.off_stage = static_cast<int>(off);
        off = align_up(off + static_cast<size_t>(a.stage_rows) * a.stage_stride, 16);
        a.off_pool = static_cast<int>(off);
        off = align_up(off + 8 * static_cast<size_t>(p->L), 16);
        a.off_ptop = static_cast<int>(off);
        off = align_up(off + 8 * ANN_MAX_W, 16);
        a.off_cbuf = static_cast<int>(off);
        off = align_up(off + 8 * ANN_MAX_STEP_CAND, 16);
        a.off_hash = static_cast<int>(off);
        off = align_up(off + (hb > 0 ? static_cast<size_t>(4) << hb : 0), 128);
        a.per_warp = static_cast<int>(off);
        return off;
    };
    // Visited table and rows per gather round when the caller leaves them
    // open.  Full SMs hide latency better than a shared table or long rounds
    // shorten it, and a lone query wants both.  So: the shared table and then
    // the longest round that still let every SM hold its share of the queries
    // (up to kFullTeams, where registers end; rounds past 24 rows gain only on
    // part-full SMs), else no table, and rounds of eight rows, or of four when
    // rows pass 1 KB (d = 384 fp32: 2,770 us with four, 3,240 with eight), but
    // never fewer than the warp takes at once, which are many when the caller
    // fixed a small team (6,000 queries at d = 960 fp16, teams of two: 2,285 us
    // with four rows, 1,300 with the sixteen that it takes).
    // Measured (us, shared table sized for 12 evaluations per
    // pool slot and rounds of 16 before, this rule after): 100,000 queries of
    // mixed L <= 512 at d = 96: 78,600 -> 28,300; 10,000 at d = 200, L = 256:
    // 8,220 -> 4,290; 100 uint8 queries, L = 64: 497 -> 382; one query: 230 ->
    // 188.
    size_t off = 0;
    {
        int dev_smem = 0, cta_smem = 0;
        cudaDeviceGetAttribute(&dev_smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, idx->device);
        cudaDeviceGetAttribute(&cta_smem, cudaDevAttrReservedSharedMemoryPerBlock, idx->device);
        const int64_t want = std::min<int64_t>(kFullTeams, (L.nq + idx->num_sms - 1) / idx->num_sms);
        auto holds = [&](size_t per_warp) {  // teams an SM holds, two to a CTA when more than one is wanted
            const int64_t w = want > 1 ? kMaxSearchWarps : 1;
            return static_cast<int64_t>(dev_smem) / static_cast<int64_t>(per_warp * w + cta_smem) * w >= want;
        };
        // a table for three times the typical evaluations, at most 32 KB
        const int table = std::min(13, default_spill_bits(p->L));
        // without it the visited set has the global tables only, which must hold as
        // much (they do unless the caller asks for small ones)
        const int none = sb + 2 >= table ? -1 : table;
        // a full shared table hands its keys to the first global one, which must
        // have room for them; the second one then holds what it would have held
        // itself (if not, the query fails, as it says)
        auto within = [&](int hb) { return hb > sb && hb <= sb + 2 ? sb : hb; };
        const int tables[2] = {within(p->hash_bits ? p->hash_bits : table), within(p->hash_bits ? p->hash_bits : none)};
        const int kRows[] = {32, 24, 16, 12, 8, 4};
        int r0 = want < kFullTeams ? 0 : 1, r1 = a.stage_stride > 1024 ? 6 : 5;
        while (r1 > 1 && kRows[r1 - 1] < 32 >> a.team_lg)
            --r1;
        r0 = std::min(r0, r1 - 1);
        bool fits = false;
        for (int t = 0; t < 2 && !fits; ++t) {
            if (p->stage_rows > 0) {
                fits = holds(off = layout(tables[t], p->stage_rows));
            } else {
                for (int r = r0; r < r1 && !fits; ++r)
                    fits = holds(off = layout(tables[t], kRows[r]));
            }
        }
    }

    // persistent grid: occupancy-limited, at most one team per query
    int teams = 0, wpc = 1;
    ann_status st = ANN_OK;
    ANN_DISPATCH(teams_for, idx, off, maxc, form, L.nq, &teams, &wpc);
    if (st != ANN_OK)
        return st;
    if (L.max_teams > 0)
        teams = std::min(teams, L.max_teams);
    teams = static_cast<int>(std::min<long long>(teams, L.nq));
    if (teams < 1)
        return ANN_OK;
    teams = (teams + wpc - 1) / wpc * wpc;  // whole CTAs
    const size_t smem = off * wpc;

    // scratch: work counter, then two spill tables per team, then the grouped
    // work order (when asked for, with seeds given and item indices in int32)
    const bool group = (p->flags & ANN_SEARCH_GROUP_ENTRIES) && L.entries && L.nq <= INT32_MAX;
    size_t need = search_scratch_bytes(teams, a.spill_bits, group ? L.nq : 0);
    void *scratch = L.scratch;
    const bool own = scratch == nullptr;
    if (own) {
        // a nearly full device still searches, with fewer teams and tables
        while ((st = scratch_alloc(idx, need, s, &scratch)) == ANN_ERR_OOM && teams > idx->num_sms) {
            cudaGetLastError();
            teams = std::max(idx->num_sms, teams / 2) / wpc * wpc;
            need = search_scratch_bytes(teams, a.spill_bits, group ? L.nq : 0);
        }
        if (st != ANN_OK)
            return st;
    } else if (L.scratch_bytes < need) {
        return ANN_ERR_CAPACITY;
    }
    a.counter = static_cast<unsigned long long *>(scratch);
    a.nteams = teams;
    a.spill = reinterpret_cast<uint32_t *>(static_cast<uint8_t *>(scratch) + 256);
    int32_t *order = nullptr;
    if (group)
        order = reinterpret_cast<int32_t *>(static_cast<uint8_t *>(scratch) +
                                            search_scratch_bytes(teams, a.spill_bits, 0));
    a.order = order;
    // exact rerank: the search hands its whole pool to rerank_kernel
    const bool rerank = (p->flags & ANN_SEARCH_RERANK) != 0;
    void *pool_buf = nullptr;
    if (rerank) {
        st = scratch_alloc(idx, static_cast<size_t>(L.nq) * p->L * 4, s, &pool_buf);
        if (st != ANN_OK) {
            if (own)
                scratch_free(idx, scratch, s);
            return st;
        }
        a.pool_out = static_cast<int32_t *>(pool_buf);
    }
    // L2-resident first-level visited tables, when asked for and they fit
    size_t window = 0;
    float hit_ratio = 1.f;
    if (p->flags & ANN_SEARCH_VISITED_L2) {
        const size_t tbytes = static_cast<size_t>(teams) * (static_cast<size_t>(4) << a.spill_bits);
        int maxwin = 0;
        cudaDeviceGetAttribute(&maxwin, cudaDevAttrMaxAccessPolicyWindowSize, idx->device);
        const size_t setaside = persisting_l2_bytes(idx->device, s);
        if (tbytes <= setaside && tbytes <= static_cast<size_t>(maxwin))
            window = tbytes;
    }
    cudaError_t e = cudaMemsetAsync(scratch, 0, 8, s);
    if (e == cudaSuccess && group) {
        group_by_seed_kernel<<<1, kGroupThreads, 0, s>>>(L.entries, a.n_entries, L.nq, order);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) {
        ANN_DISPATCH(launch_typed, a, maxc, form, smem, teams, wpc, s, window, hit_ratio);
    } else {
        st = cuda_status(e);
    }
    if (st == ANN_OK && rerank) {
        int P = 32;
        while (P < p->L)
            P <<= 1;
        const size_t rs = static_cast<size_t>(P) * 8;
        const unsigned grid = static_cast<unsigned>(std::min<int64_t>(L.nq, static_cast<int64_t>(idx->num_sms) * 16));
        auto rk = idx->metric == ANN_IP ? rerank_kernel<ANN_IP> : rerank_kernel<ANN_L2>;
        static_assert(ANN_MAX_L * 8 <= 48 * 1024, "within every kernel's limit");
        rk<<<grid, 32 * kRerankWarps, rs, s>>>(idx->d_base_f32, idx->dim, static_cast<const float *>(L.queries), L.nq,
                                                a.qdiv, a.pool_out, p->L, P, p->k, p->d_k, L.ids,
                                                static_cast<float *>(L.dists));
        st = cuda_status(cudaGetLastError());
    }
    if (pool_buf)
        scratch_free(idx, pool_buf, s);
    if (own)
        scratch_free(idx, scratch, s);
    return st;
}

}  // namespace ann
