// train.cu -- contrastive training of the two-tower entry model on the GPU
// (Sec. 4.3 Eq. loss; Sec. 5.1: Adam, batch 8,192).
//
// One step on a batch of B training queries with hub label rows (+1 positive,
// -1 negative, 0 unused):
//   forward   q_hat = tower(q) (tower_forward_kernel, saving Z1, A1, |Z2|);
//             e_hat = E / |E|; S = q_hat e_hat^T / tau        (tcgen05 GEMM)
//   loss      per query: -(1/|P|) sum_{v in P} log softmax_{P u N}(S)_v,
//             averaged over queries with |P| > 0          (infonce_rows_kernel)
//   backward  dS = (softmax - 1[P]/|P|) / n_valid; dP = dS / tau
//             dq_hat = dP e_hat, de_hat = dP^T q_hat            (tcgen05 GEMMs)
//             through the normalisations, dZ2 -> dW2 = A1^T dZ2, db2,
//             dZ1 = (dZ2 W2^T) * [Z1 > 0] -> dW1 = X^T dZ1, db1 (tcgen05 GEMMs)
//   update    Adam with bias correction on W1, b1, W2, b2, E     (adam_kernel)
// Every GEMM runs BF16 x BF16 -> FP32 on the tensor cores.  Whatever produces
// an operand writes it as BF16 in the layouts its GEMMs read (row-major, and
// transposed where a GEMM reduces over the batch), so that a step moves each
// matrix about once: the tower leaves A1^T, q_hat^T and the ReLU mask, the
// loss kernel dS, the dZ1 GEMM's epilogue dZ1^T and db1's partial sums.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <new>
#include <numeric>
#include <vector>

#include "entry.h"
#include "fusion.h"
#include "internal.h"
#include "tc.cuh"

namespace ann {
namespace {

// hubs a trainer takes: one InfoNCE block holds a row's labels in shared memory
constexpr int kMaxTrainHubs = 65536;

// ---- generic tensor-core GEMM ------------------------------------------------

enum Epi { EPI_STORE = 0, EPI_HIDDEN = 1 };

// A BF16 matrix read along its rows (K): element (r, k) = p[r * ld + k], zero
// outside rows x K; ld a multiple of 8 and p 16-byte aligned.
struct Mat {
    const __nv_bfloat16 *p;
    int64_t ld, rows;
};

struct GemmArgs {
    Mat A, B;               // A: M x K, B: N x K
    int64_t M, N, K;
    float alpha;            // out = alpha * scale[0] * acc (scale may be null)
    const float *scale;
    float *out;             // EPI_STORE
    int64_t ldo;
    // EPI_HIDDEN: x = alpha * acc where the row's mask bit is set, else 0;
    // outT[c * ldt + r] = bf16(x), part[warp][c] = sum of the warp's 32 rows
    const uint32_t *mask;   // [N / 32][ldt]
    __nv_bfloat16 *outT;
    int64_t ldt;
    float *part;            // [M / 32, rounded up to 4][256]
    int *status;
    int64_t ksplit;         // > 0: blockIdx.z takes K range [z*ksplit, (z+1)*ksplit) and adds into out
    int stages;             // ring of operand stages, 1 to kGemmStages
};

constexpr int kGemmStages = 4;

// Rows [r0, r0 + ROWS) x k [k0, k0 + 64) of m into a canonical K-major tile by
// 16-byte asynchronous copies (chunk c holds row (c / 64) * 8 + c % 8, k-chunk
// (c / 8) % 8); what lies past the matrix is filled with zeros.
template <int ROWS>
__device__ __forceinline__ void load_tile(uint8_t *tile, const Mat &m, int64_t r0, int64_t k0, int64_t K)
{
    const uint32_t to = smem_addr(tile);
#pragma unroll
    for (int i = 0; i < ROWS * 8 / 128; ++i) {
        const int c = i * 128 + static_cast<int>(threadIdx.x);
        const int64_t r = r0 + (c >> 6) * 8 + (c & 7), k = k0 + ((c >> 3) & 7) * 8;
        const int64_t left = r < m.rows ? K - k : 0;
        const int bytes = left >= 8 ? 16 : left > 0 ? static_cast<int>(left) * 2 : 0;
        const __nv_bfloat16 *src = bytes ? m.p + r * m.ld + k : m.p;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to + c * 16), "l"(src), "r"(bytes)
                     : "memory");
    }
}

// One 128 x BN tile of out = A B^T (or its share of K).  The operands stream
// through a ring of 64-wide K stages filled by asynchronous copies up to
// three stages ahead, thread 0 issues each stage's four MMAs as it lands, and
// the epilogue goes through shared memory so that whole lines are written.
// Staging each K chunk, waiting for its MMAs and storing a row per lane took
// 339 us for the six GEMMs of a step (8,192 rows, 1,024 hubs); 108 us here,
// bounded by load latency and, for the logits, by the 34 MB they write.
template <int BN, int EPI>
__global__ void __launch_bounds__(128) gemm_kernel(const GemmArgs g)
{
    begin_chained();
    extern __shared__ __align__(1024) uint8_t smem[];
    constexpr int kStage = 16384 + BN * 128;
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem + g.stages * kStage);
    uint32_t *slot = reinterpret_cast<uint32_t *>(bar + kGemmStages);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t r0 = static_cast<int64_t>(blockIdx.x) * 128;
    const int64_t c0 = static_cast<int64_t>(blockIdx.y) * BN;
    constexpr uint32_t NCOL = BN < 32 ? 32 : BN;
    if (threadIdx.x == 0) {
        for (int i = 0; i < kGemmStages; ++i)
            mbar_init(bar + i, 1);
        fence_mbar_init();
    }
    if (warp == 0)
        tmem_alloc(slot, NCOL);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *slot;
    const int64_t kb = g.ksplit > 0 ? static_cast<int64_t>(blockIdx.z) * g.ksplit : 0;
    const int64_t ke = g.ksplit > 0 ? min(kb + g.ksplit, g.K) : g.K;
    const int nc = static_cast<int>((ke - kb + 63) / 64), S = g.stages;
    auto load = [&](int c) {
        if (c < nc) {
            uint8_t *st = smem + (c % S) * kStage;
            load_tile<128>(st, g.A, r0, kb + static_cast<int64_t>(c) * 64, ke);
            load_tile<BN>(st + 16384, g.B, c0, kb + static_cast<int64_t>(c) * 64, ke);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    constexpr uint32_t IDESC = idesc_bf16_f32(128, BN);
    bool ok = true;
    for (int c = 0; c < kGemmStages - 1; ++c)
        if (c < S)
            load(c);
        else
            asm volatile("cp.async.commit_group;" ::: "memory");
    // (S < kGemmStages only when all nc chunks fit the ring: nothing is refilled)
    for (int c = 0; c < nc; ++c) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kGemmStages - 2) : "memory");
        fence_proxy_async_smem();
        tc_fence_before();
        __syncthreads();
        if (threadIdx.x == 0) {
            tc_fence_after();
            const uint8_t *sA = smem + (c % S) * kStage, *sB = sA + 16384;
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
                tc_mma(tmem, smem_desc(sA + kk * 256, 128, 1024), smem_desc(sB + kk * 256, 128, 1024), IDESC,
                       (c > 0 || kk > 0) ? 1u : 0u);
            tc_commit(bar + c % S);
        }
        const int next = c + kGemmStages - 1;
        if (next < nc && c > 0) {
            // the stage to refill was read by the previous chunk's MMAs
            uint32_t phase = static_cast<uint32_t>((c - 1) / S) & 1u;
            if (!(ok = tc_wait(bar + (c - 1) % S, phase)))
                break;
        }
        load(next);
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (ok) {
        uint32_t phase = static_cast<uint32_t>((nc - 1) / S) & 1u;
        ok = tc_wait(bar + (nc - 1) % S, phase);
    }
    if (ok) {
        const float a = g.alpha * (g.scale ? g.scale[0] : 1.f);
        const uint32_t my_lane = tmem + (static_cast<uint32_t>(warp * 32) << 16);
        const int64_t row = r0 + warp * 32 + lane;
        float *tw = reinterpret_cast<float *>(smem) + warp * (32 * 33);  // the operands are read
        for (int cc = 0; cc < BN && c0 + cc < g.N; cc += 32) {
            float v[32];
            tmem_ld32(my_lane + cc, v);
            if constexpr (EPI == EPI_HIDDEN) {
                const uint32_t mask = row < g.M ? g.mask[((c0 + cc) >> 5) * g.ldt + row] : 0u;
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    const float x = (mask >> j) & 1u ? a * v[j] : 0.f;
                    tw[lane * 33 + j] = x;
                    if (row < g.M)
                        g.outT[(c0 + cc + j) * g.ldt + row] = __float2bfloat16_rn(x);
                }
                __syncwarp();
                float sum = 0.f;
#pragma unroll
                for (int r = 0; r < 32; ++r)
                    sum += tw[r * 33 + lane];
                g.part[(static_cast<int64_t>(blockIdx.x) * 4 + warp) * 256 + c0 + cc + lane] = sum;
            } else {
#pragma unroll
                for (int j = 0; j < 32; ++j)
                    tw[lane * 33 + j] = a * v[j];
                __syncwarp();
                const int64_t col = c0 + cc + lane;
                const int rows = static_cast<int>(min(static_cast<int64_t>(32), g.M - r0 - warp * 32));
                if (col < g.N) {
                    float *o = g.out + (r0 + warp * 32) * g.ldo + col;
                    for (int r = 0; r < rows; ++r) {
                        if (g.ksplit > 0)
                            atomicAdd(o + r * g.ldo, tw[r * 33 + lane]);  // a partial sum over its K range
                        else
                            o[r * g.ldo] = tw[r * 33 + lane];
                    }
                }
            }
            __syncwarp();
        }
    } else if (threadIdx.x == 0) {
        atomicOr(g.status, kStatusTimeoutBit);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, NCOL);
    }
}

// Shared memory of a GEMM with `stages` stages: at most 512 / BN CTAs fit an SM's
// 228 KB, so that they never ask for more than its 512 TMEM columns.
template <int BN>
constexpr int gemm_smem(int stages)
{
    return std::max(stages * (16384 + BN * 128) + 64, 228 * 1024 / (512 / BN + 1) + 1);
}

// The kernel's limit, which belongs to the device and not to a launch: the most
// that any of its GEMMs takes, so that trainers of several threads never lower
// it between another one's look at it and its launch.  (No more than that: with
// the limit of the 256-wide split GEMM on the one with the hidden layer's
// epilogue too, a step took 1 % longer.)
template <int BN, int EPI>
cudaError_t gemm_limit(int stages)
{
    return cudaFuncSetAttribute(gemm_kernel<BN, EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                gemm_smem<BN>(stages));
}

// Queues one GEMM.  With EPI_STORE and few output tiles over a long reduction
// K is split over CTAs, at least min_k columns each, that add into `out`, which
// the caller has zeroed.
template <int BN, int EPI = EPI_STORE>
ann_status gemm(const GemmArgs &g, cudaStream_t s, bool chained, int64_t min_k = 512)
{
    dim3 grid(static_cast<unsigned>((g.M + 127) / 128), static_cast<unsigned>((g.N + BN - 1) / BN));
    // up to about two CTAs per SM
    GemmArgs h = g;
    h.ksplit = 0;
    const int64_t tiles = static_cast<int64_t>(grid.x) * grid.y;
    if (EPI == EPI_STORE && tiles < 128 && g.K >= 1024) {
        const int64_t want = std::min<int64_t>(g.K / min_k, std::max<int64_t>(1, 256 / tiles));
        if (want > 1) {
            h.ksplit = ((g.K + want - 1) / want + 63) / 64 * 64;
            grid.z = static_cast<unsigned>((g.K + h.ksplit - 1) / h.ksplit);
        }
    }
    const int64_t chunks = ((h.ksplit ? h.ksplit : g.K) + 63) / 64;
    h.stages = static_cast<int>(std::min<int64_t>(kGemmStages, chunks));
    launch_next(chained, gemm_kernel<BN, EPI>, grid, 128, gemm_smem<BN>(h.stages), s, h);
    return cuda_status(cudaGetLastError());
}

// ---- elementwise / row kernels --------------------------------------------

// The two transposes over the batch that no producer can write itself, in
// 64 x 64 tiles: blockIdx.z = 0: dst[c][r] = dS(r, c), BF16 both; 1: xT[c][r] =
// bf16(X(row r of the batch, c)).
struct TransposeArgs {
    const __nv_bfloat16 *dS;
    int64_t ldS;
    int H;
    __nv_bfloat16 *dST;
    const float *X;
    const int32_t *rowmap;
    int D;
    __nv_bfloat16 *xT;
    int64_t B, ldB;
};

__global__ void __launch_bounds__(256) transpose_kernel(const TransposeArgs a)
{
    begin_chained();
    __shared__ __nv_bfloat16 tile[64][66];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int64_t c0 = static_cast<int64_t>(blockIdx.x) * 64, r0 = static_cast<int64_t>(blockIdx.y) * 64;
    const bool logits = blockIdx.z == 0;
    const int cols = logits ? a.H : a.D;
    if (c0 >= cols)
        return;
    for (int i = ty; i < 64; i += 8) {
        const int64_t r = r0 + i;
        __nv_bfloat162 v;
        v.x = v.y = __float2bfloat16_rn(0.f);
        const int64_t c = c0 + 2 * tx;
        if (r < a.B) {
            if (logits) {
                // pairs are 4-byte aligned (ldS even); past H the row's padding is read, never used
                if (c < a.ldS)
                    v = *reinterpret_cast<const __nv_bfloat162 *>(a.dS + r * a.ldS + c);
            } else {
                const float *x = a.X + static_cast<int64_t>(a.rowmap ? a.rowmap[r] : r) * a.D;
                if (c < cols)
                    v.x = __float2bfloat16_rn(x[c]);
                if (c + 1 < cols)
                    v.y = __float2bfloat16_rn(x[c + 1]);
            }
        }
        *reinterpret_cast<__nv_bfloat162 *>(&tile[i][2 * tx]) = v;
    }
    __syncthreads();
    __nv_bfloat16 *dst = logits ? a.dST : a.xT;
    for (int i = ty; i < 64; i += 8) {
        const int64_t c = c0 + i, r = r0 + 2 * tx;
        if (c >= cols || r >= a.B)
            continue;
        if (r + 1 < a.B) {
            __nv_bfloat162 v;
            v.x = tile[2 * tx][i];
            v.y = tile[2 * tx + 1][i];
            *reinterpret_cast<__nv_bfloat162 *>(dst + c * a.ldB + r) = v;  // ldB and r are even
        } else {
            dst[c * a.ldB + r] = tile[2 * tx][i];
        }
    }
}

// The block's sum of b and its maximum (MAX) or sum of a, one value of each per
// thread; every thread gets both.  red holds 64 slots; blockDim.x is a multiple
// of 32.
template <bool MAX>
__device__ __forceinline__ void block_reduce2(float &a, float &b, float *red)
{
    auto warp = [&]() {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float w = __shfl_xor_sync(kFull, a, o);
            a = MAX ? fmaxf(a, w) : a + w;
            b += __shfl_xor_sync(kFull, b, o);
        }
    };
    warp();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __syncthreads();  // red is free again
    if (lane == 0) {
        red[wid] = a;
        red[32 + wid] = b;
    }
    __syncthreads();
    a = lane < nw ? red[lane] : (MAX ? -INFINITY : 0.f);
    b = lane < nw ? red[32 + lane] : 0.f;
    warp();
}

// One block per batch row: masked multi-positive InfoNCE over the labelled
// hubs.  The row's labels come as its M listed hubs (cand, lab); every hub
// not listed is a negative, so the row's H labels are first laid out in
// shared memory (all -1, then the listed ones).  Writes the row loss, a
// validity flag (|P| > 0) and the unscaled gradient softmax_{P u N}(S) -
// 1[P]/|P| (0 outside P u N and on invalid rows), rounded to BF16 as the GEMMs
// that read it need it.
__global__ void infonce_kernel(const float *S, int64_t B, int H, const int32_t *cand, const int8_t *lab, int M,
                               const int32_t *rowmap, __nv_bfloat16 *dS, int64_t ldS, float *row_loss, int *valid)
{
    begin_chained();
    extern __shared__ int8_t lrow[];
    __shared__ float red[64];
    const int64_t r = blockIdx.x;
    const int64_t mr = rowmap ? rowmap[r] : r;
    for (int c = threadIdx.x; c < H; c += blockDim.x)
        lrow[c] = -1;
    __syncthreads();
    for (int j = threadIdx.x; j < M; j += blockDim.x) {
        const int32_t h = cand[mr * M + j];
        if (h >= 0 && h < H)
            lrow[h] = lab[mr * M + j];
    }
    __syncthreads();
    const float *s = S + r * H;
    float mx = -INFINITY, np = 0.f;
    for (int c = threadIdx.x; c < H; c += blockDim.x) {
        if (lrow[c] != 0)
            mx = fmaxf(mx, s[c]);
        np += lrow[c] > 0 ? 1.f : 0.f;
    }
    block_reduce2<true>(mx, np, red);
    const int npos = static_cast<int>(np);
    float z = 0.f, sp = 0.f;
    for (int c = threadIdx.x; c < H; c += blockDim.x) {
        if (lrow[c] != 0)
            z += expf(s[c] - mx);
        if (lrow[c] > 0)
            sp += s[c];
    }
    block_reduce2<false>(z, sp, red);
    const float lse = mx + logf(z);
    const bool ok = npos > 0;
    const float inv_np = ok ? 1.f / static_cast<float>(npos) : 0.f;
    for (int c = threadIdx.x; c < H; c += blockDim.x) {
        float g = 0.f;
        if (ok && lrow[c] != 0)
            g = expf(s[c] - lse) - (lrow[c] > 0 ? inv_np : 0.f);
        dS[r * ldS + c] = __float2bfloat16_rn(g);
    }
    if (threadIdx.x == 0) {
        row_loss[r] = ok ? -(sp - npos * lse) * inv_np : 0.f;
        valid[r] = ok ? 1 : 0;
    }
}

// infonce_kernel with a warp per row, for up to kRowHubs hubs: no barriers, and
// up to 1,024 hubs a row's logits are read once into registers.  Every sum runs
// as the block's does (its thread t = 32 w + lane adds columns t, t + 256, ...;
// lanes by xor-shuffles; warps 4 apart, 2 apart, 1 apart), so that the
// logarithm of the partition sum, which decides how dS rounds to BF16, has the
// same bits.  8,192 rows x 1,024 hubs: 39 us by blocks, 33 us here.
constexpr int kRowHubs = 8192;
constexpr int kRowWarps = 8;

template <bool REG>
__global__ void __launch_bounds__(32 * kRowWarps)
    infonce_rows_kernel(const float *S, int64_t B, int H, const int32_t *cand, const int8_t *lab, int M,
                        const int32_t *rowmap, __nv_bfloat16 *dS, int64_t ldS, float *row_loss, int *valid)
{
    begin_chained();
    extern __shared__ __align__(16) int8_t lrow_all[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t r = blockIdx.x * static_cast<int64_t>(kRowWarps) + wid;
    if (r >= B)
        return;
    const int hp = (H + 15) / 16 * 16;
    int8_t *lrow = lrow_all + wid * hp;
    const int64_t mr = rowmap ? rowmap[r] : r;
    for (int c = lane; c < hp / 16; c += 32)
        reinterpret_cast<uint4 *>(lrow)[c] = make_uint4(~0u, ~0u, ~0u, ~0u);
    __syncwarp();
    for (int j = lane; j < M; j += 32) {
        const int32_t h = cand[mr * M + j];
        if (h >= 0 && h < H)
            lrow[h] = lab[mr * M + j];
    }
    __syncwarp();
    const float *s = S + r * H;
    constexpr int kReg = REG ? 32 : 1;
    float sv[kReg];
    if constexpr (REG) {
#pragma unroll
        for (int i = 0; i < 32; ++i)
            sv[i] = lane + 32 * i < H ? s[lane + 32 * i] : 0.f;
    }
    // f(i, c, logit) over the lane's columns c = lane + 32 i < H, eight i at a time
    auto each = [&](auto f) {
        if constexpr (REG) {
#pragma unroll
            for (int i = 0; i < 32; ++i)
                if (lane + 32 * i < H)
                    f(i & 7, lane + 32 * i, sv[i]);
        } else {
            for (int i0 = 0; 32 * i0 < H; i0 += 8) {
#pragma unroll
                for (int w = 0; w < 8; ++w) {
                    const int c = lane + 32 * (i0 + w);
                    if (c < H)
                        f(w, c, s[c]);
                }
            }
        }
    };
    auto add = [&](float (&v)[8]) {
#pragma unroll
        for (int w = 0; w < 8; ++w)
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                v[w] += __shfl_xor_sync(kFull, v[w], o);
        return ((v[0] + v[4]) + (v[2] + v[6])) + ((v[1] + v[5]) + (v[3] + v[7]));
    };
    float mx = -INFINITY;
    int npos = 0;
    each([&](int, int c, float x) {
        const int8_t l = lrow[c];
        if (l != 0)
            mx = fmaxf(mx, x);
        npos += l > 0;
    });
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, o));
    npos = __reduce_add_sync(kFull, npos);
    float zs[8], ps[8];
#pragma unroll
    for (int w = 0; w < 8; ++w)
        zs[w] = ps[w] = 0.f;
    each([&](int w, int c, float x) {
        const int8_t l = lrow[c];
        if (l != 0)
            zs[w] += expf(x - mx);
        if (l > 0)
            ps[w] += x;
    });
    const float z = add(zs), sp = add(ps);
    const float lse = mx + logf(z);
    const bool ok = npos > 0;
    const float inv_np = ok ? 1.f / static_cast<float>(npos) : 0.f;
    each([&](int, int c, float x) {
        const int8_t l = lrow[c];
        float g = 0.f;
        if (ok && l != 0)
            g = expf(x - lse) - (l > 0 ? inv_np : 0.f);
        dS[r * ldS + c] = __float2bfloat16_rn(g);
    });
    if (lane == 0) {
        row_loss[r] = ok ? -(sp - npos * lse) * inv_np : 0.f;
        valid[r] = ok ? 1 : 0;
    }
}

// loss = mean row loss over valid rows; scale[0] = 1 / (n_valid * tau)
__global__ void finalize_loss_kernel(const float *row_loss, const int *valid, int64_t B, float tau, float *loss,
                                     float *scale)
{
    begin_chained();
    __shared__ float sl[1024];
    __shared__ int sv[1024];
    float l = 0.f;
    int v = 0;
    for (int64_t i = threadIdx.x; i < B; i += blockDim.x) {
        l += row_loss[i];
        v += valid[i];
    }
    sl[threadIdx.x] = l;
    sv[threadIdx.x] = v;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) {
            sl[threadIdx.x] += sl[threadIdx.x + o];
            sv[threadIdx.x] += sv[threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const int nv = sv[0];
        loss[0] = nv > 0 ? sl[0] / nv : 0.f;
        scale[0] = nv > 0 ? 1.f / (nv * tau) : 0.f;
    }
}

// dZ = (dY - Y (Y . dY)) / n per row of width W (gradient of y = z / |z|)
__global__ void norm_backward_kernel(const float *Y, const float *n, const float *dY, int64_t rows, int W,
                                     float *dZ)
{
    begin_chained();
    const int lane = threadIdx.x & 31;
    const int64_t r = (blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) >> 5;
    if (r >= rows)
        return;
    float dot = 0.f;
    for (int c = lane; c < W; c += 32)
        dot = fmaf(Y[r * W + c], dY[r * W + c], dot);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        dot += __shfl_xor_sync(kFull, dot, o);
    const float inv = n[r] > 0.f ? 1.f / n[r] : 0.f;
    for (int c = lane; c < W; c += 32)
        dZ[r * W + c] = (dY[r * W + c] - Y[r * W + c] * dot) * inv;
}

// norm_backward_kernel for the queries (64 columns), 32 rows per block, with
// what the next GEMMs read: dZ2 in BF16, by rows and transposed, and the
// block's column sums (db2's partial sums).
__global__ void __launch_bounds__(256)
    query_backward_kernel(const float *Y, const float *n, const float *dY, int64_t rows, __nv_bfloat16 *dZ,
                          __nv_bfloat16 *dZT, int64_t ld, float *part)
{
    begin_chained();
    __shared__ float dz[32][65];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t r0 = static_cast<int64_t>(blockIdx.x) * 32;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int64_t r = r0 + 4 * w + i;
        float z0 = 0.f, z1 = 0.f;
        if (r < rows) {
            const float y0 = Y[r * 64 + lane], y1 = Y[r * 64 + 32 + lane];
            const float g0 = dY[r * 64 + lane], g1 = dY[r * 64 + 32 + lane];
            float dot = fmaf(y1, g1, fmaf(y0, g0, 0.f));
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                dot += __shfl_xor_sync(kFull, dot, o);
            const float inv = n[r] > 0.f ? 1.f / n[r] : 0.f;
            z0 = (g0 - y0 * dot) * inv;
            z1 = (g1 - y1 * dot) * inv;
            dZ[r * 64 + lane] = __float2bfloat16_rn(z0);
            dZ[r * 64 + 32 + lane] = __float2bfloat16_rn(z1);
        }
        dz[4 * w + i][lane] = z0;
        dz[4 * w + i][32 + lane] = z1;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int c = w + 8 * i;
        const float v = dz[lane][c];
        if (r0 + lane < rows)
            dZT[c * ld + r0 + lane] = __float2bfloat16_rn(v);
        float sum = v;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            sum += __shfl_xor_sync(kFull, sum, o);
        if (lane == 0)
            part[static_cast<int64_t>(blockIdx.x) * 64 + c] = sum;
    }
}

// db1 and db2 from their partial sums, 32 columns per block (blocks 0..7: db1,
// 8 and 9: db2), in a fixed order.  (One block that walked all rows took
// 230 us per bias.)
__global__ void __launch_bounds__(1024)
    bias_sum_kernel(const float *part1, int64_t n1, const float *part2, int64_t n2, float *b1, float *b2)
{
    begin_chained();
    __shared__ float sh[32][33];
    const bool first = blockIdx.x < 8;
    const float *part = first ? part1 : part2;
    const int64_t n = first ? n1 : n2;
    const int width = first ? 256 : 64, c0 = static_cast<int>(first ? blockIdx.x : blockIdx.x - 8) * 32;
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
    float s = 0.f;
#pragma unroll 4
    for (int64_t p = g; p < n; p += 32)
        s += part[p * width + c0 + lane];
    sh[g][lane] = s;
    __syncthreads();
    if (g == 0) {
        float t = 0.f;
#pragma unroll
        for (int i = 0; i < 32; ++i)
            t += sh[i][lane];
        (first ? b1 : b2)[c0 + lane] = t;
    }
}

// Adam with bias correction (Kingma & Ba), fp32 state
__global__ void adam_kernel(float *p, const float *g, float *m, float *v, int64_t n, float lr, float b1, float b2,
                            float eps, float bc1, float bc2)
{
    begin_chained();
    const int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
    if (i >= n)
        return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float mh = mi / bc1, vh = vi / bc2;
    p[i] -= lr * mh / (sqrtf(vh) + eps);
}

inline unsigned blocks_for(int64_t n, int per) { return static_cast<unsigned>((n + per - 1) / per); }

}  // namespace
}  // namespace ann

using namespace ann;

// Trainer: parameters (flat fp32: W1 | b1 | W2 | b2 | E), Adam state, and
// per-batch scratch.  The model struct reuses the inference launchers.
struct ann_trainer {
    int device = 0;
    int64_t batch = 0;
    int in_dim = 0, H = 0;
    float tau = 0.07f, lr = 5e-5f, beta1 = 0.9f, beta2 = 0.999f, eps = 1e-8f;
    int64_t step = 0;
    int64_t n_params = 0;
    float *params = nullptr, *grads = nullptr, *m = nullptr, *v = nullptr;
    ann_entry_model model;  // views into params + BF16 copies
    // scratch
    float *qhat = nullptr, *S = nullptr, *row_loss = nullptr;
    float *dQ = nullptr, *dEh = nullptr, *part1 = nullptr, *part2 = nullptr;
    float *loss = nullptr, *scale = nullptr;
    int *valid = nullptr, *status = nullptr;
    int64_t ldB = 0, ldH = 0;  // batch and hubs rounded up to whole 16-byte pieces
    TowerTrain tower{};
    __nv_bfloat16 *qbf = nullptr, *dS = nullptr, *dST = nullptr, *dZ2 = nullptr, *dZ2T = nullptr, *xT = nullptr,
                  *dZ1T = nullptr;
    std::vector<void *> owned;
    ann::Fusion *fu = nullptr;  // topology-aware hub tower: hub rows are E + F
};

namespace {

template <typename T>
T *talloc(ann_trainer *t, size_t count, cudaError_t &e)
{
    T *p = nullptr;
    if (e == cudaSuccess) {
        e = cudaMalloc(reinterpret_cast<void **>(&p), std::max<size_t>(count, 1) * sizeof(T));
        if (e == cudaSuccess)
            t->owned.push_back(p);
    }
    return p;
}

void trainer_free(ann_trainer *t)
{
    if (!t)
        return;
    // the trainer's device, whichever is current: its kernels are waited for and
    // its builder scratch is given back
    int prev = 0;
    cudaGetDevice(&prev);
    cudaSetDevice(t->device);
    cudaDeviceSynchronize();
    for (void *p : t->owned)
        cudaFree(p);
    fusion_free(t->fu);
    delete t;
    builder_trim();
    cudaSetDevice(prev);
}

// A step is a chain of some fifteen short kernels: each one's launch overlaps
// the one before, except under capture, which records plain dependencies.  A
// step at batch 8,192: 323 us without, 294 here.
bool may_chain(cudaStream_t s)
{
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    return cudaStreamIsCapturing(s, &cs) == cudaSuccess && cs == cudaStreamCaptureStatusNone;
}

// one Adam step over every parameter block
void adam_all(ann_trainer *t, cudaStream_t s)
{
    const bool chained = may_chain(s);
    t->step += 1;
    const float bc1 = 1.f - powf(t->beta1, static_cast<float>(t->step));
    const float bc2 = 1.f - powf(t->beta2, static_cast<float>(t->step));
    launch_next(chained, adam_kernel, blocks_for(t->n_params, 256), 256, 0, s, t->params, t->grads, t->m, t->v,
                t->n_params, t->lr, t->beta1, t->beta2, t->eps, bc1, bc2);
    if (t->fu)
        adam_kernel<<<blocks_for(t->fu->n_params, 256), 256, 0, s>>>(t->fu->params, t->fu->grads, t->fu->m,
                                                                     t->fu->v, t->fu->n_params, t->lr, t->beta1,
                                                                     t->beta2, t->eps, bc1, bc2);
}

// offsets of the parameter blocks inside the flat vector
struct Offs {
    int64_t W1, b1, W2, b2, E, total;
};
Offs offsets(int in_dim, int H)
{
    Offs o;
    o.W1 = 0;
    o.b1 = o.W1 + static_cast<int64_t>(in_dim) * 256;
    o.W2 = o.b1 + 256;
    o.b2 = o.W2 + 256 * 64;
    o.E = o.b2 + 64;
    o.total = o.E + static_cast<int64_t>(H) * 64;
    return o;
}

// forward + loss + backward for one batch; grads written to t->grads
ann_status trainer_grads(ann_trainer *t, const float *d_queries, const int32_t *rows, int64_t B,
                         const int32_t *d_cand, const int8_t *d_lab, int n_listed, cudaStream_t s)
{
    ann_entry_model &M = t->model;
    const Offs o = offsets(t->in_dim, t->H);
    const int H = t->H, D = t->in_dim;
    const bool chained = may_chain(s);
    // what split GEMMs add into: the weight gradients, de_hat and dq_hat lie together
    cudaError_t e = cudaMemsetAsync(t->grads, 0, static_cast<size_t>(o.total + (H + B) * 64) * 4, s);
    if (e != cudaSuccess)
        return cuda_status(e);
    ann_status st = ANN_OK;
    if (t->fu) {
        // the hub rows the model scores: E + F (Eq. fusion)
        if ((st = fusion_forward(t->fu, t->params + o.E, s)) != ANN_OK)
            return st;
        M.E = t->fu->Eeff;
    }
    st = prepare_model(&M, s);
    M.E = t->params + o.E;
    if (st != ANN_OK)
        return st;
    const Operand X{d_queries, OP_F32, D, 1, B, D, rows};
    if ((st = launch_tower(&M, X, B, t->qhat, t->qbf, &t->tower, t->status, s, chained)) != ANN_OK)
        return st;
    // logits
    GemmArgs g{};
    g.status = t->status;
    g.A = Mat{t->qbf, 64, B};
    g.B = Mat{M.Eb, 64, H};
    g.M = B;
    g.N = H;
    g.K = 64;
    g.alpha = 1.f / t->tau;
    g.out = t->S;
    g.ldo = H;
    if ((st = gemm<128>(g, s, chained)) != ANN_OK)
        return st;
    if (H <= kRowHubs) {
        auto kern = H <= 1024 ? infonce_rows_kernel<true> : infonce_rows_kernel<false>;
        launch_next(chained, kern, blocks_for(B, kRowWarps), 32 * kRowWarps, kRowWarps * ((H + 15) / 16 * 16), s,
                    t->S, B, H, d_cand, d_lab, n_listed, rows, t->dS, t->ldH, t->row_loss, t->valid);
    } else {
        launch_next(chained, infonce_kernel, static_cast<unsigned>(B), 256, H, s, t->S, B, H, d_cand, d_lab, n_listed,
                    rows, t->dS, t->ldH, t->row_loss, t->valid);
    }
    launch_next(chained, finalize_loss_kernel, 1, 1024, 0, s, t->row_loss, t->valid, B, t->tau, t->loss, t->scale);
    // dq_hat = scale * dS e_hat  (B x 64, K = H)
    g = GemmArgs{};
    g.status = t->status;
    g.A = Mat{t->dS, t->ldH, B};
    g.B = Mat{M.EnT, M.ldE, 64};
    g.M = B;
    g.N = 64;
    g.K = H;
    g.alpha = 1.f;
    g.scale = t->scale;
    g.out = t->dQ;
    g.ldo = 64;
    if ((st = gemm<64>(g, s, chained)) != ANN_OK)
        return st;
    // de_hat = scale * dS^T q_hat  (H x 64, K = B)
    const TransposeArgs ta{t->dS, t->ldH, H, t->dST, d_queries, rows, D, t->xT, B, t->ldB};
    launch_next(chained, transpose_kernel, dim3(blocks_for(std::max(H, D), 64), blocks_for(B, 64), 2), 256, 0, s,
                ta);
    g.A = Mat{t->dST, t->ldB, H};
    g.B = Mat{t->tower.qT, t->ldB, 64};
    g.M = H;
    g.N = 64;
    g.K = B;
    g.out = t->dEh;
    // (sums that no later rounding to BF16 reads are split further)
    if ((st = gemm<64>(g, s, chained, 256)) != ANN_OK)
        return st;
    // through the normalisations
    launch_next(chained, query_backward_kernel, blocks_for(B, 32), 256, 0, s, t->qhat, t->tower.nrm, t->dQ, B, t->dZ2,
                t->dZ2T, t->ldB, t->part2);
    launch_next(chained, norm_backward_kernel, blocks_for(static_cast<int64_t>(H) * 32, 256), 256, 0, s, M.En, M.Enrm,
                t->dEh, H, 64, t->grads + o.E);
    // dL/dF = dL/d(E + F) = dL/dE
    if (t->fu && (st = fusion_backward(t->fu, t->grads + o.E, s)) != ANN_OK)
        return st;
    // dW2 = A1^T dZ2 (256 x 64, K = B)
    g = GemmArgs{};
    g.status = t->status;
    g.A = Mat{t->tower.a1T, t->ldB, 256};
    g.B = Mat{t->dZ2T, t->ldB, 64};
    g.M = 256;
    g.N = 64;
    g.K = B;
    g.alpha = 1.f;
    g.out = t->grads + o.W2;
    g.ldo = 64;
    if ((st = gemm<64>(g, s, chained, 256)) != ANN_OK)
        return st;
    // dZ1 = (dZ2 W2^T) * [Z1 > 0]  (B x 256, K = 64), written transposed, with db1's partial sums
    g = GemmArgs{};
    g.status = t->status;
    g.A = Mat{t->dZ2, 64, B};
    g.B = Mat{M.W2b, 64, 256};
    g.M = B;
    g.N = 256;
    g.K = 64;
    g.alpha = 1.f;
    g.mask = t->tower.zmask;
    g.outT = t->dZ1T;
    g.ldt = t->ldB;
    g.part = t->part1;
    if ((st = gemm<256, EPI_HIDDEN>(g, s, chained)) != ANN_OK)
        return st;
    launch_next(chained, bias_sum_kernel, 10, 1024, 0, s, t->part1, (B + 127) / 128 * 4, t->part2, (B + 31) / 32,
                t->grads + o.b1, t->grads + o.b2);
    // dW1 = X^T dZ1  (D x 256, K = B)
    g = GemmArgs{};
    g.status = t->status;
    g.A = Mat{t->xT, t->ldB, D};
    g.B = Mat{t->dZ1T, t->ldB, 256};
    g.M = D;
    g.N = 256;
    g.K = B;
    g.alpha = 1.f;
    g.out = t->grads + o.W1;
    g.ldo = 256;
    if ((st = gemm<256>(g, s, chained, 256)) != ANN_OK)
        return st;
    return cuda_status(cudaGetLastError());
}

}  // namespace

extern "C" {

ann_status ann_trainer_create(int device, int32_t in_dim, int32_t n_hubs, const float *W1, const float *b1,
                              const float *W2, const float *b2, const float *hub_emb, int64_t max_batch,
                              float tau, float lr, float beta1, float beta2, float eps, ann_trainer **out)
{
    if (!out || !W1 || !b1 || !W2 || !b2 || !hub_emb || in_dim < 1 || in_dim > 512 || n_hubs < 2 ||
        n_hubs > kMaxTrainHubs ||
        max_batch < 1 || max_batch > (1 << 20) || !(tau > 0.f) || !(lr > 0.f) || !(beta1 >= 0.f && beta1 < 1.f) ||
        !(beta2 >= 0.f && beta2 < 1.f) || !(eps > 0.f))
        return ANN_ERR_INVALID_ARG;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev)
        return ANN_ERR_CUDA;
    cudaSetDevice(device);
    if (cudaFuncSetAttribute(infonce_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxTrainHubs) !=
            cudaSuccess ||
        cudaFuncSetAttribute(infonce_rows_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kRowWarps * kRowHubs) != cudaSuccess ||
        gemm_limit<64, EPI_STORE>(kGemmStages) != cudaSuccess ||
        gemm_limit<128, EPI_STORE>(1) != cudaSuccess ||   // the logits: K = 64
        gemm_limit<256, EPI_HIDDEN>(1) != cudaSuccess ||  // dZ1: K = 64
        gemm_limit<256, EPI_STORE>(kGemmStages) != cudaSuccess)
        return ANN_ERR_CUDA;
    ann_trainer *t = new (std::nothrow) ann_trainer();
    if (!t)
        return ANN_ERR_OOM;
    t->device = device;
    t->batch = max_batch;
    t->in_dim = in_dim;
    t->H = n_hubs;
    t->tau = tau;
    t->lr = lr;
    t->beta1 = beta1;
    t->beta2 = beta2;
    t->eps = eps;
    const Offs o = offsets(in_dim, n_hubs);
    t->n_params = o.total;
    const int64_t B = max_batch, H = n_hubs;
    cudaError_t e = cudaSuccess;
    t->params = talloc<float>(t, o.total, e);
    t->grads = talloc<float>(t, o.total + (H + B) * 64, e);
    t->dEh = t->grads + o.total;
    t->dQ = t->dEh + H * 64;
    t->m = talloc<float>(t, o.total, e);
    t->v = talloc<float>(t, o.total, e);
    t->ldB = (B + 7) / 8 * 8;
    t->ldH = (H + 7) / 8 * 8;
    t->tower.ld = t->ldB;
    t->tower.zmask = talloc<uint32_t>(t, 8 * t->ldB, e);
    t->tower.a1T = talloc<__nv_bfloat16>(t, 256 * t->ldB, e);
    t->tower.qT = talloc<__nv_bfloat16>(t, 64 * t->ldB, e);
    t->tower.nrm = talloc<float>(t, B, e);
    t->qhat = talloc<float>(t, B * 64, e);
    t->qbf = talloc<__nv_bfloat16>(t, B * 64, e);
    t->S = talloc<float>(t, B * H, e);
    t->dS = talloc<__nv_bfloat16>(t, B * t->ldH, e);
    t->dST = talloc<__nv_bfloat16>(t, H * t->ldB, e);
    t->row_loss = talloc<float>(t, B, e);
    t->valid = talloc<int>(t, B, e);
    t->part1 = talloc<float>(t, (B + 127) / 128 * 4 * 256, e);
    t->part2 = talloc<float>(t, (B + 31) / 32 * 64, e);
    t->loss = talloc<float>(t, 2, e);
    t->scale = talloc<float>(t, 2, e);
    t->status = talloc<int>(t, 4, e);
    t->dZ2 = talloc<__nv_bfloat16>(t, B * 64, e);
    t->dZ2T = talloc<__nv_bfloat16>(t, 64 * t->ldB, e);
    t->xT = talloc<__nv_bfloat16>(t, in_dim * t->ldB, e);
    t->dZ1T = talloc<__nv_bfloat16>(t, 256 * t->ldB, e);
    ann_entry_model &M = t->model;
    M.in_dim = in_dim;
    M.H = n_hubs;
    M.W1t = talloc<__nv_bfloat16>(t, static_cast<size_t>(in_dim) * 256, e);
    M.W2t = talloc<__nv_bfloat16>(t, 256 * 64, e);
    M.En = talloc<float>(t, H * 64, e);
    M.Eb = talloc<__nv_bfloat16>(t, H * 64, e);
    M.Enrm = talloc<float>(t, H, e);
    M.W2b = talloc<__nv_bfloat16>(t, 256 * 64, e);
    M.EnT = talloc<__nv_bfloat16>(t, 64 * t->ldH, e);
    M.ldE = t->ldH;
    if (e == cudaSuccess) {
        M.W1 = t->params + o.W1;
        M.b1 = t->params + o.b1;
        M.W2 = t->params + o.W2;
        M.b2 = t->params + o.b2;
        M.E = t->params + o.E;
        e = cudaMemcpy(M.W1, W1, static_cast<size_t>(in_dim) * 256 * 4, cudaMemcpyDefault);
    }
    if (e == cudaSuccess)
        e = cudaMemcpy(M.b1, b1, 256 * 4, cudaMemcpyDefault);
    if (e == cudaSuccess)
        e = cudaMemcpy(M.W2, W2, 256 * 64 * 4, cudaMemcpyDefault);
    if (e == cudaSuccess)
        e = cudaMemcpy(M.b2, b2, 64 * 4, cudaMemcpyDefault);
    if (e == cudaSuccess)
        e = cudaMemcpy(M.E, hub_emb, static_cast<size_t>(H) * 64 * 4, cudaMemcpyDefault);
    if (e == cudaSuccess)
        e = cudaMemset(t->m, 0, o.total * 4);
    if (e == cudaSuccess)
        e = cudaMemset(t->v, 0, o.total * 4);
    if (e == cudaSuccess)
        e = cudaMemset(t->grads, 0, o.total * 4);
    if (e == cudaSuccess)
        e = cudaMemset(t->status, 0, 16);
    if (e != cudaSuccess) {
        ann_status st = cuda_status(e);
        trainer_free(t);
        return st;
    }
    *out = t;
    return ANN_OK;
}

ann_status ann_trainer_free(ann_trainer *t)
{
    trainer_free(t);
    return ANN_OK;
}

ann_status ann_trainer_step(ann_trainer *t, const float *d_queries, const int32_t *d_rows, int64_t nb,
                            const int32_t *d_cand, const int8_t *d_labels, int32_t M, int32_t apply_update,
                            float *loss_out, void *stream)
{
    if (!t || !d_queries || !d_cand || !d_labels || M < 1 || M > t->H || nb < 1 || nb > t->batch ||
        (reinterpret_cast<uintptr_t>(d_queries) & 15))
        return ANN_ERR_INVALID_ARG;
    cudaSetDevice(t->device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    ann_status st = trainer_grads(t, d_queries, d_rows, nb, d_cand, d_labels, M, s);
    if (st != ANN_OK)
        return st;
    if (apply_update) {
        adam_all(t, s);
        st = cuda_status(cudaGetLastError());
    }
    if (st == ANN_OK && loss_out) {
        cudaError_t e = cudaMemcpyAsync(loss_out, t->loss, 4, cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess)
            e = cudaStreamSynchronize(s);
        st = cuda_status(e);
    }
    return st;
}

ann_status ann_trainer_get(const ann_trainer *t, float *W1, float *b1, float *W2, float *b2, float *hub_emb,
                           int32_t gradients)
{
    if (!t)
        return ANN_ERR_INVALID_ARG;
    const Offs o = offsets(t->in_dim, t->H);
    const float *src = gradients ? t->grads : t->params;
    cudaError_t e = cudaDeviceSynchronize();
    auto cp = [&](float *dst, int64_t off, int64_t count) {
        if (dst && e == cudaSuccess)
            e = cudaMemcpy(dst, src + off, count * 4, cudaMemcpyDefault);
    };
    cp(W1, o.W1, static_cast<int64_t>(t->in_dim) * 256);
    cp(b1, o.b1, 256);
    cp(W2, o.W2, 256 * 64);
    cp(b2, o.b2, 64);
    if (hub_emb && t->fu && !gradients && e == cudaSuccess) {
        // the hub rows the model scores: E + F with the current weights
        ann_status st = fusion_forward(t->fu, t->params + o.E, nullptr);
        if (st != ANN_OK)
            return st;
        e = cudaMemcpy(hub_emb, t->fu->Eeff, static_cast<size_t>(t->H) * 64 * 4, cudaMemcpyDefault);
    } else {
        cp(hub_emb, o.E, static_cast<int64_t>(t->H) * 64);
    }
    if (e == cudaSuccess) {
        int st = 0;
        e = cudaMemcpy(&st, t->status, 4, cudaMemcpyDeviceToHost);
        if (e == cudaSuccess && st)
            return ANN_ERR_TIMEOUT;
    }
    return cuda_status(e);
}

ann_status ann_trainer_fit(ann_trainer *t, const float *d_queries, int64_t nt, const int32_t *d_cand,
                           const int8_t *d_labels, int32_t M, const int32_t *d_order, int32_t epochs,
                           float *d_losses, void *stream)
{
    if (!t || !d_queries || !d_cand || !d_labels || M < 1 || M > t->H || nt < 1 || epochs < 0 ||
        (reinterpret_cast<uintptr_t>(d_queries) & 15))
        return ANN_ERR_INVALID_ARG;
    cudaSetDevice(t->device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int32_t *iota = nullptr;
    if (!d_order) {
        std::vector<int32_t> h(nt);
        std::iota(h.begin(), h.end(), 0);
        cudaError_t e = cudaMallocAsync(reinterpret_cast<void **>(&iota), nt * 4, s);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(iota, h.data(), nt * 4, cudaMemcpyHostToDevice, s);
        if (e == cudaSuccess)
            e = cudaStreamSynchronize(s);
        if (e != cudaSuccess)
            return cuda_status(e);
    }
    const int64_t spe = (nt + t->batch - 1) / t->batch;
    ann_status st = ANN_OK;
    for (int ep = 0; ep < epochs && st == ANN_OK; ++ep) {
        const int32_t *ord = d_order ? d_order + static_cast<int64_t>(ep) * nt : iota;
        for (int64_t i = 0; i < spe && st == ANN_OK; ++i) {
            const int64_t nb = std::min<int64_t>(t->batch, nt - i * t->batch);
            st = trainer_grads(t, d_queries, ord + i * t->batch, nb, d_cand, d_labels, M, s);
            if (st != ANN_OK)
                break;
            adam_all(t, s);
            if (d_losses)
                cudaMemcpyAsync(d_losses + ep * spe + i, t->loss, 4, cudaMemcpyDeviceToDevice, s);
            st = cuda_status(cudaGetLastError());
        }
    }
    if (iota)
        cudaFreeAsync(iota, s);
    if (st == ANN_OK)
        st = cuda_status(cudaStreamSynchronize(s));
    return st;
}

ann_status ann_trainer_attach(const ann_trainer *t, ann_index *idx, const int32_t *hub_nodes, int32_t hub_degree,
                              void *stream)
{
    if (!t || !idx || !hub_nodes)
        return ANN_ERR_INVALID_ARG;
    cudaError_t e = cudaDeviceSynchronize();
    if (e != cudaSuccess)
        return cuda_status(e);
    ann_entry_model_desc d{};
    d.in_dim = t->in_dim;
    d.hidden = 256;
    d.out_dim = 64;
    d.W1 = t->model.W1;
    d.b1 = t->model.b1;
    d.W2 = t->model.W2;
    d.b2 = t->model.b2;
    d.n_hubs = t->H;
    d.hub_nodes = hub_nodes;
    d.hub_emb = t->model.E;
    if (t->fu) {
        ann_status st = fusion_forward(t->fu, t->model.E, nullptr);
        if (st == ANN_OK)
            st = cuda_status(cudaDeviceSynchronize());
        if (st != ANN_OK)
            return st;
        d.hub_emb = t->fu->Eeff;
    }
    d.hub_degree = hub_degree;
    d.hub_graph = nullptr;
    d.hub_entry = -1;
    return ann_set_entry_model(idx, &d, stream);
}

ann_status ann_trainer_set_fusion(ann_trainer *t, const float *d_hub_vecs, const float *d_tokens, int32_t T,
                                  int32_t token_dim, int32_t heads, int32_t head_dim, const float *WQ, const float *WK,
                                  const float *WV, const float *WO)
{
    if (!t || !d_hub_vecs || !d_tokens || !WQ || !WK || !WV || !WO || t->fu || t->step != 0 || T < 1 || T > 64 ||
        token_dim < 1 || token_dim > 64 || heads < 1 || head_dim < 1 || heads * head_dim > 256)
        return ANN_ERR_INVALID_ARG;
    cudaSetDevice(t->device);
    cudaError_t e = cudaSuccess;
    t->fu = fusion_create(t->H, T, token_dim, heads, head_dim, t->in_dim, d_hub_vecs, d_tokens, WQ, WK, WV, WO, e);
    return cuda_status(e);
}

ann_status ann_trainer_get_fusion(const ann_trainer *t, float *WQ, float *WK, float *WV, float *WO, int32_t gradients)
{
    if (!t || !t->fu)
        return ANN_ERR_INVALID_ARG;
    const Fusion *f = t->fu;
    const float *src = gradients ? f->grads : f->params;
    cudaError_t e = cudaDeviceSynchronize();
    auto cp = [&](float *dst, int64_t off, int64_t count) {
        if (dst && e == cudaSuccess)
            e = cudaMemcpy(dst, src + off, count * 4, cudaMemcpyDefault);
    };
    cp(WQ, f->oWQ(), static_cast<int64_t>(f->dp) * f->E);
    cp(WK, f->oWK(), static_cast<int64_t>(f->dU) * f->E);
    cp(WV, f->oWV(), static_cast<int64_t>(f->dU) * f->E);
    cp(WO, f->oWO(), static_cast<int64_t>(f->E) * f->dF);
    return cuda_status(e);
}

ann_status ann_adam_update(float *d_params, const float *d_grads, float *d_m, float *d_v, int64_t n, int64_t step,
                           float lr, float beta1, float beta2, float eps, void *stream)
{
    if (!d_params || !d_grads || !d_m || !d_v || n < 0 || step < 1 || !(lr > 0.f) || !(eps > 0.f))
        return ANN_ERR_INVALID_ARG;
    if (n == 0)
        return ANN_OK;
    const float bc1 = 1.f - powf(beta1, static_cast<float>(step));
    const float bc2 = 1.f - powf(beta2, static_cast<float>(step));
    adam_kernel<<<blocks_for(n, 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(d_params, d_grads, d_m, d_v, n, lr,
                                                                                     beta1, beta2, eps, bc1, bc2);
    return cuda_status(cudaGetLastError());
}

}  // extern "C"
