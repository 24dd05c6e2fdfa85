// Router of a large batch on the tensor cores (step a1 of the layer: Sec. 3.1
// of arxiv 2506.23635 feeds every token's router output to the expert
// selection): logits[t, e] = sum_d x[t, d] W_r[d, e] as a [T x D] . [D x E]
// product with E <= 16, then the softmax, top-K and renormalised gates.
//
// k_route_tc: the 8 CTAs of a cluster take the 128 tokens of a tile, CTA r the
//   r-th of 8 equal shares of the 64-column blocks of d.  Its slice of W_r is
//   written by the threads, transposed, into shared memory in the 128-byte
//   swizzled K-major layout (16 expert rows per 64-column panel); the token rows
//   arrive by TMA, all of a share in flight where the SM has room; one lane
//   issues tcgen05.mma (M = 128 tokens, N = 16 experts, K = 16) into 16
//   accumulators in turn (the tensor core truncates when it adds to an
//   accumulator: chains of 3 roundings instead of 48 at d_model 6144; relative
//   error of the logits against 64 bits 0.80e-7, with four accumulators
//   1.84e-7, k_route 0.87e-7).  Four warps read their 32 tokens' rows from
//   tensor memory and store the share's partial logits into the shared memory
//   of the CTA that finishes the token, 16 tokens each: half a warp per token
//   adds the shares (in 64 bits) and selects the top-k (ties to the lower
//   index, NaN ranked as -inf).
// Bound by latency (one kernel after the other, event pairs): 128-600 tokens
// 16 us, 2048 tokens 24 us with x in HBM (17.5 + 10.7 us as two kernels, the
// second for the top-k), 3000 tokens 18-23 us (k_route, which re-reads W_r from
// L2 for every 4 tokens: 48-79 us).
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>

#include "tc.cuh"

namespace moe {
namespace {

using namespace tc;

constexpr int kRtThreads = 256;
constexpr int kRtCluster = 8;                             // shares of d
constexpr int kRtM = 128;                                 // tokens per tile
constexpr int kRtOwn = kRtM / kRtCluster;                 // tokens a CTA finishes
constexpr int kRtBK = 64;                                 // d per k-block (one 128 B row)
constexpr int kRtMaxStages = 12;
constexpr uint32_t kRtStageBytes = kRtM * kRtBK * 2;      // 16 KB of token rows
constexpr uint32_t kRtPanelBytes = 16 * kRtBK * 2;        // 16 expert rows x 128 B
constexpr int kRtAcc = 16;                                // accumulators of 16 columns
constexpr uint32_t kRtTmemCols = kRtAcc * 16;
// kind::f16: bf16 A and B, fp32 D, both K-major, N = 16, M = 128
constexpr uint32_t kRtIdesc =
    (1u << 4) | (1u << 7) | (1u << 10) | ((16u >> 3) << 17) | ((uint32_t)(kRtM >> 4) << 24);

struct RtHeader {
    float part[kRtCluster][kRtOwn][16];  // the shares' logits of this CTA's tokens
    float pk[kRtOwn][16];
    uint64_t full[kRtMaxStages];
    uint64_t empty[kRtMaxStages];
    uint64_t done;
    uint32_t tmem;
    int gave_up;  // the issuer's wait ran out: some accumulators were not written
};

// Ring stages for nkb k-blocks a share: as many as fit beside the router's slice
// in a whole SM's shared memory where every CTA has an SM, in half of it where
// there are more CTAs (0: the slice itself does not fit).
constexpr size_t kRtMaxSmem = 227 * 1024;
size_t rt_smem(int nkb, int n_stage) {
    return 1024 + n_stage * kRtStageBytes + (size_t)nkb * kRtPanelBytes + sizeof(RtHeader);
}
int rt_stages(int nkb, bool shared_sm) {
    int n = std::min(kRtMaxStages, nkb);
    while (n > 0 && rt_smem(nkb, n) > (shared_sm && n > 2 ? kRtMaxSmem / 2 : kRtMaxSmem)) --n;
    return n;
}
// k-blocks of the largest share
int rt_blocks(int D) { return ((D + kRtBK - 1) / kRtBK + kRtCluster - 1) / kRtCluster; }

__device__ __forceinline__ void st_cluster_v4(uint32_t addr, float a, float b, float c, float d) {
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(a), "f"(b),
                 "f"(c), "f"(d)
                 : "memory");
}

// select_topk for up to 16 experts by half a warp, lane e (of 16) with expert
// e's logit: the same operations in the same order.
__device__ __forceinline__ void half_warp_topk(int E, int K, bool live, int t, int e, float l,
                                               float *pk, float *__restrict__ logits_opt,
                                               int32_t *__restrict__ topk_idx,
                                               float *__restrict__ topk_gate) {
    const bool has = e < E;
    if (logits_opt && live && has) logits_opt[(size_t)t * E + e] = l;
    float m = has ? fmaxf(-INFINITY, l) : -INFINITY;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    float z = has ? expf(l - m) : 0.f;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
    bool taken = !has;
    float psel = 0.f;
    for (int k = 0; k < K; ++k) {
        float bv = taken || isnan(l) ? -INFINITY : l;
        int bi = taken ? 0x7fffffff : e;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) {
            const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
            const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
            if (ov > bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
        }
        taken |= bi == e;
        const float p = expf(bv - m) / z;
        psel += p;
        if (e == 0 && live) {
            topk_idx[(size_t)t * K + k] = bi;
            pk[k] = p;
        }
    }
    __syncwarp();
    if (live && e < K) topk_gate[(size_t)t * K + e] = pk[e] / psel;
}

__global__ void __launch_bounds__(kRtThreads)
k_route_tc(const __grid_constant__ CUtensorMap tmX, int T, int D, int E, int K, int n_stage,
           int max_kb, const bf16 *__restrict__ wr, float *__restrict__ logits_opt,
           int32_t *__restrict__ topk_idx, float *__restrict__ topk_gate, unsigned *err) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    unsigned char *wt = smem + n_stage * kRtStageBytes;  // W_r^T slice, max_kb panels
    RtHeader *hd = reinterpret_cast<RtHeader *>(wt + max_kb * kRtPanelBytes);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = (int)ptx::cluster_ctarank();
    const int m0 = (int)(blockIdx.x / kRtCluster) * kRtM;
    const int nkb_total = (D + kRtBK - 1) / kRtBK;
    const int kb0 = nkb_total * rank / kRtCluster;
    const int nkb = nkb_total * (rank + 1) / kRtCluster - kb0;  // <= max_kb

    ptx::launch_dependents();
    if (threadIdx.x == 0) {
        ptx::prefetch_tmap(&tmX);
        for (int s = 0; s < n_stage; ++s) {
            ptx::mbar_init(&hd->full[s], 1);
            ptx::mbar_init(&hd->empty[s], 1);
        }
        ptx::mbar_init(&hd->done, 1);
        ptx::fence_barrier_init();
        hd->gave_up = 0;
        // the token rows may come from the previous kernel (so may W_r, whose
        // layout below waits too); the first stages of them are on the way
        // while W_r is laid out
        ptx::grid_dependency_wait();
        const uint64_t pol = ptx::policy_evict_normal();
        for (int i = 0; i < min(n_stage, nkb); ++i) {
            ptx::mbar_arrive_expect_tx(&hd->full[i], kRtStageBytes);
            ptx::tma_load_2d(smem + i * kRtStageBytes, &tmX, (kb0 + i) * kRtBK, m0, &hd->full[i],
                             pol);
        }
    }
    __syncwarp();
    if (warp == 1) tmem_alloc(&hd->tmem, kRtTmemCols);
    ptx::grid_dependency_wait();
    // W_r^T slice: panel i holds d = (kb0 + i) * 64 + c, c < 64; row e of the
    // panel is expert e (zero past E or past D)
    const bool vec = E == 16;  // a router row is 32 B: two 16-byte loads
#pragma unroll 4
    for (int idx = (int)threadIdx.x - 64; idx < nkb * kRtBK; idx += kRtThreads - 64) {
        if (idx < 0) break;  // (warps 0 and 1: the copies and tensor memory)
        const int i = idx / kRtBK, c = idx - i * kRtBK;
        const int d = (kb0 + i) * kRtBK + c;
        unsigned char *panel = wt + i * kRtPanelBytes;
        uint32_t w[8];  // 16 bf16, expert e in half (e & 1) of w[e / 2]
        if (d < D && vec) {
            const uint4 a = __ldg(reinterpret_cast<const uint4 *>(wr + (size_t)d * 16));
            const uint4 b = __ldg(reinterpret_cast<const uint4 *>(wr + (size_t)d * 16 + 8));
            w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = a.w;
            w[4] = b.x; w[5] = b.y; w[6] = b.z; w[7] = b.w;
        } else {
            const unsigned short *row = reinterpret_cast<const unsigned short *>(wr) + (size_t)d * E;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const uint32_t lo = (d < D && 2 * j < E) ? row[2 * j] : 0u;
                const uint32_t hi = (d < D && 2 * j + 1 < E) ? row[2 * j + 1] : 0u;
                w[j] = lo | (hi << 16);
            }
        }
#pragma unroll
        for (int e = 0; e < 16; ++e)
            *reinterpret_cast<unsigned short *>(panel + swizzle_offset((uint32_t)e, (uint32_t)c)) =
                (unsigned short)(w[e >> 1] >> ((e & 1) * 16));
    }
    fence_proxy_async_smem();  // the slice is read by the MMA (async proxy)
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = hd->tmem;
    // every CTA of the cluster has started before the others store to it
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");

    if (warp == 0) {
        if (lane == 0) {
            const uint64_t pol = ptx::policy_evict_normal();
            int i = min(n_stage, nkb);
            for (; i < nkb; ++i) {
                const uint32_t s = i % n_stage, ph = (i / n_stage) & 1;
                if (!ptx::mbar_wait_hint(&hd->empty[s], ph ^ 1, err)) break;
                ptx::mbar_arrive_expect_tx(&hd->full[s], kRtStageBytes);
                ptx::tma_load_2d(smem + s * kRtStageBytes, &tmX, (kb0 + i) * kRtBK, m0,
                                 &hd->full[s], pol);
            }
            // let copies still in flight land before the block can exit
            for (int k = (i > n_stage ? i - n_stage : 0); k < i; ++k)
                ptx::mbar_wait_hint(&hd->full[k % n_stage], (k / n_stage) & 1, err);
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {
            for (int i = 0; i < nkb; ++i) {
                const uint32_t s = i % n_stage, ph = (i / n_stage) & 1;
                if (!ptx::mbar_wait_hint(&hd->full[s], ph, err)) {
                    hd->gave_up = 1;
                    __threadfence_block();  // ahead of the arrival on `done`
                    break;
                }
                tc_fence_after();
                const uint64_t adesc = smem_desc(ptx::smem_u32(smem + s * kRtStageBytes));
                const uint64_t bdesc = smem_desc(ptx::smem_u32(wt + i * kRtPanelBytes));
#pragma unroll
                for (int kk = 0; kk < kRtBK / 16; ++kk)
                    mma_bf16(tmem + 16 * ((4 * i + kk) % kRtAcc), adesc + 2 * kk, bdesc + 2 * kk,
                             kRtIdesc, 4 * i + kk >= kRtAcc ? 1u : 0u);
                mma_commit(&hd->empty[s]);
            }
            // `done` flips once every MMA issued here has completed
            mma_commit(&hd->done);
            ptx::mbar_wait_hint(&hd->done, 0, err);
        }
        __syncwarp();
    }
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
    if (warp < 4) {
        // the partial logits of the warp's 32 tokens, to the CTAs that finish
        // them (zero for an empty share and after a wait that gave up)
        const bool have = ptx::mbar_wait_hint(&hd->done, 0, err) && nkb > 0 &&
                          *(volatile int *)&hd->gave_up == 0;
        tc_fence_after();
        float p[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) p[e] = 0.f;
        if (__all_sync(0xffffffffu, have)) {
            const int used = min(kRtAcc, 4 * nkb);  // accumulators written: 4, 8, 12 or 16
            float q[16];
#pragma unroll
            for (int a = 0; a < kRtAcc; a += 4) {  // added pairwise
                if (a >= used) break;
                float v[2][32];
                const uint32_t base = tmem + ((uint32_t)(warp * 32) << 16) + 16 * a;
                tmem_ld32(base, v[0]);
                tmem_ld32(base + 32, v[1]);
                tmem_ld_wait();
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                    const float s = (v[0][e] + v[0][16 + e]) + (v[1][e] + v[1][16 + e]);
                    if (a == 0) p[e] = s;
                    else if (a == 4) p[e] += s;
                    else if (a == 8) q[e] = s;
                    else p[e] += q[e] + s;
                }
            }
            if (used == 12) {
#pragma unroll
                for (int e = 0; e < 16; ++e) p[e] += q[e];
            }
        }
        const int row = warp * 32 + lane;
        const uint32_t dst =
            ptx::map_rank(ptx::smem_u32(&hd->part[rank][row % kRtOwn][0]), (uint32_t)(row / kRtOwn));
#pragma unroll
        for (int q = 0; q < 4; ++q)
            st_cluster_v4(dst + 16 * q, p[4 * q], p[4 * q + 1], p[4 * q + 2], p[4 * q + 3]);
    }
    tc_fence_before();
    ptx::cluster_sync_all();  // every share's partials have arrived
    tc_fence_after();
    if (warp == 1) tmem_dealloc(tmem, kRtTmemCols);
    // half a warp for each token: lane e of it adds expert e's shares
    static_assert(2 * (kRtThreads / 32) == kRtOwn, "two tokens a warp");
    const int i = warp * 2 + (lane >> 4), e = lane & 15;
    const int t = m0 + rank * kRtOwn + i;
    double v = 0.0;
#pragma unroll
    for (int r = 0; r < kRtCluster; ++r) v += (double)hd->part[r][i][e];
    half_warp_topk(E, K, t < T, t, e, (float)v, hd->pk[i], logits_opt, topk_idx, topk_gate);
}

}  // namespace

bool route_tc_ok(const moe_dims &d, int T) {
    return T >= kRouteTcMinTokens && d.n_experts <= 16 && d.x_dtype == MOE_BF16 &&
           d.w_dtype == MOE_BF16 && rt_stages(rt_blocks(d.d_model), false) > 0 &&
           encode_fn() != nullptr;
}

cudaError_t launch_route_tc(const moe_dims &d, int T, const void *x, const void *wr,
                            float *logits, int32_t *idx, float *gate, cudaStream_t st) {
    int Tv = T, D = d.d_model, E = d.n_experts, K = d.top_k;
    const int grid = (T + kRtM - 1) / kRtM * kRtCluster;
    // (clusters of 8 fill three quarters of the SMs or more: 15 of them on 152)
    int max_kb = rt_blocks(D), n_stage = rt_stages(max_kb, 4 * grid > 3 * device_info().sm_count);
    CUtensorMap tmx;
    if (!make_map(&tmx, x, (uint64_t)T, (uint64_t)D, kRtM)) return cudaErrorInvalidValue;
    const void *kern = (const void *)k_route_tc;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kRtMaxSmem);
    if (e != cudaSuccess) return e;
    const bf16 *wp = static_cast<const bf16 *>(wr);
    unsigned *err = device_info().err;
    void *args[] = {&tmx, &Tv, &D, &E, &K, &n_stage, &max_kb, &wp, &logits, &idx, &gate, &err};
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kRtThreads);
    cfg.dynamicSmemBytes = rt_smem(max_kb, n_stage);
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = kRtCluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    LaunchScope ls("route", st);
    return cudaLaunchKernelExC(&cfg, kern, args);
}

}  // namespace moe
