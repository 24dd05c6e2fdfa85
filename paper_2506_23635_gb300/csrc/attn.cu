// Self-attention block of a DBRX-style decoder layer and whole decoder
// layers (self-attention, then the MoE block).
//
// Table 1 (note (b)) of arxiv 2506.23635 sizes the self-attention of a layer
// only by its parameters (D_qkv_hidden x D_embed + D_embed^2) and FLOPs (twice
// that); Table 2 books it under "Misc.".  The block built here is the reading
// stated in include/moe.h: grouped-query attention with head_dim 128, rotary
// embedding of queries and keys, causal softmax attention over a bf16 KV
// cache, no biases, resid += W_o . Attn(RMSNorm0(resid)).
//
// Kernels, in launch order:
//   k_sa_prenorm   RMSNorm0 of the fp32 residual -> bf16 rows; the first token's
//                  block also writes the trivial dispatch of a one-"expert" projection
//                  (offsets {0, T}), for the grouped GEMM of prefill batches;
//                  in a planned call block 0 makes the attention's plan and the
//                  tokens follow;
//                  it lets the projection launch once its own wait is over (the
//                  projection's weight loads do not depend on it);
//   projection     W_qkv . x (fp32 out): the CTA-pair tcgen05 GEMM in equal
//                  shares of its (unit, k-block)s where whole units would leave
//                  a quarter of the pairs idle (proj_split, 257 to 2048 tokens), else
//                  the tcgen05 kernel with the weights as the M operand (split
//                  reduction) for up to 512 or 640 tokens (gemm_rows_fits), else
//                  the grouped tcgen05 GEMM with E = 1;
//   k_rope_cache   rotary embedding of q and k (angles formed and reduced in
//                  fp64, evaluated in fp32), k and v written to the cache in
//                  bf16;
//   k_attn_partial one CTA per (token, key/value head, position split): the
//                  group's query heads against its positions, online softmax,
//                  partial (max, sum, weighted values) per split;
//   k_attn_merge   merges the splits, ctx in bf16 (a single split writes ctx
//                  itself); both run only where the tensor cores do not take
//                  the tokens: the prefill attention (attn_tc.cu) the tiles
//                  of consecutive positions that the plan finds (a block of
//                  k_sa_prenorm), the decode attention (attn_decode_tc.cu)
//                  every other token;
//   projection     W_o . ctx (the weights-as-M kernel or, where that does not
//                  fit, the grouped GEMM): a projection in one part is added to
//                  the residual by its epilogue, partial sums by
//                  k_residual_add or, in decoder layers, k_residual_prenorm.
#include <math.h>
#include <stdlib.h>

#include <algorithm>

#include "ptx.cuh"

namespace moe {
namespace {

constexpr int kHeadDim = 128;
constexpr int kMaxGroup = 8;       // query heads per key/value head
constexpr int kAttnThreads = 128;  // 4 warps
constexpr int kAttnWarps = kAttnThreads / 32;
constexpr int kSplitTarget = 152;     // CTAs a decode step's attention aims for at least
constexpr int kSplitPositions = 128;  // cache positions per split (a 32-position tile per warp)
constexpr int kMaxSplit = 64;
constexpr int kMaxSplitCtas = 4096;   // bound on T * Hkv * splits (sizes the workspace)
constexpr int kMaxSaTokens = 65536;
static_assert(kMaxSaTokens <= (kAttnDecodeCounts - kAttnDecodeMaxCtas) * kAttnDecodeMaxTokens,
              "a counter for every 128 tokens");

// Most position splits a call of T tokens may use (the workspace holds this many).
int split_cap(int T, int Hkv) {
    const int tg = std::max(1, T * Hkv);
    return std::max(1, std::min(kMaxSplit, kMaxSplitCtas / tg));
}

// Splits per (token, key/value head): enough CTAs to cover the SMs and at
// most kSplitPositions cache positions per split, within split_cap.
int n_split_for(int T, int Hkv, int max_len) {
    const int tg = std::max(1, T * Hkv);
    const int by_ctas = (kSplitTarget + tg - 1) / tg;
    const int by_len = (max_len + kSplitPositions - 1) / kSplitPositions;
    return std::max(1, std::min(split_cap(T, Hkv), std::max(by_ctas, by_len)));
}

// Rotary angular rates base^(-2i/dh), i < dh/2, computed on the host in
// double precision and passed by value.
struct RopeRates {
    double w[kHeadDim / 2];
};

// ---- kernels --------------------------------------------------------------------

// The trivial dispatch of a one-"expert" projection: offsets {0, T}.
__device__ __forceinline__ void write_trivial_dispatch(int T, int32_t *offsets) {
    if (threadIdx.x == 0) {
        offsets[0] = 0;
        offsets[1] = T;
    }
}

// One block per token: 1024 threads for decode batches (every thread's
// loads of the row in flight together), 256 threads with 16 float4 of the
// row each for larger batches (the 1024-thread form ran at 1.9 TB/s over
// 2048 tokens: too little work per thread between block barriers).  The row
// stays in registers between the sum of squares and the scaling.
constexpr int kNormThreads = 1024;
constexpr int kNormThreadsWide = 256;
constexpr int kNormWideMinTokens = 64;
constexpr int kNormMaxVec = 16;  // float4 per thread: D <= 4 * 16 * 256

// What the attention's plan is made from, and where it goes (plan.head null:
// the call needs none).
struct PlanArgs {
    const int32_t *seq, *pos;
    int n_seq, L;
    AttnPlan plan;
};

// The plan of an attention call, by one block of NT threads.  A run is the
// longest stretch of tokens that are consecutive positions of one sequence;
// its tiles are cut from its first token on.  Tiles of at least
// kAttnTileMinRows tokens are listed by falling length (a counting sort over
// their key/value tiles; tiles of the same length in any order: no result
// depends on it), the tokens of the others in ascending order.  Run starts are
// kept as one bit a token.  It runs beside the pre-norm's other blocks and is
// done before the projection after them ends.
constexpr int kPlanBins = 256;

template <int NT>
__device__ void plan_attention(int T, const PlanArgs &a) {
    static_assert(NT >= kPlanBins && NT % 32 == 0, "a thread for each bin");
    __shared__ uint32_t brk[kMaxSaTokens / 32];  // bit t: a run starts at token t
    __shared__ int last[kMaxSaTokens / 32];      // the last run start ahead of each word
    __shared__ int bins[kPlanBins];
    __shared__ int wsum[NT / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nw = (T + 31) / 32;
    for (int t = tid; t < nw * 32; t += NT) {
        bool b = false;
        if (t < T) {
            const int sq = a.seq[t], p = a.pos[t];
            // (a token outside the cache is a run of its own)
            b = t == 0 || sq < 0 || sq >= a.n_seq || p <= 0 || p >= a.L || a.seq[t - 1] != sq ||
                a.pos[t - 1] != p - 1;
        }
        const uint32_t m = __ballot_sync(0xffffffffu, b);
        if (lane == 0) brk[t >> 5] = m;
    }
    if (tid < kPlanBins) bins[tid] = 0;
    __syncthreads();
    if (warp == 0) {
        int run = 0;
        for (int w0 = 0; w0 < nw; w0 += 32) {
            const int w = w0 + lane;
            int v = w < nw && brk[w] ? w * 32 + 31 - __clz(brk[w]) : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v = max(v, u);
            }
            v = max(v, run);
            const int ahead = __shfl_up_sync(0xffffffffu, v, 1);
            if (w < nw) last[w] = lane == 0 ? run : ahead;
            run = __shfl_sync(0xffffffffu, v, 31);
        }
    }
    __syncthreads();
    // the tile of token t: its first token, and its tokens
    auto tile_of = [&](int t, int &ts, int &rows) {
        const uint32_t m = brk[t >> 5] & (0xffffffffu >> (31 - (t & 31)));
        const int rs = m ? (t & ~31) + 31 - __clz(m) : last[t >> 5];
        ts = rs + ((t - rs) & ~(kAttnTile - 1));
        int end = min(ts + kAttnTile, T);
        int w = (ts + 1) >> 5;
        uint32_t n = w < nw ? brk[w] & (0xffffffffu << ((ts + 1) & 31)) : 0u;
        while (n == 0 && (w + 1) * 32 < end) n = brk[++w];
        if (n) end = min(end, w * 32 + __ffs(n) - 1);
        rows = end - ts;
    };
    auto bin_of = [&](int ts, int rows) {  // falling length
        return kPlanBins - 1 - min(kPlanBins - 1, (a.pos[ts] + rows - 1) / kAttnTile);
    };
    int n_left = 0;
    for (int t0 = 0; t0 < T; t0 += NT) {
        const int t = t0 + tid;
        bool left = false;
        if (t < T) {
            int ts, rows;
            tile_of(t, ts, rows);
            left = rows < kAttnTileMinRows;
            if (!left && t == ts) atomicAdd(&bins[bin_of(ts, rows)], 1);
        }
        const uint32_t m = __ballot_sync(0xffffffffu, left);
        if (lane == 0) wsum[warp] = __popc(m);
        __syncthreads();
        int at = n_left + __popc(m & ((1u << lane) - 1u));
        for (int w = 0; w < NT / 32; ++w) {
            at += w < warp ? wsum[w] : 0;
            n_left += wsum[w];
        }
        if (left) a.plan.left[at] = t;
        __syncthreads();
    }
    if (warp == 0) {  // bins -> first place of each
        int run = 0;
        for (int b0 = 0; b0 < kPlanBins; b0 += 32) {
            const int c = bins[b0 + lane];
            int v = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += u;
            }
            bins[b0 + lane] = run + v - c;
            run += __shfl_sync(0xffffffffu, v, 31);
        }
        if (lane == 0) *a.plan.head = AttnPlanHead{run, n_left, 0, 0};
    }
    __syncthreads();
    for (int t = tid; t < T; t += NT) {
        int ts, rows;
        tile_of(t, ts, rows);
        if (t == ts && rows >= kAttnTileMinRows)
            a.plan.tiles[atomicAdd(&bins[bin_of(ts, rows)], 1)] =
                make_int4(ts, rows, a.pos[ts], a.seq[ts]);
    }
}

template <int NT, int VEC>
__global__ void __launch_bounds__(NT)
k_sa_prenorm(int T, int D, const float *__restrict__ resid, bf16 *__restrict__ xn, float eps,
             int32_t *offsets, const PlanArgs pa) {
    ptx::grid_dependency_wait();
    // the projection after this kernel may start now: its weight loads do not
    // depend on anything here, and what is ahead of the call, which may have
    // written the weights, is complete (so only after the wait)
    ptx::launch_dependents();
    __shared__ float red[NT / 32];
    int t = blockIdx.x;
    if (pa.plan.head) {  // block 0 makes the attention's plan
        if (t == 0) {
            plan_attention<NT>(T, pa);
            return;
        }
        --t;
    }
    if (t == 0) write_trivial_dispatch(T, offsets);
    const float4 *r = reinterpret_cast<const float4 *>(resid + (size_t)t * D);
    const int nv = D >> 2;
    float4 keep[VEC];
    float ss = 0.f;
#pragma unroll
    for (int u = 0; u < VEC; ++u) {
        const int i = threadIdx.x + u * NT;
        keep[u] = i < nv ? r[i] : make_float4(0.f, 0.f, 0.f, 0.f);
        ss += keep[u].x * keep[u].x + keep[u].y * keep[u].y + keep[u].z * keep[u].z +
              keep[u].w * keep[u].w;
    }
    for (int i = threadIdx.x + VEC * NT; i < nv; i += NT) {  // rows wider than the registers
        const float4 v = r[i];
        ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
    }
    ss = warp_sum(ss);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
    __syncthreads();
    float tot = 0.f;
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) tot += red[w];
    const float s = 1.0f / sqrtf(tot / (float)D + eps);
    __nv_bfloat162 *o = reinterpret_cast<__nv_bfloat162 *>(xn + (size_t)t * D);
#pragma unroll
    for (int u = 0; u < VEC; ++u) {
        const int i = threadIdx.x + u * NT;
        if (i < nv) {
            o[2 * i] = __floats2bfloat162_rn(keep[u].x * s, keep[u].y * s);
            o[2 * i + 1] = __floats2bfloat162_rn(keep[u].z * s, keep[u].w * s);
        }
    }
    for (int i = threadIdx.x + VEC * NT; i < nv; i += NT) {
        const float4 v = r[i];
        o[2 * i] = __floats2bfloat162_rn(v.x * s, v.y * s);
        o[2 * i + 1] = __floats2bfloat162_rn(v.z * s, v.w * s);
    }
}

__global__ void __launch_bounds__(256)
k_sa_setup(int T, int32_t *offsets) {
    ptx::grid_dependency_wait();
    write_trivial_dispatch(T, offsets);
}

// The decode attention's counters start at zero (threads of one block).
__device__ __forceinline__ void zero_dec_count(int *count) {
    if (count)
        for (int i = threadIdx.x; i < kAttnDecodeCounts; i += blockDim.x) count[i] = 0;
}

// qkv [T, (Hq + 2 Hkv) 128] fp32 (the sum of n_part partial projections
// part_stride floats apart) -> q [T, Hq, 128] rotated, in fp32 and in bf16
// (either may be left out); rotated keys
// and the values to the caches [n_seq, Hkv, L, 128] in bf16.  A block holds
// kRopeRows head rows of kRopeTokens tokens, a warp a head row: lane l turns
// the pairs (2l, 2l + 64) and (2l + 1, 2l + 65) of a query or key head, or
// copies those values.  Bound by memory latency: two 8-byte loads a token in
// flight for each lane, the angles of a token formed by four blocks (with one
// pair a thread and eight blocks 25 instead of 22 us at 1000 tokens, 16.6
// instead of 13.9 at 529).
constexpr int kRopeRows = 16;   // head rows per block
constexpr int kRopeTokens = 4;  // tokens per block
constexpr int kRopeThreads = kRopeRows * 32;

__device__ __forceinline__ void store_bf16x2(bf16 *p, float a, float b) {
    *reinterpret_cast<__nv_bfloat162 *>(p) = __floats2bfloat162_rn(a, b);
}

__global__ void __launch_bounds__(kRopeThreads)
k_rope_cache(int T, int Hq, int Hkv, int n_seq, int L, RopeRates rates,
             const int32_t *__restrict__ seq, const int32_t *__restrict__ pos,
             const float *__restrict__ qkv, int n_part, long long part_stride,
             const ProjSplit split, float *__restrict__ q, bf16 *__restrict__ q16, bf16 *__restrict__ kc,
             bf16 *__restrict__ vc, int *__restrict__ dec_count, unsigned *err) {
    // the tensor-core attention, one CTA per SM on the SMs that this grid
    // leaves free, may launch now and set itself up while this kernel runs
    // (ahead of this kernel's own wait: the projection before it ends without
    // a trigger, so all that is ahead of the call is complete)
    ptx::launch_dependents();
    ptx::grid_dependency_wait();
    if (blockIdx.x == 0 && blockIdx.y == 0) zero_dec_count(dec_count);
    constexpr int H2 = kHeadDim / 2;
    static_assert(kRopeTokens * H2 <= kRopeThreads, "one thread per (token, pair)");
    __shared__ __align__(8) float cs_s[kRopeTokens][H2], sn_s[kRopeTokens][H2];
    __shared__ int seq_s[kRopeTokens], pos_s[kRopeTokens];
    const int hr = blockIdx.x * kRopeRows + threadIdx.x / 32;
    const int i = 2 * (threadIdx.x % 32);
    const int nq = Hq * kHeadDim, nkv = Hkv * kHeadDim;
    const int tb = blockIdx.y * kRopeTokens;
    const int nt = min(kRopeTokens, T - tb);
    // every token's pairs first (independent loads in flight together, and
    // in flight while the angles are formed), the projection's partial sums
    // added in order
    const bool row_ok = hr < Hq + 2 * Hkv;
    // n_part 0: as many parts as the projection's split left each (row, token)
    __shared__ int np_s[kRopeTokens][kRopeRows];
    if (n_part == 0) {
        if (threadIdx.x < kRopeTokens * kRopeRows) {
            const int u = threadIdx.x / kRopeRows, r = threadIdx.x % kRopeRows;
            np_s[u][r] = split.parts(T, min(tb + u, T - 1),
                                     min((int)blockIdx.x * kRopeRows + r, Hq + 2 * Hkv - 1) * kHeadDim);
        }
        __syncthreads();
    }
    float2 av[kRopeTokens], bv[kRopeTokens];
#pragma unroll
    for (int u = 0; u < kRopeTokens; ++u) {
        av[u] = bv[u] = make_float2(0.f, 0.f);
        if (row_ok && u < nt) {
            const float *row = qkv + (size_t)(tb + u) * (nq + 2 * nkv) + (size_t)hr * kHeadDim + i;
            const int np = n_part > 0 ? n_part : np_s[u][threadIdx.x / 32];
            for (int k = 0; k < np; ++k) {
                const float2 a = *reinterpret_cast<const float2 *>(row + k * part_stride);
                const float2 b = *reinterpret_cast<const float2 *>(row + k * part_stride + H2);
                av[u].x += a.x;
                av[u].y += a.y;
                bv[u].x += b.x;
                bv[u].y += b.y;
            }
        }
    }
    // the angles of every token of the block: pair i of token tb+u turns by
    // pos * rate_i, formed and reduced to [-pi, pi] in fp64 (exact to far
    // below fp32 resolution at any cache position), evaluated in fp32
    if (threadIdx.x < nt * H2) {
        const int u = threadIdx.x / H2, k = threadIdx.x % H2;
        const int sq = seq[tb + u], p = pos[tb + u];
        const bool ok = sq >= 0 && sq < n_seq && p >= 0 && p < L;
        if (k == 0) {
            seq_s[u] = ok ? sq : -1;
            pos_s[u] = p;
            if (!ok && blockIdx.x == 0) set_error(err, kErrIndex);
        }
        constexpr double kTwoPi = 6.283185307179586;
        const double ang = (double)(ok ? p : 0) * rates.w[k];
        const double red = fma(-rint(ang * (1.0 / kTwoPi)), kTwoPi, ang);
        sincosf((float)red, &sn_s[u][k], &cs_s[u][k]);
    }
    __syncthreads();
    if (!row_ok) return;
#pragma unroll
    for (int u = 0; u < kRopeTokens; ++u) {
        if (u >= nt) break;
        const int t = tb + u, sq = seq_s[u], p = pos_s[u];
        const float2 a = av[u], b = bv[u];
        if (hr >= Hq + Hkv) {  // a value head: stored as it is
            if (sq < 0) continue;
            bf16 *vd = vc + (((size_t)sq * Hkv + (hr - Hq - Hkv)) * L + p) * kHeadDim + i;
            store_bf16x2(vd, a.x, a.y);
            store_bf16x2(vd + H2, b.x, b.y);
            continue;
        }
        const float2 cs = *reinterpret_cast<const float2 *>(&cs_s[u][i]);
        const float2 sn = *reinterpret_cast<const float2 *>(&sn_s[u][i]);
        const float2 x0 = make_float2(a.x * cs.x - b.x * sn.x, a.y * cs.y - b.y * sn.y);
        const float2 x1 = make_float2(b.x * cs.x + a.x * sn.x, b.y * cs.y + a.y * sn.y);
        if (hr < Hq) {
            if (q) {
                float *qo = q + (size_t)t * nq + (size_t)hr * kHeadDim + i;
                *reinterpret_cast<float2 *>(qo) = x0;
                *reinterpret_cast<float2 *>(qo + H2) = x1;
            }
            if (q16) {  // the tensor-core attention's copy
                bf16 *qh = q16 + (size_t)t * nq + (size_t)hr * kHeadDim + i;
                store_bf16x2(qh, x0.x, x0.y);
                store_bf16x2(qh + H2, x1.x, x1.y);
            }
        } else if (sq >= 0) {
            bf16 *kd = kc + (((size_t)sq * Hkv + (hr - Hq)) * L + p) * kHeadDim + i;
            store_bf16x2(kd, x0.x, x0.y);
            store_bf16x2(kd + H2, x1.x, x1.y);
        }
    }
}

// 8-byte asynchronous global -> shared copy (per thread) and its group wait.
__device__ __forceinline__ void cp_async8(void *dst_smem, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(ptx::smem_u32(dst_smem)),
                 "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
    asm volatile("cp.async.commit_group;" ::: "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

__device__ __forceinline__ void unpack4(uint2 u, float (&o)[4]) {
    unpack_bf16x2(u.x, o[0], o[1]);
    unpack_bf16x2(u.y, o[2], o[3]);
}

// One CTA per (split s, token t, key/value head g); the split covers cache
// positions [j0, j1) of token t's sequence.  Each warp takes tiles of 32
// positions (tile i of warp w starts at j0 + 32*(w + kAttnWarps*i)):
//   scores: lane l owns position l of the tile and computes the full dot
//     products with the G query heads (queries pre-scaled in shared memory),
//     so no cross-lane reduction per position;
//   softmax: per head, one warp max and one warp sum per tile update the
//     running (max m, sum l) and rescale the accumulator;
//   values: lane l owns dims [4l, 4l+4); for each position of the tile the
//     head weights are broadcast from the owning lane and the value row is
//     read coalesced.
// Partial results per (t, query head, s): m, l, and the weighted value sum
// (relative to m).
template <int G>
__global__ void __launch_bounds__(kAttnThreads)
k_attn_partial(int Hq, int Hkv, int n_seq, int L, int n_split, int n_tg,
               const int32_t *__restrict__ seq, const int32_t *__restrict__ pos,
               const float *__restrict__ q, const bf16 *__restrict__ kc,
               const bf16 *__restrict__ vc, float *__restrict__ part_ml,
               float *__restrict__ part_acc, bf16 *__restrict__ ctx,
               const AttnPlan plan) {
    ptx::grid_dependency_wait();
    __shared__ __align__(16) float qs[G][kHeadDim];
    __shared__ float sm_m[kAttnWarps][G], sm_l[kAttnWarps][G];
    __shared__ float sm_acc[kAttnWarps][G][kHeadDim];
    __shared__ __align__(16) bf16 vtile[kAttnWarps][32][kHeadDim];  // each warp's value tile
    const int s = blockIdx.x;
    // (token, key/value head) items blockIdx.y, + gridDim.y, ...: with a plan
    // only those of the tokens that no tensor-core tile holds
    if (plan.head) n_tg = plan.head->n_left * Hkv;
    for (int tg = blockIdx.y; tg < n_tg; tg += gridDim.y) {
        const int i0 = tg / Hkv, g = tg - i0 * Hkv;
        const int t = plan.head ? plan.left[i0] : i0;
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        const int sq = seq[t], p = pos[t];
        const bool ok = sq >= 0 && sq < n_seq && p >= 0 && p < L;
        const int n = ok ? p + 1 : 0;
        const int chunk = (n + n_split - 1) / n_split;
        const int j0 = min(n, s * chunk), j1 = min(n, j0 + chunk);
        const float scale = 1.0f / sqrtf((float)kHeadDim);
        // the queries as stored activations: rounded to bf16, as the
        // tensor-core kernels read them
        for (int i = threadIdx.x; i < G * kHeadDim; i += blockDim.x)
            qs[i / kHeadDim][i % kHeadDim] =
                __bfloat162float(
                    __float2bfloat16_rn(q[((size_t)t * Hq + g * G) * kHeadDim + i])) *
                scale;
        __syncthreads();

        float m[G], l[G], acc[G][4];
#pragma unroll
        for (int h = 0; h < G; ++h) {
            m[h] = -INFINITY;
            l[h] = 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[h][i] = 0.f;
        }
        const size_t base = ok ? ((size_t)sq * Hkv + g) * L * kHeadDim : 0;
        const bf16 *kb = kc + base;
        const bf16 *vb = vc + base;
        for (int jt = j0 + warp * 32; jt < j1; jt += kAttnWarps * 32) {
            const int jl = jt + lane;  // this lane's position
            const bool live = jl < j1;
            const int nt = min(32, j1 - jt);
            // the tile's value rows land in shared memory while the scores are
            // computed: lane l copies bytes [8l, 8l+8) of every row
            __syncwarp();
            for (int u = 0; u < nt; ++u)
                cp_async8(&vtile[warp][u][lane * 4], vb + (size_t)(jt + u) * kHeadDim + lane * 4);
            cp_async_commit();
            float sc[G];
#pragma unroll
            for (int h = 0; h < G; ++h) sc[h] = 0.f;
            if (live) {
                const uint4 *kr = reinterpret_cast<const uint4 *>(kb + (size_t)jl * kHeadDim);
#pragma unroll
                for (int c = 0; c < kHeadDim / 32; ++c) {  // 32 dims per step
                    uint4 u[4];
#pragma unroll
                    for (int v = 0; v < 4; ++v) u[v] = __ldg(kr + c * 4 + v);
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        float k8[8];
                        unpack_bf16x2(u[v].x, k8[0], k8[1]);
                        unpack_bf16x2(u[v].y, k8[2], k8[3]);
                        unpack_bf16x2(u[v].z, k8[4], k8[5]);
                        unpack_bf16x2(u[v].w, k8[6], k8[7]);
                        const int d0 = c * 32 + v * 8;
#pragma unroll
                        for (int h = 0; h < G; ++h) {
                            const float4 qa = *reinterpret_cast<const float4 *>(&qs[h][d0]);
                            const float4 qb = *reinterpret_cast<const float4 *>(&qs[h][d0 + 4]);
                            sc[h] = fmaf(qa.x, k8[0], sc[h]);
                            sc[h] = fmaf(qa.y, k8[1], sc[h]);
                            sc[h] = fmaf(qa.z, k8[2], sc[h]);
                            sc[h] = fmaf(qa.w, k8[3], sc[h]);
                            sc[h] = fmaf(qb.x, k8[4], sc[h]);
                            sc[h] = fmaf(qb.y, k8[5], sc[h]);
                            sc[h] = fmaf(qb.z, k8[6], sc[h]);
                            sc[h] = fmaf(qb.w, k8[7], sc[h]);
                        }
                    }
                }
            }
            float w[G];
#pragma unroll
            for (int h = 0; h < G; ++h) {
                float tm = live ? sc[h] : -INFINITY;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
                    tm = fmaxf(tm, __shfl_xor_sync(0xffffffffu, tm, o));
                const float mn = fmaxf(m[h], tm);  // finite: the tile has a live lane
                const float corr = expf(m[h] - mn);  // 0 while m is -inf
                w[h] = live ? expf(sc[h] - mn) : 0.f;
                l[h] = l[h] * corr + warp_sum(w[h]);
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[h][i] *= corr;
                m[h] = mn;
            }
            cp_async_wait_all();
            __syncwarp();
#pragma unroll 4
            for (int u = 0; u < nt; ++u) {
                float v4[4];
                unpack4(*reinterpret_cast<const uint2 *>(&vtile[warp][u][lane * 4]), v4);
#pragma unroll
                for (int h = 0; h < G; ++h) {
                    const float wu = __shfl_sync(0xffffffffu, w[h], u);
#pragma unroll
                    for (int i = 0; i < 4; ++i) acc[h][i] = fmaf(wu, v4[i], acc[h][i]);
                }
            }
        }
#pragma unroll
        for (int h = 0; h < G; ++h) {
            if (lane == 0) {
                sm_m[warp][h] = m[h];
                sm_l[warp][h] = l[h];
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) sm_acc[warp][h][lane * 4 + i] = acc[h][i];
        }
        __syncthreads();
        const int d = threadIdx.x;
#pragma unroll 1
        for (int h = 0; h < G; ++h) {
            float M = -INFINITY;
#pragma unroll
            for (int w = 0; w < kAttnWarps; ++w) M = fmaxf(M, sm_m[w][h]);
            float Ls = 0.f, A = 0.f;
            if (M != -INFINITY) {
#pragma unroll
                for (int w = 0; w < kAttnWarps; ++w) {
                    const float c = expf(sm_m[w][h] - M);
                    Ls = fmaf(sm_l[w][h], c, Ls);
                    A = fmaf(sm_acc[w][h][d], c, A);
                }
            }
            if (n_split == 1) {  // the only split: this is the result
                ctx[((size_t)t * Hq + g * G + h) * kHeadDim + d] =
                    __float2bfloat16_rn(Ls > 0.f ? A / Ls : 0.f);
                continue;
            }
            const size_t o = ((size_t)t * Hq + g * G + h) * n_split + s;
            if (d == 0) {
                part_ml[2 * o] = M;
                part_ml[2 * o + 1] = Ls;
            }
            part_acc[o * kHeadDim + d] = A;
        }
    }
}

// ctx[t, h*128 + d] = merged weighted values / merged sum, over the splits:
// ctx = sum_s e^(M_s - M) A_s[d] / sum_s e^(M_s - M) L_s.  The splits'
// (max, sum) pairs are read once into shared memory; kMergeGroups groups of
// 128 threads each sum every kMergeGroups-th split of their dimension with
// independent loads, and the groups' sums are added in group order.
constexpr int kMergeGroups = 4;

__global__ void __launch_bounds__(kHeadDim * kMergeGroups)
k_attn_merge(int n_split, const float *__restrict__ part_ml, const float *__restrict__ part_acc,
             bf16 *__restrict__ ctx) {
    static_assert(kMaxSplit <= kHeadDim * kMergeGroups, "one thread per split");
    ptx::launch_dependents();  // the output projection may start streaming its weights
    ptx::grid_dependency_wait();
    __shared__ float sm[kMaxSplit], sl[kMaxSplit], sc[kMaxSplit];
    __shared__ float sa[kMergeGroups][kHeadDim], sls[kMergeGroups][kHeadDim];
    const int th = blockIdx.x, tid = threadIdx.x;
    const int d = tid % kHeadDim, grp = tid / kHeadDim;
    const float *ml = part_ml + (size_t)th * n_split * 2;
    if (tid < n_split) {
        sm[tid] = ml[2 * tid];
        sl[tid] = ml[2 * tid + 1];
    }
    __syncthreads();
    float M = -INFINITY;
    for (int k = 0; k < n_split; ++k) M = fmaxf(M, sm[k]);
    if (tid < n_split) sc[tid] = M != -INFINITY ? expf(sm[tid] - M) : 0.f;
    __syncthreads();
    float Ls = 0.f, A = 0.f;
    const float *pa = part_acc + (size_t)th * n_split * kHeadDim + d;
#pragma unroll 4
    for (int k = grp; k < n_split; k += kMergeGroups) {
        Ls = fmaf(sl[k], sc[k], Ls);
        A = fmaf(pa[(size_t)k * kHeadDim], sc[k], A);
    }
    sa[grp][d] = A;
    sls[grp][d] = Ls;
    __syncthreads();
    if (grp != 0) return;
    for (int g = 1; g < kMergeGroups; ++g) {
        A += sa[g][d];
        Ls += sls[g][d];
    }
    ctx[(size_t)th * kHeadDim + d] = __float2bfloat16_rn(Ls > 0.f ? A / Ls : 0.f);
}

// The tensor-core attention's bf16 copy of fp32 queries, for a call that
// brings its own queries (moe_sa_attend); in the whole block the rotary
// kernel writes it.  n4 groups of four elements.  It lets no launch start before
// its wait: the decode attention reads seq and pos ahead of its own.
__global__ void __launch_bounds__(256)
k_q_bf16(int T, long long n4, const float *__restrict__ q, bf16 *__restrict__ q16,
         int *__restrict__ dec_count, const PlanArgs pa) {
    ptx::grid_dependency_wait();
    if (blockIdx.x == 0) zero_dec_count(dec_count);
    if (blockIdx.x == 0 && pa.plan.head) plan_attention<256>(T, pa);
    const float4 *a = reinterpret_cast<const float4 *>(q);
    __nv_bfloat162 *o = reinterpret_cast<__nv_bfloat162 *>(q16);
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n4;
         i += (long long)gridDim.x * blockDim.x) {
        const float4 v = a[i];
        o[2 * i] = __floats2bfloat162_rn(v.x, v.y);
        o[2 * i + 1] = __floats2bfloat162_rn(v.z, v.w);
    }
}

// resid += y_0 + ... + y_{n_part-1} (partial projections n4 float4 apart,
// added in order before the residual).
__global__ void __launch_bounds__(256)
k_residual_add(long long n4, int n_part, float *__restrict__ resid, const float *__restrict__ y) {
    ptx::grid_dependency_wait();
    float4 *r = reinterpret_cast<float4 *>(resid);
    const float4 *a = reinterpret_cast<const float4 *>(y);
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n4;
         i += (long long)gridDim.x * blockDim.x) {
        float4 w = a[i];
        for (int k = 1; k < n_part; ++k) {
            const float4 u = a[k * n4 + i];
            w.x += u.x;
            w.y += u.y;
            w.z += u.z;
            w.w += u.w;
        }
        float4 v = r[i];
        v.x += w.x;
        v.y += w.y;
        v.z += w.z;
        v.w += w.w;
        r[i] = v;
    }
}

// Decoder layers: resid[t] += sum of the n_part partial projections (0: they
// have been added), then the MoE
// block's input xn[t] = bf16(RMSNorm0(resid[t])) -- the residual add of the
// attention block and the pre-norm of the MoE block in one pass, one block
// per token with the row in registers (NT threads x VEC float4: 1024 x 4 for
// decode batches, 256 x 16 for larger ones, as k_sa_prenorm; D <= 16384).
constexpr int kResNormCap = 4 * 4 * kNormThreads;  // row length the fused form holds

template <int NT, int VEC>
__global__ void __launch_bounds__(NT)
k_residual_prenorm(int T, int D, int n_part, float *__restrict__ resid, const float *__restrict__ y,
                   bf16 *__restrict__ xn, float eps) {
    static_assert(4 * NT * VEC == kResNormCap, "both forms hold a row of kResNormCap");
    ptx::grid_dependency_wait();
    __shared__ float red[NT / 32];
    const int t = blockIdx.x;
    const int nv = D >> 2;
    const long long stride4 = (long long)T * nv;  // between partial projections, in float4
    float4 *r = reinterpret_cast<float4 *>(resid + (size_t)t * D);
    const float4 *a = reinterpret_cast<const float4 *>(y + (size_t)t * D);
    float4 keep[VEC];
    float ss = 0.f;
#pragma unroll
    for (int u = 0; u < VEC; ++u) {
        const int i = threadIdx.x + u * NT;
        keep[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i < nv) {
            float4 v = r[i];
            if (n_part > 0) {
                float4 w = a[i];
                for (int k = 1; k < n_part; ++k) {
                    const float4 v1 = a[k * stride4 + i];
                    w.x += v1.x;
                    w.y += v1.y;
                    w.z += v1.z;
                    w.w += v1.w;
                }
                v.x += w.x;
                v.y += w.y;
                v.z += w.z;
                v.w += w.w;
                r[i] = v;
            }
            keep[u] = v;
            ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
        }
    }
    ss = warp_sum(ss);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
    __syncthreads();
    float tot = 0.f;
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) tot += red[w];
    const float sc = 1.0f / sqrtf(tot / (float)D + eps);
    __nv_bfloat162 *o = reinterpret_cast<__nv_bfloat162 *>(xn + (size_t)t * D);
#pragma unroll
    for (int u = 0; u < VEC; ++u) {
        const int i = threadIdx.x + u * NT;
        if (i < nv) {
            o[2 * i] = __floats2bfloat162_rn(keep[u].x * sc, keep[u].y * sc);
            o[2 * i + 1] = __floats2bfloat162_rn(keep[u].z * sc, keep[u].w * sc);
        }
    }
}

// ---- host ------------------------------------------------------------------------

struct SaWs {
    size_t offsets, xn, qkv, q, q16, plan_head, plan_tiles, plan_left, part_ml, part_acc,
        dec_count, dec_part, ctx, total;
};

SaWs sa_ws(const moe_sa_dims &d, int64_t T) {
    auto up = [](size_t v) { return (v + 255) & ~size_t(255); };
    const size_t nq = (size_t)d.n_heads * kHeadDim;
    const size_t nr = nq + 2 * (size_t)d.n_kv_heads * kHeadDim;
    const size_t splits = (size_t)T * d.n_heads * split_cap((int)T, d.n_kv_heads);
    SaWs L{};
    size_t o = 0;
    L.offsets = o; o += up(2 * 4);
    L.xn = o; o += up((size_t)T * d.d_model * 2);
    // projection outputs: qkv first, later the output projection's rows, as many
    // as any call of up to T tokens needs: partial sums of a split reduction for up
    // to kRowsMaxTokens tokens, two parts of the equal shares for up to
    // kProjSplitMaxTokens (whatever proj_split says of this shape: it asks the
    // device and the environment, and the size must not depend on either)
    const size_t part_rows =
        std::max({(size_t)T, (size_t)kRowsMaxParts * std::min<int64_t>(T, kRowsMaxTokens),
                  (size_t)2 * std::min<int64_t>(T, kProjSplitMaxTokens)});
    L.qkv = o; o += up(part_rows * std::max(nr, (size_t)d.d_model) * 4);
    L.q = o; o += up((size_t)T * nq * 4);
    L.q16 = o; o += up((size_t)T * nq * 2);
    L.plan_head = o; o += up(sizeof(AttnPlanHead));
    L.plan_tiles = o; o += up((size_t)(T / kAttnTileMinRows) * sizeof(int4));
    L.plan_left = o; o += up((size_t)T * 4);
    L.part_ml = o; o += up(splits * 2 * 4);
    L.part_acc = o; o += up(splits * kHeadDim * 4);
    L.dec_count = o; o += up(kAttnDecodeCounts * 4);
    L.dec_part = o; o += up(kAttnDecodePartFloats * 4);
    L.ctx = o; o += up((size_t)T * nq * 2);
    L.total = o;
    return L;
}

template <typename P>
P *at(void *ws, size_t off) {
    return reinterpret_cast<P *>(static_cast<char *>(ws) + off);
}

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
bool ok_ptr(const void *p) { return p != nullptr && aligned16(p); }
moe_status cuda_status(cudaError_t e) { return e == cudaSuccess ? MOE_OK : MOE_ERR_CUDA; }

moe_status check_sa(const moe_sa_dims *d) {
    if (!d) return MOE_ERR_INVALID_ARG;
    if (d->d_model < 8 || d->d_model > 49152 || d->d_model % 8) return MOE_ERR_INVALID_ARG;
    if (d->head_dim != kHeadDim) return MOE_ERR_UNSUPPORTED;
    if (d->n_kv_heads < 1 || d->n_heads < d->n_kv_heads || d->n_heads % d->n_kv_heads)
        return MOE_ERR_INVALID_ARG;
    if (d->n_heads / d->n_kv_heads > kMaxGroup) return MOE_ERR_UNSUPPORTED;
    if ((int64_t)(d->n_heads + 2 * d->n_kv_heads) * kHeadDim > 49152) return MOE_ERR_INVALID_ARG;
    if (!(d->rope_base > 1.f) || !isfinite(d->rope_base)) return MOE_ERR_INVALID_ARG;
    return MOE_OK;
}

moe_status check_sa_call(const moe_sa_dims *d, int32_t T, const int32_t *seq, const int32_t *pos,
                         int32_t n_seq, int32_t max_len) {
    moe_status s = check_sa(d);
    if (s != MOE_OK) return s;
    if (T < 0 || T > kMaxSaTokens || n_seq < 1 || max_len < 1) return MOE_ERR_INVALID_ARG;
    if (T > 0 && (!ok_ptr(seq) || !ok_ptr(pos))) return MOE_ERR_INVALID_ARG;
    return MOE_OK;
}

// The one-"expert" projection dims: Nw output rows, Kdim inputs.
moe_dims proj_dims(int Nw, int Kdim) {
    moe_dims p{};
    p.d_model = Nw;
    p.ffn_hidden = Kdim;
    p.n_experts = 1;
    p.top_k = 1;
    p.w_dtype = MOE_BF16;
    p.x_dtype = MOE_BF16;
    p.out_dtype = MOE_F32;
    return p;
}

struct SaCall {
    const moe_sa_dims &d;
    int T;
    cudaStream_t st;
    void *ws;
    SaWs L;
    int nq() const { return d.n_heads * kHeadDim; }
    int nr() const { return (d.n_heads + 2 * d.n_kv_heads) * kHeadDim; }
};

// W_qkv . xn -> qkv (fp32), then the rotary embedding and the cache writes.
cudaError_t qkv_rope(const SaCall &c, const void *xn, const void *w_qkv, const int32_t *seq,
                     const int32_t *pos, int n_seq, int L, float *q, void *kc, void *vc,
                     bf16 *q16 = nullptr) {
    const moe_dims pd = proj_dims(c.nr(), c.d.d_model);
    const int32_t *offsets = at<int32_t>(c.ws, c.L.offsets);
    float *qkv = at<float>(c.ws, c.L.qkv);
    cudaError_t e;
    int n_part = 1;
    ProjSplit split{};
    if (proj_split(c.T, c.d.d_model, c.nr(), &split)) {
        n_part = 0;
        e = launch_proj_wm(c.T, c.d.d_model, c.nr(), xn, w_qkv, qkv, split, c.st, "qkv_gemm_tc");
    } else if (gemm_rows_fits(c.T, c.nr())) {
        n_part = gemm_rows_parts(c.T, c.d.d_model, c.nr());
        e = launch_gemm_rows_tc(c.T, c.d.d_model, c.nr(), xn, w_qkv, n_part, qkv, c.st,
                                "qkv_rows_tc");
    } else {
        e = launch_gemm_down_wm(pd, c.T, xn, offsets, w_qkv, qkv, c.st, "qkv_gemm_tc");
    }
    if (e != cudaSuccess) return e;
    long long pstride = (long long)c.T * c.nr();
    int Hq = c.d.n_heads, Hkv = c.d.n_kv_heads, ns = n_seq, Lv = L;
    RopeRates rates;
    for (int i = 0; i < kHeadDim / 2; ++i)
        rates.w[i] = pow((double)c.d.rope_base, -2.0 * i / (double)kHeadDim);
    const float *qkvc = qkv;
    bf16 *kcp = static_cast<bf16 *>(kc), *vcp = static_cast<bf16 *>(vc);
    unsigned *err = device_info().err;
    int Tv = c.T;
    int *dec_count = q16 ? at<int>(c.ws, c.L.dec_count) : nullptr;
    void *args[] = {&Tv,     &Hq,      &Hkv, &ns,  &Lv,  &rates, &seq, &pos,
                    &qkvc,   &n_part,  &pstride, &split, &q, &q16, &kcp, &vcp, &dec_count, &err};
    LaunchScope ls("rope_cache", c.st);
    const int rows = Hq + 2 * Hkv;
    return launch_pdl((const void *)k_rope_cache,
                      dim3((rows + kRopeRows - 1) / kRopeRows, (c.T + kRopeTokens - 1) / kRopeTokens),
                      dim3(kRopeThreads), 0, c.st, args);
}

// Whether tokens that no prefill tile holds attend on the tensor cores;
// MOE_ATTN_CUDA_CORES=1 keeps them on the CUDA-core kernel.
bool decode_tc() {
    static const bool off = [] {
        const char *v = getenv("MOE_ATTN_CUDA_CORES");
        return v && v[0] == '1';
    }();
    return !off && attn_decode_tc_ok();
}

// Whether a call's tokens are sorted into prefill tiles and the rest.  A call
// that cannot hold a full tile, with hardly more tokens than the caches have
// sequences, is taken as a decode step: every token goes to the decode kernel,
// which takes any, and the launch of the other is saved.  (The caches' sequences
// are all that the host knows of how the tokens are spread: a chunk over caches
// of many idle sequences is so taken one by one up to 127 tokens, as any call
// below 128 was before there were ragged tiles: 127 tokens from position 512 on
// over 96 sequences 92.8 us, 128 tokens there as a tile 65.4.)  The attention
// block of DBRX, one by one and as a tile: 100 tokens at 0 72 and 70 us; 40
// tokens at 300, and 30 tokens beside 40 decode tokens, the same either way; 16
// tokens at 0 48.6 and 50.6 us, four runs of 9 at 600 beside 40 decode tokens
// 100 and 104 us.
constexpr int kPlanMinTokens = 48;  // beyond one for each sequence

bool planned(int T, int n_seq) {
    if (!attn_prefill_tc_ok()) return false;
    return T >= kAttnTile || (decode_tc() && T - n_seq >= kPlanMinTokens);
}

AttnPlan plan_at(const SaCall &c) {
    return AttnPlan{at<AttnPlanHead>(c.ws, c.L.plan_head), at<int4>(c.ws, c.L.plan_tiles),
                    at<int>(c.ws, c.L.plan_left)};
}

PlanArgs plan_args(const SaCall &c, const int32_t *seq, const int32_t *pos, int n_seq, int L) {
    return PlanArgs{seq, pos, n_seq, L, planned(c.T, n_seq) ? plan_at(c) : AttnPlan{}};
}

// Whether a call wants the bf16 copy of its queries (one of the tensor-core
// attention kernels reads it).
bool wants_q16(int T, int n_seq) { return decode_tc() || planned(T, n_seq); }

// Attention over the caches.  A planned call: its tiles on the tensor cores,
// then its other tokens; any other call: every token by the decode kernel.
// The CUDA-core kernel's per-split partials, when there are several splits,
// are merged last.
cudaError_t attend(const SaCall &c, const float *q, const int32_t *seq, const int32_t *pos,
                   int n_seq, int L, const void *kc, const void *vc, void *ctx,
                   const bf16 *q16 = nullptr) {
    const int Hq = c.d.n_heads, Hkv = c.d.n_kv_heads, G = Hq / Hkv;
    int ns = n_split_for(c.T, Hkv, L);
    AttnPlan plan{};
    float *ml = at<float>(c.ws, c.L.part_ml), *acc = at<float>(c.ws, c.L.part_acc);
    bf16 *cp = static_cast<bf16 *>(ctx);
    if (q16 && planned(c.T, n_seq)) {
        plan = plan_at(c);
        cudaError_t e =
            launch_attn_prefill_tc(c.T, Hq, Hkv, n_seq, L, plan, q16, kc, vc, ctx, c.st);
        if (e != cudaSuccess) return e;
        ns = 1;
    }
    if (q16 && decode_tc())
        return launch_attn_decode_tc(c.T, Hq, Hkv, n_seq, L, seq, pos, q16, kc, vc, ctx,
                                     at<float>(c.ws, c.L.dec_part), at<int>(c.ws, c.L.dec_count),
                                     c.st, plan.head ? &plan : nullptr);
    const void *kern = nullptr;
    switch (G) {
        case 1: kern = (const void *)k_attn_partial<1>; break;
        case 2: kern = (const void *)k_attn_partial<2>; break;
        case 3: kern = (const void *)k_attn_partial<3>; break;
        case 4: kern = (const void *)k_attn_partial<4>; break;
        case 5: kern = (const void *)k_attn_partial<5>; break;
        case 6: kern = (const void *)k_attn_partial<6>; break;
        case 7: kern = (const void *)k_attn_partial<7>; break;
        default: kern = (const void *)k_attn_partial<8>; break;
    }
    int Hqv = Hq, Hkvv = Hkv, nsq = n_seq, Lv = L;
    const bf16 *kcp = static_cast<const bf16 *>(kc), *vcp = static_cast<const bf16 *>(vc);
    {
        int n_tg = c.T * Hkv;
        // (a planned call usually leaves few tokens: one wave of CTAs;
        // otherwise a block per item up to the grid's y limit, the kernel
        // looping past it)
        const int gy = std::min(n_tg, plan.head ? 2 * device_info().sm_count : 65535);
        void *args[] = {&Hqv, &Hkvv, &nsq, &Lv, &ns, &n_tg, &seq, &pos, &q, &kcp, &vcp, &ml,
                        &acc, &cp, &plan};
        LaunchScope ls("attention", c.st);
        cudaError_t e = launch_pdl(kern, dim3(ns, gy), dim3(kAttnThreads), 0, c.st, args);
        if (e != cudaSuccess || ns == 1) return e;
    }
    const float *mlc = ml, *accc = acc;
    void *args[] = {&ns, &mlc, &accc, &cp};
    LaunchScope ls("attn_merge", c.st);
    return launch_pdl((const void *)k_attn_merge, dim3(c.T * Hq), dim3(kHeadDim * kMergeGroups), 0,
                      c.st, args);
}

// resid += W_o . ctx; with xn_next (decoder layers, D <= 4 * 4 * 1024) the
// MoE block's normalised input is written in the same pass.
cudaError_t out_proj(const SaCall &c, const void *ctx, const void *w_o, float *resid,
                     bf16 *xn_next = nullptr, float eps = 0.f) {
    const moe_dims pd = proj_dims(c.d.d_model, c.nq());
    const int32_t *offsets = at<int32_t>(c.ws, c.L.offsets);
    float *y = at<float>(c.ws, c.L.qkv);
    const bool rows = gemm_rows_fits(c.T, c.d.d_model);
    int n_part = rows ? gemm_rows_parts(c.T, c.nq(), c.d.d_model) : 1;
    // a projection in one part is added to the residual by its epilogue
    const bool add = n_part == 1;
    float *dst = add ? resid : y;
    cudaError_t e =
        rows
            ? launch_gemm_rows_tc(c.T, c.nq(), c.d.d_model, ctx, w_o, n_part, dst, c.st,
                                  "o_rows_tc", add)
            : launch_gemm_down_wm(pd, c.T, ctx, offsets, w_o, dst, c.st, "o_gemm_tc", add);
    if (e != cudaSuccess) return e;
    if (add) n_part = 0;
    if (xn_next) {
        int Tv = c.T, D = c.d.d_model;
        const float *yc = y;
        void *args[] = {&Tv, &D, &n_part, &resid, &yc, &xn_next, &eps};
        LaunchScope ls("residual_prenorm", c.st);
        if (c.T >= kNormWideMinTokens)
            return launch_pdl((const void *)k_residual_prenorm<kNormThreadsWide, kNormMaxVec>,
                              dim3(c.T), dim3(kNormThreadsWide), 0, c.st, args);
        return launch_pdl((const void *)k_residual_prenorm<kNormThreads, 4>, dim3(c.T),
                          dim3(kNormThreads), 0, c.st, args);
    }
    if (add) return cudaSuccess;
    long long n4 = (long long)c.T * c.d.d_model / 4;
    const long long cap = (long long)device_info().sm_count * 8;
    const int grid = (int)std::max(1LL, std::min((n4 + 255) / 256, cap));
    const float *yc = y;
    void *args[] = {&n4, &n_part, &resid, &yc};
    LaunchScope ls("residual_add", c.st);
    return launch_pdl((const void *)k_residual_add, dim3(grid), dim3(256), 0, c.st, args);
}

moe_status check_ws(const moe_sa_dims *d, int T, void *ws, size_t ws_bytes) {
    size_t need = sa_ws(*d, T).total;
    if (!ws || !aligned16(ws) || ws_bytes < need) return MOE_ERR_WORKSPACE;
    return MOE_OK;
}

moe_status setup_dispatch(const SaCall &c) {
    int Tv = c.T;
    int32_t *off = at<int32_t>(c.ws, c.L.offsets);
    void *args[] = {&Tv, &off};
    LaunchScope ls("sa_setup", c.st);
    return cuda_status(launch_pdl((const void *)k_sa_setup, dim3(1), dim3(256), 0, c.st, args));
}

}  // namespace
}  // namespace moe

using namespace moe;

namespace {

moe_status sa_forward_impl(const moe_sa_dims *dims, int32_t T, const int32_t *seq,
                           const int32_t *pos, int32_t n_seq, int32_t max_len, float *resid,
                           const void *w_qkv, const void *w_o, void *k_cache, void *v_cache,
                           float eps, void *ws, size_t ws_bytes, moe_stream_t stream,
                           bf16 *xn_next) {
    moe_status s = check_sa_call(dims, T, seq, pos, n_seq, max_len);
    if (s != MOE_OK) return s;
    if (T == 0) return MOE_OK;
    if (!ok_ptr(resid) || !ok_ptr(w_qkv) || !ok_ptr(w_o) || !ok_ptr(k_cache) ||
        !ok_ptr(v_cache) || !(eps > 0.f))
        return MOE_ERR_INVALID_ARG;
    if ((s = check_ws(dims, T, ws, ws_bytes)) != MOE_OK) return s;
    SaCall c{*dims, T, (cudaStream_t)stream, ws, sa_ws(*dims, T)};
    if (!tc_path_ok(proj_dims(c.nr(), dims->d_model)) ||
        !tc_path_ok(proj_dims(dims->d_model, c.nq())))
        return MOE_ERR_UNSUPPORTED;
    bf16 *xn = at<bf16>(ws, c.L.xn);
    float *q = at<float>(ws, c.L.q);
    bf16 *ctx = at<bf16>(ws, c.L.ctx);
    {
        int Tv = T, D = dims->d_model;
        const float *rc = resid;
        int32_t *off = at<int32_t>(ws, c.L.offsets);
        PlanArgs pa = plan_args(c, seq, pos, n_seq, max_len);
        void *args[] = {&Tv, &D, &rc, &xn, &eps, &off, &pa};
        const dim3 grid(T + (pa.plan.head ? 1 : 0));
        LaunchScope ls("sa_prenorm", c.st);
        const cudaError_t e =
            T >= kNormWideMinTokens
                ? launch_pdl((const void *)k_sa_prenorm<kNormThreadsWide, kNormMaxVec>, grid,
                             dim3(kNormThreadsWide), 0, c.st, args)
                : launch_pdl((const void *)k_sa_prenorm<kNormThreads, 4>, grid,
                             dim3(kNormThreads), 0, c.st, args);
        if (e != cudaSuccess) return MOE_ERR_CUDA;
    }
    bf16 *q16 = wants_q16(T, n_seq) ? at<bf16>(ws, c.L.q16) : nullptr;
    // (only the CUDA-core attention reads the fp32 queries)
    cudaError_t e = qkv_rope(c, xn, w_qkv, seq, pos, n_seq, max_len, decode_tc() ? nullptr : q,
                             k_cache, v_cache, q16);
    if (e == cudaSuccess) e = attend(c, q, seq, pos, n_seq, max_len, k_cache, v_cache, ctx, q16);
    if (e == cudaSuccess) e = out_proj(c, ctx, w_o, resid, xn_next, eps);
    return cuda_status(e);
}

}  // namespace

extern "C" {

moe_status moe_sa_workspace_size(const moe_sa_dims *dims, int32_t max_tokens, size_t *bytes) {
    moe_status s = check_sa(dims);
    if (s != MOE_OK) return s;
    if (!bytes || max_tokens < 0 || max_tokens > kMaxSaTokens) return MOE_ERR_INVALID_ARG;
    *bytes = sa_ws(*dims, max_tokens).total;
    return MOE_OK;
}

moe_status moe_sa_qkv(const moe_sa_dims *dims, int32_t T, const void *x_norm, const void *w_qkv,
                      const int32_t *seq, const int32_t *pos, int32_t n_seq, int32_t max_len,
                      float *q, void *k_cache, void *v_cache, void *ws, size_t ws_bytes,
                      moe_stream_t stream) {
    MOE_INJECT("moe_sa_qkv");
    moe_status s = check_sa_call(dims, T, seq, pos, n_seq, max_len);
    if (s != MOE_OK) return s;
    if (T == 0) return MOE_OK;
    if (!ok_ptr(x_norm) || !ok_ptr(w_qkv) || !ok_ptr(q) || !ok_ptr(k_cache) || !ok_ptr(v_cache))
        return MOE_ERR_INVALID_ARG;
    if ((s = check_ws(dims, T, ws, ws_bytes)) != MOE_OK) return s;
    SaCall c{*dims, T, (cudaStream_t)stream, ws, sa_ws(*dims, T)};
    if (!tc_path_ok(proj_dims(c.nr(), dims->d_model))) return MOE_ERR_UNSUPPORTED;
    if ((s = setup_dispatch(c)) != MOE_OK) return s;
    return cuda_status(qkv_rope(c, x_norm, w_qkv, seq, pos, n_seq, max_len, q, k_cache, v_cache));
}

moe_status moe_sa_attend(const moe_sa_dims *dims, int32_t T, const float *q, const int32_t *seq,
                         const int32_t *pos, int32_t n_seq, int32_t max_len, const void *k_cache,
                         const void *v_cache, void *ctx, void *ws, size_t ws_bytes,
                         moe_stream_t stream) {
    MOE_INJECT("moe_sa_attend");
    moe_status s = check_sa_call(dims, T, seq, pos, n_seq, max_len);
    if (s != MOE_OK) return s;
    if (T == 0) return MOE_OK;
    if (!ok_ptr(q) || !ok_ptr(k_cache) || !ok_ptr(v_cache) || !ok_ptr(ctx))
        return MOE_ERR_INVALID_ARG;
    if ((s = check_ws(dims, T, ws, ws_bytes)) != MOE_OK) return s;
    SaCall c{*dims, T, (cudaStream_t)stream, ws, sa_ws(*dims, T)};
    // the same kernels as the whole block: the tensor-core attention
    // kernels, from a bf16 copy of the queries
    bf16 *q16 = nullptr;
    if (wants_q16(T, n_seq)) {
        q16 = at<bf16>(ws, c.L.q16);
        int Tv = T;
        PlanArgs pa = plan_args(c, seq, pos, n_seq, max_len);
        long long n4 = (long long)T * dims->n_heads * dims->head_dim / 4;
        const float *qc = q;
        int *dec_count = at<int>(ws, c.L.dec_count);
        void *args[] = {&Tv, &n4, &qc, &q16, &dec_count, &pa};
        const int blocks = (int)std::min<long long>((n4 + 255) / 256, 4LL * device_info().sm_count);
        LaunchScope ls("q_bf16", c.st);
        cudaError_t e = launch_pdl((const void *)k_q_bf16, dim3(std::max(blocks, 1)), dim3(256), 0,
                                   c.st, args);
        if (e != cudaSuccess) return cuda_status(e);
    }
    return cuda_status(attend(c, q, seq, pos, n_seq, max_len, k_cache, v_cache, ctx, q16));
}

moe_status moe_sa_forward(const moe_sa_dims *dims, int32_t T, const int32_t *seq,
                          const int32_t *pos, int32_t n_seq, int32_t max_len, float *resid,
                          const void *w_qkv, const void *w_o, void *k_cache, void *v_cache,
                          float eps, void *ws, size_t ws_bytes, moe_stream_t stream) {
    MOE_INJECT("moe_sa_forward");
    return sa_forward_impl(dims, T, seq, pos, n_seq, max_len, resid, w_qkv, w_o, k_cache, v_cache,
                           eps, ws, ws_bytes, stream, nullptr);
}


moe_status moe_decoder_workspace_size(const moe_sa_dims *attn, const moe_dims *moe_d,
                                      int32_t max_tokens, size_t *bytes) {
    if (!bytes) return MOE_ERR_INVALID_ARG;
    size_t a = 0, b = 0, c = 0;
    moe_status s = moe_sa_workspace_size(attn, max_tokens, &a);
    if (s != MOE_OK) return s;
    if ((s = moe_workspace_size(moe_d, max_tokens, &b)) != MOE_OK) return s;
    if ((s = moe_stack_workspace_size(moe_d, max_tokens, &c)) != MOE_OK) return s;
    // the MoE block's normalised input, then the attention block's or the
    // MoE layer's scratch (never live together)
    const size_t xn = ((size_t)max_tokens * attn->d_model * 2 + 255) & ~size_t(255);
    *bytes = std::max(xn + std::max(a, b), std::max(a, c));
    return MOE_OK;
}

moe_status moe_decoder_forward(const moe_sa_dims *attn, const moe_dims *moe_d, int32_t n_layers,
                               int32_t T, const int32_t *seq, const int32_t *pos, int32_t n_seq,
                               int32_t max_len, float *resid, const void *const *w_qkv,
                               const void *const *w_o, const void *const *w_router,
                               const void *const *w1, const void *const *v1,
                               const void *const *w2, void *const *k_cache,
                               void *const *v_cache, float eps, void *ws, size_t ws_bytes,
                               moe_stream_t stream) {
    MOE_INJECT("moe_decoder_forward");
    moe_status s = check_sa_call(attn, T, seq, pos, n_seq, max_len);
    if (s != MOE_OK) return s;
    if (!moe_d || moe_d->d_model != attn->d_model || moe_d->w_dtype != MOE_BF16 ||
        moe_d->x_dtype != MOE_BF16 || moe_d->out_dtype != MOE_F32 || n_layers < 0)
        return MOE_ERR_INVALID_ARG;
    if (T == 0 || n_layers == 0) return MOE_OK;
    if (!w_qkv || !w_o || !w_router || !w1 || !v1 || !w2 || !k_cache || !v_cache)
        return MOE_ERR_INVALID_ARG;
    size_t need = 0;
    if ((s = moe_decoder_workspace_size(attn, moe_d, T, &need)) != MOE_OK) return s;
    if (!ws || !aligned16(ws) || ws_bytes < need) return MOE_ERR_WORKSPACE;
    // the attention block's residual add and the MoE block's pre-norm run as
    // one kernel when a row fits its registers; otherwise as the stack does
    const bool fused = attn->d_model <= kResNormCap;
    const size_t xn_bytes = ((size_t)T * attn->d_model * 2 + 255) & ~size_t(255);
    bf16 *xn = static_cast<bf16 *>(ws);
    void *inner = static_cast<char *>(ws) + xn_bytes;
    for (int l = 0; l < n_layers; ++l) {
        if (fused) {
            s = sa_forward_impl(attn, T, seq, pos, n_seq, max_len, resid, w_qkv[l], w_o[l],
                                k_cache[l], v_cache[l], eps, inner, ws_bytes - xn_bytes, stream,
                                xn);
            if (s != MOE_OK) return s;
            // resid <- resid + MoE_l(xn): the combine reads each residual
            // element before it writes the same element
            s = moe_layer_forward(moe_d, T, xn, w_router[l], w1[l], v1[l], w2[l], resid, resid,
                                  inner, ws_bytes - xn_bytes, stream);
        } else {
            s = moe_sa_forward(attn, T, seq, pos, n_seq, max_len, resid, w_qkv[l], w_o[l],
                               k_cache[l], v_cache[l], eps, ws, ws_bytes, stream);
            if (s != MOE_OK) return s;
            s = moe_stack_forward(moe_d, 1, T, &w_router[l], &w1[l], &v1[l], &w2[l], resid, eps,
                                  ws, ws_bytes, stream);
        }
        if (s != MOE_OK) return s;
    }
    return MOE_OK;
}

}  // extern "C"
