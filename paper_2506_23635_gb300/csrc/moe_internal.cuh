// Internal helpers shared by the CUDA translation units of libmoe.
// Nothing here is part of the C ABI (include/moe.h).
#pragma once

#include <algorithm>

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "moe.h"

namespace moe {

typedef __nv_bfloat16 bf16;

// Device error word: the first error a kernel meets is stored here with an
// atomic compare-and-swap and read back by moe_get_last_error.
enum : unsigned { kErrNone = 0, kErrIndex = 1, kErrTimeout = 2 };

__device__ __forceinline__ void set_error(unsigned *err, unsigned code) {
    if (err) atomicCAS(err, 0u, code);
}

__device__ __forceinline__ float to_f(float v) { return v; }
__device__ __forceinline__ float to_f(bf16 v) { return __bfloat162float(v); }

template <typename T> __device__ __forceinline__ T from_f(float v);
template <> __device__ __forceinline__ float from_f<float>(float v) { return v; }
template <> __device__ __forceinline__ bf16 from_f<bf16>(float v) { return __float2bfloat16_rn(v); }

// Two bf16 packed in a 32-bit word -> two floats (exact).
__device__ __forceinline__ void unpack_bf16x2(uint32_t u, float &lo, float &hi) {
    lo = __uint_as_float(u << 16);
    hi = __uint_as_float(u & 0xffff0000u);
}

// 16-byte read-only load that does not allocate in L1 (weights are streamed
// once per call; keeping them out of L1 leaves it to the token vectors).
__device__ __forceinline__ uint4 ld_stream16(const void *p) {
    uint4 r;
    asm("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
        : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
        : "l"(p));
    return r;
}

// Eight consecutive weights (streamed) -> float[8].
__device__ __forceinline__ void stream8(const bf16 *p, float (&o)[8]) {
    uint4 u = ld_stream16(p);
    unpack_bf16x2(u.x, o[0], o[1]);
    unpack_bf16x2(u.y, o[2], o[3]);
    unpack_bf16x2(u.z, o[4], o[5]);
    unpack_bf16x2(u.w, o[6], o[7]);
}
__device__ __forceinline__ void stream8(const float *p, float (&o)[8]) {
    uint4 a = ld_stream16(p), b = ld_stream16(p + 4);
    o[0] = __uint_as_float(a.x); o[1] = __uint_as_float(a.y);
    o[2] = __uint_as_float(a.z); o[3] = __uint_as_float(a.w);
    o[4] = __uint_as_float(b.x); o[5] = __uint_as_float(b.y);
    o[6] = __uint_as_float(b.z); o[7] = __uint_as_float(b.w);
}

// Eight consecutive values through the normal cached path -> float[8].
__device__ __forceinline__ void load8(const bf16 *p, float (&o)[8]) {
    uint4 u = __ldg(reinterpret_cast<const uint4 *>(p));
    unpack_bf16x2(u.x, o[0], o[1]);
    unpack_bf16x2(u.y, o[2], o[3]);
    unpack_bf16x2(u.z, o[4], o[5]);
    unpack_bf16x2(u.w, o[6], o[7]);
}
__device__ __forceinline__ void load8(const float *p, float (&o)[8]) {
    float4 a = __ldg(reinterpret_cast<const float4 *>(p));
    float4 b = __ldg(reinterpret_cast<const float4 *>(p) + 1);
    o[0] = a.x; o[1] = a.y; o[2] = a.z; o[3] = a.w;
    o[4] = b.x; o[5] = b.y; o[6] = b.z; o[7] = b.w;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ float silu(float a) { return a / (1.0f + expf(-a)); }

// An expert whose slot range is not inside [0, S] is recorded as an index
// error and given no work, so a corrupt offsets array cannot move an access
// out of bounds.
template <int NS>
__device__ __forceinline__ void chunk_prefix(const int32_t *offsets, int E, int S, int *prefix,
                             unsigned *err) {
    const int lane = threadIdx.x & 31;
    int run = 0;
    for (int base = 0; base < E; base += 32) {
        int e = base + lane;
        int c = 0;
        if (e < E) {
            const int lo = offsets[e], hi = offsets[e + 1];
            if (lo < 0 || hi < lo || hi > S) set_error(err, kErrIndex);
            else c = (hi - lo + NS - 1) / NS;
        }
        int incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        if (e < E) prefix[e] = run + incl - c;
        run += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (lane == 0) prefix[E] = run;
}


// Expert e of chunk q: the largest e with prefix[e] <= q (prefix from
// chunk_prefix; experts without chunks have prefix[e] == prefix[e+1]).
__device__ __forceinline__ int chunk_expert(const int *prefix, int E, int q) {
    int lo = 0, hi = E - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (prefix[mid] <= q) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Warp-level softmax + top-k of one token's logits l[0..E); writes
// topk_idx/topk_gate[t*K + k] (and sidx[k] if non-null).  A NaN logit (a
// token with a NaN or infinite component) ranks as -inf, so the K picks are
// always distinct experts in [0, E) (K <= E): the indices that address the
// dispatch arrays stay in range whatever the data; such a token's gates
// are NaN.
__device__ inline void select_topk(int E, int K, int t, const float *l, float *pk,
                            float *__restrict__ logits_opt, int32_t *__restrict__ topk_idx,
                            float *__restrict__ topk_gate, int *sidx) {
    const int lane = threadIdx.x & 31;
    if (logits_opt)
        for (int e = lane; e < E; e += 32) logits_opt[(size_t)t * E + e] = l[e];
    float m = -INFINITY;
    for (int e = lane; e < E; e += 32) m = fmaxf(m, l[e]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    float z = 0.f;
    for (int e = lane; e < E; e += 32) z += expf(l[e] - m);
    z = warp_sum(z);

    uint32_t taken = 0;  // bit i: expert lane + 32*i already selected
    float psel = 0.f;
    for (int k = 0; k < K; ++k) {
        float bv = -INFINITY;
        int bi = 0x7fffffff;
        for (int i = 0, e = lane; e < E; ++i, e += 32) {
            if ((taken >> i) & 1u) continue;
            const float v = isnan(l[e]) ? -INFINITY : l[e];
            if (v > bv || (v == bv && e < bi)) { bv = v; bi = e; }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
            const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
            if (ov > bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
        }
        if ((bi & 31) == lane) taken |= 1u << (bi >> 5);
        const float p = expf(bv - m) / z;
        psel += p;
        if (lane == 0) {
            topk_idx[(size_t)t * K + k] = bi;
            pk[k] = p;
            if (sidx) sidx[k] = bi;
        }
    }
    __syncwarp();
    for (int k = lane; k < K; k += 32) topk_gate[(size_t)t * K + k] = pk[k] / psel;
}

// ---- host side -----------------------------------------------------------

struct DeviceInfo {
    int sm_count;
    unsigned *err;  // device address of the error word
};

// Per-device facts, looked up once per device (current device).
const DeviceInfo &device_info();

// Host-side fault injection for callers' error paths: MOE_INJECT_FAILURE
// "<entry point>:<status>" makes that entry return the status at once,
// before anything is validated or launched.  Read on every call (tests set
// it per process); nothing is injected when it is unset.
moe_status injected_failure(const char *entry);

#define MOE_INJECT(name)                                 \
    do {                                                 \
        moe_status inj_ = ::moe::injected_failure(name); \
        if (inj_ != MOE_OK) return inj_;                 \
    } while (0)

// Launch bookkeeping: counts every launch and, when profiling is on,
// brackets it with CUDA events on its stream.
struct LaunchScope {
    LaunchScope(const char *name, cudaStream_t stream);
    ~LaunchScope();
    const char *name;
    cudaStream_t stream;
    int slot;
};

// Workspace layout of moe_layer_forward / moe_expert_ffn for T tokens.
struct WsLayout {
    size_t idx, gate, counts, offsets, perm, inv_perm, h, xs, y, y_tail, ctr, total;
};
// Decode batches of up to this many tokens take the stream-K down projection
// (a second [T*K, D] fp32 output, added by the combine).
constexpr int kStreamKMaxTokens = 64;
WsLayout ws_layout(const moe_dims &d, int64_t T);

// Decode-path launchers (ffn_gemv.cu).
cudaError_t launch_up_glu_gemv(const moe_dims &d, int T, const void *x,
                               const int32_t *perm, const int32_t *offsets,
                               const void *w1, const void *v1, float *h,
                               cudaStream_t st);
cudaError_t launch_down_gemv(const moe_dims &d, int T, const float *h,
                             const int32_t *perm, const int32_t *offsets,
                             const void *w2, const float *gate, float *y_sorted,
                             const void *residual, void *out, bool fused,
                             cudaStream_t st);

// Launch with programmatic stream serialisation: the kernel may begin while
// the previous kernel in the stream finishes, and must execute
// griddepcontrol.wait before touching memory that kernel writes or reads.
inline cudaError_t launch_pdl(const void *func, dim3 grid, dim3 block, size_t smem,
                              cudaStream_t st, void **args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelExC(&cfg, func, args);
}

constexpr int kFusedCombineMaxTokens = 64;

// tcgen05 grouped GEMMs (ffn_tc.cu), bf16 only; h is bf16, y_sorted fp32.
bool tc_path_ok(const moe_dims &d);
cudaError_t launch_gather_rows(const moe_dims &d, int T, const void *x, const int32_t *perm,
                               void *x_sorted, cudaStream_t st, const int32_t *range = nullptr,
                               int n_range = 0);
cudaError_t launch_gemm_up_tc(const moe_dims &d, int T, const void *x_sorted,
                              const int32_t *offsets, const void *w1, const void *v1, void *h,
                              cudaStream_t st);
// One bf16 weight matrix w [Nw, Kdim] against T <= kRowsMaxTokens token rows
// x [T, Kdim]: y = x . w^T in fp32, weights as the MMA's M operand, the
// reduction split into `parts` (<= kRowsMaxParts) shares whose partial sums
// land in y + p*T*Nw for p < parts (the caller adds them in order).
// gemm_rows_parts: the split that keeps the SMs streaming for this shape.
// The sizes at which the CTA-pair GEMM does not beat it (gemm_rows_fits):
// measured on attention blocks, this kernel and that one: DBRX (QKV 8192 rows,
// d_model 6144) 300 tokens 85 and 101 us, 400: 100 and 112, 512: 115 and 117,
// 700: 170 and 161; 6144 rows, d_model 4096: 300: 61 and 79, 640: 83 and 95; 10,240
// rows, d_model 8192: 300: 124 and 129, 512: 152 and 148.  Above 512 tokens (three
// runs of tokens) only where its CTAs, one for each 128 rows and run, fit one round
// on the SMs: 10,240 rows at 600 tokens, 240 CTAs, 220 and 204 us.  (Smaller
// matrices would gain from it up to 1024 tokens: 3072 rows, d_model 2048, 900
// tokens 72 and 82 us.)
constexpr int kRowsMaxTokens = 640;
constexpr int kRowsMaxParts = 4;
bool gemm_rows_fits(int T, int Nw);
int gemm_rows_parts(int T, int Kdim, int Nw);
// add (one part): the result is added to y.
cudaError_t launch_gemm_rows_tc(int T, int Kdim, int Nw, const void *x, const void *w, int parts,
                                float *y, cudaStream_t st, const char *name = nullptr,
                                bool add = false);
// How the tokens of an attention call are shared between the kernels, found on
// the device (plan_attention in attn.cu): the tiles of the tensor-core prefill
// attention, longest first, and the tokens that none of them holds.
constexpr int kAttnTile = 128;  // tokens of a tile at most
// and at least: fewer consecutive tokens are attended one by one (a tile costs
// its (head pair)s ~2.75 us of an SM for each 128 cache positions whatever its
// rows, a token its key/value heads ~1 us: DBRX's heads break even at ~8-10)
constexpr int kAttnTileMinRows = 16;
struct AttnPlanHead {
    int n_tiles, n_left;
    int next;  // units taken from the tiles beyond each CTA's first
    int pad;
};
struct AttnPlan {
    AttnPlanHead *head;
    int4 *tiles;  // first token, tokens, position of the first, sequence
    int *left;    // tokens in ascending order
};
// Causal attention of the plan's tiles on the tensor cores (attn_tc.cu).  q16
// [T, Hq*128] bf16 queries (rotated, unscaled), caches [n_seq, Hkv, L, 128]
// bf16, head_dim 128.
bool attn_prefill_tc_ok();
cudaError_t launch_attn_prefill_tc(int T, int Hq, int Hkv, int n_seq, int L, const AttnPlan &plan,
                                   const void *q16, const void *k_cache, const void *v_cache,
                                   void *ctx, cudaStream_t st);
// Decode attention on the tensor cores (attn_decode_tc.cu): every token of a
// call of up to kAttnDecodeMaxTokens over positions 0..pos[t] of its
// sequence; ctx written.  Queries as above; query heads per key/value head
// <= 8.  part: kAttnDecodePartFloats floats for the results of (token,
// key/value head)s that several CTAs share; count: kAttnDecodeCounts ints,
// zero at the start (the kernel that writes q16 zeroes them).  With a plan,
// only its tokens that no tile holds, any number of them; the launch ahead is
// then the plan's prefill attention, which this one overlaps.
constexpr int kAttnDecodeMaxTokens = 128;
constexpr int kAttnDecodeMaxCtas = 160;
// a counter of finished parts for each CTA, one of (token, head)s taken for
// every 128 listed tokens of the largest call
constexpr int kAttnDecodeCounts = kAttnDecodeMaxCtas + 65536 / kAttnDecodeMaxTokens;
constexpr size_t kAttnDecodePartFloats = (size_t)2 * kAttnDecodeMaxCtas * 8 * (128 + 2);
bool attn_decode_tc_ok();
cudaError_t launch_attn_decode_tc(int T, int Hq, int Hkv, int n_seq, int L, const int32_t *seq,
                                  const int32_t *pos, const void *q16, const void *k_cache,
                                  const void *v_cache, void *ctx, float *part, int *count,
                                  cudaStream_t st, const AttnPlan *plan = nullptr);

// name: the profiling name of the launch (default "gemm_down_tc").  y_tail
// (optional, [T*K, D]): the stream-K schedule's second output; the result is
// then y_sorted + y_tail.  The 128-slot-tile kernels of both projections read
// the offsets before their dependency wait: the launch ahead of the up
// projection is launch_gather_rows, that ahead of the down projection the up
// projection, and either lets the next one launch after its own wait.
cudaError_t launch_gemm_down_tc(const moe_dims &d, int T, const void *h, const int32_t *offsets,
                                const void *w2, float *y_sorted, cudaStream_t st,
                                const char *name = nullptr, float *y_tail = nullptr);

// Prefill forms of the two grouped GEMMs (ffn_tc_wm.cu): the expert weights
// as the MMA's M operand, the slots as a per-tile N; chosen by
// launch_gemm_up_tc / launch_gemm_down_tc when the batch is not a decode
// batch and gives the experts at least 128 slots each on average (fewer
// slots per weight tile stream the weights faster through the 128-slot
// tiles of ffn_tc.cu: 609 vs 641 us for the up projection at 128 tokens).
constexpr int kWmMinTokens = 65;
inline bool use_wm(const moe_dims &d, int T) {
    return T >= kWmMinTokens && (long long)T * d.top_k >= 128LL * d.n_experts;
}
// One weight matrix against many token rows (ffn_tc_wm.cu): y = x . w^T in fp32,
// its units (256 weight rows x a run of up to 256 tokens) x k-blocks shared out
// evenly, CTA pair p taking the blocks [W p / P, W (p + 1) / P) of all W, at
// least a unit each: a unit that two pairs have a piece of comes in two parts,
// which the caller adds in order: part k of it lies at y + k T Nw.
struct ProjSplit {
    static constexpr int kMaxPairs = 80;
    static constexpr int kMaxUnits = 640;
    int pairs, nk, nwt, nst;  // k-blocks of a unit, weight tiles, token runs
    __host__ __device__ int owner(int block) const {
        return ((block + 1) * pairs - 1) / (nwt * nst * nk);
    }
    __host__ __device__ int run_start(int T, int st) const {
        return (int)((long long)st * T / nst);
    }
    // parts of output row n (of Nw) of token t
    __host__ __device__ int parts(int T, int t, int n) const {
        const int st = ((t + 1) * nst - 1) / T;  // the run that holds t
        const int first = ((n >> 8) * nst + st) * nk;
        return owner(first + nk - 1) - owner(first) + 1;
    }
};
// (up to 256 tokens the weights-as-M kernel splits the reduction itself; above
// 2048, nine runs of tokens and more, whole units leave a quarter of 76 pairs idle
// only with 18 weight tiles, 4608 rows, or fewer, and the two parts of every
// output would go on widening the workspace; the share of idle pairs is what
// decides between, measured on the widths that proj_split names)
constexpr int kProjSplitMinTokens = 257;
constexpr int kProjSplitMaxTokens = 2048;
bool proj_split(int T, int Kdim, int Nw, ProjSplit *split);
cudaError_t launch_proj_wm(int T, int Kdim, int Nw, const void *x, const void *w, float *y,
                           const ProjSplit &split, cudaStream_t st, const char *name);

cudaError_t launch_gemm_up_wm(const moe_dims &d, int T, const void *x_sorted,
                              const int32_t *offsets, const void *w1, const void *v1, void *h,
                              cudaStream_t st);
cudaError_t launch_gemm_down_wm(const moe_dims &d, int T, const void *h, const int32_t *offsets,
                                const void *w2, float *y_sorted, cudaStream_t st,
                                const char *name, bool add = false);

// Router of larger batches on the tensor cores (route_tc.cu), E <= 16, bf16:
// logits, top-k and gates as moe_route.
constexpr int kRouteTcMinTokens = 128;
bool route_tc_ok(const moe_dims &d, int T);
cudaError_t launch_route_tc(const moe_dims &d, int T, const void *x, const void *wr,
                            float *logits, int32_t *idx, float *gate, cudaStream_t st);

// Bulk-copy pipelined decode kernels (ffn_stream.cu), bf16 only, up to
// kStreamMaxSlots slots; the GLU hidden vectors h are bf16.  Batches of at
// most kStreamMaxTokens tokens take them; larger ones take the tcgen05 GEMMs.
constexpr int kStreamMaxSlots = 64;
constexpr int kStreamMaxTokens = 1;
bool stream_path_ok(const moe_dims &d, int T);
// ctr (optional, one token only): a counter the routing kernel zeroed; the
// rows are then shared out as the SMs free their stages instead of in equal
// static shares.
cudaError_t launch_up_glu_stream(const moe_dims &d, int T, const void *x, const int32_t *perm,
                                 const int32_t *offsets, const void *w1, const void *v1, void *h,
                                 cudaStream_t st, int *ctr = nullptr);
cudaError_t launch_down_stream(const moe_dims &d, int T, const void *h, const int32_t *offsets,
                               const int32_t *inv_perm, const void *w2, const float *gate,
                               const void *residual, void *out, float *y_sorted, bool fused,
                               cudaStream_t st);

}  // namespace moe
