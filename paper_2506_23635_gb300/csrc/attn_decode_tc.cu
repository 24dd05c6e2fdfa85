// Decode attention on the tcgen05 tensor cores: tokens that attend to a key/
// value cache one by one (a decode step: one token per sequence).
//
// A decode token's grouped-query attention is small in the query dimension
// (the G <= 8 query heads that share one key/value head) and long in the
// position dimension, so the positions are the MMA's M and the heads its N:
//
//   S^T = K_j Q^T       M = 128 positions, N = 16 (the G heads, zero-
//                       padded), K = 128 dims; K_j and Q both K-major
//   O^T += V_j^T P_j^T  M = 128 dims, N = 16, K = 128 positions; V_j
//                       as it lies in the cache (dims contiguous: an
//                       MN-major A operand), P_j K-major in shared memory:
//                       rows h the heads' probabilities rounded to bf16, rows
//                       8 + h the rounded rests, whose columns of O^T are
//                       added at the end of a piece
//
// with S^T and O^T in tensor memory (lane = position, resp. dim; column =
// head).  Schedules (template parameter MODE):
//
//   shares   the position tiles (128 positions each) of every (token,
//            key/value head), token by token, are one list; CTA b of G (one
//            per SM) takes the contiguous share [W b / G, W (b + 1) / G) of its
//            W tiles, so every SM streams the same number of bytes whatever
//            the sequences' lengths.  A share is a run of pieces: the end of
//            one (token, head)'s tiles, whole ones, the start of another's.
//            Where they are of like length, or no more than a CTA each, a CTA
//            has one whole; where there are many to a CTA, it takes them whole,
//            longest first and one after the other from a counter: parts and
//            their merges cost more than the uneven ends (attention block at
//            48 sequences of 512-2048 positions and a chunk of 8: 97 us with
//            a CTA for each (token, head), 102 in equal shares, 91 so; up to
//            4096 positions 139 and 125; taking the next one at the start of
//            its predecessor, in the call's order, 147).
//            (One CTA per (token, head) before: 88 of 152 SMs with 11
//            sequences, all waiting for the longest; 1488-4096 positions, 118
//            MB of keys and values: 42.2 us before, 30.6 us, of which ~8 us are
//            launch, first load and drain.)
//   splits   few (token, head)s: the n_split (up to 8) CTAs of a cluster share
//            the tiles of one: split c takes tiles c, c + n_split, c + 2
//            n_split first, then one at a time from a counter in the cluster's
//            CTA 0, so a split whose share of the memory bandwidth runs ahead
//            takes more.
//   listed   the same for the tokens that a plan lists (the tokens of a call
//            that no prefill tile holds), 128 tokens after the other.  More than
//            128 are taken whole: batches in equal shares would need slots and
//            counters of their own, and with 8 key/value heads there are 6 or
//            more (token, head)s to a CTA.  With 1 or 2 a batch has about
//            one for each CTA, and a sequence far longer than the others keeps
//            one CTA busy while the rest idle (1 key/value head, 160 tokens, one
//            of 32,768 positions: 294 us; 1,050 on the CUDA cores).  The CTAs start as the prefill
//            attention ahead leaves them SMs: that kernel started after the
//            queries and cache rows were complete, and its own results are not
//            read here, so they wait for it only at their end (for the kernels
//            that follow).
//
//   warp 0      TMA: a piece's bf16 query rows into one of four buffers, key
//               and value tiles into three-stage rings (each 32 KB: two boxes
//               of 64 dims with the 128-byte swizzle), the first three right
//               after the dependency wait; each tile is described
//               to the other warps in a ring of DecDesc;
//   warp 1      tensor memory (S^T twice, O^T: 48 of 64 columns) and the
//               MMAs: S_{j+1} is issued as soon as its key tile has landed
//               and the softmax has read S_{j-1}, O += P_j V_j once P_j is
//               written (a piece's first tile overwrites O);
//   warps 2-5   softmax, one thread per position of the tile (its tensor-
//               memory lane): the tile maximum of every head across the
//               128 positions (a warp maximum, then the four warps' through
//               shared memory), the base-2 exponent of the 1/sqrt(128)-
//               scaled scores against a per-head base that moves only when
//               the maximum passes it by more than 8 (then O^T is rescaled
//               in tensor memory, each thread its dim's row), both terms
//               of the probabilities written into P_j (positions
//               contiguous, 128-byte swizzle), rows of V_j past the
//               sequence's last position zeroed (0 * NaN is NaN; those cache
//               rows may hold anything).
//
// The end of a piece: each thread owns dim r of O^T; per head the row sums of
// the four warps are added.  Shares: a (token, head) that lies in one share is
// written to ctx at once; otherwise every share that holds a piece of it
// leaves (base, sum) and O^T in the workspace and, its share done, counts
// itself on the (token, head)'s counter; the one that counts last merges the
// pieces in order and writes ctx (no CTA waits for another).  Splits: CTA c of
// the cluster owns the heads h = c, c + n_split, ...; every CTA stores its
// (base, sum) and O^T row of each head straight into the owner's shared
// memory with asynchronous stores that count their bytes on the owner's merge
// barrier (the owner expects all splits' bytes from its start), so no sender
// waits for its stores or fences them; the owner's acquire wait on the barrier
// sees every split's partials, then it combines its heads and writes their
// ctx.  (The stores wait until every CTA of the cluster has initialised its
// barriers: each arrives on the cluster barrier at its start and waits on it
// before storing, by when the wait is long satisfied.)
//
// The kernel launches while the one ahead of it (which writes the call's new
// cache rows and the queries) runs, and asks for its first tiles' lines in L2
// meanwhile; it loads nothing before it has waited.  (Loads of tiles that the
// call does not write were sent before the wait for a time: the wait then lasts
// until these copies have landed, 3 us by clock stamps where every SM sends three
// tiles.  Attention block of DBRX, no early copies, loads, lines asked for: 9
// sequences of up to 2048 positions 52.2, 53.3 and 50.8 us, 16 60.2, 60.0 and 58.4,
// 11 up to 4096 79.7 (other schedule), 68.1 and 66.2.)
//
// Numerics: bf16 queries, fp32 scores and accumulation, probabilities in two
// bf16 terms (2^-17 of each at most unaccounted for: the padding rows of N hold
// the second, so it costs no MMA and no time that could be measured); the row
// sum takes the probabilities as stored.  Every wait is bounded (ptx.cuh); once one gives up the thread
// skips the later waits and the kernel ends.
#include <math.h>

#include <algorithm>
#include <mutex>

#include "tc.cuh"

namespace moe {
namespace {

using namespace tc;

constexpr int kDecPos = 128;   // positions per key/value tile: the MMA's M
constexpr int kDecN = 16;      // the MMA's N: the group's query heads, zero-padded
constexpr int kDecMaxG = 8;    // query heads per key/value head
constexpr int kDecThreads = 6 * 32;
constexpr int kDecMaxTokens = kAttnDecodeMaxTokens;
static_assert(kDecMaxTokens == 4 * 32, "four tokens a lane in the set-up");
constexpr int kDecStages = 3;     // key and value tiles in flight
constexpr int kDecMaxSplit = 8;   // splits of one (token, key/value head): a portable cluster
// query buffers: a piece's rows replace those of the piece four before it,
// whose last tile is at least four tiles back; the stage the new piece's
// first key tile goes to is free once the tile three back has been scored
constexpr int kDecQBufs = 4;
// the tiles of a CTA are described in a ring: the producer publishes its tile
// j once S_{j-3} has been computed (after the softmax took S_{j-5}, so after
// it read description j-5), so a slot is rewritten long after both its
// readers (issuer, softmax) took it
constexpr int kDecRing = 8;
constexpr uint32_t kDecHalf = kDecPos * 128;  // one 64-dim box of a key/value tile: 16 KB
constexpr uint32_t kDecTile = 2 * kDecHalf;   // 32 KB
constexpr uint32_t kDecNHalf = kDecN * 128;   // 16 rows x 64 elements: 2 KB
constexpr uint32_t kDecQ = 2 * kDecNHalf;     // query rows, 128 dims
constexpr uint32_t kDecP = 2 * kDecNHalf;     // probabilities, 128 positions
// shared memory (1024-byte aligned): K[3], V[3], Q[4], P[2], header
constexpr uint32_t kDecOffK = 0;
constexpr uint32_t kDecOffV = kDecOffK + kDecStages * kDecTile;
constexpr uint32_t kDecOffQ = kDecOffV + kDecStages * kDecTile;
constexpr uint32_t kDecOffP = kDecOffQ + kDecQBufs * kDecQ;
constexpr uint32_t kDecOffHdr = kDecOffP + 2 * kDecP;
// cluster: the O^T rows the splits store for the heads this CTA merges, where
// the second to fourth query buffers are otherwise (a split has one piece):
// [heads this CTA owns <= ceil(8 / n_split)][n_split][128] floats, at most 14
// rows (8 heads over 7 splits)
constexpr uint32_t kDecOffX = kDecOffQ + kDecQ;
static_assert(14 * 128 * 4 <= (kDecQBufs - 1) * kDecQ, "the merge rows fit the query buffers");
constexpr uint32_t kDecHdrBytes = 4096;
constexpr size_t kDecSmem = 1024 + kDecOffHdr + kDecHdrBytes;
static_assert(kDecSmem <= 227 * 1024, "shared memory");
// kind::f16: bf16 A and B, fp32 D, M = 128, N = 16; A and B K-major
constexpr uint32_t kDecIdescQK = (1u << 4) | (1u << 7) | (1u << 10) |
                                 ((uint32_t)(kDecN >> 3) << 17) | ((uint32_t)(kDecPos >> 4) << 24);
// the same with A MN-major (bit 15): O^T += V^T P^T with V as stored
constexpr uint32_t kDecIdescPV = kDecIdescQK | (1u << 15);
constexpr uint32_t kDecTmemCols = 64;
constexpr uint32_t kDecColS = 0, kDecColO = 2 * kDecN;
// base-2 distance the tile maximum may run ahead of a head's exponent base
constexpr float kDecRescale = 8.f;

// One position tile of a CTA's share.
struct DecDesc {
    int tile;     // position tile of the sequence; -1: the share has ended
    int tg;       // token * Hkv + key/value head
    int n;        // positions the token attends to (0: outside the cache)
    int flags;    // kDecFirst, kDecLast: of its piece; kDecWhole: the piece is the
                  // whole (token, head), kDecEnd: of its share; from bit 4: the query buffer
    int b0, parts;  // not whole: the first share with a piece of it, and how many have one
    int start;      // not whole: this piece is its start
    int share;
};
// a part's slot in the workspace: 8 rows of O^T, 8 pairs (base, sum)
constexpr int kDecSlot = kDecMaxG * (128 + 2);
static_assert(2 * kAttnDecodeMaxCtas * kDecSlot <= (int)kAttnDecodePartFloats,
              "two slots a share");
// shares of fewer tiles than this leave SMs out: two tiles' copies are in
// flight together and cost little more than one's, a part to merge 2-3 us
constexpr int kDecMinTiles = 2;
// a share's end inside a (token, head) of at most this many tiles moves to the
// nearer end of it
constexpr int kDecMaxWhole = 4;
// from this many (token, head)s for each CTA on they are taken whole (32
// tokens of DBRX, 1.7, up to 4096 positions: 102 us in equal shares, 112 with
// a CTA each)
constexpr int kDecWholeMin = 2;
// and where there is a CTA for each unless the longest has more tiles than an
// equal share and this many: parts and their merges cost about as much as
// these tiles take (attention block of DBRX, a CTA each and equal shares: 16
// sequences of up to 864 positions, longest 4 tiles over the share, 49.3 and 51.4
// us, 2047 each: 3 over, 62.0 and 64.5, up to 2048: 8 over, 59.4 and 58.1, 4096: 15
// over, 76.2 and 70.9; 18 of up to 1400: 5 over, 54.5 and 56.2, 2048: 7 over, 59.8
// and 60.4; 12 of up to 1400: 7 over, 54.1 and 52.5)
constexpr int kDecWholeSlack = 5;
// listed tokens: taken whole unless the longest has more tiles than twice an
// equal share and this many.  The CTAs start one by one as the prefill
// attention leaves them SMs, and an equal share that starts late ends late
// (attention block of DBRX, a chunk of 200 beside decode tokens of 512-2048
// positions, equal shares and taken whole: 2 tokens 75 and 79 us, 4: 90 and 80,
// 8: 93 and 81, 16: 100 and 85, 24: 109 and 89)
constexpr int kDecListedSlack = 12;
enum : int { kDecFirst = 1, kDecLast = 2, kDecWhole = 4, kDecEnd = 8, kDecQShift = 4 };

struct DecHeader {
    uint64_t k_full[kDecStages], k_empty[kDecStages];  // key tile j in stage j % 3
    uint64_t v_full[kDecStages], v_empty[kDecStages];  // value tile j in stage j % 3
    uint64_t s_full[2];              // S_j written (buffer j % 2)
    uint64_t s_empty[2];             // S_j read by the four softmax warps
    uint64_t p_ready[2];             // P_j written (four softmax warps)
    uint64_t p_empty[2];             // P_j V_j finished
    uint64_t t_full[kDecRing];       // description of tile j published (producer)
    uint64_t done;
    uint64_t merge_full;             // cluster: every split's partials stored here (their bytes)
    uint32_t tmem_base;
    uint32_t next_tile;              // the cluster's tile counter (in CTA 0)
    int last;                        // this CTA counted last on its first (1), last (2) piece
    alignas(16) DecDesc desc[kDecRing];
    float red[4][kDecMaxG];     // the warps' tile maxima
    float lsum[4][kDecMaxG];    // the warps' row sums at the end
    alignas(8) float ml[kDecMaxG][kDecMaxSplit][2];  // cluster: (base, sum) of the owned heads
    // the call's tokens: row of the caches' sequence, positions, and the
    // position tiles of the tokens before it (entry T: of all of them)
    int seq[kDecMaxTokens], n[kDecMaxTokens];
    int before[kDecMaxTokens + 1];
    int tok[kDecMaxTokens];    // listed: the token
    int order[kDecMaxTokens];  // taken whole: the tokens by falling length
    int gave_up;             // listed: a wait ran out
};
static_assert(sizeof(DecHeader) <= kDecHdrBytes, "decode attention header");

// Waits spin on the non-blocking test (bounded by the wall-time limit of
// ptx.cuh): the pipeline is a chain of short steps, and a thread that
// suspends in try_wait resumes later than the phase completes.
__device__ __forceinline__ bool dec_test(uint64_t *bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(ptx::smem_u32(bar)), "r"(parity)
        : "memory");
    return done != 0;
}

__device__ __forceinline__ bool dec_wait(uint64_t *bar, uint32_t parity, unsigned *err) {
    if (dec_test(bar, parity)) return true;
    const uint64_t t0 = ptx::globaltimer();
    for (uint32_t it = 1;; ++it) {
        if (dec_test(bar, parity)) return true;
        if ((it & 255u) == 0 && ptx::globaltimer() - t0 > ptx::kWaitLimitNs) {
            set_error(err, kErrTimeout);
            return false;
        }
    }
}

__device__ __forceinline__ float dec_exp2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// 16 fp32 columns of this warp's 32 tensor-memory lanes.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float (&v)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
        "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])),
        "r"(__float_as_uint(v[3])), "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])),
        "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])), "r"(__float_as_uint(v[8])),
        "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])), "r"(__float_as_uint(v[11])),
        "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])), "r"(__float_as_uint(v[14])),
        "r"(__float_as_uint(v[15]))
        : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// Asynchronous stores into CTA `rank`'s shared memory that count their bytes
// on that CTA's barrier `bar` (complete-tx, released at cluster scope): the
// receiver's acquire wait on `bar` sees them, and the sender waits for
// nothing.
__device__ __forceinline__ void st_async_f32(float *p, uint32_t rank, uint64_t *bar, float v) {
    asm volatile(
        "st.async.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];" ::"r"(
            ptx::map_rank(ptx::smem_u32(p), rank)),
        "f"(v), "r"(ptx::map_rank(ptx::smem_u32(bar), rank))
        : "memory");
}

__device__ __forceinline__ void st_async_v2f32(float *p, uint32_t rank, uint64_t *bar, float a,
                                               float b) {
    asm volatile(
        "st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(
            ptx::map_rank(ptx::smem_u32(p), rank)),
        "f"(a), "f"(b), "r"(ptx::map_rank(ptx::smem_u32(bar), rank))
        : "memory");
}

__device__ __forceinline__ void cluster_arrive_release() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
// Take the next value of a counter in a cluster CTA's shared memory.
__device__ __forceinline__ uint32_t dec_take(uint32_t cluster_addr) {
    uint32_t old;
    asm volatile("atom.shared::cluster.add.u32 %0, [%1], 1;" : "=r"(old) : "r"(cluster_addr)
                 : "memory");
    return old;
}
__device__ __forceinline__ void cluster_wait() {
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
}

// MN-major operand written by TMA with the 128-byte swizzle (the value tile
// as A = V^T): a 128-byte row holds 64 consecutive dims of one position, 8
// positions make a 1024-byte atom (stride offset), the next 64 dims are the
// second box, 16 KB on (leading offset).
__device__ __forceinline__ uint64_t dec_desc_mn(uint32_t saddr) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(kDecHalf >> 4) << 16) |
           ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

// S^T = K Q^T: 128 positions x 16 heads over 128 dims.
__device__ __forceinline__ void dec_issue_qk(uint32_t d_tmem, uint32_t k_smem, uint32_t q_smem) {
#pragma unroll
    for (int half = 0; half < 2; ++half) {
        const uint64_t ad = smem_desc(k_smem + half * kDecHalf);
        const uint64_t bd = smem_desc(q_smem + half * kDecNHalf);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
            mma_bf16(d_tmem, ad + 2 * kk, bd + 2 * kk, kDecIdescQK, (half | kk) != 0 ? 1u : 0u);
    }
}

// O^T (+)= V^T P^T: 128 dims x 16 heads over 128 positions, 16 a step.
__device__ __forceinline__ void dec_issue_pv(uint32_t d_tmem, uint32_t v_smem, uint32_t p_smem,
                                             bool accumulate) {
#pragma unroll
    for (int ks = 0; ks < 8; ++ks) {
        const uint64_t ad = dec_desc_mn(v_smem + ks * 16 * 128);
        const uint64_t bd = smem_desc(p_smem + (ks >> 2) * kDecNHalf) + 2 * (ks & 3);
        mma_bf16(d_tmem, ad, bd, kDecIdescPV, (accumulate || ks != 0) ? 1u : 0u);
    }
}

// The maximum over the warp (NaN scores give way to numbers, as with fmaxf).
__device__ __forceinline__ float warp_max(float v) {
    float m;
    asm("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(m) : "f"(v));
    return m;
}

// Barrier over `threads` threads that also tells whether any of them had p.
__device__ __forceinline__ bool named_bar_or(uint32_t id, uint32_t threads, bool p) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %3, 0;\n\t"
        "barrier.cta.red.or.pred q, %1, %2, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"(id), "r"(threads), "r"((uint32_t)p)
        : "memory");
    return r != 0;
}

// Shares of W tiles among G CTAs: CTA c starts at tile W c / G, and tile x is
// in CTA ((x + 1) G - 1) / W.  (In 32 bits where the products fit: a 64-bit
// division takes a few hundred cycles.)
__device__ __forceinline__ long long dec_start(long long W, int c, int G) {
    if (W < (1 << 24)) return (unsigned)W * (unsigned)c / (unsigned)G;
    return W * c / G;
}
__device__ __forceinline__ int dec_owner(long long x, long long W, int G) {
    if (W < (1 << 24)) return (int)((((unsigned)x + 1u) * (unsigned)G - 1u) / (unsigned)W);
    return (int)(((x + 1) * G - 1) / W);
}
static_assert(kAttnDecodeMaxCtas < 256, "the 32-bit products of dec_start and dec_owner");

// Row 0 of the group's heads in ctx.
template <int G>
__device__ __forceinline__ bf16 *dec_ctx(bf16 *ctx, int tg, int Hq, int Hkv) {
    const int t = tg / Hkv, g = tg - t * Hkv;
    return ctx + ((size_t)t * Hq + g * G) * 128;
}

// Weighted values over the sum of weights (a sum of probabilities of at most
// 2^8 each: far inside the fast division's range); zero where nothing is.
__device__ __forceinline__ bf16 dec_mean(float a, float s) {
    return __float2bfloat16_rn(s > 0.f ? __fdividef(a, s) : 0.f);
}

// The parts of a (token, head) in the workspace, merged in order, thread r its
// dim: part q is CTA b0 + q's, in its first slot (the start of the (token,
// head), which ends CTA b0's share, in its second).  Four parts' loads go out
// together, past L1.
template <int G>
__device__ __forceinline__ void dec_merge(const float *part, int b0, int parts, int r, bf16 *dst) {
    float M[G], A[G], S[G];
#pragma unroll
    for (int h = 0; h < G; ++h) {
        M[h] = -INFINITY;
        A[h] = S[h] = 0.f;
    }
    for (int q0 = 0; q0 < parts; q0 += 4) {
        float2 bl[4][G];
        float ov[4][G];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int q = q0 + u;
            const float *pq = part + (size_t)(2 * (b0 + q) + (q == 0 ? 1 : 0)) * kDecSlot;
#pragma unroll
            for (int h = 0; h < G; ++h) {
                bl[u][h] = make_float2(-INFINITY, 0.f);
                ov[u][h] = 0.f;
                if (q < parts) {
                    bl[u][h] = __ldcg(reinterpret_cast<const float2 *>(pq + kDecMaxG * 128 + 2 * h));
                    ov[u][h] = __ldcg(pq + h * 128 + r);
                }
            }
        }
#pragma unroll
        for (int h = 0; h < G; ++h) {
            const float mn = fmaxf(M[h], fmaxf(fmaxf(bl[0][h].x, bl[1][h].x),
                                               fmaxf(bl[2][h].x, bl[3][h].x)));
            if (mn == -INFINITY) continue;  // parts of a wait that gave up
            const float c = dec_exp2(M[h] - mn);
            M[h] = mn;
            A[h] *= c;
            S[h] *= c;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float w = dec_exp2(bl[u][h].x - mn);
                S[h] = fmaf(w, bl[u][h].y, S[h]);
                A[h] = fmaf(w, ov[u][h], A[h]);
            }
        }
    }
#pragma unroll
    for (int h = 0; h < G; ++h) dst[h * 128] = dec_mean(A[h], S[h]);
}

// The token that holds tile x: the last with `before` tiles ahead of it.
__device__ __forceinline__ int dec_token(const int *before, int T, int Hkv, long long x) {
    int t = 0;
    for (int step = kDecMaxTokens / 2; step > 0; step >>= 1)
        if (t + step < T && (long long)before[t + step] * Hkv <= x) t += step;
    return t;
}

// kDecSplits: the n_split >= 2 CTAs of a cluster share one (token, key/value
// head); otherwise n_split is 1 and every CTA has a share of all tiles.  (One
// kernel that held both forms took 11.5-12.3 us where the cluster form alone
// takes 10.6-12.0, one sequence of 300-2048 positions.)
enum : int { kDecShares = 0, kDecSplits = 1, kDecListed = 2 };

template <int G, int MODE>
__global__ void __launch_bounds__(kDecThreads, 1)
k_attn_decode_tc(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                 const __grid_constant__ CUtensorMap tmV, int T, int Hq, int Hkv, int n_seq, int L,
                 const int32_t *__restrict__ seq, const int32_t *__restrict__ pos,
                 bf16 *__restrict__ ctx, float *__restrict__ part, int *__restrict__ count,
                 int n_split, const AttnPlan plan, unsigned *err) {
    static_assert(G >= 1 && G <= kDecMaxG, "query heads per key/value head");
    constexpr bool SPLIT = MODE == kDecSplits, LISTED = MODE == kDecListed;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    DecHeader *hd = reinterpret_cast<DecHeader *>(smem + kDecOffHdr);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    const int cta = (int)blockIdx.x;
    // the output projection may launch now: it streams its weights into the
    // SMs this grid leaves free while the attention runs
    ptx::launch_dependents();

    const int n_listed = LISTED ? __ldcg(&plan.head->n_left) : 0;
    if (LISTED && n_listed == 0) {
        ptx::grid_dependency_wait();
        return;
    }
#pragma unroll 1
    for (int t_base = 0; !LISTED || t_base < n_listed; t_base += kDecMaxTokens) {
    if (LISTED) T = min(kDecMaxTokens, n_listed - t_base);
    // The producer warp sets up the barriers and finds the CTA's share before
    // the block-wide barrier.
    // the next tile to send: token, head, tile of its sequence, and the
    // sequence's tiles
    struct At {
        int t, g, tile, nt;
    } at = {0, 0, 0, 1};
    long long lo = 0;  // the share's first tile
    long long W = 0;
    int n_share = 1;
    bool whole_only = false;  // the shares are the (token, head)s
    bool taking = false;      // and a CTA takes more than one
    int cur = cta, total = 0;  // the share, its tiles
    int n_pre = 0;             // tiles sent right after the wait
    const uint64_t pol_kv = ptx::policy_evict_first();  // key and value tiles are read once
    // the tile after a, its share's j-th; false: there is none.  A split's
    // first kDecStages tiles are fixed (c, c + n_split, ...); `taken` is then
    // the next one from the cluster's counter
    auto advance = [&](At &a, int j, int taken) -> bool {
        if constexpr (SPLIT) {
            a.tile = j < kDecStages ? a.tile + n_split : taken;
            return a.tile < a.nt;
        }
        if (j >= total) return false;
        if (++a.tile == a.nt) {
            a.tile = 0;
            if (++a.g == Hkv) {
                a.g = 0;
                ++a.t;
                a.nt = hd->before[a.t + 1] - hd->before[a.t];
            }
        }
        return true;
    };
    auto token = [&](int t) { return LISTED ? hd->tok[t] : t; };
    // the next (token, head) that no CTA has taken (the first ones are the
    // CTAs' own, unless the CTAs start at different times)
    auto take = [&]() {
        return atomicAdd(&count[kAttnDecodeMaxCtas + t_base / kDecMaxTokens], 1) +
               (LISTED ? 0 : (int)gridDim.x);
    };
    // where share c starts (c - 1 ends): moved to the nearer end of a (token,
    // head) of few tiles
    auto share_end = [&](int c) -> long long {
        if (c >= n_share) return W;
        const long long x = dec_start(W, c, n_share);
        const int t = dec_token(hd->before, T, Hkv, x);
        const int ntx = hd->before[t + 1] - hd->before[t];
        if (ntx > kDecMaxWhole) return x;
        const int o = (int)((unsigned)(x - (long long)hd->before[t] * Hkv) % (unsigned)ntx);
        return x + (2 * o < ntx ? -o : ntx - o);
    };
    // (token, head) c of those taken whole, longest first
    auto find_whole = [&](At &a, int c) {
        total = 0;
        if (c >= n_share) return;
        a.t = hd->order[c / Hkv];
        a.g = c % Hkv;
        a.tile = 0;
        a.nt = total = hd->before[a.t + 1] - hd->before[a.t];
    };
    // the share's first tile: lo
    auto find = [&](At &a) {
        a.t = dec_token(hd->before, T, Hkv, lo);
        a.nt = hd->before[a.t + 1] - hd->before[a.t];
        const long long in_t = lo - (long long)hd->before[a.t] * Hkv;
        a.g = in_t < (1 << 30) ? (int)((unsigned)in_t / (unsigned)a.nt) : (int)(in_t / a.nt);
        a.tile = (int)(in_t - (long long)a.g * a.nt);
    };
    if (warp == 0) {
        // the tokens' sequences and positions are inputs of the call, complete
        // before it in stream order (no kernel of the library writes them):
        // read first, their latency behind the set-up of the barriers.  A token
        // outside the cache is given one tile with no valid position: its ctx
        // is zero.
        int tok_seq[4], tok_n[4];  // tokens 4 lane + i
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int t = 4 * lane + i;
            int tok = t;
            if (LISTED && t < T) hd->tok[t] = tok = __ldcg(plan.left + t_base + t);
            tok_seq[i] = t < T ? seq[tok] : -1;
            tok_n[i] = t < T ? pos[tok] : -1;
        }
        if (lane == 0) {
            if (LISTED) {
                hd->gave_up = 0;
                if (t_base > 0)
                    for (uint64_t *b = hd->k_full; b <= &hd->merge_full; ++b) ptx::mbar_inval(b);
            }
            for (int b = 0; b < kDecStages; ++b) {
                ptx::mbar_init(&hd->k_full[b], 1);
                ptx::mbar_init(&hd->k_empty[b], 1);
                ptx::mbar_init(&hd->v_full[b], 1);
                ptx::mbar_init(&hd->v_empty[b], 1);
            }
            for (int b = 0; b < 2; ++b) {
                ptx::mbar_init(&hd->s_full[b], 1);
                ptx::mbar_init(&hd->s_empty[b], 4);
                ptx::mbar_init(&hd->p_ready[b], 4);
                ptx::mbar_init(&hd->p_empty[b], 1);
            }
            for (int b = 0; b < kDecRing; ++b) ptx::mbar_init(&hd->t_full[b], 1);
            ptx::mbar_init(&hd->done, 1);
            ptx::mbar_init(&hd->merge_full, 1);
            hd->next_tile = 0u;
            if constexpr (SPLIT) {
                // the bytes every split stores here: an O^T row and (base, sum)
                // for each head this CTA merges
                const int c = cta % n_split;
                const int owned = c < G ? (G - 1 - c) / n_split + 1 : 0;
                ptx::mbar_arrive_expect_tx(&hd->merge_full,
                                           (uint32_t)(n_split * owned * (kDecPos * 4 + 8)));
            }
            ptx::fence_barrier_init();
            ptx::prefetch_tmap(&tmK);
            ptx::prefetch_tmap(&tmV);
            ptx::prefetch_tmap(&tmQ);
        }
        int nt[4], sum = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int t = 4 * lane + i;
            const bool ok = tok_seq[i] >= 0 && tok_seq[i] < n_seq && tok_n[i] >= 0 && tok_n[i] < L;
            tok_seq[i] = ok ? tok_seq[i] : -1;
            tok_n[i] = ok ? tok_n[i] + 1 : 0;
            nt[i] = t < T ? max(1, (tok_n[i] + kDecPos - 1) / kDecPos) : 0;
            sum += nt[i];
            if (t < T) {
                hd->seq[t] = ok ? tok_seq[i] : 0;
                hd->n[t] = tok_n[i];
            }
        }
        if constexpr (SPLIT) {
            // a split: its first tile of the cluster's (token, head)
            __syncwarp();
            const int tg = cta / n_split;
            at.t = tg / Hkv;
            at.g = tg - at.t * Hkv;
            at.tile = cta - tg * n_split;
            at.nt = max(1, (hd->n[at.t] + kDecPos - 1) / kDecPos);
            total = at.tile < at.nt ? 1 : 0;  // (whether it has any)
        } else {
            // the tiles before each token, and this CTA's share of all
            int incl = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += v;
            }
            int run = incl - sum;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                hd->before[4 * lane + i] = run;
                run += nt[i];
            }
            if (lane == 31) hd->before[kDecMaxTokens] = run;
            __syncwarp();
            W = (long long)hd->before[kDecMaxTokens] * Hkv;
            const int longest =
                __reduce_max_sync(0xffffffffu, max(max(nt[0], nt[1]), max(nt[2], nt[3])));
            if (LISTED)
                whole_only = n_listed > kDecMaxTokens ||
                             longest <= 2 * W / (int)gridDim.x + kDecListedSlack;
            else
                whole_only = T * Hkv >= kDecWholeMin * (int)gridDim.x ||
                             (T * Hkv <= (int)gridDim.x &&
                              longest <= W / (int)gridDim.x + kDecWholeSlack);
            taking = whole_only && (LISTED || T * Hkv > (int)gridDim.x);
            n_share = whole_only ? T * Hkv
                                 : (int)min((long long)gridDim.x,
                                            max(1LL, W < (1 << 24)
                                                         ? (unsigned)W / (unsigned)kDecMinTiles
                                                         : W / kDecMinTiles));
            if (whole_only) {
                // the tokens by falling length, ties in their order: each
                // lane counts those ahead of its four
                int rank[4] = {0, 0, 0, 0};
                int b0 = 0;
                for (int u = 0; u < T; ++u) {
                    const int b1 = hd->before[u + 1], nu = b1 - b0;
                    b0 = b1;
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        rank[i] += nu > nt[i] || (nu == nt[i] && u < 4 * lane + i) ? 1 : 0;
                }
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (4 * lane + i < T) hd->order[rank[i]] = 4 * lane + i;
                __syncwarp();
                if (LISTED) cur = __shfl_sync(0xffffffffu, lane == 0 ? take() : 0, 0);
                find_whole(at, cur);
            } else {
                // even lanes: the share's start, odd lanes: its end
                const long long x = share_end(cur + (lane & 1));
                lo = __shfl_sync(0xffffffffu, x, 0);
                total = (int)(__shfl_sync(0xffffffffu, x, 1) - lo);
                find(at);
            }
        }
        // the lines of the first stages' tiles, on their way into L2 while the
        // kernel ahead runs
        At a = at;
        bool have = !LISTED && total > 0;
#pragma unroll 1
        for (int j = 0; j < kDecStages && have; ++j) {
            if (lane < 4)
                ptx::tma_prefetch_2d(lane < 2 ? &tmK : &tmV, (lane & 1) * 64,
                                     (hd->seq[a.t] * Hkv + a.g) * L + a.tile * kDecPos);
            n_pre = j + 1;
            have = n_pre < kDecStages && advance(a, n_pre, 0);
        }
    }
    if (warp == 1 && (!LISTED || t_base == 0)) tmem_alloc(&hd->tmem_base, kDecTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // this CTA's barriers are initialised: the cluster's other CTAs may store
    // to it once they pass the matching wait (the arrival releases the
    // initialising thread's stores at cluster scope)
    if constexpr (SPLIT) cluster_arrive_release();
    const uint32_t tmem = hd->tmem_base;
    const uint32_t sbase = ptx::smem_u32(smem);
    // queries and new cache rows come from the previous kernel
    if (!LISTED) ptx::grid_dependency_wait();

    if (warp == 0) {
        // ------------------------------------------------------------ producer
        const uint64_t pol_q = ptx::policy_evict_normal();
        // the first stages' keys and values and their pieces' query rows, at once
        if (lane == 0) {
            At a = at;
            int piece = -1;
            for (int j = 0; j < n_pre; ++j) {
                const bool first = j == 0 || (!SPLIT && a.tile == 0);
                const int row = (hd->seq[a.t] * Hkv + a.g) * L + a.tile * kDecPos;
                ptx::mbar_arrive_expect_tx(&hd->k_full[j], kDecTile + (first ? kDecQ : 0u));
                if (first) {
                    ++piece;
                    for (int half = 0; half < 2; ++half)
                        ptx::tma_load_2d(smem + kDecOffQ + piece * kDecQ + half * kDecNHalf, &tmQ,
                                         half * 64, a.t * Hq + a.g * G, &hd->k_full[j], pol_q);
                }
                for (int half = 0; half < 2; ++half)
                    ptx::tma_load_2d(smem + kDecOffK + j * kDecTile + half * kDecHalf, &tmK,
                                     half * 64, row, &hd->k_full[j], pol_kv);
                ptx::mbar_arrive_expect_tx(&hd->v_full[j], kDecTile);
                for (int half = 0; half < 2; ++half)
                    ptx::tma_load_2d(smem + kDecOffV + j * kDecTile + half * kDecHalf, &tmV,
                                     half * 64, row, &hd->v_full[j], pol_kv);
                advance(a, j + 1, 0);
            }
        }
        if constexpr (SPLIT) cluster_wait();  // CTA 0's counter is initialised before the first take
        if (lane == 0) {
            const uint32_t counter = ptx::map_rank(ptx::smem_u32(&hd->next_tile), 0u);
            int piece = -1, k_issued = 0, v_issued = 0, taken = 0;
            DecDesc d;
            // (a (token, head)'s successor is taken two tiles before its end:
            // the counter's answer is there in time, and the CTAs that are
            // done first take the next ones)
            int share = n_share;
            int jj = 0;  // tiles of the share before this one
            auto next_share = [&]() {
                cur = share;
                find_whole(at, cur);
                jj = 0;
                return total > 0;
            };
            // values of tile v_issued: sent after the keys of the tile that
            // follows, so that their stage is free again soon after they land
            // (their P is formed while they are on the way)
            int v_row = 0;
            bool v_sent = false;
            auto send_v = [&]() -> bool {
                const int b = v_issued % kDecStages;
                if (!dec_wait(&hd->v_empty[b], ((v_issued / kDecStages) & 1) ^ 1, err)) return false;
                if (!v_sent) {
                    ptx::mbar_arrive_expect_tx(&hd->v_full[b], kDecTile);
                    for (int half = 0; half < 2; ++half)
                        ptx::tma_load_2d(smem + kDecOffV + b * kDecTile + half * kDecHalf, &tmV,
                                         half * 64, v_row, &hd->v_full[b], pol_kv);
                }
                ++v_issued;
                return true;
            };
            bool have = total > 0;
            At nxt = at;
            bool more = have && advance(nxt, 1, 0), good = true;
            for (int j = 0;; ++j) {
                const int b = j % kDecStages;
                const uint32_t ph = ((j / kDecStages) & 1) ^ 1;
                if (!have) {
                    hd->desc[j % kDecRing].tile = -1;
                    ptx::mbar_arrive(&hd->t_full[j % kDecRing]);
                    if (j > 0) good = send_v();
                    break;
                }
                // (taken two tiles ahead: the counter's round trip runs while
                // a stage frees)
                if (SPLIT && more && j + 2 >= kDecStages)
                    taken = kDecStages * n_split + (int)dec_take(counter);
                if (!SPLIT && taking && at.tile == std::max(0, at.nt - 3)) share = take();
                const bool first = jj == 0 || (!SPLIT && at.tile == 0);
                const bool last = !more || (!SPLIT && at.tile == at.nt - 1);
                if (first) {
                    ++piece;
                    d.tg = token(at.t) * Hkv + at.g;
                    d.n = hd->n[at.t];
                    const bool whole = !SPLIT && at.tile == 0 && at.nt <= total - jj;
                    d.b0 = d.parts = d.start = 0;
                    d.share = cur;
                    if (!whole && !SPLIT) {
                        const long long f0 = lo + jj - at.tile;  // the (token, head)'s first tile
                        d.b0 = dec_owner(f0, W, n_share);
                        d.parts = dec_owner(f0 + at.nt - 1, W, n_share) - d.b0 + 1;
                        d.start = at.tile == 0 ? 1 : 0;
                    }
                    d.flags = (whole ? kDecWhole : 0) | ((piece % kDecQBufs) << kDecQShift);
                }
                d.tile = at.tile;
                d.flags = (d.flags & ~(kDecFirst | kDecLast | kDecEnd)) | (first ? kDecFirst : 0) |
                          (last ? kDecLast : 0) | (more ? 0 : kDecEnd);
                const int row = (hd->seq[at.t] * Hkv + at.g) * L + at.tile * kDecPos;
                const bool sent = j < n_pre;  // above
                if (!(good = dec_wait(&hd->k_empty[b], ph, err))) break;
                if (!sent)
                    ptx::mbar_arrive_expect_tx(&hd->k_full[b], kDecTile + (first ? kDecQ : 0u));
                if (first && !sent)
                    for (int half = 0; half < 2; ++half)
                        ptx::tma_load_2d(smem + kDecOffQ + (piece % kDecQBufs) * kDecQ +
                                             half * kDecNHalf,
                                         &tmQ, half * 64, token(at.t) * Hq + at.g * G, &hd->k_full[b],
                                         pol_q);
                if (!sent)
                    for (int half = 0; half < 2; ++half)
                        ptx::tma_load_2d(smem + kDecOffK + b * kDecTile + half * kDecHalf, &tmK,
                                         half * 64, row, &hd->k_full[b], pol_kv);
                k_issued = j + 1;
                hd->desc[j % kDecRing] = d;
                ptx::mbar_arrive(&hd->t_full[j % kDecRing]);
                if (j > 0 && !(good = send_v())) break;
                v_row = row;
                v_sent = sent;
                at = nxt;
                have = more;
                ++jj;
                if (!SPLIT && !have) {
                    have = taking && next_share();
                    nxt = at;
                }
                more = have && advance(nxt, SPLIT ? j + 2 : jj + 1, taken);
            }
            // copies still in flight land before the block can exit
            for (int j = std::max(0, k_issued - kDecStages); j < k_issued; ++j)
                dec_wait(&hd->k_full[j % kDecStages], (j / kDecStages) & 1, err);
            for (int j = std::max(0, v_issued - kDecStages); j < v_issued; ++j)
                dec_wait(&hd->v_full[j % kDecStages], (j / kDecStages) & 1, err);
            if (LISTED) {  // and the MMAs' last arrivals, before the barriers start anew
                for (int j = std::max(0, k_issued - kDecStages); good && j < k_issued; ++j)
                    good = dec_wait(&hd->k_empty[j % kDecStages], (j / kDecStages) & 1, err);
                for (int j = std::max(0, v_issued - kDecStages); good && j < v_issued; ++j)
                    good = dec_wait(&hd->v_empty[j % kDecStages], (j / kDecStages) & 1, err);
                if (!good) hd->gave_up = 1;
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        if (lane == 0) {
            bool good = dec_wait(&hd->t_full[0], 0, err);
            const bool any = good && hd->desc[0].tile >= 0;
            good = good && (!any || dec_wait(&hd->k_full[0], 0, err));
            if (good && any) {
                tc_fence_after();
                dec_issue_qk(tmem + kDecColS, sbase + kDecOffK, sbase + kDecOffQ);
                mma_commit(&hd->s_full[0]);
                mma_commit(&hd->k_empty[0]);
            }
            bool first = true;  // tile j is its piece's first
            for (int j = 0; good && any; ++j) {
                // is there a tile j + 1 (published by the producer)?
                const int r1 = (j + 1) % kDecRing;
                if (!(good = dec_wait(&hd->t_full[r1], ((j + 1) / kDecRing) & 1, err))) break;
                const bool more = hd->desc[r1].tile >= 0;
                const int fl1 = more ? hd->desc[r1].flags : 0;
                if (more) {
                    // S_{j+1} into the buffer of S_{j-1}, once the softmax has read it
                    const int sb1 = (j + 1) & 1, kb1 = (j + 1) % kDecStages;
                    good = dec_wait(&hd->k_full[kb1], ((j + 1) / kDecStages) & 1, err) &&
                           (j < 1 || dec_wait(&hd->s_empty[sb1], ((j - 1) >> 1) & 1, err));
                    if (!good) break;
                    tc_fence_after();
                    dec_issue_qk(tmem + kDecColS + sb1 * kDecN, sbase + kDecOffK + kb1 * kDecTile,
                                 sbase + kDecOffQ + (uint32_t)(fl1 >> kDecQShift) * kDecQ);
                    mma_commit(&hd->s_full[sb1]);
                    mma_commit(&hd->k_empty[kb1]);
                }
                const int pb = j & 1, vb = j % kDecStages;
                good = dec_wait(&hd->v_full[vb], (j / kDecStages) & 1, err) &&
                       dec_wait(&hd->p_ready[pb], (j >> 1) & 1, err);
                if (!good) break;
                tc_fence_after();
                // (P_j of a piece's first tile comes after the softmax has
                // taken the piece before it out of O)
                dec_issue_pv(tmem + kDecColO, sbase + kDecOffV + vb * kDecTile,
                             sbase + kDecOffP + pb * kDecP, !first);
                mma_commit(&hd->p_empty[pb]);
                mma_commit(&hd->v_empty[vb]);
                if (!more) break;
                first = (fl1 & kDecFirst) != 0;
            }
            mma_commit(&hd->done);
            good &= dec_wait(&hd->done, 0, err);
            if (LISTED && !good) hd->gave_up = 1;
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------ softmax
        {
            // probability rows G..7 and 8 + G..15 of both buffers stay zero
            // (the MMA's padding heads; no thread writes them later, and each
            // thread's proxy fence before it releases P_0 covers its zeros)
            for (int i = threadIdx.x - 64; i < 2 * (int)(kDecP / 16); i += 128)
                if ((i / 8) % 8 >= G)  // (16-byte chunk i, eight to a row)
                    reinterpret_cast<uint4 *>(smem + kDecOffP)[i] = make_uint4(0u, 0u, 0u, 0u);
        }
        const int qd = warp & 3;       // tensor-memory lane quarter
        const int r = qd * 32 + lane;  // position of the tile; dim of O^T
        const uint32_t lane_base = (uint32_t)(qd * 32) << 16;
        const float sl2 = 1.4426950408889634f / sqrtf(128.f);
        // every CTA of the cluster has initialised its barriers before this
        // one's merge stores (waited here, long before they are needed)
        if constexpr (SPLIT) cluster_wait();
        float base[G], l[G], o[16], Ls[G];
#pragma unroll
        for (int h = 0; h < G; ++h) {
            base[h] = -INFINITY;
            l[h] = Ls[h] = 0.f;
        }
#pragma unroll
        for (int h = 0; h < 16; ++h) o[h] = 0.f;
        // the share's first and last piece where they are parts of a (token,
        // head) of which other CTAs hold parts too (parts > 0): which, the
        // first CTA with a part, how many
        int pend_tg[2], pend_b0[2], pend_parts[2] = {0, 0};
        bool good = true;
        for (int j = 0;; ++j) {
            const int b = j & 1;
            good = good && dec_wait(&hd->t_full[j % kDecRing], (j / kDecRing) & 1, err);
            // (lane 0's reading steers the warp: its loop stays converged)
            const DecDesc *dj = &hd->desc[j % kDecRing];
            const int tile = __shfl_sync(0xffffffffu, good ? dj->tile : -1, 0);
            if (tile < 0) break;
            const int n = dj->n, flags = dj->flags, tg = dj->tg;  // (one value for the warp)
            const int b0 = dj->b0, parts = dj->parts, start = dj->start, share = dj->share;
            if (flags & kDecFirst) {
#pragma unroll
                for (int h = 0; h < G; ++h) {
                    base[h] = -INFINITY;
                    l[h] = 0.f;
                }
            }
            const int pj = tile * kDecPos + r;
            const bool valid = pj < n;
            // (the load runs on every lane whatever its waits returned: it is
            // warp-collective; after a failed wait the values are not used)
            float v[16];
            good = good && dec_wait(&hd->s_full[b], (j >> 1) & 1, err);
            tc_fence_after();
            tmem_ld16(tmem + lane_base + kDecColS + b * kDecN, v);
            tmem_ld_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&hd->s_empty[b]);
            // the exponent base of a head moves when a score of the tile
            // passes it by more than 8 (always on a piece's first tile, whose
            // bases are -inf); only then the tile maxima are formed: a warp
            // maximum, then the four warps' through shared memory.  (A token
            // outside the cache has no valid position: nothing moves.)
            float x[G], corr[G];
            bool over = false;
#pragma unroll
            for (int h = 0; h < G; ++h) {
                x[h] = valid ? v[h] * sl2 : -INFINITY;
                corr[h] = 1.f;
                over |= x[h] > base[h] + kDecRescale;
            }
            const bool bump_any = (flags & kDecFirst) || named_bar_or(1, 128, over);
            if (bump_any) {
#pragma unroll
                for (int h = 0; h < G; ++h) {
                    const float m = warp_max(x[h]);
                    if (lane == 0) hd->red[qd][h] = m;
                }
                ptx::named_bar_sync(1, 128);
#pragma unroll
                for (int h = 0; h < G; ++h) {
                    const float tm = fmaxf(fmaxf(hd->red[0][h], hd->red[1][h]),
                                           fmaxf(hd->red[2][h], hd->red[3][h]));
                    const bool bump = tm > base[h] + kDecRescale;
                    corr[h] = bump ? exp2f(base[h] - tm) : 1.f;  // 0 on the first tile
                    if (bump) base[h] = tm;
                }
            }
            // P_j into buffer b, free once P_{j-2} V_{j-2} has finished
            good = good && (j < 2 || dec_wait(&hd->p_empty[b], ((j - 2) >> 1) & 1, err));
            unsigned char *pb = smem + kDecOffP + b * kDecP + (r >> 6) * kDecNHalf;
#pragma unroll
            for (int h = 0; h < G; ++h) {
                const float pv = valid ? dec_exp2(x[h] - base[h]) : 0.f;
                const bf16 p1 = __float2bfloat16_rn(pv);
                const bf16 p2 = __float2bfloat16_rn(pv - __bfloat162float(p1));
                if (good) {
                    unsigned char *row = pb + swizzle_offset((uint32_t)h, (uint32_t)(r & 63));
                    *reinterpret_cast<bf16 *>(row) = p1;
                    *reinterpret_cast<bf16 *>(row + 8 * 128) = p2;  // (rows 8 apart swizzle alike)
                }
                l[h] = fmaf(l[h], corr[h], __bfloat162float(p1) + __bfloat162float(p2));
            }
            // a value tile that runs past the sequence's last position: its
            // rows there are zeroed before P_j V_j reads them
            if (tile * kDecPos + kDecPos > n) {
                const int vb = j % kDecStages;
                good = good && dec_wait(&hd->v_full[vb], (j / kDecStages) & 1, err);
                if (good && !valid) {
                    unsigned char *vt = smem + kDecOffV + vb * kDecTile;
#pragma unroll
                    for (int c = 0; c < 128; c += 8)
                        *reinterpret_cast<uint4 *>(
                            vt + (c >> 6) * kDecHalf +
                            swizzle_offset((uint32_t)r, (uint32_t)(c & 63))) =
                            make_uint4(0u, 0u, 0u, 0u);
                }
            }
            // a moved base rescales O^T (each thread its dim's row) once
            // P_{j-1} V_{j-1} has finished; P_j V_j waits for this warp
            if (!(flags & kDecFirst) && bump_any) {
                good = good && dec_wait(&hd->p_empty[(j - 1) & 1], ((j - 1) >> 1) & 1, err);
                if (__all_sync(0xffffffffu, good)) {
                    tc_fence_after();
                    float so[16];
                    tmem_ld16(tmem + lane_base + kDecColO, so);
                    tmem_ld_wait();
#pragma unroll
                    for (int h = 0; h < G; ++h) {
                        so[h] *= corr[h];
                        so[8 + h] *= corr[h];
                    }
                    tmem_st16(tmem + lane_base + kDecColO, so);
                }
            }
            fence_proxy_async_smem();  // P_j and the zeroed value rows
            tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&hd->p_ready[b]);
            if (!(flags & kDecLast)) continue;

            // the piece's result: O^T row r (dim r) of every head, the row
            // sums of the four warps added in warp order
            bool fin = good && dec_wait(&hd->p_empty[b], (j >> 1) & 1, err);
            fin = __all_sync(0xffffffffu, fin);
            good = good && fin;
#pragma unroll
            for (int h = 0; h < G; ++h) {
                const float ws = warp_sum(l[h]);
                if (lane == 0) hd->lsum[qd][h] = ws;
            }
            ptx::named_bar_sync(1, 128);
            if (fin) {
                tc_fence_after();
                tmem_ld16(tmem + lane_base + kDecColO, o);
                tmem_ld_wait();
                tc_fence_before();
#pragma unroll
                for (int h = 0; h < G; ++h) o[h] += o[8 + h];
            }
#pragma unroll
            for (int h = 0; h < G; ++h)
                Ls[h] = fin ? (hd->lsum[0][h] + hd->lsum[1][h]) + (hd->lsum[2][h] + hd->lsum[3][h])
                            : 0.f;
            if (LISTED && !fin) hd->gave_up = 1;
            if constexpr (SPLIT) continue;  // (the share's only piece)
            if (flags & kDecWhole) {
                bf16 *dst = dec_ctx<G>(ctx, tg, Hq, Hkv) + r;
#pragma unroll
                for (int h = 0; h < G; ++h) dst[h * 128] = dec_mean(o[h], Ls[h]);
            } else {
                // a part: its slot holds G rows of O^T, then G pairs (base, sum)
                float *mine = part + (size_t)(2 * share + start) * kDecSlot;
#pragma unroll
                for (int h = 0; h < G; ++h) {
                    mine[h * 128 + r] = o[h];
                    if (r == 0)
                        *reinterpret_cast<float2 *>(mine + kDecMaxG * 128 + 2 * h) =
                            make_float2(fin ? base[h] : -INFINITY, Ls[h]);
                }
                // (start 0: the share begins inside the (token, head))
                if (start) pend_tg[1] = tg, pend_b0[1] = b0, pend_parts[1] = parts;
                else pend_tg[0] = tg, pend_b0[0] = b0, pend_parts[0] = parts;
            }
            if (!(flags & kDecEnd) || (pend_parts[0] == 0 && pend_parts[1] == 0)) continue;
            // the share is done: its parts are counted, and the CTA that
            // counts last on a (token, head) finds every part of it stored
            ptx::named_bar_sync(1, 128);
            if (r == 0) {
                __threadfence();  // the warps' stores (ordered by the barrier) before the counts
                int last = 0;
#pragma unroll
                for (int i = 0; i < 2; ++i)
                    if (pend_parts[i] > 0 &&
                        atomicAdd(&count[pend_b0[i]], 1) == pend_parts[i] - 1)
                        last |= 1 << i;
                hd->last = last;
                __threadfence();  // the counts before the loads of the other parts
            }
            ptx::named_bar_sync(1, 128);
#pragma unroll 1
            for (int i = 0; i < 2; ++i)
                if ((hd->last >> i) & 1)
                    dec_merge<G>(part, pend_b0[i], pend_parts[i], r,
                                 dec_ctx<G>(ctx, pend_tg[i], Hq, Hkv) + r);
            pend_parts[0] = pend_parts[1] = 0;
        }
        if constexpr (SPLIT) {
            // every split sends its part of head h to the CTA that owns it,
            // h % n_split, row slot h / n_split; the stores count their bytes
            // on the owner's merge barrier
            float *xo = reinterpret_cast<float *>(smem + kDecOffX);
            const int tg = cta / n_split, c = cta - tg * n_split;
#pragma unroll
            for (int h = 0; h < G; ++h) {
                const uint32_t owner = (uint32_t)(h % n_split);
                const int slot = h / n_split;
                st_async_f32(&xo[((size_t)slot * n_split + c) * 128 + r], owner, &hd->merge_full,
                             good ? o[h] : 0.f);
                if (r == 0)
                    st_async_v2f32(&hd->ml[slot][c][0], owner, &hd->merge_full,
                                   good ? base[h] : -INFINITY, good ? Ls[h] : 0.f);
            }
            // the heads this CTA owns (base 2: split weight 2^(base_s - M)),
            // once every split's bytes have landed
            const bool got = ptx::mbar_wait_cluster(&hd->merge_full, 0, err);
            bf16 *dst = dec_ctx<G>(ctx, tg, Hq, Hkv) + r;
            // (unrolled to the bounds and predicated, so that the heads' and
            // the splits' loads go out together: n_split >= 2 leaves at most
            // (G + 1) / 2 heads to a CTA)
#pragma unroll
            for (int slot = 0; slot < (G + 1) / 2; ++slot) {
                const int h = c + slot * n_split;
                if (!got || h >= G) continue;
                float bq[kDecMaxSplit], M = -INFINITY;
#pragma unroll
                for (int q = 0; q < kDecMaxSplit; ++q) {
                    bq[q] = q < n_split ? hd->ml[slot][q][0] : -INFINITY;
                    M = fmaxf(M, bq[q]);
                }
                float A = 0.f, S = 0.f;
                if (M != -INFINITY) {
#pragma unroll
                    for (int q = 0; q < kDecMaxSplit; ++q) {
                        if (q < n_split) {
                            const float w = dec_exp2(bq[q] - M);
                            S = fmaf(w, hd->ml[slot][q][1], S);
                            A = fmaf(w, xo[(slot * n_split + q) * 128 + r], A);
                        }
                    }
                }
                dst[h * 128] = dec_mean(A, S);
            }
        }
    }
    // (the aligned wait of every thread: the others waited at their start)
    if (SPLIT && warp == 1) cluster_wait();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (!LISTED || hd->gave_up) break;
    __syncthreads();  // (read by all before the next tokens' set-up)
    }
    if (warp == 1) tmem_dealloc(hd->tmem_base, kDecTmemCols);
    if (LISTED) ptx::grid_dependency_wait();
}

template <int MODE>
const void *dec_kernel(int G) {
    switch (G) {
        case 1: return (const void *)k_attn_decode_tc<1, MODE>;
        case 2: return (const void *)k_attn_decode_tc<2, MODE>;
        case 3: return (const void *)k_attn_decode_tc<3, MODE>;
        case 4: return (const void *)k_attn_decode_tc<4, MODE>;
        case 5: return (const void *)k_attn_decode_tc<5, MODE>;
        case 6: return (const void *)k_attn_decode_tc<6, MODE>;
        case 7: return (const void *)k_attn_decode_tc<7, MODE>;
        default: return (const void *)k_attn_decode_tc<8, MODE>;
    }
}

// Clusters of c CTAs of this kernel the current device keeps resident at once
// (GPCs hold a whole number of clusters: 15 of 8 CTAs and 23 of 6 on a GB300's
// 152 SMs; a call that needs one more waits for a whole wave), looked up once
// per device.
struct DecClusters {
    int resident[kDecMaxSplit + 1];
};

const DecClusters &dec_clusters() {
    static DecClusters info[64];
    static std::once_flag once[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
    std::call_once(once[dev], [dev] {
        const void *kern = (const void *)k_attn_decode_tc<1, kDecSplits>;
        const bool ok = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)kDecSmem) == cudaSuccess;
        for (int c = 2; c <= kDecMaxSplit; ++c) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(c * kAttnDecodeMaxCtas);
            cfg.blockDim = dim3(kDecThreads);
            cfg.dynamicSmemBytes = kDecSmem;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = c;
            attr[0].val.clusterDim.y = 1;
            attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            int n = 0;
            if (!ok || cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) n = 0;
            info[dev].resident[c] = n;
        }
        (void)cudaGetLastError();
    });
    return info[dev];
}

// CTAs for each of `pairs` (token, key/value head)s: the largest cluster that
// is resident for all of them at once (attention block of DBRX at 2 sequences
// of 2048 positions: 6 CTAs 50.0 us, 8 CTAs, one cluster left over, 54.3 us).
// 1: whole ones or the shares of all tiles, chosen on the device.  Clusters of
// two beat the shares up to 76 pairs, also where they leave a third of the SMs
// out (6 sequences of up to 864, 2048 and 4096 positions: 45.9, 50.3 and 59.1
// us against 49.5, 53.1 and 56.9; 7: 46.0, 50.6 and 59.2 against 50.0, 53.7
// and 58.1; 9: 47.1, 51.2 and 59.6 against 50.1, 54.2 and 61.0): a part left in
// the workspace costs its CTA a fence and a count, the merging CTA two more
// trips to L2.
int dec_splits(int pairs, int max_tiles) {
    const DecClusters &dc = dec_clusters();
    int n = std::min(max_tiles, kDecMaxSplit);
    while (n > 1 && dc.resident[n] < pairs) --n;
    return std::max(1, n);
}

}  // namespace

bool attn_decode_tc_ok() { return encode_fn() != nullptr; }

cudaError_t launch_attn_decode_tc(int T, int Hq, int Hkv, int n_seq, int L, const int32_t *seq,
                                  const int32_t *pos, const void *q16, const void *k_cache,
                                  const void *v_cache, void *ctx, float *part, int *count,
                                  cudaStream_t st, const AttnPlan *plan) {
    const int G = Hq / Hkv;
    if (G < 1 || G > kDecMaxG || G * Hkv != Hq || T < 1 || (!plan && T > kDecMaxTokens))
        return cudaErrorInvalidValue;
    CUtensorMap mq, mk, mv;
    const uint64_t rows = (uint64_t)n_seq * Hkv * L;
    if (!make_map(&mq, q16, (uint64_t)T * Hq, 128, kDecN) ||
        !make_map(&mk, k_cache, rows, 128, kDecPos) || !make_map(&mv, v_cache, rows, 128, kDecPos))
        return cudaErrorInvalidValue;
    unsigned *err = device_info().err;
    bf16 *cp = static_cast<bf16 *>(ctx);
    int Tv = T, Hqv = Hq, Hkvv = Hkv, ns = n_seq, Lv = L;
    // few (token, key/value head)s: a cluster of CTAs for each; otherwise one
    // share of all tiles per SM
    // (listed tokens are counted on the device: one CTA per SM)
    const int pairs = T * Hkv, sms = std::min(device_info().sm_count, kAttnDecodeMaxCtas);
    const int max_tiles = (L + kDecPos - 1) / kDecPos;
    int n_split = plan ? 1 : dec_splits(pairs, max_tiles);
    AttnPlan pl = plan ? *plan : AttnPlan{};
    const void *kern = plan          ? dec_kernel<kDecListed>(G)
                       : n_split > 1 ? dec_kernel<kDecSplits>(G)
                                     : dec_kernel<kDecShares>(G);
    cudaError_t e =
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDecSmem);
    if (e != cudaSuccess) return e;
    void *args[] = {&mq,  &mk,  &mv, &Tv,   &Hqv,   &Hkvv,    &ns, &Lv,
                    &seq, &pos, &cp, &part, &count, &n_split, &pl, &err};
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(n_split > 1 ? (unsigned)(n_split * pairs)
                                   : (unsigned)std::min<long long>((long long)pairs * max_tiles, sms));
    cfg.blockDim = dim3(kDecThreads);
    cfg.dynamicSmemBytes = kDecSmem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = n_split;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = n_split > 1 ? 2 : 1;
    LaunchScope ls("attention_decode_tc", st);
    return cudaLaunchKernelExC(&cfg, kern, args);
}

}  // namespace moe
