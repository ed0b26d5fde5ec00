// Decode-attention kernels of the hot/cold KV tiering hot path, for sm_103a.
//
//   decode_split_kernel    data path 1 (Section 3): split-KV paged GQA decode
//                          attention with an fp32 online softmax; KV tiles are
//                          staged by TMA (cp.async.bulk.tensor, 128-byte
//                          swizzle) into a per-warp mbarrier ring, and the
//                          group-by-tile products run on mma.sync bf16.
//                          In a long grid, the last CTA of a kv-head of a
//                          session of at most 4 splits to finish merges them
//                          (log-sum-exp in a fixed order).
//   decode_combine_small_kernel, decode_combine_kernel, decode_combine_shared_kernel
//                          the same merge for the other multi-split sessions
//                          (one warp per query head from registers, up to 16
//                          splits; four warps per head for more, and where
//                          several CTAs shared a split), launched as a
//                          programmatic dependent of the split kernel.
//
// Hot pool: hot[NB][L][2][Hkv][bt][128] bf16. A (block, layer, K|V, head)
// run is bt rows of 256 B, row = ((blk*L + l)*2 + kv)*Hkv + g)*bt + slot. The
// decode kernel views the pool as a 4-D tensor (64 columns, row, column half,
// K|V) and loads one box per 16-token tile: its 16 K rows and 16 V rows.
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <type_traits>

#include "decode_launch.h"
#include "kvt_internal.h"

namespace kvt {
namespace {

#ifndef KVT_STAGES
#define KVT_STAGES 2   // 4 warps x 2 x 8 KiB: 3 CTAs (24 tiles in flight) per SM
#endif
constexpr int kCombineWarps = 4;
static_assert(kCombineWarps == kMergeChains && kRegMergeMax == kMergeChains * 4 &&
                  kSplitKernelMerge <= kRegMergeMax,
              "four splits per chain in a register merge, one chain per combine warp");
constexpr int kTileBytes = 8192;           // K 4 KiB + V 4 KiB
constexpr int kHalfBytes = 2048;           // 16 rows x 128 B (64 dims)
// The plan of one split: its tiles are dealt round robin to kAccs running
// softmax states (accumulator v takes tiles v, v + kAccs, ...), which merge
// at the end, first each half of them, then the halves (join_accs).
// That plan fixes the result; how the accumulators map to warps and CTAs is a
// launch choice, and every choice gives bit-identical results:
//   <4 warps, KVT_STAGES slots, 1>  3 CTAs per SM; a warp owns accumulators w
//                                   and w + 4 and alternates between them, so
//                                   consecutive tiles of a warp are independent
//   <4 warps, 3 slots, 1>           2 CTAs per SM
//   these two, kLongestFirst        their CTAs take the longest sessions first
//   these two, kOneSplit            tables of one split (kernel forms, below)
//   <8 warps, 3 slots, 1, kOneSplit>   1 CTA per SM: one accumulator per warp,
//                                   twice the warps per SM
//   <8 / kSub warps, slots, kSub>   a split shared by kSub = 2 or 8 CTAs, one
//                                   accumulator per warp: grids of up to
//                                   three CTAs per SM once shared
// Lazy softmax maximum: the reference moves when a logit exceeds it by more
// than this many powers of two (P then stays at most 2^8 = 256).
constexpr float kLazyLog2 = 8.f;
constexpr int kWarpsNarrow = 4;
constexpr int kStagesFull = KVT_STAGES;    // 3 CTAs per SM
constexpr int kStagesHalf = 3;             // 2 CTAs per SM
__host__ __device__ constexpr int decode_smem(int warps, int stages) {
    return warps * stages * kTileBytes + 1024 + 256;   // rings, alignment, barriers
}
constexpr unsigned long long kWaitLimitNs = 2000000000ull;   // 2 s

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Non-blocking form: has the phase completed?
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Wait for a phase with a wall-clock limit; false means the limit expired.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = global_ns();
    while (!mbar_try_wait(bar, parity)) {
        if (global_ns() - t0 > kWaitLimitNs) return false;
    }
    return true;
}

// L2 policy of the K and V copies: each byte is read once per step, so its
// line is the first to leave. Otherwise a layer's stream (over three times the
// L2 for 32 sessions of 20K tokens) also pushes out the partials, which the
// combine then reads from HBM behind the next call's copies: us per layer with
// the default policy and this one, 16 x 14K tokens 72.7 and 70.2, 32 x 20K 191
// and 185.5, 64 x 8K 154.3 and 150.4, 8 x 16K 45.2 and 44.1, 256 x 4K (merged
// in the split kernel) 309 and 302; sessions whose layer fits the L2 the same.
// Sessions of one split leave no partials and keep the normal policy (256 x 1 000
// 80.3 and 81.2 with evict-first); tables of one split name none at all: with
// K and V in the L2 a call over 48 layers of one session of 1K tokens takes 18.4 us
// with the normal policy spelled out and 16.5 without.
__device__ __forceinline__ uint64_t copy_policy(bool stream) {
    uint64_t p, q;
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    asm("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(q));
    return stream ? p : q;
}

// One tile: the box (64 columns, 16 rows, 2 column halves, K and V) of the
// hot pool's 4-D view, starting at K row `row`.
template <bool kPolicy>
__device__ __forceinline__ void tma_load_tile(uint32_t dst, const CUtensorMap *map, int row,
                                              uint32_t bar, uint64_t policy) {
    if constexpr (!kPolicy) {
        asm volatile(
            "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
            " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst),
            "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(row), "r"(0), "r"(0), "r"(bar)
            : "memory");
        return;
    }
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        ".L2::cache_hint [%0], [%1, {%2, %3, %4, %5}], [%6], %7;" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(row), "r"(0), "r"(0), "r"(bar),
        "l"(policy)
        : "memory");
}

__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t &r0, uint32_t &r1, uint32_t &r2,
                                        uint32_t &r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr));
}

__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t &r0, uint32_t &r1,
                                          uint32_t &r2, uint32_t &r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr));
}

// D = A(16x16 bf16, row) * B(16x8 bf16, col) + D, fp32 accumulate.
__device__ __forceinline__ void mma_bf16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                         uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
        "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t movmatrix_t(uint32_t x) {
    uint32_t y;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
    return y;
}

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi, float &rlo, float &rhi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    rlo = __low2float(v);
    rhi = __high2float(v);
    return *reinterpret_cast<uint32_t *>(&v);
}

// Byte offset, inside a 16-row x 128-byte box written with the 128-byte
// swizzle, of 16-byte unit `c` (0..7) of row `r`.
__device__ __forceinline__ uint32_t swz(int r, int c) {
    return static_cast<uint32_t>(r * 128 + ((c ^ (r & 7)) << 4));
}

// Acquire-release add at GPU scope: orders this CTA's partial writes (made
// visible to thread 0 by the preceding barrier) before its arrival, and the
// last arrival's reads of the other partials after it.
__device__ __forceinline__ int arrive(int32_t *counter) {
    int prev;
    asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], 1;"
                 : "=r"(prev)
                 : "l"(counter)
                 : "memory");
    return prev;
}

// One step of a running log-sum-exp merge: fold the partial (m, l) = v with
// accumulator o into (m, lsum, acc). The roundings are spelled out (one
// product, then one fused multiply-add), so that the split kernel and the
// combine kernel, which both run this, give the same bits.
__device__ __forceinline__ float fold(float x, float c, float w, float y) {
    return __fmaf_rn(x, c, __fmul_rn(w, y));
}
__device__ __forceinline__ void lse_step(float &m, float &lsum, float4 &acc, const float2 v,
                                         const float4 o) {
    const float mn = fmaxf(m, v.x);
    const float ref = mn == -INFINITY ? 0.f : mn;  // two empty states stay (-inf, 0, 0)
    const float c = ex2(m - ref);                  // rescale what is summed so far
    const float w = ex2(v.x - ref);
    m = mn;
    lsum = fold(lsum, c, w, v.y);
    acc.x = fold(acc.x, c, w, o.x);
    acc.y = fold(acc.y, c, w, o.y);
    acc.z = fold(acc.z, c, w, o.z);
    acc.w = fold(acc.w, c, w, o.w);
}

// The merge of a split's accumulators: each half (0-3 and 4-7) by its largest
// maximum, then the two halves. kN = 8 is a whole split, 4 a half, 2 the two
// halves; the result is in place 0. (Pairs, then pairs of pairs, would suit
// every way of sharing, but its three levels cost a one-split call 0.1-0.2 us.)
template <int kN>
__device__ __forceinline__ void join_accs(float (&m)[kN], float (&l)[kN], float4 (&acc)[kN]) {
    static_assert(kN == 1 || kN == 2 || kN == 4 || kN == 8, "parts of a split");
    if constexpr (kN >= 4) {
#pragma unroll
        for (int h = 0; h < kN; h += 4) {
            const float mx = fmaxf(fmaxf(m[h], m[h + 1]), fmaxf(m[h + 2], m[h + 3]));
            const float ref = mx == -INFINITY ? 0.f : mx;   // empty states stay (-inf, 0, 0)
            float lsum = 0.f;
            float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int v = h; v < h + 4; ++v) {
                const float c = ex2(m[v] - ref);
                lsum = __fmaf_rn(c, l[v], lsum);
                r.x = __fmaf_rn(c, acc[v].x, r.x);
                r.y = __fmaf_rn(c, acc[v].y, r.y);
                r.z = __fmaf_rn(c, acc[v].z, r.z);
                r.w = __fmaf_rn(c, acc[v].w, r.w);
            }
            m[h] = mx;
            l[h] = lsum;
            acc[h] = r;
        }
    }
    if constexpr (kN == 2 || kN == 8)
        lse_step(m[0], l[0], acc[0], make_float2(m[kN / 2], l[kN / 2]), acc[kN / 2]);
}

// Dims 4*lane .. 4*lane + 3 of output row `row`.
__device__ __forceinline__ void store_out(const DecodeArgs &a, int64_t row, int lane,
                                          const float4 y) {
    if (a.out_bf16) {
        float r0, r1;
        uint2 pk;
        pk.x = pack_bf16(y.x, y.y, r0, r1);
        pk.y = pack_bf16(y.z, y.w, r0, r1);
        reinterpret_cast<uint2 *>(reinterpret_cast<uint16_t *>(a.out) + row * kHeadDim)[lane] = pk;
    } else {
        reinterpret_cast<float4 *>(a.out + row * kHeadDim)[lane] = y;
    }
}

// The chains' states merged in chain order and normalised; lane t writes
// dims 4t..4t+3 of output row `row`.
__device__ __forceinline__ void merge_chains_store(const DecodeArgs &a, int64_t row, int lane,
                                                   const float (&m)[kMergeChains],
                                                   const float (&l)[kMergeChains],
                                                   const float4 (&acc)[kMergeChains]) {
    float M = m[0];
#pragma unroll
    for (int q = 1; q < kMergeChains; ++q) M = fmaxf(M, m[q]);
    float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
    float lt = 0.f;
#pragma unroll
    for (int q = 0; q < kMergeChains; ++q) {
        const float c = ex2(m[q] - M);             // an empty chain has m = -inf: c = 0
        r.x = __fmaf_rn(c, acc[q].x, r.x);
        r.y = __fmaf_rn(c, acc[q].y, r.y);
        r.z = __fmaf_rn(c, acc[q].z, r.z);
        r.w = __fmaf_rn(c, acc[q].w, r.w);
        lt = __fmaf_rn(c, l[q], lt);
    }
    const float inv = __frcp_rn(lt);
    store_out(a, row, lane, make_float4(__fmul_rn(r.x, inv), __fmul_rn(r.y, inv),
                                        __fmul_rn(r.z, inv), __fmul_rn(r.w, inv)));
}

// The merge of one query head's ns (2 .. 4 * kPer) split partials by one warp. Every
// load is issued before the first is used (indices clamped into the row, so
// the loads need no guard): lane t loads split t's (m, l), shared by shuffle,
// and each lane its 4 dims of every split's accumulator. Partials that other
// CTAs of the same grid wrote are read from L2 (.cg); after a grid's end plain
// loads are right, and cheaper under the next call's copies (16 x 4K tokens
// per layer 23.8 -> 23.4 us, 32 x 4K 44.6 -> 43.9 us).
template <int kPer, bool kSameGrid>   // kPer: splits per chain, at most
__device__ __forceinline__ void merge_head_regs(const DecodeArgs &a, int64_t row, int ns,
                                                int lane) {
    const int64_t base = row * a.max_splits;
    auto load = [](auto *p) { return kSameGrid ? __ldcg(p) : *p; };
    const float2 mine = load(reinterpret_cast<const float2 *>(a.part_ml) + base + min(lane, ns - 1));
    const float4 *po = reinterpret_cast<const float4 *>(a.part_o + base * kHeadDim) + lane;
    float4 o[kMergeChains][kPer];
    int s0[kMergeChains], n[kMergeChains];
#pragma unroll
    for (int q = 0; q < kMergeChains; ++q) {
        s0[q] = (q * ns) / kMergeChains;
        n[q] = ((q + 1) * ns) / kMergeChains - s0[q];
#pragma unroll
        for (int i = 0; i < kPer; ++i) o[q][i] = load(po + min(s0[q] + i, ns - 1) * (kHeadDim / 4));
    }
    float m[kMergeChains], l[kMergeChains];
    float4 acc[kMergeChains];
#pragma unroll
    for (int q = 0; q < kMergeChains; ++q) {
        m[q] = -INFINITY;
        l[q] = 0.f;
        acc[q] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int sp = min(s0[q] + i, ns - 1);
            const float2 v = make_float2(__shfl_sync(0xffffffffu, mine.x, sp),
                                         __shfl_sync(0xffffffffu, mine.y, sp));
            if (i < n[q]) lse_step(m[q], l[q], acc[q], v, o[q][i]);
        }
    }
    merge_chains_store(a, row, lane, m, l, acc);
}

// Q^T fragments (mma B operand): head n = lane/4 of the group, dims
// 16*ks + 2*(lane%4) + {0,1} and +8. `row0` is the group's first q row.
__device__ __forceinline__ void load_q(const DecodeArgs &a, int64_t row0, int G, int lane,
                                       uint32_t (&qb)[8][2]) {
    const int n = lane >> 2;
    const bool live = n < G;
    const uint32_t *qrow = reinterpret_cast<const uint32_t *>(a.q + (row0 + (live ? n : 0)) *
                                                                        kHeadDim) + (lane & 3);
#pragma unroll
    for (int ks = 0; ks < 8; ++ks) {
        qb[ks][0] = live ? qrow[ks * 8] : 0u;
        qb[ks][1] = live ? qrow[ks * 8 + 4] : 0u;
    }
}

// Offset of a lane's ldmatrix row in a tile, for 16-dim step i of K (A operand
// of S^T, row = token) and of V (A operand of O^T, loaded transposed, row =
// token). Steps i and i + 4 lie one half apart.
__device__ __forceinline__ uint32_t k_offset(int lane, int i) {
    return (i >> 2) * kHalfBytes + swz((lane & 7) + ((lane >> 3) & 1) * 8, 2 * (i & 3) + (lane >> 4));
}
__device__ __forceinline__ uint32_t v_offset(int lane, int i) {
    return (2 + (i >> 2)) * kHalfBytes + swz((lane & 7) + (lane >> 4) * 8, 2 * (i & 3) + ((lane >> 3) & 1));
}

// The session's last tile, in `slot` (one warp), in two steps; no copy is
// issued into the slot afterwards, so neither needs ordering against the async
// proxy. Fused append: token T-1 arrives with this call; its K and V rows
// replace whatever the copy brought for that slot and are stored to the
// reserved pool slot. Lanes 0-15 move K, 16-31 V, 16 B each.
__device__ __forceinline__ void splice_new(const DecodeArgs &a, const int32_t *trow, int T,
                                           int tok_base, int l, int lb, int g, uint8_t *slot,
                                           int lane) {
    const Shape &sh = a.s;
    const int r = T - 1 - tok_base;
    const int u = lane & 15;
    const int isv = lane >> 4;
    const uint4 val = *reinterpret_cast<const uint4 *>(
        (isv ? a.v_new : a.k_new) + (static_cast<int64_t>(lb) * sh.Hkv + g) * kHeadDim + u * 8);
    *reinterpret_cast<uint4 *>(slot + isv * 2 * kHalfBytes + (u >> 3) * kHalfBytes +
                               swz(r, u & 7)) = val;
    const int j = (T - 1) / sh.bt;
    const int blk = trow[j];
    if (blk >= 0 && blk < sh.num_blocks) {   // a bad id was flagged by the copy
        const int row = ((blk * sh.L + l) * 2 * sh.Hkv + g) * sh.bt + (T - 1 - j * sh.bt) +
                        isv * sh.Hkv * sh.bt;   // the pool has fewer than 2^31 rows
        *reinterpret_cast<uint4 *>(a.hot + static_cast<int64_t>(row) * kHeadDim + u * 8) = val;
    }
    __syncwarp();
}
// Slots past T may hold anything (NaN); P is 0 there but 0 * NaN is not, so
// their V rows are cleared.
__device__ __forceinline__ void clear_tail_v(int T, int tok_base, uint8_t *slot, int lane) {
    const int row = T - tok_base + (lane >> 4);   // this lane's rows: row, row + 2, ...
    uint8_t *vp = slot + (2 + ((lane >> 3) & 1)) * kHalfBytes + row * 128 + (lane & 7) * 16;
#pragma unroll
    for (int j = 0; j < kTileTokens / 2; ++j)
        if (row + 2 * j < kTileTokens)
            *reinterpret_cast<uint4 *>(vp + j * 256) = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
}

constexpr int kOStride = kHeadDim + 4;   // floats per head row of a state in shared memory (bank skew)
constexpr int kAccFloats = kMaxGroup * kOStride + 2 * kMaxGroup;   // O rows, m[8], l[8]

// The CTA's kHere accumulator states (state(v), in shared memory): a whole
// split or a half of one is merged, fewer are left to the combine. One warp per
// head, four dims per lane, so a warp reads one head's row of a state as 32
// consecutive float4. A session of one split held by one CTA is finished here;
// others leave partials.
template <int kHere, int kSub, int kWarps, bool kOne, typename State>
__device__ __forceinline__ void merge_states(const DecodeArgs &a, int64_t row_base, int G,
                                             int nsplit, int split, int sub, State state) {
    constexpr int kParts = parts_per_split(kSub);   // of the split
    constexpr int kMine = kParts / kSub;            // of this CTA
    const int lane = threadIdx.x & 31;
    const int d0 = lane * 4;
#pragma unroll 1
    for (int h = threadIdx.x >> 5; h < G; h += kWarps) {
        float m[kHere], l[kHere];
        float4 acc[kHere];
#pragma unroll
        for (int v = 0; v < kHere; ++v) {
            const float *ws = state(v);
            m[v] = ws[kMaxGroup * kOStride + h];
            l[v] = ws[kMaxGroup * kOStride + kMaxGroup + h];
            acc[v] = *reinterpret_cast<const float4 *>(ws + h * kOStride + d0);
        }
        if constexpr (kMine == 1) join_accs<kHere>(m, l, acc);
        if (kOne || (kSub == 1 && nsplit == 1)) {
            const float inv = __frcp_rn(l[0]);
            store_out(a, row_base + h, lane,
                      make_float4(__fmul_rn(acc[0].x, inv), __fmul_rn(acc[0].y, inv),
                                  __fmul_rn(acc[0].z, inv), __fmul_rn(acc[0].w, inv)));
        } else {
            const int64_t prow = ((row_base + h) * a.max_splits + split) * kParts + sub * kMine;
#pragma unroll
            for (int v = 0; v < kMine; ++v) {
                *reinterpret_cast<float4 *>(a.part_o + (prow + v) * kHeadDim + d0) = acc[v];
                if (lane == 0)
                    *reinterpret_cast<float2 *>(a.part_ml + (prow + v) * 2) = make_float2(m[v], l[v]);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// K1: kSub CTAs = (split s, kv-head g, layer-batch row lb = li*B + b).
// The split's tiles go round robin to kAccs = 8 accumulators; warp w of the
// split's kStep = kWarps * kSub consumes tiles w, w + kStep, ... through its
// own ring of kStages 8 KiB slots, tile k of the warp feeding its accumulator
// k % (8 / kStep).
// Per tile (16 tokens):
//   S^T[16 tok x 8 heads] = K[16 x 128] . Q^T       8 x mma m16n8k16
//   online softmax over tokens (columns = heads)
//   O^T[128 x 8] += V^T[128 x 16] . P^T[16 x 8]     8 x mma, P^T via movmatrix
// The CTA's accumulators merge in shared memory; a one-split session held by
// one CTA writes its normalised output, others write (m, l, acc) partials,
// which the group's last CTA to finish merges when the launch allows it
// (a.merge_max_splits), else a combine kernel.
//
// Large grids are bound by HBM. A small one (a layer of one or a few
// sessions) is a chain of latencies: the previous call's end, q, a warp's
// tiles one after another (0.36 us each), the merge, the combine. So a warp of
// a shared split takes tiles that have landed in twos (tile_batch): 48 layers of
// one session of 3 001 tokens with peaked scores 295 us in fours that went back
// to single tiles where a maximum moved, 263 in fours, 258 in twos; of 16 391
// tokens 372, 377 and 367.
// Such a call also runs every instruction once or twice, so its code has to stay in
// the instruction cache (straight-line code of over about 32 KB is fetched at
// 2.7 cycles an instruction): loops that are not on the tile path stay rolled
// and the rare steps are in one place.
// ---------------------------------------------------------------------------
struct AccState {
    float m0, m1;   // running max, heads 2(lane%4) and +1 (log2 units)
    float l0, l1;   // this lane's share of the normaliser
    float o[8][4];  // O^T fragments
};

// Forms of the kernel, each of its own so that the others do not carry its code:
// kLongestFirst takes the sessions by length (launch_decode); kOneSplit is for
// tables of one split, whose calls are a chain of latencies: no L2 policy, no
// pacing, no partials or arrival, and a ring that is filled without a loop. us in
// the form for any table and in this one: 48 layers one after another, one session of 1K tokens
// 303.5 and 290.1, of 300 151.4 and 149.1, 8 of 1K 327.5 and 320.3, 40 of 1 000 741
// and 726, 128 of 1 000 2 000 and 1 983, but 12 of 300 174.3 and 180.4; all
// layers in one call, one session of 1K 18.2 and 16.5 with K and V in the L2, 21.5
// and 21.0 from HBM, 12 of 300 67.4 and 64.2.
enum Form { kAny, kLongestFirst, kOneSplit };

template <int kWarps, int kStages, int kSub, Form kForm = kAny>
__global__ void __launch_bounds__(kWarps * 32, kWarps != kWarpsNarrow ? 1 : kStages == 2 ? 3 : kStages == 3 ? 2 : 1)
    decode_split_kernel(const __grid_constant__ CUtensorMap map, const DecodeArgs a) {
    constexpr int kStep = kWarps * kSub;  // warps of the split's CTAs
    constexpr int kA = kAccs / kStep;     // accumulators per warp
    static_assert(kWarps * kStages * 8 <= 256, "mbarriers must fit their 256-byte area");
    constexpr bool kOne = kForm == kOneSplit;
    static_assert(!kOne || kSub == 1, "one split: unshared");
    constexpr bool kPaced = kForm == kAny && (kSub == 2 || (kSub == 1 && kStages == kStagesHalf));
    static_assert(kA * kStep == kAccs, "accumulators divide among the warps");
    static_assert(kA == 1 || (kA == 2 && kSub == 1), "two accumulators only in an unshared split");
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + kWarps * kStages * kTileBytes);

    // The grid is (splits, kv-heads, rows); its blocks go out in linear order,
    // read here head-fastest so the CTAs of one split's kv-heads, whose runs
    // sit side by side in each block, start together (measured slightly
    // faster than split-fastest; the work of each CTA is the same).
    const uint32_t lin = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
    const uint32_t run = lin / gridDim.y;
    const int g = static_cast<int>(lin - run * gridDim.y);
    const int slice = static_cast<int>(run % gridDim.x);
    const int split = slice / kSub;
    const int sub = slice % kSub;           // which of the split's CTAs
    int lb = static_cast<int>(run / gridDim.x);
    int b = lb % a.B;
    const int li = lb / a.B;
    const int l = a.layer0 + li;
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int first = sub * kWarps + warp;  // this warp's first tile of the split
    const Shape sh = a.s;
    const int G = sh.Hq / sh.Hkv;

    // The combine kernel, or the next call launched with the overlap option,
    // may be scheduled once every CTA of this grid has started; it still
    // waits for this grid to finish before reading.
    asm volatile("griddepcontrol.launch_dependents;");
    if constexpr (kForm == kLongestFirst) {
        // Row r of the grid is the r-th longest session (ties by batch row).
        // Behind a test in the other forms, where it never ran, 48 layers of 12
        // sessions of 300 tokens took 167 us and 159 without it, of 40 of 1 000
        // (fused) 779 and 773.
        const int t = lane < a.B ? a.seq_lens[lane] : 0;
        int rank = 0;
        for (int j = 0; j < a.B; ++j) {
            const int tj = __shfl_sync(0xffffffffu, t, j);
            rank += tj > t || (tj == t && j < lane);
        }
        b = lb = __ffs(__ballot_sync(0xffffffffu, lane < a.B && rank == lb)) - 1;
    }
    const int32_t *trow = a.tables + static_cast<int64_t>(b) * a.max_blocks;
    // Tables at most KVT_SPLIT_TARGET x KVT_SPLIT_MIN_TILES tiles wide split
    // every session every KVT_SPLIT_MIN_TILES tiles, so this warp's tiles are
    // known before T: their block ids load alongside T instead of after it.
    // Lanes past the session's tiles may read table entries past its blocks
    // (never used).
    constexpr int kMinWarpTiles = KVT_SPLIT_MIN_TILES / kStep;
    const bool fixed_split = kOne || split_tiles(a.max_blocks * sh.bt) == KVT_SPLIT_MIN_TILES;
    int early_blk = 0;
    if (fixed_split && lane < kMinWarpTiles) {
        const int j = (split * KVT_SPLIT_MIN_TILES + first + lane * kStep) * kTileTokens / sh.bt;
        if (j < a.max_blocks) early_blk = trow[j];
    }
    const int T = a.seq_lens[b];
    if (T < 1 || T > a.max_blocks * sh.bt) {
        if (slice == 0 && g == 0 && threadIdx.x == 0) atomicOr(a.err, kErrBadLength);
        // The end of a call of such rows alone is also the end of the call before:
        // a third one waits for nothing else.
        asm volatile("griddepcontrol.wait;" ::: "memory");
        return;
    }
    const int nsplit = kOne ? 1 : num_splits(T);
    if (split >= nsplit) return;
    const int st = split_tiles(T);
    const int tile0 = kOne ? 0 : split * st;
    const int tile1 = kOne ? tiles_of(T) : min(tiles_of(T), tile0 + st);
    int my_tiles = (tile1 - tile0 - first + kStep - 1) / kStep;  // may be <= 0

    uint8_t *ring = smem + warp * kStages * kTileBytes;
    const uint32_t ring_s = smem_u32(ring);
    const uint32_t bar0 = smem_u32(bars + warp * kStages);

    // Block ids of this warp's tiles, fetched together up front: lane t
    // holds the block of the warp's tile t, so no table load waits in front
    // of a tile copy (one CTA per SM has no other warps to hide it behind).
    static_assert((KVT_SPLIT_MAX_TILES + kStep - 1) / kStep <= 32,
                  "a warp's tiles of one split must fit one block id per lane");
    static_assert(KVT_SPLIT_MIN_TILES % kStep == 0, "whole tiles per warp");
    int lane_blk = early_blk;
    if (!fixed_split && lane < my_tiles)
        lane_blk = trow[(tile0 + first + lane * kStep) * kTileTokens / sh.bt];

    if (lane == 0) {
        for (int i = 0; i < kStages; ++i) mbar_init(bar0 + 8 * i, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();

    const uint64_t policy = copy_policy(nsplit > 1);
    // Producer step (lane 0): tile k of this warp, in block blk, into slot
    // k % kStages.
    auto issue = [&](int k, int blk) {
        const int ti = tile0 + first + k * kStep;
        const int tok = ti * kTileTokens;
        const int j = tok / sh.bt;
        if (blk < 0 || blk >= sh.num_blocks) {
            atomicOr(a.err, kErrBadBlock);
            blk = 0;
        }
        const int rowk = ((blk * sh.L + l) * 2 * sh.Hkv + g) * sh.bt + (tok - j * sh.bt);
        const uint32_t slot = ring_s + (k % kStages) * kTileBytes;
        const uint32_t bar = bar0 + 8 * (k % kStages);
        // inject_extra_tx (a test of the bounded wait, 0 in normal calls): this
        // one barrier then never completes its phase, although every copy lands.
        const bool injected = k == 0 && warp == 0 && slice == 0 && g == 0 && lb == 0;
        mbar_expect_tx(bar, kTileBytes + (injected ? a.inject_extra_tx : 0));
        tma_load_tile<!kOne>(slot, &map, rowk, bar, policy);
    };
    // The block of tile k, for every lane (k < 32 wherever it is used).
    auto blk_of = [&](int k) { return __shfl_sync(0xffffffffu, lane_blk, k & 31); };
    // A wait ran out: tiles from .. to - 1 were issued and not consumed, so wait
    // (again bounded) for them, that no copy lands after the CTA exits.
    auto give_up = [&](int from, int to) {
        if (lane == 0) atomicOr(a.err, kErrTimeout);
#pragma unroll 1
        for (int k = from; k < to; ++k) mbar_wait(bar0 + 8 * (k % kStages), (k / kStages) & 1);
    };
    // The ring's first tiles. a.pace > 0 (decode_shape; the other forms do not carry
    // it): at most that many of the warp's tiles in flight while the previous
    // kernel may still be running. A warp whose wait runs out here issues no more,
    // and has no tiles to consume.
    if constexpr (kOne) {
#pragma unroll
        for (int k = 0; k < kStages; ++k) {
            const int blk = blk_of(k);
            if (lane == 0 && k < my_tiles) issue(k, blk);
        }
    } else {
#pragma unroll 1
        for (int k = 0; k < kStages && k < my_tiles; ++k) {
            const int blk = blk_of(k);
            if (kPaced && a.pace > 0 && k >= a.pace &&
                !__all_sync(0xffffffffu, mbar_wait(bar0 + 8 * (k - a.pace), 0))) {
                give_up(k - a.pace, k);
                my_tiles = 0;
                break;
            }
            if (lane == 0) issue(k, blk);
        }
    }

    uint32_t koff[4], voff[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        koff[j] = k_offset(lane, j);
        voff[j] = v_offset(lane, j);
    }

    // Everything above reads only the hot pool, the block table and seq_lens.
    // When this grid is launched as a programmatic dependent (the caller's
    // overlap option) it may run while the previous decode call drains; Q is
    // read, and partials/outputs written, only after that call completes.
    asm volatile("griddepcontrol.wait;" ::: "memory");

    // Q^T fragments (mma B operand): head n = lane/4 of the group, dims
    // 16*ks + 2*(lane%4) + {0,1} and +8.
    uint32_t qb[8][2];
    load_q(a, static_cast<int64_t>(lb) * sh.Hq + g * G, G, lane, qb);

    AccState acc_state[kA];
#pragma unroll
    for (int i = 0; i < kA; ++i) {
        acc_state[i].m0 = acc_state[i].m1 = -INFINITY;
        acc_state[i].l0 = acc_state[i].l1 = 0.f;
#pragma unroll
        for (int r = 0; r < 8; ++r)
            acc_state[i].o[r][0] = acc_state[i].o[r][1] = acc_state[i].o[r][2] = acc_state[i].o[r][3] = 0.f;
    }
    const float sl = a.scale_log2;
    int fail_k = -1;

    auto load_k = [&](uint32_t slot, int ks, uint32_t (&f)[4]) {
        ldsm_x4(slot + koff[ks & 3] + (ks >> 2) * kHalfBytes, f[0], f[1], f[2], f[3]);
    };
    auto load_v = [&](uint32_t slot, int i, uint32_t (&f)[4]) {
        ldsm_x4_t(slot + voff[i & 3] + (i >> 2) * kHalfBytes, f[0], f[1], f[2], f[3]);
    };
    auto load_values = [&](uint32_t slot, uint32_t (&f)[8][4]) {
#pragma unroll
        for (int i = 0; i < 8; ++i) load_v(slot, i, f[i]);
    };
    // One k-step (16 dims) of S^T = K . Q^T into acc.
    auto qk_step = [&](const uint32_t (&f)[4], int ks, float (&acc)[4]) {
        mma_bf16(acc, f[0], f[1], f[2], f[3], qb[ks][0], qb[ks][1]);
    };
    // Logits in log2 units; tokens at or past T are -inf.
    auto logits = [&](const float (&sa)[4], const float (&sb)[4], int tok_base, float (&x)[4]) {
        const bool v0 = tok_base + (lane >> 2) < T;
        const bool v1 = tok_base + (lane >> 2) + 8 < T;
        x[0] = v0 ? (sa[0] + sb[0]) * sl : -INFINITY;
        x[1] = v0 ? (sa[1] + sb[1]) * sl : -INFINITY;
        x[2] = v1 ? (sa[2] + sb[2]) * sl : -INFINITY;
        x[3] = v1 ? (sa[3] + sb[3]) * sl : -INFINITY;
    };
    auto tile_base = [&](int k) { return (tile0 + first + k * kStep) * kTileTokens; };

    // Online-softmax step with a lazy maximum: the reference point m moves
    // only when a logit of the tile exceeds it by more than kLazyLog2 (the
    // first tile always does, m starting at -inf); otherwise P = 2^(x - m)
    // stays at most 2^kLazyLog2 and neither m, l nor the accumulator are
    // rescaled. When it moves, m becomes the exact running maximum (a
    // quad-shuffle reduction over the tile's columns) and l and O are
    // rescaled by 2^(m_old - m_new). The decision is the warp's and depends
    // only on the tile's logits and the state, so every launch variant takes
    // it alike.
    auto grows = [&](const float (&x)[4], const AccState &s) {
        return (x[0] > s.m0 + kLazyLog2) | (x[2] > s.m0 + kLazyLog2) |
               (x[1] > s.m1 + kLazyLog2) | (x[3] > s.m1 + kLazyLog2);
    };
    auto move_max = [&](const float (&x)[4], AccState &s) {
        float mx0 = fmaxf(x[0], x[2]), mx1 = fmaxf(x[1], x[3]);
#pragma unroll
        for (int off = 4; off < 32; off <<= 1) {
            mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, off));
            mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, off));
        }
        const float mn0 = fmaxf(s.m0, mx0), mn1 = fmaxf(s.m1, mx1);
        const float al0 = ex2(s.m0 - mn0), al1 = ex2(s.m1 - mn1);
        s.m0 = mn0;
        s.m1 = mn1;
        s.l0 *= al0;
        s.l1 *= al1;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            s.o[i][0] *= al0;
            s.o[i][1] *= al1;
            s.o[i][2] *= al0;
            s.o[i][3] *= al1;
        }
    };
    // P of a tile (rounded to bf16, as the PV product sees it) as the PV
    // product's B fragment; its rounded values join the normaliser.
    auto weights = [&](const float (&x)[4], AccState &s, uint32_t &pb0, uint32_t &pb1) {
        float q0, q1, q2, q3;
        const uint32_t p01 = pack_bf16(ex2(x[0] - s.m0), ex2(x[1] - s.m1), q0, q1);
        const uint32_t p23 = pack_bf16(ex2(x[2] - s.m0), ex2(x[3] - s.m1), q2, q3);
        s.l0 += q0 + q2;
        s.l1 += q1 + q3;
        pb0 = movmatrix_t(p01);   // P^T tokens 0-7  -> B fragment
        pb1 = movmatrix_t(p23);   // P^T tokens 8-15
    };
    // O^T += V^T . P^T
    auto add_values = [&](const uint32_t (&f)[8][4], AccState &s, uint32_t pb0, uint32_t pb1) {
#pragma unroll
        for (int i = 0; i < 8; ++i) mma_bf16(s.o[i], f[i][0], f[i][1], f[i][2], f[i][3], pb0, pb1);
    };
    auto slot_of = [&](int k) { return ring_s + (k % kStages) * kTileBytes; };
    // Without a branch around the shuffle, except where the ring holds a whole split
    // of 64 tiles: one layer after another of 48, one session of 16 391 tokens 366.7 us
    // with the branch and 355.4 without, 16 of 14 000 3 368 and 3 366, but one of
    // 3 001 in splits shared by 8 CTAs 235.5 and 239.1.
    auto refill = [&](int k) {
        if (kSub == 8 && k + kStages >= my_tiles) return;
        const int nblk = blk_of(k + kStages);
        if (lane == 0 && k + kStages < my_tiles) issue(k + kStages, nblk);
    };

    // One tile into accumulator s. False: its wait timed out.
    auto one_tile = [&](int k, AccState &s) -> bool {
        if (!mbar_wait(bar0 + 8 * (k % kStages), (k / kStages) & 1)) return false;
        const int tok_base = tile_base(k);
        const uint32_t slot = slot_of(k);
        uint8_t *const tile = ring + (k % kStages) * kTileBytes;
        if (a.k_new != nullptr && tok_base + kTileTokens >= T)
            splice_new(a, trow, T, tok_base, l, lb, g, tile, lane);
        if (kSub > 1 && tok_base + kTileTokens > T) clear_tail_v(T, tok_base, tile, lane);
        // S^T = K . Q^T, two accumulators to shorten the mma chain.
        float sa[4] = {0.f, 0.f, 0.f, 0.f}, sb[4] = {0.f, 0.f, 0.f, 0.f}, x[4];
        uint32_t kf[8][4], vf[8][4];
        if constexpr (kSub > 1) {
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) load_k(slot, ks, kf[ks]);
        }
#pragma unroll
        for (int ks = 0; ks < 8; ks += 2) {
            if constexpr (kSub == 1) {
                load_k(slot, ks, kf[ks]);
                load_k(slot, ks + 1, kf[ks + 1]);
            }
            qk_step(kf[ks], ks, sa);
            qk_step(kf[ks + 1], ks + 1, sb);
        }
        // The warps of a shared split have no others to hide behind: V comes in
        // while the softmax runs.
        if constexpr (kSub > 1) load_values(slot, vf);
        logits(sa, sb, tok_base, x);
        if (__any_sync(0xffffffffu, grows(x, s))) move_max(x, s);
        uint32_t pb0, pb1;
        weights(x, s, pb0, pb1);
        if constexpr (kSub == 1) {
            if (tok_base + kTileTokens > T) clear_tail_v(T, tok_base, tile, lane);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                load_v(slot, i, vf[i]);
                mma_bf16(s.o[i], vf[i][0], vf[i][1], vf[i][2], vf[i][3], pb0, pb1);
            }
        } else {
            add_values(vf, s, pb0, pb1);
        }
        __syncwarp();
        refill(k);
        return true;
    };

    // kN consecutive tiles that have all landed, none of them the session's
    // last, into the one accumulator of a warp: the values of one_tile on each
    // in turn, with the score products side by side and the next fragments on
    // their way while a step's products run. The weights follow together too,
    // unless a tile after the first of all moves the maximum (peaked scores):
    // then the tiles go one by one from their scores on, in a rolled loop.
    auto tile_batch = [&](auto n_const, int k, AccState &s) {
        constexpr int kN = decltype(n_const)::value;
        float sa[kN][4], sb[kN][4], x[kN][4];
#pragma unroll
        for (int i = 0; i < kN; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) sa[i][j] = sb[i][j] = 0.f;
        uint32_t f[2][2 * kN][4];
        auto load_step = [&](int ks) {
#pragma unroll
            for (int i = 0; i < kN; ++i) {
                load_k(slot_of(k + i), ks, f[(ks >> 1) & 1][2 * i]);
                load_k(slot_of(k + i), ks + 1, f[(ks >> 1) & 1][2 * i + 1]);
            }
        };
        load_step(0);
#pragma unroll
        for (int ks = 0; ks < 8; ks += 2) {
            if (ks + 2 < 8) load_step(ks + 2);
#pragma unroll
            for (int i = 0; i < kN; ++i) {
                qk_step(f[(ks >> 1) & 1][2 * i], ks, sa[i]);
                qk_step(f[(ks >> 1) & 1][2 * i + 1], ks + 1, sb[i]);
            }
        }
        uint32_t vf[2][8][4];
        load_values(slot_of(k), vf[0]);
#pragma unroll
        for (int i = 0; i < kN; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) x[i][j] = (sa[i][j] + sb[i][j]) * sl;
        if (k == 0 && __any_sync(0xffffffffu, grows(x[0], s))) move_max(x[0], s);
        bool grow = false;
#pragma unroll
        for (int i = 0; i < kN; ++i) grow |= grows(x[i], s);
        if (__any_sync(0xffffffffu, grow)) {
#pragma unroll 1
            for (int i = 0; i < kN; ++i) {
                float y[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    y[j] = x[0][j];
#pragma unroll
                    for (int t = 1; t < kN; ++t) y[j] = i == t ? x[t][j] : y[j];
                }
                if (__any_sync(0xffffffffu, grows(y, s))) move_max(y, s);
                uint32_t pb0, pb1;
                weights(y, s, pb0, pb1);
                load_values(slot_of(k + i), vf[0]);
                add_values(vf[0], s, pb0, pb1);
            }
        } else {
            uint32_t pb[kN][2];
#pragma unroll
            for (int i = 0; i < kN; ++i) weights(x[i], s, pb[i][0], pb[i][1]);
#pragma unroll
            for (int i = 0; i < kN; ++i) {
                if (i + 1 < kN) load_values(slot_of(k + i + 1), vf[(i + 1) & 1]);
                add_values(vf[i & 1], s, pb[i][0], pb[i][1]);
            }
        }
        __syncwarp();
#pragma unroll 1
        for (int i = 0; i < kN; ++i) refill(k + i);
    };

    if constexpr (kA == 2) {
        // Consecutive tiles of a warp feed different accumulators, so the
        // second tile's work does not wait for the first tile's products.
#pragma unroll 1
        for (int k = 0; k < my_tiles; k += 2) {
            if (!one_tile(k, acc_state[0])) {
                fail_k = k;
                break;
            }
            if (k + 1 < my_tiles && !one_tile(k + 1, acc_state[1])) {
                fail_k = k + 1;
                break;
            }
        }
    } else if constexpr (kSub == 1) {
#pragma unroll 1
        for (int k = 0; k < my_tiles; ++k) {
            if (!one_tile(k, acc_state[0])) {
                fail_k = k;
                break;
            }
        }
    } else {
        constexpr int kBatch = 2;
        // The warp's tiles before the session's last one need no length mask.
        const int plain = tile_base(my_tiles - 1) + kTileTokens >= T ? my_tiles - 1 : my_tiles;
#pragma unroll 1
        for (int k = 0; k < my_tiles;) {
            bool batch = k + kBatch <= plain;
            if (batch) {
#pragma unroll
                for (int i = 0; i < kBatch; ++i)
                    batch &= mbar_test(bar0 + 8 * ((k + i) % kStages), ((k + i) / kStages) & 1);
                batch = __all_sync(0xffffffffu, batch);
            }
            if (batch) {
                tile_batch(std::integral_constant<int, kBatch>{}, k, acc_state[0]);
                k += kBatch;
                continue;
            }
            if (!one_tile(k, acc_state[0])) {
                fail_k = k;
                break;
            }
            ++k;
        }
    }

    if (fail_k >= 0) give_up(fail_k, min(fail_k + kStages, my_tiles));

    // Accumulator states -> this warp's own ring (all of its loads have
    // completed): accumulator v = warp + kWarps * i at float offset
    // i * kAccFloats of warp (v % kWarps)'s ring.
    static_assert(kA * kAccFloats * 4 <= kStages * kTileBytes, "states fit the ring");
#pragma unroll
    for (int i = 0; i < kA; ++i) {
        AccState &s = acc_state[i];
        // Normaliser: reduce the per-lane shares over the 8 lanes of a column.
#pragma unroll
        for (int off = 4; off < 32; off <<= 1) {
            s.l0 += __shfl_xor_sync(0xffffffffu, s.l0, off);
            s.l1 += __shfl_xor_sync(0xffffffffu, s.l1, off);
        }
        float *ws = reinterpret_cast<float *>(ring) + i * kAccFloats;
        float *wm = ws + kMaxGroup * kOStride;   // m[8], l[8]
        const int h0 = 2 * (lane & 3);
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int d = 16 * r + (lane >> 2);
            ws[h0 * kOStride + d] = s.o[r][0];
            ws[(h0 + 1) * kOStride + d] = s.o[r][1];
            ws[h0 * kOStride + d + 8] = s.o[r][2];
            ws[(h0 + 1) * kOStride + d + 8] = s.o[r][3];
        }
        if (lane < 4) {
            wm[h0] = s.m0;
            wm[h0 + 1] = s.m1;
            wm[8 + h0] = s.l0;
            wm[8 + h0 + 1] = s.l1;
        }
    }
    __syncthreads();

    const int64_t row_base = static_cast<int64_t>(lb) * sh.Hq + g * G;
    merge_states<kAccs / kSub, kSub, kWarps, kOne>(
        a, row_base, G, nsplit, split, sub, [&](int v) {
            return reinterpret_cast<const float *>(smem + (v % kWarps) * kStages * kTileBytes) +
                   (v / kWarps) * kAccFloats;
        });
    if (kOne || kWarps != kWarpsNarrow || kSub > 1) return;
    if (nsplit == 1 || nsplit > a.merge_max_splits) return;

    // Arrival. Every split of the group arrives once, whatever happened in
    // it; the last one merges the group's G heads (a warp per head) and
    // resets the counter for the next call, which touches it only after this
    // grid has completed.
    __shared__ int s_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        int32_t *counter = a.counters + static_cast<int64_t>(lb) * sh.Hkv + g;
        const bool last = arrive(counter) == nsplit - 1;
        if (last) *counter = 0;
        s_last = last;
    }
    __syncthreads();
    if (!s_last) return;
#pragma unroll 1
    for (int h = warp; h < G; h += kWarps) merge_head_regs<kSplitKernelMerge / kMergeChains, true>(a, row_base + h, nsplit, lane);
}

// Splits of batch row b that a combine kernel has to merge; 0: none, its length
// being bad or its splits merged by K1 (all sessions of one split, and of up to
// `merged`; -1 where K1 leaves partials of every session, as shared splits do).
// seq_lens is read before the combine's wait, as K1 reads it: no decode kernel
// writes it, so only the partials have to wait for K1 to finish.
// A row without splits to merge may leave at once, except in block 0: every
// combine grid has a block that waits for K1, so that the end of the combine is
// the end of the call. Where no row of a batch waited (sessions much shorter
// than their table), the combine would end while K1's last CTAs still ran, and
// what comes next, whose only predecessor is the combine (an overlapped call's
// wait, a graph's next node), would start beside them: on the partials and
// arrival counters that they still use, or before the outputs are written.
__device__ __forceinline__ int splits_to_merge(const DecodeArgs &a, int b, int merged) {
    const int T = a.seq_lens[b];
    if (T < 1 || T > a.max_blocks * a.s.bt) return 0;
    const int ns = num_splits(T);
    return ns <= merged || (merged >= 0 && ns == 1) ? 0 : ns;
}

// K2 for tables of at most kRegMergeMax splits: one warp per (layer-batch
// row, q-head), four per CTA, folding the four chains side by side from
// registers (merge_head_regs), so no shared memory or CTA barrier sits
// between its loads and its store.
__global__ void __launch_bounds__(128) decode_combine_small_kernel(const DecodeArgs a) {
    asm volatile("griddepcontrol.launch_dependents;");   // a following overlapped call
    const int64_t row = static_cast<int64_t>(blockIdx.x) * 4 + (threadIdx.x >> 5);
    if (row >= static_cast<int64_t>(a.nlayers) * a.B * a.s.Hq) return;
    const int ns = splits_to_merge(a, static_cast<int>((row / a.s.Hq) % a.B), a.merge_max_splits);
    if (ns == 0 && blockIdx.x != 0) return;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (ns == 0) return;
    merge_head_regs<kRegMergeMax / kMergeChains, false>(a, row, ns, threadIdx.x & 31);
}

// K2 for wider tables: one CTA (4 warps) per (layer-batch row, q-head) of a
// multi-split session the split kernel did not merge. Warp w folds chain w, the
// contiguous quarter [w*ns/4, (w+1)*ns/4) of the splits (split order), each
// split's kParts states joined first as the split kernel joins them, then
// warp 0 merges the four chains in order. The result depends only on the
// partials and ns. Launched as a programmatic dependent of K1: it waits for
// K1's completion with griddepcontrol.wait, so its CTAs can already be resident
// while K1 drains. Batches of kBatch splits: every load of a batch is issued
// before the first is folded (indices clamped into the quarter, no guards).
template <int kParts, int kBatch>
__global__ void __launch_bounds__(128) decode_combine_kernel(const DecodeArgs a) {
    asm volatile("griddepcontrol.launch_dependents;");   // a following overlapped call
    const int64_t row = blockIdx.x;                // lb * Hq + h
    const int ns = splits_to_merge(a, static_cast<int>((row / a.s.Hq) % a.B),
                                   kParts == 1 ? a.merge_max_splits : -1);
    if (ns == 0 && blockIdx.x != 0) return;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (ns == 0) return;
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int64_t base = row * a.max_splits * kParts;
    const float2 *ml = reinterpret_cast<const float2 *>(a.part_ml) + base;
    const float4 *po = reinterpret_cast<const float4 *>(a.part_o + base * kHeadDim) + lane;
    __shared__ float s_m[kCombineWarps], s_l[kCombineWarps];
    __shared__ float4 s_acc[kCombineWarps][kHeadDim / 4];
    const int s0 = (warp * ns) / kCombineWarps;
    const int s1 = ((warp + 1) * ns) / kCombineWarps;
    float m = -INFINITY, lsum = 0.f;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int sb = s0; sb < s1; sb += kBatch) {
        float2 v[kBatch][kParts];
        float4 o[kBatch][kParts];
#pragma unroll
        for (int j = 0; j < kBatch; ++j) {
            const int sp = min(sb + j, s1 - 1) * kParts;
#pragma unroll
            for (int r = 0; r < kParts; ++r) {
                v[j][r] = ml[sp + r];
                o[j][r] = po[(sp + r) * (kHeadDim / 4)];
            }
        }
#pragma unroll
        for (int j = 0; j < kBatch; ++j) {
            float mr[kParts], lr[kParts];
#pragma unroll
            for (int r = 0; r < kParts; ++r) {
                mr[r] = v[j][r].x;
                lr[r] = v[j][r].y;
            }
            join_accs<kParts>(mr, lr, o[j]);
            if (sb + j < s1) lse_step(m, lsum, acc, make_float2(mr[0], lr[0]), o[j][0]);
        }
    }
    s_acc[warp][lane] = acc;
    if (lane == 0) {
        s_m[warp] = m;
        s_l[warp] = lsum;
    }
    __syncthreads();
    if (warp == 0) {
        float mq[kMergeChains], lq[kMergeChains];
        float4 aq[kMergeChains];
#pragma unroll
        for (int q = 0; q < kMergeChains; ++q) {
            mq[q] = s_m[q];
            lq[q] = s_l[q];
            aq[q] = s_acc[q][lane];
        }
        merge_chains_store(a, row, lane, mq, lq, aq);
    }
}

// K2 for shared splits, tables of at most kRegMergeMax splits: as above, with
// all of a chain's partials (at most four splits of 2 halves or 8 accumulators)
// loaded at once. Latency-bound: one round trip to L2 (0.13 us, several times
// that under the next call's copies), then 0.4 us of dependent steps. The loop
// above in its place keeps fewer registers and starts its loads after each
// other: 6.2 instead of 5.3 us per layer for one session of 3 001 tokens, 13.3
// instead of 12.5 for 8 x 4K.
template <int kParts>
__global__ void __launch_bounds__(128) decode_combine_shared_kernel(const DecodeArgs a) {
    asm volatile("griddepcontrol.launch_dependents;");   // a following overlapped call
    const int64_t row = blockIdx.x;                // lb * Hq + h
    const int ns = splits_to_merge(a, static_cast<int>((row / a.s.Hq) % a.B), -1);
    if (ns == 0 && blockIdx.x != 0) return;
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int s0 = (warp * ns) / kMergeChains;
    const int n = ((warp + 1) * ns) / kMergeChains - s0;
    const int64_t base = row * a.max_splits * kParts;
    const float2 *ml = reinterpret_cast<const float2 *>(a.part_ml) + base;
    const float4 *po = reinterpret_cast<const float4 *>(a.part_o + base * kHeadDim) + lane;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (ns == 0) return;
    __shared__ float s_m[kMergeChains], s_l[kMergeChains];
    __shared__ float4 s_acc[kMergeChains][kHeadDim / 4];
    constexpr int kPer = kRegMergeMax / kMergeChains;
    float2 v[kPer][kParts];
    float4 o[kPer][kParts];
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        if (i < n) {
#pragma unroll
            for (int r = 0; r < kParts; ++r) {
                const int p = (s0 + i) * kParts + r;
                v[i][r] = __ldcg(ml + p);
                o[i][r] = __ldcg(po + p * (kHeadDim / 4));
            }
        }
    }
    float m = -INFINITY, lsum = 0.f;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        if (i < n) {
            float mr[kParts], lr[kParts];
#pragma unroll
            for (int r = 0; r < kParts; ++r) {
                mr[r] = v[i][r].x;
                lr[r] = v[i][r].y;
            }
            join_accs<kParts>(mr, lr, o[i]);
            lse_step(m, lsum, acc, make_float2(mr[0], lr[0]), o[i][0]);
        }
    }
    s_acc[warp][lane] = acc;
    if (lane == 0) {
        s_m[warp] = m;
        s_l[warp] = lsum;
    }
    __syncthreads();
    if (warp == 0) {
        float mq[kMergeChains], lq[kMergeChains];
        float4 aq[kMergeChains];
#pragma unroll
        for (int q = 0; q < kMergeChains; ++q) {
            mq[q] = s_m[q];
            lq[q] = s_l[q];
            aq[q] = s_acc[q][lane];
        }
        merge_chains_store(a, row, lane, mq, lq, aq);
    }
}

}  // namespace

bool encode_hot_tensor_map(CUtensorMap *map, void *hot_base, int64_t rows, int64_t run_rows,
                           const char **why) {
    // Resolved once; a function-local static is initialised exactly once even
    // when pools are created, or allocation-free decodes issued, on several
    // host threads at the same moment.
    static const PFN_cuTensorMapEncodeTiled_v12000 encode = [] {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000,
                                             cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            fn = nullptr;
        return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    }();
    if (!encode) {
        *why = "cuTensorMapEncodeTiled entry point unavailable";
        return false;
    }
    // A 4-D view of the pool: (64 columns, row, column half, K|V) with byte
    // strides (2, 256, 128, run_rows * 256). A tile is one box of it: 16 rows
    // of both halves of K and of V, landing in shared memory as [K|V][half]
    // [row][64] with the 128-byte swizzle, the layout the kernel reads.
    cuuint64_t dims[4] = {64, static_cast<cuuint64_t>(rows), 2, 2};
    cuuint64_t strides[3] = {static_cast<cuuint64_t>(kRowBytes), 128,
                             static_cast<cuuint64_t>(run_rows) * kRowBytes};
    cuuint32_t box[4] = {64, kTileTokens, 2, 2};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, hot_base, dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        *why = "cuTensorMapEncodeTiled rejected the hot pool";
        return false;
    }
    return true;
}

template <int kWarps, int kStages, int kSub, Form kForm = kAny>
static cudaError_t prepare_split() {
    return cudaFuncSetAttribute(decode_split_kernel<kWarps, kStages, kSub, kForm>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize,
                                decode_smem(kWarps, kStages));
}

cudaError_t prepare_kernels() {
    // Set in order, the last one telling that all of them are set: every pool
    // asks, and each set costs a pool's creation some 15 us.
    cudaFuncAttributes set;
    cudaError_t e = cudaFuncGetAttributes(&set, decode_split_kernel<1, 8, 8>);
    if (e == cudaSuccess && set.maxDynamicSharedSizeBytes >= decode_smem(1, 8)) return e;
    if (e == cudaSuccess) e = prepare_split<kWarpsNarrow, kStagesFull, 1>();
    if (e == cudaSuccess) e = prepare_split<kWarpsNarrow, kStagesHalf, 1>();
    if (e == cudaSuccess) e = prepare_split<kWarpsNarrow, kStagesFull, 1, kLongestFirst>();
    if (e == cudaSuccess) e = prepare_split<kWarpsNarrow, kStagesHalf, 1, kLongestFirst>();
    if (e == cudaSuccess) e = prepare_split<8, 3, 1, kOneSplit>();
    if (e == cudaSuccess) e = prepare_split<kWarpsNarrow, kStagesHalf, 1, kOneSplit>();
    if (e == cudaSuccess) e = prepare_split<kWarpsNarrow, kStagesFull, 1, kOneSplit>();
    if (e == cudaSuccess) e = prepare_split<4, 6, 2>();
    if (e == cudaSuccess) e = prepare_split<4, 3, 2>();
    if (e == cudaSuccess) e = prepare_split<4, 2, 2>();
    if (e == cudaSuccess) e = prepare_split<1, 8, 8>();
    return e;
}

template <int kWarps, int kStages, int kSub, Form kForm = kAny>
static cudaError_t launch_split(cudaLaunchConfig_t &c, const CUtensorMap &map, const DecodeArgs &a) {
    c.gridDim.x *= kSub;
    c.blockDim = dim3(kWarps * 32);
    c.dynamicSmemBytes = decode_smem(kWarps, kStages);
    return cudaLaunchKernelEx(&c, decode_split_kernel<kWarps, kStages, kSub, kForm>, map, a);
}

template <int kStages>
static cudaError_t launch_unshared(const DecodeShape &d, cudaLaunchConfig_t &c, const CUtensorMap &map,
                                   const DecodeArgs &a) {
    if (d.one_split) return launch_split<kWarpsNarrow, kStages, 1, kOneSplit>(c, map, a);
    if (d.by_length) return launch_split<kWarpsNarrow, kStages, 1, kLongestFirst>(c, map, a);
    return launch_split<kWarpsNarrow, kStages, 1>(c, map, a);
}

cudaError_t launch_decode(const CUtensorMap &map, const DecodeArgs &a, int num_sms,
                          cudaStream_t st, bool overlap_previous) {
    // Every session of the batch has T <= max_blocks * bt, so its splits fit.
    const int splits = max_splits_for(static_cast<int64_t>(a.max_blocks) * a.s.bt);
    if (splits > a.max_splits) return cudaErrorInvalidValue;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;

    cudaLaunchConfig_t c1 = {};
    c1.gridDim = dim3(splits, a.s.Hkv, a.nlayers * a.B);
    c1.blockDim = dim3(kWarpsNarrow * 32);
    c1.stream = st;
    c1.attrs = overlap_previous ? attr : nullptr;
    c1.numAttrs = overlap_previous ? 1 : 0;
    const DecodeShape d = decode_shape(a, splits, num_sms, overlap_previous);
    DecodeArgs ka = a;
    ka.pace = d.pace;
    ka.merge_max_splits = d.merge_max_splits;
    cudaError_t e;
    if (d.sub == 8)
        e = launch_split<1, 8, 8>(c1, map, ka);
    else if (d.sub == 2 && d.per_sm == 1)
        e = launch_split<4, 6, 2>(c1, map, ka);
    else if (d.sub == 2 && d.per_sm == 2)
        e = launch_split<4, 3, 2>(c1, map, ka);
    else if (d.sub == 2)
        e = launch_split<4, 2, 2>(c1, map, ka);
    else if (d.per_sm == 1)
        e = launch_split<8, 3, 1, kOneSplit>(c1, map, ka);
    else if (d.per_sm == 2)
        e = launch_unshared<kStagesHalf>(d, c1, map, ka);
    else
        e = launch_unshared<kStagesFull>(d, c1, map, ka);
    if (e != cudaSuccess) return e;
    // Else the split kernel writes every session's output: one split each, or
    // few enough splits to merge there.
    if (!d.combine) return cudaSuccess;

    const int64_t rows = static_cast<int64_t>(a.nlayers) * a.B * a.s.Hq;
    cudaLaunchConfig_t c2 = {};
    c2.blockDim = dim3(kCombineWarps * 32);
    c2.dynamicSmemBytes = 0;
    c2.stream = st;
    c2.attrs = attr;
    c2.numAttrs = 1;
    if (d.sub == 1 && !d.wide) {
        c2.gridDim = dim3(static_cast<unsigned>((rows + 3) / 4));
        return cudaLaunchKernelEx(&c2, decode_combine_small_kernel, ka);
    }
    c2.gridDim = dim3(static_cast<unsigned>(rows));
    if (d.wide)
        return d.sub == 2 ? cudaLaunchKernelEx(&c2, decode_combine_kernel<2, 8>, ka)
                        : cudaLaunchKernelEx(&c2, decode_combine_kernel<1, 16>, ka);
    if (d.sub == 8) return cudaLaunchKernelEx(&c2, decode_combine_shared_kernel<8>, ka);
    return cudaLaunchKernelEx(&c2, decode_combine_shared_kernel<2>, ka);
}

}  // namespace kvt
