// Copy kernels of the hot/cold KV tiering hot path, for sm_103a.
//
//   migrate_kernel<false>  data path 2: resume-unpack, cold image -> blocks.
//   resume_inline_kernel   the same for a resume of up to 2 048 blocks whose
//                          ids ride in the launch (it also writes the row).
//   migrate_kernel<true>   data path 4: pause-pack, blocks -> cold image,
//                          tokens [t0, T) only (write-on-evict, Section 3).
//   block_jobs_kernel<>    the same moves for explicit (slot, block, token
//                          range) lists: residency-mode evictions and fetches.
//   append_kernel          data path 3: fresh tokens into the tail blocks.
//   append_inline_kernel   the same with up to 2 048 new block ids in the launch.
//   table_write_kernel / gather_tables_kernel: block-table bookkeeping.
//
// Hot pool: hot[NB][L][2][Hkv][bt][128] bf16. A (block, layer, K|V, head)
// run is bt rows of 256 B. The image of a session is img[L][2][Hkv][T_cap][128].
#include <cstdint>

#include "kvt_internal.h"

namespace kvt {
namespace {

// Migration copy shape: one warp per 8-token chunk of a run (2 KiB on both
// sides), moved by one round of 32-byte loads, two per lane, and stores. Bound
// by HBM. The warps are not reused, unless decode may run beside the move
// (migration_ctas): a grid-stride loop over 32 CTAs per SM moved three sessions of
// 20K-30K tokens in 2.26 ms, one warp per chunk in 2.19 ms (16-byte loads in
// that loop 2.31 ms). Four loads
// per lane over 16 tokens need 48 registers, so five CTAs an SM instead of
// six, and a move of 29 MB ends with a second wave of a few CTAs: two resumes of
// 892 tokens, 16 layers, 28.4 us, now 26.1 (27.6 with 16-byte loads); of 1 000
// 29.0 and 27.5; of 24K, 48 layers, 1 339 and 1 335; three of 892 in a row 80.3
// and 82.2 (82.2). Held to 40 registers they spill (31.5).
// Moves larger than kOnceBytes touch image and blocks once and let both leave
// the L2 first, which leaves room for what others keep there: of a turn of
// 1 536 tokens, appended and then packed, the pack finds most of the appended
// blocks in the L2 (96.1 -> 87.4 us with both hints, 94.4 with one of them).
// Smaller ones may be used again while they are there (two resumes of 300
// tokens 26.4 us, 28.0 with the hints).
constexpr int kMigChunkTokens = 8;      // tokens per migration item (divides bt)
constexpr int kMigUnroll = 2;           // 32-byte loads in flight per lane
static_assert(kMigChunkTokens * kRowBytes == 32 * 32 * kMigUnroll, "one round moves a chunk");
constexpr int64_t kOnceBytes = int64_t(32) << 20;   // a quarter of the L2
constexpr int kAppendRows = 16;         // head rows an append warp moves
constexpr int append_group(int Hkv) {   // tokens that make them up
    return Hkv * 2 >= kAppendRows ? 1 : kAppendRows / (2 * Hkv);
}
// head_inv of a shape: (w * head_inv) >> 8 == w / Hkv for the rows w of an item.
constexpr int head_inv(int Hkv) { return (256 + Hkv - 1) / Hkv; }
constexpr bool head_inv_exact() {
    for (int h = 1; h <= 8; ++h)
        for (int w = 0; w < append_group(h) * h; ++w)
            if ((w * head_inv(h)) >> 8 != w / h) return false;
    return true;
}
static_assert(head_inv_exact(), "kv-heads 1 to 8");

struct alignas(32) Row32 {
    uint32_t w[8];
};

// L2 policies of a move: its lines leave first, or as any others.
__device__ __forceinline__ uint64_t move_policy(bool once) {
    uint64_t p, q;
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    asm("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(q));
    return once ? p : q;
}

__device__ __forceinline__ Row32 ld_row(const Row32 *p, uint64_t policy) {
    Row32 v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8], %9;"
                 : "=r"(v.w[0]), "=r"(v.w[1]), "=r"(v.w[2]), "=r"(v.w[3]), "=r"(v.w[4]),
                   "=r"(v.w[5]), "=r"(v.w[6]), "=r"(v.w[7])
                 : "l"(p), "l"(policy));
    return v;
}

__device__ __forceinline__ void st_row(Row32 *p, const Row32 &v, uint64_t policy) {
    asm volatile("st.global.L2::cache_hint.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8}, %9;" ::"l"(p),
                 "r"(v.w[0]), "r"(v.w[1]), "r"(v.w[2]), "r"(v.w[3]), "r"(v.w[4]), "r"(v.w[5]),
                 "r"(v.w[6]), "r"(v.w[7]), "l"(policy)
                 : "memory");
}

__device__ __forceinline__ uint4 ld_stream(const uint4 *p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}

// Up to one chunk of rows from `from` to `to` by a warp.
__device__ __forceinline__ void move_rows(const uint8_t *from, uint8_t *to, int rows, int lane,
                                          uint64_t policy) {
    const Row32 *src = reinterpret_cast<const Row32 *>(from) + lane;
    Row32 *dst = reinterpret_cast<Row32 *>(to) + lane;
    const int units = rows * (kRowBytes / 32) - lane;
    Row32 v[kMigUnroll];
#pragma unroll
    for (int k = 0; k < kMigUnroll; ++k)
        if (k * 32 < units) v[k] = ld_row(src + k * 32, policy);
#pragma unroll
    for (int k = 0; k < kMigUnroll; ++k)
        if (k * 32 < units) st_row(dst + k * 32, v[k], policy);
}

// K3 / K4: the chunks of the token range of every (layer, K|V, kv-head) run.
// Both sides of a chunk are contiguous rows of 256 B. Items are ordered
// run-major so that consecutive warps walk the image sequentially (the eight
// runs of a block next to each other instead: 4.39 against 4.37 ms for the
// sessions above).
// The copy loop of a session's migration; block_of(j) gives logical block j's slot.
template <bool kPack, typename BlockOf>
__device__ __forceinline__ void migrate_runs(const MigArgs &a, BlockOf block_of) {
    const Shape sh = a.s;
    const int runs = sh.L * 2 * sh.Hkv;
    // Items are chunks of a run, so a 64-token block is as many warps' work as
    // four of 16 tokens.
    const int q0 = a.t_begin / kMigChunkTokens;
    const int q1 = (a.t_end + kMigChunkTokens - 1) / kMigChunkTokens;
    const int nq = q1 - q0;
    const int items = runs * nq;
    const int lane = threadIdx.x & 31;
    const uint64_t policy = move_policy(a.once);
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int it = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; it < items; it += nwarps) {
        const int c = it / nq;
        const int q = q0 + (it - c * nq);
        const int j = q * kMigChunkTokens / sh.bt;
        const int blk = block_of(j);
        if (blk < 0 || blk >= sh.num_blocks) {
            if (lane == 0) atomicOr(a.err, kErrBadBlock);
            continue;
        }
        const int t_lo = max(a.t_begin, q * kMigChunkTokens);
        const int t_hi = min(a.t_end, (q + 1) * kMigChunkTokens);
        uint8_t *hp = a.hot + ((static_cast<int64_t>(blk) * runs + c) * sh.bt + (t_lo - j * sh.bt)) *
                                  kRowBytes;
        uint8_t *ip = a.img + (static_cast<int64_t>(c) * a.T_cap + t_lo) * kRowBytes;
        move_rows(kPack ? hp : ip, kPack ? ip : hp, t_hi - t_lo, lane, policy);
    }
}

template <bool kPack>
__global__ void __launch_bounds__(kCopyThreads) migrate_kernel(const MigArgs a) {
    migrate_runs<kPack>(a, [&](int j) { return a.table[j]; });
}

// Resume-unpack with the new block ids in the launch parameters: the grid
// also writes them to the session's table row (read by later work only).
__global__ void __launch_bounds__(kCopyThreads) resume_inline_kernel(const __grid_constant__ ResumeArgs r) {
    const int nthreads = gridDim.x * blockDim.x;
    int32_t *row = const_cast<int32_t *>(r.m.table);   // the pool's own row: writable
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < r.n; j += nthreads)
        row[j] = r.blocks[j];
    migrate_runs<false>(r.m, [&](int j) { return j < r.n ? r.blocks[j] : -1; });
}

// K3'/K4': block-granular moves for the residency mode: one warp per chunk of a
// (job, layer, K|V, kv-head) run; a job moves tokens [t0, t1) of one block.
template <bool kPack>
__global__ void __launch_bounds__(kCopyThreads) block_jobs_kernel(const __grid_constant__ BlockJobs a) {
    const Shape sh = a.s;
    const int runs = sh.L * 2 * sh.Hkv;
    const int cpb = sh.bt / kMigChunkTokens;      // chunks per block
    const int items = a.n * runs * cpb;
    const int lane = threadIdx.x & 31;
    const uint64_t policy = move_policy(a.once);
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int it = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; it < items; it += nwarps) {
        const int jb = it / (runs * cpb);
        const int rem = it - jb * runs * cpb;
        const int c = rem / cpb;
        const int ch = rem - c * cpb;
        const BlockJob &b = a.job[jb];
        if (b.slot < 0 || b.slot >= sh.num_blocks || b.t0 < 0 || b.t1 > sh.bt) {
            if (lane == 0 && ch == 0 && c == 0) atomicOr(a.err, kErrBadBlock);
            continue;
        }
        if (!kPack && b.sid >= 0 && c == 0 && ch == 0 && lane == 0)   // a fetch: its table entry
            a.tables[static_cast<int64_t>(b.sid) * a.table_stride + b.j] = b.slot;
        const int t_lo = max(b.t0, ch * kMigChunkTokens);
        const int t_hi = min(b.t1, (ch + 1) * kMigChunkTokens);
        if (t_hi <= t_lo) continue;
        uint8_t *hp = a.hot + ((static_cast<int64_t>(b.slot) * runs + c) * sh.bt + t_lo) * kRowBytes;
        uint8_t *ip = b.img + (static_cast<int64_t>(c) * b.T_cap + static_cast<int64_t>(b.j) * sh.bt +
                               t_lo) * kRowBytes;
        move_rows(kPack ? hp : ip, kPack ? ip : hp, t_hi - t_lo, lane, policy);
    }
}

// K5: one warp per (layer, group of tokens). A token's K (or V) rows for all
// kv-heads are Hkv*256 contiguous bytes in the source, and so are the next
// token's; each 256-byte head row goes to its (layer, K|V, head) run of the
// token's block, beside the token before. A group is the tokens that make up 16
// head rows (4 KiB, one token of 8 kv-heads, four of 2), so that a warp moves as
// much whatever the shape, in one round of 16-byte loads, eight per lane, half a
// warp per row (k and v need be aligned to no more). Items are layer-major so that
// consecutive warps read k and v sequentially. Bound by HBM; one token per warp
// in its place: a turn of 16 000 tokens of 2 kv-heads, 16 layers, appended and
// packed, 180 -> 155 us.
// A short append is a chain of latencies: the block ids are on their way before
// the rows, and nothing in front of a load is divided but the item's number. With
// group counts, positions and row numbers divided here, 8 tokens of 4 kv-heads, 48
// layers, took 6.2 us and one of 8 kv-heads 6.2 (both 4.2 now; one token per
// warp in two launches 5.2 and 4.3), 100 tokens 7.8 (6.4).
// block_of(j) gives logical block j's slot.
template <typename BlockOf>
__device__ __forceinline__ void append_tokens(const AppendArgs &a, BlockOf block_of) {
    const Shape sh = a.s;
    const int items = sh.L * a.groups;
    const int lane = threadIdx.x & 31;
    const int c = lane & 15;                         // 16-byte unit of a row
    const int shift = sh.bt == 64 ? 6 : 4;           // blocks hold 16 or 64 tokens
    const int run_bytes = kRowBytes << shift;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int it = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; it < items; it += nwarps) {
        const int l = it / a.groups;
        const int i = (it - l * a.groups) * a.group;
        const int tokens = min(a.group, a.n - i);
        const int rows = tokens * sh.Hkv;            // of K, and again of V
        // The group lies in one block, or in two.
        const int t = a.pos0 + i;
        const int j = t >> shift;
        const int slot0 = t - (j << shift);
        const bool two = slot0 + tokens > sh.bt;
        const int blk[2] = {block_of(j), two ? block_of(j + 1) : 0};
        const int64_t src_off = (static_cast<int64_t>(l) * a.n + i) * sh.Hkv * kRowBytes;
        const uint4 *ks = reinterpret_cast<const uint4 *>(a.k + src_off) + c;
        const uint4 *vs = reinterpret_cast<const uint4 *>(a.v + src_off) + c;
        uint4 v[kAppendRows / 2];
#pragma unroll
        for (int k = 0; k < kAppendRows / 2; ++k) {
            const int r = 2 * k + (lane >> 4);
            if (r < 2 * rows) v[k] = ld_stream(r < rows ? ks + r * 16 : vs + (r - rows) * 16);
        }
        uint8_t *base[2];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const bool ok = blk[s] >= 0 && blk[s] < sh.num_blocks;
            if (!ok && lane == 0) atomicOr(a.err, kErrBadBlock);
            base[s] = ok ? a.hot + (static_cast<int64_t>(blk[s]) * sh.L + l) * 2 * sh.Hkv * run_bytes + c * 16
                         : nullptr;
        }
#pragma unroll
        for (int k = 0; k < kAppendRows / 2; ++k) {
            const int r = 2 * k + (lane >> 4);
            if (r >= 2 * rows) continue;
            const int kv = r >= rows;
            const int w = r - kv * rows;             // token and head of the row
            const int ti = (w * a.head_inv) >> 8;    // w / Hkv (append_shape)
            const int slot = slot0 + ti;
            const int next = slot >= sh.bt;
            uint8_t *to = next ? base[1] : base[0];
            if (to != nullptr)
                *reinterpret_cast<uint4 *>(to + (kv * sh.Hkv + (w - ti * sh.Hkv)) * run_bytes +
                                           (slot - next * sh.bt) * kRowBytes) = v[k];
        }
    }
}

__global__ void __launch_bounds__(kCopyThreads) append_kernel(const AppendArgs a) {
    append_tokens(a, [&](int j) { return a.table[j]; });
}

// An append whose new block ids ride in the launch: the grid also writes them
// to the session's table row (read by later work only), which saves the
// table-write launch in front of it: a turn of 1 536 tokens, appended and
// packed, 98.0 -> 94.3 us.
__global__ void __launch_bounds__(kCopyThreads) append_inline_kernel(const __grid_constant__ AppendInlineArgs r) {
    const int nthreads = gridDim.x * blockDim.x;
    int32_t *row = const_cast<int32_t *>(r.m.table);   // the pool's own row: writable
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < r.n; j += nthreads)
        row[r.from + j] = r.blocks[j];
    append_tokens(r.m, [&](int j) {
        return j < r.from ? r.m.table[j] : j < r.from + r.n ? r.blocks[j - r.from] : -1;
    });
}

__global__ void table_write_kernel(const __grid_constant__ TableWriteArgs a) {
    for (int i = threadIdx.x; i < a.n; i += blockDim.x) a.dst[i] = a.vals[i];
}

__global__ void gather_tables_kernel(const __grid_constant__ GatherArgs a) {
    const int r = blockIdx.x;
    if (r >= a.count) return;
    int32_t *src = a.arena + static_cast<int64_t>(a.sids[r]) * a.stride;
    int32_t *dst = a.tables + static_cast<int64_t>(a.row0 + r) * a.max_blocks;
    const int n = a.nblk[r];
    const int32_t nb = a.new_blk[r];   // a block the row just gained, not yet in the arena
    for (int e = threadIdx.x; e < a.max_blocks; e += blockDim.x)
        dst[e] = e < n ? (e == n - 1 && nb >= 0 ? nb : src[e]) : -1;
    if (threadIdx.x == 0) {
        if (nb >= 0) src[n - 1] = nb;
        a.seq_lens[a.row0 + r] = a.lens[r];
    }
}

}  // namespace

// Chunks of a session's move, and whether it goes through the L2 once.
static int64_t move_items(const MigArgs &a) {
    const int64_t nq = (a.t_end + kMigChunkTokens - 1) / kMigChunkTokens - a.t_begin / kMigChunkTokens;
    return nq * a.s.L * 2 * a.s.Hkv;
}
static int32_t moves_once(int64_t items) {
    return items * kMigChunkTokens * kRowBytes > kOnceBytes;
}

cudaError_t launch_unpack(MigArgs a, int max_ctas, cudaStream_t st) {
    if (a.t_end <= a.t_begin) return cudaSuccess;
    a.once = moves_once(move_items(a));
    migrate_kernel<false><<<item_grid(move_items(a), max_ctas), kCopyThreads, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_unpack_inline(ResumeArgs &r, int max_ctas, cudaStream_t st) {
    if (r.m.t_end <= r.m.t_begin || r.n < 1 || r.n > kResumeInlineMax) return cudaErrorInvalidValue;
    r.m.once = moves_once(move_items(r.m));
    resume_inline_kernel<<<item_grid(move_items(r.m), max_ctas), kCopyThreads, 0, st>>>(r);
    return cudaGetLastError();
}

cudaError_t launch_pack(MigArgs a, int max_ctas, cudaStream_t st) {
    if (a.t_end <= a.t_begin) return cudaSuccess;
    a.once = moves_once(move_items(a));
    migrate_kernel<true><<<item_grid(move_items(a), max_ctas), kCopyThreads, 0, st>>>(a);
    return cudaGetLastError();
}

// The items of an append: groups of tokens, per layer. Worked out here, since the
// divisions would stand in front of a short append's loads.
static int64_t append_shape(AppendArgs &a) {
    a.group = append_group(a.s.Hkv);
    a.groups = (a.n + a.group - 1) / a.group;
    a.head_inv = head_inv(a.s.Hkv);
    return static_cast<int64_t>(a.s.L) * a.groups;
}

cudaError_t launch_append(AppendArgs a, int max_ctas, cudaStream_t st) {
    const int64_t items = append_shape(a);
    append_kernel<<<item_grid(items, max_ctas), kCopyThreads, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_append_inline(AppendInlineArgs &r, int max_ctas, cudaStream_t st) {
    if (r.n < 1 || r.n > kResumeInlineMax) return cudaErrorInvalidValue;
    const int64_t items = append_shape(r.m);
    append_inline_kernel<<<item_grid(items, max_ctas), kCopyThreads, 0, st>>>(r);
    return cudaGetLastError();
}

cudaError_t launch_block_jobs(BlockJobs &a, bool pack, int max_ctas, cudaStream_t st) {
    if (a.n <= 0) return cudaSuccess;
    const int64_t items = static_cast<int64_t>(a.n) * a.s.L * 2 * a.s.Hkv *
                          (a.s.bt / kMigChunkTokens);
    const unsigned grid = item_grid(items, max_ctas);
    a.once = moves_once(items);
    if (pack)
        block_jobs_kernel<true><<<grid, kCopyThreads, 0, st>>>(a);
    else
        block_jobs_kernel<false><<<grid, kCopyThreads, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_table_write(const TableWriteArgs &a, cudaStream_t st) {
    table_write_kernel<<<1, 256, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_gather(const GatherArgs &a, cudaStream_t st) {
    gather_tables_kernel<<<a.count, 128, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace kvt
