// The sparse expert MLPs (Eq. 1) in ONE persistent launch, for tokens grouped by expert:
//
//   up    h[r,:] = GeLU(x[row_token[r],:] . W1[e])                 tile = (expert, 128 rows, <= 256 hidden units)
//   down  rows[r,:] = row_gate[r] * (h[r,:] . W2[e])  in fp32      tile = (expert, 128 rows, <= 256 output columns)
//
//   warp 0       TMA producer          (one lane)
//   warp 1       MMA issuer            (one lane); owns the TMEM allocation
//   warps 2..5   epilogue              (warp w reads TMEM lanes 32*(w%4) .. +31)
//   warps 6..13  gather the up-projection's rows of x
//   warp 14      dealer: claims this CTA's next tile and hands it to the others
//
// One list of tiles -- every up tile, then the down tiles -- is claimed in order, a tile at a time, by one CTA per SM: no round of
// tiles is left incomplete at the end of the up-projection (448 tiles on 148 CTAs for 7001 tokens of 4096, 32 experts of 512, top-4:
// four rounds for the work of three) and no launch gap lies between the projections.  A down tile waits (on a counter) until its
// own 128 rows of h are complete, nothing else; its weights are on their way meanwhile.
// Every up tile that a down tile may wait for is in the hands of a CTA that runs, and no CTA has a down tile before its last up
// tile.  So the waits end with any number of resident CTAs: in a context that owns a part of the SMs, and beside other streams'
// kernels, whose SMs join in as they become free.  (Dealt out by CTA index, as it was first, the list needed every SM at once, a
// cooperative launch.)  Claimed against dealt out: 32 shapes of 150 to 1500 tokens 1.01 times as fast (0.98 to 1.09), 48 of 1024 to
// 8192 1.02 (0.97 to 1.09): a CTA that is done early takes more.
// The first round alone is not first come, first served: tile b is CTA b's, and goes to another only if CTA b has not begun.  CTAs of
// neighbouring indices sit on SMs far apart, so that 64 up tiles do not share the 74 SM pairs' ways to L2 by chance (150 tokens
// of 4096, 512 wide: 120 us first come, 113 so).
// Against two launches of umma_gemm_kernel (dealt out, cooperative), layers of 32 experts (us): 300 tokens of 2048, 1024 wide, by
// threshold 91 -> 86; 1500 of 3072, 384 wide, by threshold 214 -> 180; 3333 of 3072, 384 wide, top-6 237 -> 205; 7001 of 4096, 512 wide,
// top-4 441 -> 422; 8192 of 6144, 768 wide, top-4 904 -> 882 (76 shapes of 150 to 8192 tokens: 1.06 times on average, 0.98 to 1.22).
// Bound by the latency of the operands' way out of L2 (2048 tokens of 4096, 512 wide, top-4: tensor pipe 42 % busy, L2 at 37 % of its
// throughput, DRAM at 47 %; the issuer waits while four ring slots are under way) and, with narrow experts, the fp32 rows' way to memory
// (7001 tokens of that shape: the down tiles 158 us, 108 without their stores).
// Up to 2048 tokens (1024 of more than 32 experts: what the selection words' table may take of the shared memory) there is no row-index
// kernel before this one: every CTA turns the selection words into a bit per expert, chunk and token and finds its tiles' rows there.
// Without that kernel, its launch and the one that cannot be chained to it, whole calls (us): 300 tokens of 2048, 256 wide, 32 experts,
// top-4 53.1 -> 45.1; 1500 of 4096, 512 wide 132.8 -> 121.9; 700 of 128, 192 wide, 8 experts 35.0 -> 28.8 (130 shapes of 130 to
// 2048 tokens: 1.02 to 1.30 times).  Beyond that the 8 us are a per cent or two.
// The weighted sum of Eq. 1 inside this launch, over groups of columns whose rows were to stay in L2, was slower than its own launch
// in every form (355 us and more against 248 + 78): beside a 200 KB ring an SM has too few bytes of rows under way, and handing
// small groups from stores to sums and back costs more than the rows' way to memory and back.
#include <algorithm>

#include "common.cuh"
#include "mlp_device.cuh"

namespace dsmoe {

namespace {

constexpr int kStageRow = 144;                   // bytes of a row of the tiles through which the epilogue's rows leave

struct GroupedParams {
    int E, d, H, T, W;
    long long amax;
    GroupedFold fold;              // FOLD: in place of offsets, row_token and row_gate
    const int32_t* offsets;
    const int32_t* row_token;
    const float* row_gate;
    const __nv_bfloat16* x;
    __nv_bfloat16* h;              // [amax, H]
    float* rows;                   // [amax, d]
    int* sync;                     // zero at launch: [0] row tiles of h that are complete; [kSyncNext] tiles claimed beyond the first round; from
                                   // kSyncTaken on, a bit per tile of the first round; from kSyncH on, per row tile, its finished epilogue warps
    int max_row_tiles;             // ... and so many of these there are
    int32_t* dev_status;
};
constexpr int kSyncNext = 8, kSyncTaken = 16, kSyncH = 24;
constexpr int kGroupedMaxCtas = 32 * (kSyncH - kSyncTaken);

struct alignas(16) GroupedTile {
    int up, e, row0, rows_valid, rt, n0, bn, nk;      // e < 0: no more tiles
};
constexpr int kTileSlots = 4;                          // claimed tiles that the CTA's roles have not all seen yet
// Blocks of a tile's reduction still to be loaded when the next tile is claimed: the claim, finding the tile and its rows' tokens take
// some 2 us, 8 blocks and the ring's 4 some 3.  (2 or 4 blocks: the same within 0.5 %.  As soon as the roles' slots are free, with up to
// four tiles in hand: 0.93, the last ones wait in some CTAs while others have none.)
constexpr int kClaimAhead = 8;
constexpr int kGroupedThreads = GATHER_THREADS + 32;   // ... and the dealer
constexpr int kTileReaders = 2 + 4 + GATHER_WARPS;

struct GroupedShared {
    uint64_t full[STAGES], empty[STAGES], tfull[2], tempty[2];
    uint64_t tile_full[kTileSlots], tile_empty[kTileSlots], want;      // the dealer's: a tile is there; all have seen it; claim the next
    GroupedTile tile[kTileSlots];
    uint32_t tmem_base;
    volatile int abort_flag;
    int row_tiles, up_tiles, down_tiles;   // totals
    int bad_offsets;
    int seg0[kMaxExperts], seg1[kMaxExperts];      // rows of each expert
    int rt0[kMaxExperts + 1];                      // its first row tile
    int rowtok[GATHER_WARPS * (BM / 2)];
};
constexpr size_t kGroupedShared = 4096;
static_assert(sizeof(GroupedShared) <= kGroupedShared, "barriers and tables");
// FOLD (1: up to 1024 tokens, 2: up to 2048 of at most 32 experts): which of a chunk's tokens selected an expert, [chunk][expert]
constexpr size_t kFoldBytes = kGroupedFoldWords * sizeof(uint32_t);
template <int FOLD>
struct FoldTable {
    static constexpr int CHUNKS = 32 * FOLD, LD = FOLD == 2 ? 33 : 65;      // (odd: a column's words lie in different banks)
    static_assert(CHUNKS * LD <= kGroupedFoldWords, "");
};
constexpr size_t kGroupedSmem = 1024 + (size_t)RING_BYTES + kGroupedShared + 4 * 32 * kStageRow;
static_assert(kGroupedSmem + kFoldBytes <= 227 * 1024, "shared memory of one CTA");

#ifdef DSMOE_TRACE
// Diagnostic build only, per CTA.  Time stamps (globaltimer): [0] start, [1] last up tile multiplied, [2] last tile multiplied, [3] epilogue
// done.  Cycles waited: [4] MMA issuer for operands of up tiles, [5] of down tiles, [6] for an accumulator, [7] producer for h.
__device__ long long g_grouped_trace[192][8];
#define GT_NOW() (long long)ptx::globaltimer_ns()
#define GT_SET(i) do { if (blockIdx.x < 192) g_grouped_trace[blockIdx.x][i] = GT_NOW(); } while (0)
#define GT_T0(v) const long long v = clock64()
#define GT_ADD(var, v) var += clock64() - (v)
#define GT_PUT(i, var) do { if (blockIdx.x < 192) g_grouped_trace[blockIdx.x][i] = (var); } while (0)
#else
#define GT_SET(i)
#define GT_T0(v)
#define GT_ADD(var, v)
#define GT_PUT(i, var)
#endif


// Tile `id` of the list (the whole warp asks); e < 0: the list is shorter.  Experts ascend, then column ranges; the row tiles of one
// weight tile follow one another.
__device__ __forceinline__ GroupedTile tile_at(const GroupedParams& P, const GroupedShared& sh, int id, int lane) {
    GroupedTile t;
    t.up = id < sh.up_tiles;
    if (!t.up) id -= sh.up_tiles;
    const int N = t.up ? P.H : P.d, ntn = ceil_div(N, BN);
    const unsigned lo = __ballot_sync(0xffffffffu, lane < P.E && id >= sh.rt0[min(lane, P.E)] * ntn);
    const unsigned hi = __ballot_sync(0xffffffffu, lane + 32 < P.E && id >= sh.rt0[min(lane + 32, P.E)] * ntn);
    const int e = __popc(lo) + __popc(hi) - 1;      // (the last expert that begins at or before id: one with rows)
    const int local = id - sh.rt0[e] * ntn, mtiles = max(sh.rt0[e + 1] - sh.rt0[e], 1);
    const int nt = local / mtiles, mt = local - nt * mtiles;
    t.e = !t.up && id >= sh.down_tiles ? -1 : e;
    t.rt = sh.rt0[e] + mt;
    t.row0 = sh.seg0[e] + mt * BM;
    t.rows_valid = min(BM, sh.seg1[e] - t.row0);
    t.n0 = nt * BN;
    t.bn = min(BN, N - t.n0);
    t.nk = (t.up ? P.d : P.H) / BK;
    return t;
}

// A role's place in the sequence of tiles that the dealer hands to this CTA.  Finding a tile takes some hundred cycles, which in
// series with a tile of 8 reduction blocks (4096 cycles of the tensor core) cost the MMA issuer a third of its time: the
// dealer does it, ahead of the others.
struct TileReader {
    int k = 0;
    // the next tile (the whole warp asks); false: no more, or given up
    __device__ __forceinline__ bool next(GroupedShared& sh, int lane, GroupedTile& t) {
        const int slot = k % kTileSlots;
        const bool there = ptx::mbar_wait(ptx::smem_u32(&sh.tile_full[slot]), (uint32_t)(k / kTileSlots) & 1u, &sh.abort_flag);
        if (!__all_sync(0xffffffffu, there)) return false;
        t = sh.tile[slot];
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&sh.tile_empty[slot]));
        ++k;
        return t.e >= 0;
    }
};

// Counters in global memory that other CTAs wait for.  An arrival releases this thread's writes and, after a __syncwarp, its
// warp's.  Waiting polls with relaxed loads and acquires once at the end: an acquiring load empties the SM's L1.
__device__ __forceinline__ void counter_add(int* c, int n) {
    asm volatile("red.release.gpu.global.add.s32 [%0], %1;" ::"l"(c), "r"(n) : "memory");
}
__device__ __forceinline__ int counter_now(const int* c) {
    int v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(c) : "memory");
    return v;
}
__device__ __forceinline__ int counter_acquire(const int* c) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(c) : "memory");
    return v;
}
// Bounded wait until the counter is at least `target`; false: gave up (limit reached, or another thread of the CTA already had)
__device__ __forceinline__ bool counter_wait(const int* c, int target, volatile int* abort_flag) {
    uint64_t t0 = 0;
    while (counter_now(c) < target) {
        __nanosleep(100);
        const uint64_t now = ptx::globaltimer_ns();
        if (t0 == 0) t0 = now;
        if (*abort_flag || now - t0 > ptx::kWaitLimitNs) {
            *abort_flag = 1;
            return false;
        }
    }
    return counter_acquire(c) >= target;
}

// The first round of tiles: tile b is CTA b's if it comes for it.  false: another CTA has taken it
__device__ __forceinline__ bool take_first_round(int* sync, int b) {
    const unsigned bit = 1u << (b & 31);
    return (atomicOr(reinterpret_cast<unsigned*>(sync) + kSyncTaken + (b >> 5), bit) & bit) == 0;
}
// Before its first down tile a CTA sees to it that the first n tiles (the up tiles of the first round) are all taken: those whose
// CTAs have not begun within kGraceNs it takes itself, one a call.  -1: none is left.  (The whole warp calls; t0: when it first
// found one missing, 0 before.)
constexpr uint64_t kGraceNs = 5000;     // (the CTAs of a launch begin within 0.5 us of each other where there is room)
__device__ __forceinline__ int left_over(int* sync, int n, int lane, uint64_t& t0) {
    for (;;) {
        unsigned missing = 0;
        if (lane * 32 < n) {
            missing = ~(unsigned)counter_now(sync + kSyncTaken + lane);
            if (n - lane * 32 < 32) missing &= (1u << (n - lane * 32)) - 1u;
        }
        const unsigned words = __ballot_sync(0xffffffffu, missing != 0);
        if (!words) return -1;
        const uint64_t now = __shfl_sync(0xffffffffu, ptx::globaltimer_ns(), 0);
        if (t0 == 0) t0 = now;
        if (now - t0 > kGraceNs) {
            const int word = __ffs(words) - 1;
            const int b = word * 32 + __ffs(__shfl_sync(0xffffffffu, missing, word)) - 1;
            if (__shfl_sync(0xffffffffu, lane == 0 && take_first_round(sync, b) ? 1 : 0, 0)) return b;
        } else {
            __nanosleep(200);
        }
    }
}

// 32 words of 32 bits, one a lane, transposed: bit i of lane e's result is bit e of lane i's word
__device__ __forceinline__ uint32_t transpose_bits(uint32_t x, int lane) {
    uint32_t low = 0xffffu;                          // the low half of every 2 j bits
#pragma unroll
    for (int j = 16; j > 0; j >>= 1) {
        const uint32_t y = __shfl_xor_sync(0xffffffffu, x, j);
        x = lane & j ? (x & ~low) | ((y >> j) & low) : (x & low) | ((y << j) & ~low);
        low ^= low << (j >> 1);
    }
    return x;
}

// The tokens of an expert's rows min(first + lane + 32 j, last), counted within the expert, whose rows ascend by token (the whole warp asks).
template <int FOLD, int N>
__device__ __forceinline__ void find_tokens(const uint32_t* bits, int e, int first, int last, int lane, int (&tok)[N]) {
    uint32_t w[FOLD];
    int n = 0;
#pragma unroll
    for (int i = 0; i < FOLD; ++i) {
        w[i] = bits[(lane * FOLD + i) * FoldTable<FOLD>::LD + e];
        n += __popc(w[i]);
    }
    int before = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, before, o);
        if (lane >= o) before += v;
    }
    before -= n;
#pragma unroll
    for (int j = 0; j < N; ++j) {
        const int r = min(first + lane + 32 * j, last);
        int c = 0;                                   // the last lane whose chunks begin at or before r: the one that has it
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            if (__shfl_sync(0xffffffffu, before, c + o) <= r) c += o;
        int k = r - __shfl_sync(0xffffffffu, before, c), at = c * FOLD * kChunk;
        uint32_t b = __shfl_sync(0xffffffffu, w[0], c);
        if (FOLD == 2) {
            const uint32_t b1 = __shfl_sync(0xffffffffu, w[FOLD - 1], c);
            if (const int n0 = __popc(b); k >= n0) {
                k -= n0;
                b = b1;
                at += kChunk;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {           // its k-th bit
            const int low = __popc(b & ((1u << o) - 1u));
            if (k >= low) {
                k -= low;
                b >>= o;
                at += o;
            }
        }
        tok[j] = at;
    }
}

template <int FOLD>
__global__ void __launch_bounds__(kGroupedThreads, 1)
grouped_layer_kernel(const __grid_constant__ BMaps tmW1, const __grid_constant__ CUtensorMap tmH,
                     const __grid_constant__ BMaps tmW2, const GroupedParams P) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = ptx::smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;             // 128-byte swizzle wants 1024-byte aligned tiles
    const uint32_t smA = base, smB = base + STAGES * A_STAGE_BYTES;
    GroupedShared& sh = *reinterpret_cast<GroupedShared*>(smem_raw + (base - raw) + RING_BYTES);
    uint8_t* const stage = smem_raw + (base - raw) + RING_BYTES + kGroupedShared;
    uint32_t* const bits = reinterpret_cast<uint32_t*>(stage + 4 * 32 * kStageRow);       // (FOLD only)
    using Table = FoldTable<FOLD ? FOLD : 1>;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            ptx::mbar_init(ptx::smem_u32(&sh.full[s]), 3);      // the producer and two gathering warps (down: the producer thrice)
            ptx::mbar_init(ptx::smem_u32(&sh.empty[s]), 1);
        }
        for (int a = 0; a < 2; ++a) {
            ptx::mbar_init(ptx::smem_u32(&sh.tfull[a]), 1);
            ptx::mbar_init(ptx::smem_u32(&sh.tempty[a]), 4);
        }
        for (int s = 0; s < kTileSlots; ++s) {
            ptx::mbar_init(ptx::smem_u32(&sh.tile_full[s]), 1);
            ptx::mbar_init(ptx::smem_u32(&sh.tile_empty[s]), kTileReaders);
        }
        ptx::mbar_init(ptx::smem_u32(&sh.want), 1);
        sh.abort_flag = 0;
        sh.bad_offsets = 0;
        ptx::fence_barrier_init();
        ptx::prefetch_tensormap(&tmH);
        for (int i = 2; i < 5; ++i) ptx::prefetch_tensormap(&tmW1.m[i]);
        for (int i = 2; i < 5; ++i) ptx::prefetch_tensormap(&tmW2.m[i]);
    }
    if (warp == 1) {
        ptx::tmem_alloc(ptx::smem_u32(&sh.tmem_base), TMEM_COLS);
        ptx::tmem_relinquish();
    }
    if (FOLD) chain_wait();
    // (the dealer's; asked before the tables below are there)
    bool first_is_mine = false;
    if (warp == kGroupedThreads / 32 - 1 && lane == 0) first_is_mine = take_first_round(P.sync, blockIdx.x);
    if (FOLD) {
#pragma unroll 4
        for (int c = warp; c < Table::CHUNKS; c += kGroupedThreads / 32) {
            const uint64_t m = c * kChunk + lane < P.T ? P.fold.mask[c * kChunk + lane] : 0ull;
            bits[c * Table::LD + lane] = transpose_bits((uint32_t)m, lane);
            if (FOLD == 1) bits[c * Table::LD + lane + 32] = transpose_bits((uint32_t)(m >> 32), lane);
        }
        __syncthreads();
    }
    if (warp == 0) {
        __syncwarp();
        int first[2], count[2] = {0, 0};             // FOLD: experts lane, lane + 32
        if (FOLD) {
#pragma unroll
            for (int c = 0; c < Table::CHUNKS; ++c) {
                count[0] += __popc(bits[c * Table::LD + lane]);
                if (FOLD == 1) count[1] += __popc(bits[c * Table::LD + lane + 32]);
            }
            first[0] = count[0];
            first[1] = count[1];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int a = __shfl_up_sync(0xffffffffu, first[0], o), b = __shfl_up_sync(0xffffffffu, first[1], o);
                if (lane >= o) {
                    first[0] += a;
                    first[1] += b;
                }
            }
            first[1] += __shfl_sync(0xffffffffu, first[0], 31);
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                first[j] -= count[j];
                if (blockIdx.x == 0 && lane + 32 * j < P.E) {
                    P.fold.counts[lane + 32 * j] = count[j];
                    P.fold.offsets[lane + 32 * j + 1] = first[j] + count[j];
                    if (P.fold.counts_out) P.fold.counts_out[lane + 32 * j] = count[j];
                }
            }
            if (blockIdx.x == 0 && lane == 0) P.fold.offsets[0] = 0;
        }
        // Segments and their row tiles.  As in umma_gemm_kernel, one that is negative, decreasing or ends beyond the rows counts as
        // empty and is reported: a corrupt array must not send a tile out of range.  Segments that overlap could still have more
        // row tiles than there are counters; then all count as empty.
        int tiles[2];
        bool bad = false;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int e = lane + 32 * j;
            int a = 0, b = 0;
            if (e < P.E) {
                a = FOLD ? first[j] : P.offsets[e];
                b = FOLD ? first[j] + count[j] : P.offsets[e + 1];
            }
            if (a < 0 || b < a || b > P.amax) {
                bad = true;
                a = b = 0;
            }
            tiles[j] = (int)(((long long)b - a + BM - 1) / BM);
            if (e < P.E) {
                sh.seg0[e] = a;
                sh.seg1[e] = b;
            }
        }
        long long sum = (long long)tiles[0] + tiles[1];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (sum > P.max_row_tiles) {
            bad = true;
            tiles[0] = tiles[1] = 0;
        }
        if (__any_sync(0xffffffffu, bad) && lane == 0) sh.bad_offsets = 1;
        int lo = tiles[0], hi = tiles[1];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int a = __shfl_up_sync(0xffffffffu, lo, o), b = __shfl_up_sync(0xffffffffu, hi, o);
            if (lane >= o) {
                lo += a;
                hi += b;
            }
        }
        const int half = __shfl_sync(0xffffffffu, lo, 31);
        if (lane == 0) sh.rt0[0] = 0;
        if (lane < P.E) sh.rt0[lane + 1] = lo;
        if (lane + 32 < P.E) sh.rt0[lane + 33] = half + hi;
        __syncwarp();
        if (lane == 0) {
            sh.row_tiles = sh.rt0[P.E];
            sh.up_tiles = sh.row_tiles * ceil_div(P.H, BN);
            sh.down_tiles = sh.row_tiles * ceil_div(P.d, BN);
        }
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem_base = sh.tmem_base;
    const int htarget = 4 * ceil_div(P.H, BN);     // arrivals that complete a row tile of h
    int* const h_done = P.sync + kSyncH;
    GroupedTile t{};

    TileReader tiles;
    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer
        int s = 0;
        uint32_t phb = 0;            // a phase bit per ring slot
        bool alive = true, h_complete = sh.up_tiles == 0;
#ifdef DSMOE_TRACE
        long long gt_h = 0;
#endif
        const auto next_slot = [&]() {
            phb ^= 1u << s;
            if (++s == STAGES) s = 0;
        };
        const auto load_b = [&](const BMaps* maps, int kb, int N) {
            const uint32_t bar = ptx::smem_u32(&sh.full[s]), dst = smB + s * B_STAGE_BYTES;
            if (t.bn == BN) ptx::tma_load_3d(dst, &maps->m[4], bar, 0, wrow(kb, t.n0, N), t.e);
            else load_weight_rows(maps, dst, bar, wrow(kb, t.n0, N), t.bn, t.e);
        };
        const auto want_next = [&]() { ptx::mbar_arrive(ptx::smem_u32(&sh.want)); };
        while (alive && tiles.next(sh, lane, t)) {
            const int claim_at = max(t.nk - kClaimAhead, 0);
            const bool elected = ptx::elect_one();
            if (elected && t.up) {
                for (int i = 0; i < t.nk; ++i) {
                    if (i == claim_at) want_next();
                    if (!ptx::mbar_wait(ptx::smem_u32(&sh.empty[s]), ((phb >> s) & 1u) ^ 1u, &sh.abort_flag)) {
                        alive = false;
                        break;
                    }
                    ptx::mbar_expect_tx(ptx::smem_u32(&sh.full[s]), (uint32_t)t.bn * BK * 2);
                    load_b(&tmW1, i, P.H);
                    next_slot();
                }
            } else if (elected) {
                // the weights do not wait for h: while its rows are being finished elsewhere, a ring of them is on its way
                int ahead = 0, s0 = s;
                if (!h_complete) {
                    for (; ahead < min(t.nk, STAGES); ++ahead) {
                        if (!ptx::mbar_wait(ptx::smem_u32(&sh.empty[s]), ((phb >> s) & 1u) ^ 1u, &sh.abort_flag)) {
                            alive = false;
                            break;
                        }
                        ptx::mbar_expect_tx(ptx::smem_u32(&sh.full[s]), A_STAGE_BYTES + (uint32_t)t.bn * BK * 2);
                        load_b(&tmW2, ahead, P.d);
                        next_slot();
                    }
                    GT_T0(t_h);
                    alive = alive && counter_wait(h_done + t.rt, htarget, &sh.abort_flag);
                    GT_ADD(gt_h, t_h);
                    h_complete = counter_acquire(P.sync) >= sh.row_tiles;
                    asm volatile("fence.proxy.async;" ::: "memory");   // h was written through the generic proxy, TMA reads it
                    for (int i = 0; alive && i < ahead; ++i) {
                        const uint32_t bar = ptx::smem_u32(&sh.full[s0]);
                        ptx::tma_load_2d(smA + s0 * A_STAGE_BYTES, &tmH, bar, i * BK, t.row0);
                        ptx::mbar_arrive(bar);
                        ptx::mbar_arrive(bar);
                        if (++s0 == STAGES) s0 = 0;
                    }
                }
                if (alive && claim_at < ahead) want_next();
                for (int i = ahead; alive && i < t.nk; ++i) {
                    if (i == claim_at) want_next();
                    if (!ptx::mbar_wait(ptx::smem_u32(&sh.empty[s]), ((phb >> s) & 1u) ^ 1u, &sh.abort_flag)) {
                        alive = false;
                        break;
                    }
                    const uint32_t bar = ptx::smem_u32(&sh.full[s]);
                    ptx::mbar_expect_tx(bar, A_STAGE_BYTES + (uint32_t)t.bn * BK * 2);
                    ptx::tma_load_2d(smA + s * A_STAGE_BYTES, &tmH, bar, i * BK, t.row0);
                    load_b(&tmW2, i, P.d);
                    ptx::mbar_arrive(bar);
                    ptx::mbar_arrive(bar);
                    next_slot();
                }
            }
            alive = __all_sync(0xffffffffu, alive);
        }
        chain_next();
#ifdef DSMOE_TRACE
        if (gt_h) GT_PUT(7, gt_h);           // (the elected lane's)
#endif
        if (!alive) {
            // copies already issued still land in this CTA's shared memory: give them time
            const uint64_t t0 = ptx::globaltimer_ns();
            while (ptx::globaltimer_ns() - t0 < 200000ull) {
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        int s = 0, acc = 0;
        uint32_t phb = 0, aph = 0;
        bool alive = true;
#ifdef DSMOE_TRACE
        long long gt_up = 0, gt_down = 0, gt_acc = 0;
        bool gt_seen = false;
        if (lane == 0) GT_SET(0);
#endif
        while (alive && tiles.next(sh, lane, t)) {
#ifdef DSMOE_TRACE
            if (!t.up && !gt_seen && lane == 0) GT_SET(1);
            gt_seen = gt_seen || !t.up;
#endif
            if (ptx::elect_one()) {
                GT_T0(t_acc);
                alive = ptx::mbar_wait(ptx::smem_u32(&sh.tempty[acc]), aph ^ 1u, &sh.abort_flag);
                GT_ADD(gt_acc, t_acc);
                ptx::tc_fence_after();
                const uint32_t idesc = ptx::make_idesc_bf16(BM, (uint32_t)t.bn);
                const uint32_t d_tmem = tmem_base + (uint32_t)(acc * BN);
                for (int i = 0; alive && i < t.nk; ++i) {
                    GT_T0(t_w);
                    if (!ptx::mbar_wait(ptx::smem_u32(&sh.full[s]), (phb >> s) & 1u, &sh.abort_flag)) {
                        alive = false;
                        break;
                    }
#ifdef DSMOE_TRACE
                    if (t.up) GT_ADD(gt_up, t_w);
                    else GT_ADD(gt_down, t_w);
#endif
                    ptx::tc_fence_after();
                    const uint32_t a0 = smA + s * A_STAGE_BYTES, b0 = smB + s * B_STAGE_BYTES;
#pragma unroll
                    for (int kk = 0; kk < BK / 16; ++kk)
                        ptx::umma_bf16(d_tmem, ptx::make_desc_k_sw128(a0 + kk * 32), ptx::make_desc_k_sw128(b0 + kk * 32), idesc,
                                       (uint32_t)((i | kk) != 0));
                    ptx::umma_commit(ptx::smem_u32(&sh.empty[s]));     // slot reusable once these MMAs have read it
                    phb ^= 1u << s;
                    if (++s == STAGES) s = 0;
                }
                if (alive) ptx::umma_commit(ptx::smem_u32(&sh.tfull[acc]));       // accumulator complete
            }
            alive = __all_sync(0xffffffffu, alive);
            if (++acc == 2) {
                acc = 0;
                aph ^= 1u;
            }
        }
#ifdef DSMOE_TRACE
        if (lane == 0) {
            GT_SET(2);
        }
        if (gt_up | gt_down | gt_acc) {      // (the elected lane's)
            GT_PUT(4, gt_up);
            GT_PUT(5, gt_down);
            GT_PUT(6, gt_acc);
        }
#endif
    } else if (warp < 6) {
        // ------------------------------------------------------------ epilogue
        const int q = warp & 3;
        int acc = 0;
        uint32_t aph = 0;
        uint8_t* const st = stage + q * 32 * kStageRow;
        while (tiles.next(sh, lane, t)) {
            const int row = q * 32 + lane;
            const bool valid = row < t.rows_valid;
            const int nrows = min(32, max(0, t.rows_valid - q * 32));       // rows of this warp
            float g = 1.f;
            if (FOLD && !t.up) {
                int tok[1];
                const int first = t.row0 - sh.seg0[t.e];
                find_tokens<FOLD ? FOLD : 1>(bits, t.e, first + q * 32, first + t.rows_valid - 1, lane, tok);
                if (valid) {
                    g = P.fold.scores[(size_t)tok[0] * P.E + t.e];
                    if (t.n0 == 0) {     // once a row: where the aggregation finds it
                        const int slot = __popcll(P.fold.mask[tok[0]] & ((1ull << t.e) - 1ull));
                        // (a token of top-K whose scores are no numbers is selected by all experts)
                        if (slot < P.W) P.fold.token_rows[(size_t)tok[0] * P.W + slot] = t.row0 + row;
                    }
                }
            } else if (!t.up && valid) {
                g = P.row_gate[t.row0 + row];
            }
            // the TMEM reads below are warp-collective: the warp leaves as one
            if (__any_sync(0xffffffffu, !ptx::mbar_wait(ptx::smem_u32(&sh.tfull[acc]), aph, &sh.abort_flag))) break;
            ptx::tc_fence_after();
            const uint32_t taddr = tmem_base + (uint32_t)(acc * BN) + ((uint32_t)(q * 32) << 16);
            if (t.up) {
                // hidden activations: a lane's 64 bytes of one row go through a shared-memory tile, 4 lanes store a row's 64
                // bytes together, eight rows per instruction
                constexpr int LDB = kStageRow;
                const int rr = lane >> 2, cc = lane & 3;
                for (int c = 0; nrows > 0 && c < t.bn; c += 32) {
                    uint32_t r[32];
                    ptx::tmem_ld32(taddr + (uint32_t)c, r);
                    ptx::tmem_ld_wait();
                    uint4 pk[4];
                    __nv_bfloat162* hv = reinterpret_cast<__nv_bfloat162*>(pk);
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        hv[j] = __floats2bfloat162_rn(gelu_erf(__uint_as_float(r[2 * j])), gelu_erf(__uint_as_float(r[2 * j + 1])));
                    uint8_t* const tb = st;
#pragma unroll
                    for (int j = 0; j < 4; ++j) *reinterpret_cast<uint4*>(tb + lane * LDB + 16 * j) = pk[j];
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int rl = i * 8 + rr;
                        if (rl < nrows)
                            *reinterpret_cast<uint4*>(P.h + ((long long)t.row0 + q * 32 + rl) * P.H + t.n0 + c + cc * 8) =
                                *reinterpret_cast<const uint4*>(tb + rl * LDB + 16 * cc);
                    }
                    __syncwarp();
                }
                ptx::tc_fence_before();
                asm volatile("fence.proxy.async;" ::: "memory");     // TMA of other CTAs reads these rows
                __syncwarp();
                if (lane == 0) {
                    ptx::mbar_arrive(ptx::smem_u32(&sh.tempty[acc]));
                    int before;
                    asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], 1;" : "=r"(before) : "l"(h_done + t.rt) : "memory");
                    if (before == htarget - 1) counter_add(P.sync, 1);
                }
            } else {
                // fp32 rows, gate applied.  Out of TMEM a lane holds 32 columns of ONE row; turned through the tile, 8 lanes store one
                // row's 128 bytes together, four whole rows per instruction
                constexpr int LD = kStageRow / 4;       // floats per staged row: 16-byte aligned, conflict-free in quarter warps
                float* const tp = reinterpret_cast<float*>(st);
                const int rr = lane >> 3, cc = lane & 7;
                for (int c = 0; nrows > 0 && c < t.bn; c += 32) {
                    uint32_t r[32];
                    ptx::tmem_ld32(taddr + (uint32_t)c, r);
                    ptx::tmem_ld_wait();
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        *reinterpret_cast<float4*>(tp + lane * LD + 4 * j) =
                            make_float4(g * __uint_as_float(r[4 * j]), g * __uint_as_float(r[4 * j + 1]),
                                        g * __uint_as_float(r[4 * j + 2]), g * __uint_as_float(r[4 * j + 3]));
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int rl = i * 4 + rr;      // row of this warp's 32
                        if (rl < nrows)
                            *reinterpret_cast<float4*>(P.rows + ((long long)t.row0 + q * 32 + rl) * P.d + t.n0 + c + cc * 4) =
                                *reinterpret_cast<const float4*>(tp + rl * LD + cc * 4);
                    }
                    __syncwarp();
                }
                ptx::tc_fence_before();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&sh.tempty[acc]));
            }
            if (++acc == 2) {
                acc = 0;
                aph ^= 1u;
            }
        }
        if (warp == 2 && lane == 0) GT_SET(3);
    } else if (warp < 6 + GATHER_WARPS) {
        // ------------------------------------------------------------ gather: the up tiles' rows of x
        // Warps j and j + 4 bring the two halves of the A tiles of the ring stages j, j + 4, ... of this CTA's sequence.  An
        // instruction covers 4 rows x 128 bytes (8 lanes x 16 bytes per row), written in the 128-byte-swizzle order
        // the MMA descriptors expect (chunk c of row r sits at chunk c ^ (r % 8)).  The warp then waits for its copies,
        // makes them visible to the tensor core's proxy and arrives at the stage's barrier; while it waits, the other
        // warps' stages are in flight.
        const int w8 = warp - 6;
        bool alive = true;
        {
            constexpr int ROWS = BM / 2;
            const int team = w8 % STAGES, part = w8 / STAGES;
            int* const rowtok = sh.rowtok + w8 * ROWS;
            const int lr = lane >> 3, lc = lane & 7;
            int n = 0;                       // stages of the sequence seen so far
            while (alive && tiles.next(sh, lane, t)) {
                if (!t.up) continue;
                // rows past the segment, which nobody reads: its last one again (all tiles' the same token: up to 1.4 times as long)
                int tok[ROWS / 32];
                if (FOLD) {
                    const int first = t.row0 - sh.seg0[t.e];
                    find_tokens<FOLD ? FOLD : 1>(bits, t.e, first + part * ROWS, first + t.rows_valid - 1, lane, tok);
                } else {
#pragma unroll
                    for (int j = 0; j < ROWS / 32; ++j) tok[j] = P.row_token[t.row0 + min(part * ROWS + lane + 32 * j, t.rows_valid - 1)];
                }
#pragma unroll
                for (int j = 0; j < ROWS / 32; ++j) rowtok[lane + 32 * j] = min(max(tok[j], 0), P.T - 1);
                __syncwarp();
                // this lane's rows (4 jj + lane / 8 of the warp's share): where they start in x, in 16-byte units
                uint32_t src_off[ROWS / 4];
#pragma unroll
                for (int jj = 0; jj < ROWS / 4; ++jj)
                    src_off[jj] = (uint32_t)(((size_t)rowtok[jj * 4 + lr] * P.d * 2) >> 4);
                for (int i = 0; i < t.nk; ++i, ++n) {
                    if (n % STAGES != team) continue;
                    const uint32_t ph = (uint32_t)(n / STAGES) & 1u;
                    if (!ptx::mbar_wait(ptx::smem_u32(&sh.empty[team]), ph ^ 1u, &sh.abort_flag)) {
                        alive = false;
                        break;
                    }
                    const uint32_t dst0 = smA + team * A_STAGE_BYTES;
                    const char* src0 = reinterpret_cast<const char*>(P.x) + (size_t)i * (BK * 2) + lc * 16;
#pragma unroll
                    for (int jj = 0; jj < ROWS / 4; ++jj) {
                        const int r = part * ROWS + jj * 4 + lr;
                        ptx::cp_async16(dst0 + (uint32_t)r * (BK * 2) + (uint32_t)((lc ^ (r & 7)) << 4), src0 + ((size_t)src_off[jj] << 4));
                    }
                    ptx::cp_async_commit();
                    ptx::cp_async_wait<0>();
                    ptx::fence_proxy_async();
                    __syncwarp();              // every lane's rows are in place and fenced: one arrival for the warp
                    if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&sh.full[team]));
                }
            }
        }
    } else {
        // ------------------------------------------------------------ dealer
        first_is_mine = __shfl_sync(0xffffffffu, first_is_mine ? 1 : 0, 0) != 0;
        int held = -1;                 // a claimed down tile that waits until the first round of up tiles is taken
        bool swept = false;
        uint64_t t0 = 0;
        for (int k = 0;; ++k) {
            if (k > 0 && !__all_sync(0xffffffffu, ptx::mbar_wait(ptx::smem_u32(&sh.want), (uint32_t)(k - 1) & 1u, &sh.abort_flag))) break;
            int id = held;
            if (held < 0) {
                id = (int)blockIdx.x;
                if (k > 0 || !first_is_mine) id = (int)gridDim.x + __shfl_sync(0xffffffffu, lane == 0 ? atomicAdd(P.sync + kSyncNext, 1) : 0, 0);
            }
            held = -1;
            if (!swept && id >= sh.up_tiles) {
                const int left = left_over(P.sync, min((int)gridDim.x, sh.up_tiles), lane, t0);
                if (left >= 0) {
                    held = id;
                    id = left;
                } else {
                    swept = true;
                }
            }
            const int slot = k % kTileSlots;
            t = tile_at(P, sh, id, lane);
            if (!__all_sync(0xffffffffu, ptx::mbar_wait(ptx::smem_u32(&sh.tile_empty[slot]), ((uint32_t)(k / kTileSlots) & 1u) ^ 1u,
                                                        &sh.abort_flag)))
                break;
            if (lane == 0) {
                sh.tile[slot] = t;
                ptx::mbar_arrive(ptx::smem_u32(&sh.tile_full[slot]));
            }
            if (t.e < 0) break;
        }
    }

    // ---------------------------------------------------------------- teardown
    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem_base, TMEM_COLS);
    }
    if (threadIdx.x == 0) {
        if (sh.abort_flag) report_status(P.dev_status, DSMOE_ERR_TIMEOUT);
        else if (sh.bad_offsets) report_status(P.dev_status, DSMOE_ERR_INVALID_ARG);
    }
}

}  // namespace

#ifdef DSMOE_TRACE
extern "C" __attribute__((visibility("default"))) int dsmoe_grouped_trace_read(long long* out) {
    return (int)cudaMemcpyFromSymbol(out, g_grouped_trace, sizeof(long long) * 192 * 8);
}
#endif

// (no more than E of the experts' last row tiles are incomplete)
static size_t max_row_tiles(const dsmoe_layer_desc& p) { return amax_of(p) / BM + p.E; }

// Counters of the grouped layer's launch: behind the hidden activations [Amax, H] if the workspace has room there (it keeps [T, E*H] for
// other paths), else none
GroupedScratch grouped_scratch(const dsmoe_layer_desc& p, const WsLayout& L) {
    GroupedScratch S{};
    S.sync = L.bwd;
    S.sync_ints = kSyncH + max_row_tiles(p);
    S.fits = umma_supported(p) && S.sync + S.sync_ints * 4 <= L.total_packed;
    return S;
}

dsmoe_status launch_grouped_layer(const dsmoe_layer_desc& p, const void* x, const void* packed, const int32_t* offsets,
                                  const int32_t* row_token, const float* row_gate, const GroupedFold* fold, float* rows, char* ws,
                                  const WsLayout& L, int32_t* dev_status, cudaStream_t s) {
    DeviceState* st = nullptr;
    DSMOE_TRY(device_state(&st));
    if (!st->attr_grouped) {
        DSMOE_CUDA_TRY(cudaFuncSetAttribute(grouped_layer_kernel<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGroupedSmem));
        for (auto* k : {grouped_layer_kernel<1>, grouped_layer_kernel<2>})
            DSMOE_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kGroupedSmem + kFoldBytes)));
        st->attr_grouped = true;
    }
    const size_t amax = amax_of(p);
    const __nv_bfloat16* w1t = static_cast<const __nv_bfloat16*>(packed);
    const __nv_bfloat16* w2t = w1t + (size_t)p.E * p.H * p.d;
    CUtensorMap mH;
    BMaps mW1, mW2;
    DSMOE_TRY(cached_bmaps(&mW1, w1t, p.E, p.H, p.d));
    DSMOE_TRY(cached_map_2d(&mH, ws + L.h, amax, p.H, BM));
    DSMOE_TRY(cached_bmaps(&mW2, w2t, p.E, p.d, p.H));
    GroupedParams P{};
    P.E = p.E; P.d = p.d; P.H = p.H; P.T = p.T; P.W = width_of(p);
    if (fold) P.fold = *fold;
    P.amax = (long long)amax;
    P.offsets = offsets; P.row_token = row_token; P.row_gate = row_gate;
    P.x = static_cast<const __nv_bfloat16*>(x);
    P.h = reinterpret_cast<__nv_bfloat16*>(ws + L.h);
    P.rows = rows;
    P.sync = reinterpret_cast<int*>(ws + grouped_scratch(p, L).sync);
    P.max_row_tiles = (int)max_row_tiles(p);
    P.dev_status = dev_status;
    int timed = -1;
    DSMOE_TRY(timing_begin(s, &timed));
    // Chained to the router, whose CTAs leave SMs free (fold, unchained: 1.06 to 1.07 times as fast as with the row-index kernel; chained:
    // 1.08 to 1.13).  Not chained to the row-index kernel: its CTAs would be set up beside that kernel's blocks, which leave no room for one on their
    // SMs, and come in another order (8 shapes of 150 to 700 tokens, two boxes: 0.3 and 1 % slower on average than this,
    // 4 % faster to 2.3 % slower).
    const int grid = std::min(sm_count(), kGroupedMaxCtas);
    if (fold) {
        DSMOE_CUDA_TRY(launch_chained(p.T <= 1024 ? grouped_layer_kernel<1> : grouped_layer_kernel<2>, grid, kGroupedThreads, kGroupedSmem + kFoldBytes, s, mW1, mH, mW2, P));
    } else {
        grouped_layer_kernel<0><<<grid, kGroupedThreads, kGroupedSmem, s>>>(mW1, mH, mW2, P);
        DSMOE_CUDA_TRY(cudaGetLastError());
    }
    DSMOE_TRY(timing_end(s, timed));
    return DSMOE_OK;
}

}  // namespace dsmoe
