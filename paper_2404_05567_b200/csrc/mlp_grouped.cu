// The sparse expert MLPs (Eq. 1) in ONE persistent launch, for tokens grouped by expert:
//
//   up    h[r,:] = GeLU(x[row_token[r],:] . W1[e])                 tile = (expert, 128 rows, <= 256 hidden units)
//   down  rows[r,:] = row_gate[r] * (h[r,:] . W2[e])  in fp32      tile = (expert, 128 rows, <= 256 output columns)
//
//   warp 0       TMA producer          (one lane)
//   warp 1       MMA issuer            (one lane); owns the TMEM allocation
//   warps 2..5   epilogue              (warp w reads TMEM lanes 32*(w%4) .. +31)
//   warps 6..13  gather the up-projection's rows of x
//
// One list of tiles -- every up tile, then the down tiles -- is dealt out to one CTA per SM: no round of tiles is left
// incomplete at the end of the up-projection (448 tiles on 148 CTAs for 7001 tokens of 4096, 32 experts of 512, top-4: four rounds
// for the work of three) and no launch gap lies between the projections.  A down tile waits (on a counter) until its own 128 rows
// of h are complete, nothing else; its weights are on their way meanwhile.
// Against two launches of umma_gemm_kernel, layers of 32 experts (us): 300 tokens of 2048, 1024 wide, by threshold 91 -> 86;
// 1500 of 3072, 384 wide, by threshold 214 -> 180; 3333 of 3072, 384 wide, top-6 237 -> 205; 7001 of 4096, 512 wide, top-4 441 -> 422;
// 8192 of 6144, 768 wide, top-4 904 -> 882 (76 shapes of 150 to 8192 tokens: 1.06 times on average, 0.98 to 1.22).
// Bound by the operands' way out of L2 (up) and, with narrow experts, the fp32 rows' way to memory (down: 158 us of which 108
// without its stores, at the first shape).
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
    int E, d, H, T;
    long long amax;
    const int32_t* offsets;
    const int32_t* row_token;
    const float* row_gate;
    const __nv_bfloat16* x;
    __nv_bfloat16* h;              // [amax, H]
    float* rows;                   // [amax, d]
    int* sync;                     // zero at launch: [0] row tiles of h that are complete; from kSyncH on, per row tile, its finished epilogue warps
    int max_row_tiles;             // ... and so many of these there are
    int32_t* dev_status;
};
constexpr int kSyncH = 16;

struct GroupedTile {
    bool up;
    int e, row0, rows_valid, rt, n0, bn, nk;
};

struct GroupedShared {
    uint64_t full[STAGES], empty[STAGES], tfull[2], tempty[2];
    uint32_t tmem_base;
    volatile int abort_flag;
    int row_tiles, up_tiles, down_tiles;   // totals
    int mine, skip;                // up tiles of this CTA; rounds of down tiles that CTAs with one more up tile sit out
    int bad_offsets;
    int seg0[kMaxExperts], seg1[kMaxExperts];      // rows of each expert
    int rt0[kMaxExperts + 1];                      // its first row tile
    int rowtok[GATHER_WARPS * (BM / 2)];
};
constexpr size_t kGroupedShared = 4096;
static_assert(sizeof(GroupedShared) <= kGroupedShared, "barriers and tables");
constexpr size_t kGroupedSmem = 1024 + (size_t)RING_BYTES + kGroupedShared + 4 * 32 * kStageRow;
static_assert(kGroupedSmem <= 227 * 1024, "shared memory of one CTA");

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


// The k-th tile of this CTA; false: it has no more.  Experts ascend, then column ranges; the row tiles of one weight tile follow
// one another.
__device__ __forceinline__ bool tile_at(const GroupedParams& P, const GroupedShared& sh, int k, GroupedTile& t) {
    const int G = gridDim.x;
    t.up = k < sh.mine;
    int id;
    if (t.up) {
        id = (int)blockIdx.x + k * G;
    } else {
        // Down tiles go round by round, starting with the CTAs that had one up tile less; those with one more sit out as many
        // rounds as their tile takes.
        const int extra = sh.up_tiles % G, fewer = G - extra;
        int r = k - sh.mine, idx = (int)blockIdx.x - extra;
        if (idx < 0) idx += G;
        if (idx < fewer) id = r < sh.skip ? r * fewer + idx : sh.skip * fewer + (r - sh.skip) * G + idx;
        else id = sh.skip * fewer + r * G + idx;
        if (id >= sh.down_tiles) return false;
    }
    const int N = t.up ? P.H : P.d, ntn = ceil_div(N, BN);
    int e = 0;
#pragma unroll
    for (int step = kMaxExperts / 2; step > 0; step >>= 1)
        if (e + step < P.E && id >= sh.rt0[e + step] * ntn) e += step;
    const int local = id - sh.rt0[e] * ntn, mtiles = sh.rt0[e + 1] - sh.rt0[e];
    const int nt = local / mtiles, mt = local - nt * mtiles;
    t.e = e;
    t.rt = sh.rt0[e] + mt;
    t.row0 = sh.seg0[e] + mt * BM;
    t.rows_valid = min(BM, sh.seg1[e] - t.row0);
    t.n0 = nt * BN;
    return true;
}

// Every role walks this CTA's list of tiles.  Finding a tile takes a bisection and two divisions, some hundred cycles, which in
// series with a tile of 8 reduction blocks (4096 cycles of the tensor core) cost the MMA issuer a third of its time; so a
// role's warp finds 32 tiles at once, one per lane, and hands them out by shuffles.
struct TileList {
    GroupedTile own;
    bool there;
    // the k-th tile (the whole warp asks); false: no more
    __device__ __forceinline__ bool get(const GroupedParams& P, const GroupedShared& sh, int k, int lane, GroupedTile& t) {
        const bool up = k < sh.mine;
        const int j = (up ? k : k - sh.mine) & 31;
        if (j == 0) there = (!up || k + lane < sh.mine) && tile_at(P, sh, k + lane, own);
        const unsigned all = 0xffffffffu;
        if (!__shfl_sync(all, there ? 1 : 0, j)) return false;
        t.up = up;
        t.e = __shfl_sync(all, own.e, j);
        t.row0 = __shfl_sync(all, own.row0, j);
        t.rows_valid = __shfl_sync(all, own.rows_valid, j);
        t.rt = __shfl_sync(all, own.rt, j);
        t.n0 = __shfl_sync(all, own.n0, j);
        t.bn = min(BN, (t.up ? P.H : P.d) - t.n0);
        t.nk = (t.up ? P.d : P.H) / BK;
        return true;
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

__global__ void __launch_bounds__(GATHER_THREADS, 1)
grouped_layer_kernel(const __grid_constant__ BMaps tmW1, const __grid_constant__ CUtensorMap tmH,
                     const __grid_constant__ BMaps tmW2, const GroupedParams P) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = ptx::smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;             // 128-byte swizzle wants 1024-byte aligned tiles
    const uint32_t smA = base, smB = base + STAGES * A_STAGE_BYTES;
    GroupedShared& sh = *reinterpret_cast<GroupedShared*>(smem_raw + (base - raw) + RING_BYTES);
    uint8_t* const stage = smem_raw + (base - raw) + RING_BYTES + kGroupedShared;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int G = gridDim.x;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            ptx::mbar_init(ptx::smem_u32(&sh.full[s]), 3);      // the producer and two gathering warps (down: the producer thrice)
            ptx::mbar_init(ptx::smem_u32(&sh.empty[s]), 1);
        }
        for (int a = 0; a < 2; ++a) {
            ptx::mbar_init(ptx::smem_u32(&sh.tfull[a]), 1);
            ptx::mbar_init(ptx::smem_u32(&sh.tempty[a]), 4);
        }
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
    chain_wait();
    if (warp == 0) {
        __syncwarp();
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
                a = P.offsets[e];
                b = P.offsets[e + 1];
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
            const int q = sh.up_tiles / G, extra = sh.up_tiles % G;
            sh.mine = q + ((int)blockIdx.x < extra ? 1 : 0);
            // (a down tile costs its reduction and the time of some 1.5 blocks; in a single round of up tiles nothing of h is there yet)
            sh.skip = q > 0 && extra > 0 ? (2 * (P.d / BK) + P.H / BK + 1) / (2 * (P.H / BK) + 3) : 0;
        }
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem_base = sh.tmem_base;
    const int htarget = 4 * ceil_div(P.H, BN);     // arrivals that complete a row tile of h
    int* const h_done = P.sync + kSyncH;
    GroupedTile t;

    TileList tiles;
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
        for (int k = 0;; ++k) {
            if (!alive || !tiles.get(P, sh, k, lane, t)) break;
            if (lane == 0 && t.up) {
                for (int i = 0; i < t.nk; ++i) {
                    if (!ptx::mbar_wait(ptx::smem_u32(&sh.empty[s]), ((phb >> s) & 1u) ^ 1u, &sh.abort_flag)) {
                        alive = false;
                        break;
                    }
                    ptx::mbar_expect_tx(ptx::smem_u32(&sh.full[s]), (uint32_t)t.bn * BK * 2);
                    load_b(&tmW1, i, P.H);
                    next_slot();
                }
            } else if (lane == 0) {
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
                for (int i = ahead; alive && i < t.nk; ++i) {
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
            alive = __shfl_sync(0xffffffffu, alive ? 1 : 0, 0) != 0;
        }
        chain_next();
        if (lane == 0) GT_PUT(7, gt_h);
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
        if (lane == 0) GT_SET(0);
#endif
        for (int k = 0;; ++k) {
#ifdef DSMOE_TRACE
            if (k == sh.mine && lane == 0) GT_SET(1);
#endif
            if (!alive || !tiles.get(P, sh, k, lane, t)) break;
            if (lane == 0) {
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
            alive = __shfl_sync(0xffffffffu, alive ? 1 : 0, 0) != 0;
            if (++acc == 2) {
                acc = 0;
                aph ^= 1u;
            }
        }
#ifdef DSMOE_TRACE
        if (lane == 0) {
            GT_SET(2);
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
        for (int k = 0; tiles.get(P, sh, k, lane, t); ++k) {
            const int row = q * 32 + lane;
            const bool valid = row < t.rows_valid;
            const int nrows = min(32, max(0, t.rows_valid - q * 32));       // rows of this warp
            const float g = !t.up && valid ? P.row_gate[t.row0 + row] : 1.f;
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
    } else {
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
            for (int k = 0; k < sh.mine && alive; ++k) {
                if (!tiles.get(P, sh, k, lane, t)) break;
#pragma unroll
                for (int j = 0; j < ROWS / 32; ++j) {
                    const int r = part * ROWS + lane + 32 * j;
                    const int tok = P.row_token[t.row0 + min(r, t.rows_valid - 1)];   // rows past the segment: nobody reads them
                    rowtok[lane + 32 * j] = min(max(tok, 0), P.T - 1);
                }
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
                                  const int32_t* row_token, const float* row_gate, float* rows, char* ws, const WsLayout& L,
                                  int32_t* dev_status, cudaStream_t s) {
    DeviceState* st = nullptr;
    DSMOE_TRY(device_state(&st));
    if (!st->attr_grouped) {
        DSMOE_CUDA_TRY(cudaFuncSetAttribute(grouped_layer_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGroupedSmem));
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
    P.E = p.E; P.d = p.d; P.H = p.H; P.T = p.T;
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
    // down tiles wait for other CTAs' up tiles: all of them must be resident
    void* args[] = {&mW1, &mH, &mW2, &P};
    DSMOE_CUDA_TRY(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(grouped_layer_kernel), dim3(sm_count()), dim3(GATHER_THREADS),
                                               args, kGroupedSmem, s));
    DSMOE_TRY(timing_end(s, timed));
    return DSMOE_OK;
}

}  // namespace dsmoe
