// The whole layer for a handful of tokens (one to a few users decoding) in one cooperative launch, with the weights as the
// multiplications' rows and the tokens as their 8 columns (mma.sync m16n8k16).
//
// With so few tokens tcgen05 is the wrong tool: an MMA of 128 rows takes some 110 cycles however few of its rows and columns are
// used, and a tile's 128 of them in series (d = 2048) took 9 of the 11 us that small_layer_kernel spent on either projection
// for one token, with the weights in L2 or not.  Here every weight is read once, 32 bytes a lane, straight into the registers that
// the warp-level MMA takes it from (the order of the reduction is free, so a lane's 16 neighbouring elements serve four
// steps); what bounds the kernel is the weights' stream and the way from one phase to the next.
//
//   router  the reduction over d of every token cut into slices, one CTA each                    -> grid barrier
//           every CTA adds every token's slices, takes softmax and selection itself (the same result everywhere)
//   up      hg[t, (e, j)] = [e in sel(t)] S[t,e] GeLU(x[t] . W1[e][:, j]) for the experts that some token selected: their hidden
//           units are cut into equal runs, one per CTA; its 16 warps share out the 64-wide blocks of d  -> grid barrier
//   down    out[t, :] = hg . W2: a CTA owns d / CTAs columns outright -- no partial sums in memory and no third barrier; its
//           warps share out the (expert, 64 hidden units) blocks
//
// A load covers 8 weight rows x 128 bytes; neighbouring rows of a packed block are neighbours in memory.  A register that has been
// used is loaded again at once, with its place in the next block: 8 KB are under way per warp, 128 KB per SM.
//
// Against small_layer_kernel (us a layer call of 32 experts, by threshold / top-4; in brackets the experts that the threshold selected):
// 1 token of 2048, 1024 wide 39.1 -> 26.1 (9) / 34.7 -> 16.8; 2 of 4096, 512 wide 51.3 -> 41.0 (20) / 47.1 -> 24.2; 4 of 3072, 384 wide
// 45.1 -> 40.7 (30) / 43.1 -> 27.9; 7 tokens 1.03 to 1.58 times as fast.  One token of 2048, 1024 wide with 13 selected experts (109 MB)
// takes 31 us: experts known at 4.9, the two streams 19 (5.7 TB/s), the barrier and reductions between them 3, and some 4 between two
// launches.
#include <algorithm>

#include "common.cuh"
#include "mlp_device.cuh"
#include "router_device.cuh"

namespace dsmoe {

namespace {

constexpr int kFewThreads = 512, kFewWarps = kFewThreads / 32;
constexpr int kFewMaxT = 7;                  // (the B operand has 8 columns; from 8 tokens on small_layer_kernel streams ahead of its router)
constexpr int kFewTiles = 4;                 // tiles of 16 rows x 64 weights that a warp has under way
constexpr int kFewChunk = 128;               // rows whose sums shared memory holds at a time
constexpr int kFewPad = 8;                   // elements between the tokens' rows in shared memory: no bank conflicts
constexpr int kFewPart = kFewWarps * kFewChunk * 8;      // the warps' partial sums of a chunk, floats
#ifdef DSMOE_TRACE
// Diagnostic build only: per CTA, globaltimer: [0] start, [1] slices written, [2] first barrier passed, [3] experts known, [4] up multiplied
// (first warp), [5] hg written, [6] second barrier passed, [7] end
__device__ unsigned long long g_few_trace[192][8];
#define FT_STAMP(i) do { if (threadIdx.x == 0 && blockIdx.x < 192) g_few_trace[blockIdx.x][i] = ptx::globaltimer_ns(); } while (0)
#else
#define FT_STAMP(i)
#endif

struct FewParams {
    int T, d, H, E;
    const __nv_bfloat16* x;
    const float* Wr;
    const float* br;
    const __nv_bfloat16 *W1, *W2;            // packed
    SelParams sel;
    float* scores;
    uint64_t* mask;
    int32_t* k_t;
    int32_t* counts_out;                     // nullable
    __nv_bfloat16* hg;                       // [T, E*H]
    float* slices;                           // [T][slices][64]
    void* out;
    int out_f32;
    int* sync;                               // zero at launch: two barrier counters, [4] an abort flag
    int32_t* dev_status;
};

// One thread, after a __syncthreads: the CTA's writes are released
__device__ __forceinline__ void few_arrive(int* counter) {
    asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(counter) : "memory");
}
// One thread; bounded
__device__ __forceinline__ bool few_wait(int* sync, int idx, int target) {
    uint64_t t0 = 0;
    for (uint32_t spin = 1;; ++spin) {
        int v;
        asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(sync + idx) : "memory");
        if (v >= target) return true;
        if ((spin & 0x3f) == 0) {
            int ab;
            asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(ab) : "l"(sync + 4) : "memory");
            const uint64_t now = ptx::globaltimer_ns();
            if (t0 == 0) t0 = now;
            if (ab || now - t0 > ptx::kWaitLimitNs) {
                atomicExch(sync + 4, 1);
                return false;
            }
        }
    }
}

// 16 neighbouring weights of a row.  They are read once: no line of L1 for them
__device__ __forceinline__ void load_weights(uint32_t (&r)[8], const __nv_bfloat16* p) {
    asm volatile("ld.global.nc.L1::no_allocate.v8.u32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "l"(p));
}
// acc (16 rows x 8 tokens) += 64 elements of 16 weight rows times the tokens': lane (g, q) holds elements 16 q .. + 15 of rows g and
// g + 8 and of token g.  Step s takes the lane's elements 4 s .. + 3 as its four elements of the reduction, in all operands alike.
__device__ __forceinline__ void mma64(float (&acc)[4], const uint32_t (&lo)[8], const uint32_t (&hi)[8], const uint32_t (&x)[8]) {
#pragma unroll
    for (int s = 0; s < 4; ++s)
        asm volatile(
            "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
            : "+f"(acc[0]), "+f"(acc[1]), "+f"(acc[2]), "+f"(acc[3])
            : "r"(lo[2 * s]), "r"(hi[2 * s]), "r"(lo[2 * s + 1]), "r"(hi[2 * s + 1]), "r"(x[2 * s]), "r"(x[2 * s + 1]));
}

__global__ void __launch_bounds__(kFewThreads, 1) few_tokens_kernel(const FewParams P) {
    extern __shared__ __align__(16) float few_smem[];
    __shared__ int active_s[kMaxExperts];
    __shared__ uint64_t mask_s[kFewMaxT];
    __shared__ float score_s[kFewMaxT][kMaxExperts];
    __shared__ int alive_s;
    float* const part = few_smem;                              // [warps][rows of a chunk][8]
    __nv_bfloat16* const xs = reinterpret_cast<__nv_bfloat16*>(few_smem + kFewPart);      // [T][d + kFewPad]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int G = gridDim.x, E = P.E, T = P.T;
    const int g8 = lane >> 2, q16 = (lane & 3) * 16;           // this lane's row of eight (and token), and its 16 of 64 reduction elements
    const int ldx = P.d + kFewPad;

    FT_STAMP(0);
    // ---------------------------------------------------------------- router, slices
    int KS = 1;
    while (KS < 16 && KS * 2 * T <= G) KS *= 2;
    if ((int)blockIdx.x < T * KS) {
        const int t = blockIdx.x / KS, sl = blockIdx.x % KS;
        const int klen = (P.d + KS - 1) / KS, kbeg = sl * klen, kend = min(P.d, kbeg + klen);
        const __nv_bfloat16* const xr = P.x + (size_t)t * P.d;
        // a row of Wr is covered by `quads` neighbouring threads, four experts each
        const int quads = (E + 3) / 4, rpp = kFewThreads / quads, qd = tid % quads, r0 = tid / quads, e0 = qd * 4;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r0 < rpp) {
#pragma unroll 4
            for (int k = kbeg + r0; k < kend; k += rpp) {
                const float xv = __bfloat162float(xr[k]);
                const float* const w = P.Wr + (size_t)k * E + e0;
                if ((E & 3) == 0) {
                    const float4 w4 = *reinterpret_cast<const float4*>(w);
                    acc.x = fmaf(xv, w4.x, acc.x);
                    acc.y = fmaf(xv, w4.y, acc.y);
                    acc.z = fmaf(xv, w4.z, acc.z);
                    acc.w = fmaf(xv, w4.w, acc.w);
                } else {
                    acc.x = fmaf(xv, w[0], acc.x);
                    if (e0 + 1 < E) acc.y = fmaf(xv, w[1], acc.y);
                    if (e0 + 2 < E) acc.z = fmaf(xv, w[2], acc.z);
                    if (e0 + 3 < E) acc.w = fmaf(xv, w[3], acc.w);
                }
            }
        }
        // the threads' sums meet: inside a warp where its lanes hold whole rows, then through shared memory
        int rows = rpp, slot = r0;
        bool writes = r0 < rpp;
        if ((32 % quads) == 0) {
            for (int o = 16; o >= quads; o >>= 1) {
                acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o);
                acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
                acc.z += __shfl_xor_sync(0xffffffffu, acc.z, o);
                acc.w += __shfl_xor_sync(0xffffffffu, acc.w, o);
            }
            rows = kFewWarps;
            slot = warp;
            writes = lane < quads;
        }
        float4* const st = reinterpret_cast<float4*>(few_smem);          // [rows][quads]: at most kFewThreads of them
        if (writes) st[slot * quads + qd] = acc;
        __syncthreads();
        if (tid < E) {
            float v = 0.f;
            for (int r = 0; r < rows; ++r) v += few_smem[(r * quads + (tid >> 2)) * 4 + (tid & 3)];
            P.slices[((size_t)t * KS + sl) * kMaxExperts + tid] = v;
        }
        __syncthreads();
    }
    FT_STAMP(1);
    if (tid == 0) few_arrive(P.sync + 0);
    // ... meanwhile the tokens go to shared memory
    for (int t = 0; t < T; ++t)
        for (int i = tid; i < P.d / 8; i += kFewThreads)
            *reinterpret_cast<uint4*>(xs + t * ldx + i * 8) = reinterpret_cast<const uint4*>(P.x + (size_t)t * P.d)[i];
    if (tid == 0) alive_s = few_wait(P.sync, 0, G) ? 1 : 0;
    __syncthreads();
    FT_STAMP(2);
    // ---------------------------------------------------------------- softmax and selection
    if (warp < T && alive_s) {
        const bool v_lo = lane < E, v_hi = lane + 32 < E;
        float lo[16], hi[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const float* const p = P.slices + ((size_t)warp * KS + j) * kMaxExperts;
            lo[j] = j < KS && v_lo ? __ldcg(p + lane) : 0.f;
            hi[j] = j < KS && v_hi ? __ldcg(p + lane + 32) : 0.f;
        }
        float l_lo = P.br && v_lo ? P.br[lane] : 0.f, l_hi = P.br && v_hi ? P.br[lane + 32] : 0.f;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            l_lo += lo[j];
            l_hi += hi[j];
        }
        float s_lo, s_hi;
        softmax_warp(l_lo, l_hi, E, lane, s_lo, s_hi);
        const uint64_t m = select_warp(s_lo, s_hi, P.sel, lane);
        score_s[warp][lane] = s_lo;
        score_s[warp][lane + 32] = s_hi;
        if (lane == 0) mask_s[warp] = m;
        if ((int)blockIdx.x == warp) {
            if (v_lo) P.scores[(size_t)warp * E + lane] = s_lo;
            if (v_hi) P.scores[(size_t)warp * E + lane + 32] = s_hi;
            if (lane == 0) {
                P.mask[warp] = m;
                if (P.k_t) P.k_t[warp] = __popcll(m);
            }
        }
    }
    __syncthreads();
    if (!alive_s) {
        if (tid == 0) report_status(P.dev_status, DSMOE_ERR_TIMEOUT);
        return;
    }
    uint64_t any = 0;
    for (int t = 0; t < T; ++t) any |= mask_s[t];
    const int n_act = __popcll(any);
    if (tid < E) {
        if ((any >> tid) & 1ull) active_s[__popcll(any & ((1ull << tid) - 1ull))] = tid;
        if (blockIdx.x == 0 && P.counts_out) {
            int n = 0;
            for (int t = 0; t < T; ++t) n += (int)((mask_s[t] >> tid) & 1ull);
            P.counts_out[tid] = n;
        }
    }
    __syncthreads();
    FT_STAMP(3);

    // ---------------------------------------------------------------- up-projection
    // A warp takes its blocks of d for one 16-row tile after the other (the run's rows are dealt out evenly to its tiles, so that
    // every load brings about as much), kFewTiles (tile, block) items under way.
    uint32_t lo[kFewTiles][8], hi[kFewTiles][8];              // rows g8 and g8 + 8 of the items under way
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    {
        const long long total = (long long)n_act * P.H;
        const int r_begin = (int)(total * blockIdx.x / G), rows = (int)(total * (blockIdx.x + 1) / G) - r_begin;
        const int nkb = P.d / BK, mine = warp < nkb ? (nkb - warp + kFewWarps - 1) / kFewWarps : 0;
        // the run's rows lie in at most two experts (it is no longer than H, few_fits): row r of it is at base + r * 64 of block 0
        const int i0 = r_begin / P.H, bound = (i0 + 1) * P.H - r_begin;
        const int ea = n_act ? active_s[min(i0, n_act - 1)] : 0, eb = n_act ? active_s[min(i0 + 1, n_act - 1)] : 0;
        const int j0 = r_begin - i0 * P.H;                    // the first row's hidden unit
        const __nv_bfloat16* const base_a = P.W1 + ((long long)ea * nkb * P.H + j0) * BK + q16;
        const __nv_bfloat16* const base_b = P.W1 + ((long long)eb * nkb * P.H - bound) * BK + q16;
        for (int done = 0; done < rows; done += kFewChunk) {      // (one chunk but for very many selected experts)
            const int n = min(kFewChunk, rows - done), tiles = (n + 15) / 16, ts = (n + tiles - 1) / tiles;      // rows of a tile
            const auto load = [&](int tile, int i, int m) {
                if (tile >= tiles) return;                        // (uniform in the warp)
                const int at = done + tile * ts, last = min(at + ts, done + n) - 1;
                const int ra = min(at + g8, last), rb = min(at + g8 + 8, last);      // rows past the tile: nobody reads the sums
                const long long block = (long long)(warp + i * kFewWarps) * P.H;
                load_weights(lo[m], (ra < bound ? base_a : base_b) + (block + ra) * BK);
                load_weights(hi[m], (rb < bound ? base_a : base_b) + (block + rb) * BK);
            };
            if (mine > 0) {
                int lt = 0, li = 0, tile = 0, i = 0;              // the item to load next, the one to multiply next
                const auto step = [&](int& t, int& k) {
                    if (++k == mine) {
                        k = 0;
                        ++t;
                    }
                };
#pragma unroll
                for (int m = 0; m < kFewTiles; ++m) {
                    load(lt, li, m);
                    step(lt, li);
                }
                while (tile < tiles) {
#pragma unroll
                    for (int m = 0; m < kFewTiles; ++m) {
                        if (tile >= tiles) break;
                        uint32_t xv[8] = {};
                        if (g8 < T) {
                            const uint4* const src = reinterpret_cast<const uint4*>(xs + g8 * ldx + (warp + i * kFewWarps) * BK + q16);
                            *reinterpret_cast<uint4*>(xv) = src[0];
                            *reinterpret_cast<uint4*>(xv + 4) = src[1];
                        }
                        mma64(acc, lo[m], hi[m], xv);
                        load(lt, li, m);
                        step(lt, li);
                        if (i + 1 == mine) {
                            float* const to = part + ((warp * kFewChunk + tile * 16 + g8) * 8 + (lane & 3) * 2);
                            *reinterpret_cast<float2*>(to) = make_float2(acc[0], acc[1]);
                            *reinterpret_cast<float2*>(to + 64) = make_float2(acc[2], acc[3]);
                            acc[0] = acc[1] = acc[2] = acc[3] = 0.f;
                        }
                        step(tile, i);
                    }
                }
            }
            FT_STAMP(4);
            __syncthreads();
            const int parts = min(kFewWarps, nkb);
            const int slot = tid % kFewChunk, in_tile = slot & 15, r = done + (slot >> 4) * ts + in_tile;
            if ((slot >> 4) < tiles && in_tile < ts && r < done + n) {
                const int e = r < bound ? ea : eb, j = r < bound ? j0 + r : r - bound;
                for (int t = tid / kFewChunk; t < T; t += kFewThreads / kFewChunk) {
                    float v = 0.f;
#pragma unroll 16
                    for (int w = 0; w < parts; ++w) v += part[(w * kFewChunk + slot) * 8 + t];
                    const float g = ((mask_s[t] >> e) & 1ull) ? score_s[t][e] : 0.f;
                    P.hg[((long long)t * E + e) * P.H + j] = __float2bfloat16_rn(g == 0.f ? 0.f : g * gelu_erf(v));
                }
            }
            if (done + kFewChunk < rows) __syncthreads();          // the sums are read before the next chunk's come
        }
    }
    __syncthreads();                            // every thread's part of hg is written
    FT_STAMP(5);
    if (tid == 0) few_arrive(P.sync + 1);

    // ---------------------------------------------------------------- down-projection
    const int c_begin = (int)((long long)P.d * blockIdx.x / G), c_end = (int)((long long)P.d * (blockIdx.x + 1) / G);
    const int jb = P.H / BK, blocks = n_act * jb, mine = warp < blocks ? (blocks - warp + kFewWarps - 1) / kFewWarps : 0;
    const int cols = c_end - c_begin, passes = (cols + 15) / 16, cs = passes ? (cols + passes - 1) / passes : 0;     // columns of a pass
    // the warp's items: its blocks warp, warp + 16, ... for one pass after the other; their expert (its place in the list) and block of
    // hidden units without a division each
    const int first_a = warp / jb, first_k = warp - first_a * jb, da = kFewWarps / jb, dk = kFewWarps - da * jb;
    struct Item {
        int pass, i, a, k;
    };
    const auto next = [&](Item& it) {
        ++it.i;
        it.a += da;
        it.k += dk;
        if (it.k >= jb) {
            it.k -= jb;
            ++it.a;
        }
        if (it.i >= mine) it = Item{it.pass + 1, 0, first_a, first_k};
    };
    Item wi{0, 0, first_a, first_k};                           // the next item whose weights are asked for
    const auto load = [&](int m) {
        if (wi.pass >= passes) return;                         // (uniform in the warp)
        const __nv_bfloat16* const base = P.W2 + ((long long)active_s[wi.a] * jb + wi.k) * P.d * BK + q16;
        const int at = c_begin + wi.pass * cs, last = min(at + cs, c_end) - 1;
        load_weights(lo[m], base + (long long)min(at + g8, last) * BK);
        load_weights(hi[m], base + (long long)min(at + g8 + 8, last) * BK);
        next(wi);
    };
    // The first weights do not wait for the other CTAs.  (More of them asked into L2 meanwhile, 32 to 512 KB a CTA: 0.5 to 2.5 % slower,
    // the requests delay the other CTAs' last up-projection loads and with them the barrier.)
    if (mine > 0) {
#pragma unroll
        for (int m = 0; m < kFewTiles; ++m) load(m);
    }
    if (tid == 0) alive_s = few_wait(P.sync, 1, G) ? 1 : 0;
    __syncthreads();
    FT_STAMP(6);
    if (!alive_s) {
        if (tid == 0) report_status(P.dev_status, DSMOE_ERR_TIMEOUT);
        return;
    }
    if (mine > 0) {
        uint32_t hv[kFewTiles][8];                              // this lane's 16 hidden activations of token g8 in the items under way
        Item hn{0, 0, first_a, first_k};                        // the next item whose activations are asked for
        const auto load_h = [&](int m) {
            if (hn.pass >= passes) return;
            if (g8 < T) {
                const uint4* const src = reinterpret_cast<const uint4*>(P.hg + ((long long)g8 * E + active_s[hn.a]) * P.H + hn.k * BK + q16);
                *reinterpret_cast<uint4*>(hv[m]) = __ldcg(src);
                *reinterpret_cast<uint4*>(hv[m] + 4) = __ldcg(src + 1);
            }
            next(hn);
        };
#pragma unroll
        for (int m = 0; m < kFewTiles; ++m) {
#pragma unroll
            for (int q = 0; q < 8; ++q) hv[m][q] = 0u;
            load_h(m);
        }
        int pass = 0, i = 0;                                    // the item to multiply
        while (pass < passes) {
#pragma unroll
            for (int m = 0; m < kFewTiles; ++m) {
                if (pass >= passes) break;
                mma64(acc, lo[m], hi[m], hv[m]);
                load(m);
                load_h(m);
                if (++i == mine) {
                    float* const to = part + ((warp * kFewChunk + pass * 16 + g8) * 8 + (lane & 3) * 2);
                    *reinterpret_cast<float2*>(to) = make_float2(acc[0], acc[1]);
                    *reinterpret_cast<float2*>(to + 64) = make_float2(acc[2], acc[3]);
                    acc[0] = acc[1] = acc[2] = acc[3] = 0.f;
                    i = 0;
                    ++pass;
                }
            }
        }
    }
    __syncthreads();
    const int slot = tid % kFewChunk, col = c_begin + (slot >> 4) * cs + (slot & 15), parts = min(kFewWarps, blocks);
    if ((slot >> 4) < passes && (slot & 15) < cs && col < c_end) {
        for (int t = tid / kFewChunk; t < T; t += kFewThreads / kFewChunk) {
            float v = 0.f;
#pragma unroll 16
            for (int w = 0; w < parts; ++w) v += part[(w * kFewChunk + slot) * 8 + t];
            if (P.out_f32) static_cast<float*>(P.out)[(long long)t * P.d + col] = v;
            else static_cast<__nv_bfloat16*>(P.out)[(long long)t * P.d + col] = __float2bfloat16_rn(v);
        }
    }
    FT_STAMP(7);
}

size_t few_smem_bytes(const dsmoe_layer_desc& p) { return (size_t)kFewPart * 4 + (size_t)p.T * (p.d + kFewPad) * 2; }
constexpr size_t kFewMaxSmem = 200 * 1024;

}  // namespace

#ifdef DSMOE_TRACE
extern "C" __attribute__((visibility("default"))) int dsmoe_few_trace_read(unsigned long long* out) {
    return (int)cudaMemcpyFromSymbol(out, g_few_trace, sizeof(unsigned long long) * 192 * 8);
}
#endif

// What `ctas` CTAs can take: a run of hidden units touches no third expert, which takes a CTA for every expert that may be
// selected (H * n_act / ctas <= H); 64 KB of partial sums hold 128 columns of a CTA; the tokens fit beside them.
bool few_fits(const dsmoe_layer_desc& p, int ctas) {
    return p.T <= kFewMaxT && p.E <= ctas && ceil_div(p.d, ctas) <= kFewChunk && few_smem_bytes(p) <= kFewMaxSmem;
}

// (weights are read 32 bytes at a time)
bool few_supported(const dsmoe_layer_desc& p, const void* packed) {
    return small_supported(p) && ((uintptr_t)packed & 31u) == 0 && few_fits(p, std::min(sm_count(), kSmallMaxCtas));
}

dsmoe_status launch_layer_few(const dsmoe_layer_desc& p, const void* x, const float* Wr, const float* br, const void* packed,
                              float* scores, uint64_t* mask, int32_t* k_t, int32_t* counts_out, void* out, char* ws, const WsLayout& L,
                              int32_t* dev_status, cudaStream_t s) {
    DeviceState* st = nullptr;
    DSMOE_TRY(device_state(&st));
    if (!st->attr_few) {
        DSMOE_CUDA_TRY(cudaFuncSetAttribute(few_tokens_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFewMaxSmem));
        st->attr_few = true;
    }
    FewParams P{};
    P.T = p.T; P.d = p.d; P.H = p.H; P.E = p.E;
    P.x = static_cast<const __nv_bfloat16*>(x);
    P.Wr = Wr;
    P.br = br;
    P.W1 = static_cast<const __nv_bfloat16*>(packed);
    P.W2 = P.W1 + (size_t)p.E * p.H * p.d;
    P.sel = SelParams{p.E, p.mode, p.eps, p.eps_normalized, p.K, p.min_k, nullptr};
    P.scores = scores;
    P.mask = mask;
    P.k_t = k_t;
    P.counts_out = counts_out;
    P.hg = reinterpret_cast<__nv_bfloat16*>(ws + L.h);
    P.slices = reinterpret_cast<float*>(ws + L.partial);
    P.out = out;
    P.out_f32 = p.out_fp32 ? 1 : 0;
    P.sync = reinterpret_cast<int*>(ws + L.sync);
    P.dev_status = dev_status;
    DSMOE_CUDA_TRY(cudaMemsetAsync(P.sync, 0, 32, s));
    int timed = -1;
    DSMOE_TRY(timing_begin(s, &timed));
    void* args[] = {&P};
    DSMOE_CUDA_TRY(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(few_tokens_kernel), dim3(std::min(sm_count(), kSmallMaxCtas)),
                                               dim3(kFewThreads), args, few_smem_bytes(p), s));
    DSMOE_TRY(timing_end(s, timed));
    return DSMOE_OK;
}

}  // namespace dsmoe
