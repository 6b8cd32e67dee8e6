// The mixture-of-attention-heads layer for a few decoding tokens (Eq. 7-8), in three chained launches:
//
//   1. query projection of all experts' heads, q[t, (e, j)] = x[t] . Wq[e], with the router beside it      moa_decode_gemm_kernel<QUERY>
//   2. attention: every token's selected experts' queries against the keys and values of its sequence     moa_decode_attention_kernel
//   3. output projection with the gates, out[t] = sum over selected e of S[t,e] (o[t,e] . Wo[e])            moa_decode_gemm_kernel
//
// Few tokens of a top-K selection touch nearly every expert, so the projections read every expert's weights and need no grouping: the
// router runs beside the first of them instead of before it.  What bounds each launch is its stream out of memory (weights; keys
// and values; weights), so each starts its own before it waits for its predecessor: the keys and values and the output weights
// come from nothing that the call itself writes.
//
// 32 tokens against 2048 positions, d 4096, 8 experts of 4 heads of 128, top-5: 75.5 us in the seven launches of the grouped form, 44.9
// here (queries 7.3, with the router the longer of the two; attention from its first keys to its last 20 for 134 MB; output 6.4; the rest
// passes from one launch to the next).  1 to 64 tokens, 100 to 3000 positions, three models' shapes: 1.44 to 2.97 times as fast, 2.2 on average.
#include <algorithm>
#include <cstdlib>

#include "common.cuh"
#include "mlp_device.cuh"
#include "router_device.cuh"

namespace dsmoe {

namespace {

__device__ __forceinline__ void mma_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldsm_x4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm_x4_trans(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}
__device__ __forceinline__ float exp2_fast(float v) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

// ---------------------------------------------------------------- the two projections
//
// out[t, n] = sum over k of X[t, k] W[n, k] with the weights as the rows of m16n8k16 and the tokens (up to 64) as its columns.  A
// CTA, or a cluster of two or four where there are few rows, owns 32 weight rows and takes the reduction in blocks of 64.  Its eight
// warps work by themselves: a warp takes every eighth block, by TMA through a ring of its own that an elected lane fills.  (With one
// thread to fill one ring for all, some 12 copies a microsecond got under way: 4096 x 4096 weights for 32 tokens took 14.6 us, 5.3 so: the
// weights at 6.3 TB/s, the tensor pipe busy for 4.3 of it.)  The warps' and the CTAs' sums meet in shared memory, in that order.  The output
// projection's sums are multiplied by the token's gate, in fp32, whenever a warp passes from one expert to the next.
constexpr int kDgRows = 32, kDgWarps = 8, kDgThreads = 32 * kDgWarps;
constexpr int kDgMaxCluster = 4;
constexpr int kDgRing = 192 * 1024;
constexpr int kDgLd = kDgRows + 4;           // floats between two tokens' sums in shared memory: no bank conflicts
constexpr int kDgMaxT = 64, kDgMaxE = 16;
constexpr int kDgRouterTokens = 4;           // tokens that share a CTA's loads of the router's weights

template <int NT>        // 8 NT tokens
struct DgGeo {
    static constexpr int W_BYTES = kDgRows * 128, X_BYTES = NT * 8 * 128, STAGE = W_BYTES + X_BYTES;
    static constexpr int STAGES = kDgRing / (STAGE * kDgWarps);        // of a warp
    static constexpr int RING = STAGES * STAGE * kDgWarps, SMEM = RING + 1024;
    static_assert(kDgWarps * NT * 8 * kDgLd * 4 <= RING, "the sums take the ring's place");
};

struct DecodeGemmParams {
    int T, d, E, H;
    int routers;                  // CTAs in front of the others that are the router's (queries)
    int cluster;
    int rows_per_expert;          // weight rows of an expert: H (queries) or d (output)
    int blocks;                   // 64-wide reduction blocks: d / 64 (queries) or E * H / 64 (output)
    int k_blocks;                 // ... of one expert
    void* out;                    // q [T, E * H] bf16, or the layer output [T, d]
    int out_f32;
    // router (queries); the output projection reads scores and mask for the gates
    const __nv_bfloat16* x;
    const float* Wr;
    const float* br;
    SelParams sel;
    float* scores;
    uint64_t* mask;
    int32_t* k_t;
    int* zero;                    // counters of the attention step
    int n_zero;
    int32_t* counts_out;          // output: the experts' counts (nullable)
    int32_t* dev_status;
};

template <int NT>
struct DgShared {
    uint64_t full[kDgWarps][DgGeo<NT>::STAGES];
    volatile int abort_flag;
    alignas(16) float red[kDgRouterTokens][kDgThreads / 4][4];       // [token][slot][expert of a quad]
    alignas(8) float gate[kDgMaxE][NT * 8];      // (read in pairs) < 0: not selected
};

__device__ __forceinline__ float4 ld_cluster4(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}

// Softmax and selection of tokens t0 .. t0 + n - 1 (at most kDgRouterTokens) by the whole CTA: a row of Wr is covered by `quads`
// neighbouring threads, four experts each
template <int TT>
__device__ __forceinline__ void decode_router(const DecodeGemmParams& P, float (*red)[kDgThreads / 4][4], int t0, int n) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, E = P.E;
    const int quads = E <= 4 ? 1 : E <= 8 ? 2 : 4, qd = tid % quads, e0 = qd * 4, rows = kDgThreads / quads;
    const __nv_bfloat16* xr[TT];
#pragma unroll
    for (int u = 0; u < TT; ++u) xr[u] = P.x + (size_t)(t0 + min(u, n - 1)) * P.d;       // past the last token: it again, unused
    float4 acc[TT];
#pragma unroll
    for (int u = 0; u < TT; ++u) acc[u] = make_float4(0.f, 0.f, 0.f, 0.f);
    // a thread takes 8 neighbouring rows at a time, two such runs' loads under way (more of them unrolled cost more in instruction
    // fetches than they hide); experts past the last: it again, unused
    const auto walk = [&](auto load) {
#pragma unroll 1
        for (int k0 = tid / quads * 8; k0 < P.d; k0 += 2 * 8 * rows) {
            float4 w[16];
            uint4 xv[TT][2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int k = min(k0 + h * 8 * rows, P.d - 8);
#pragma unroll
                for (int i = 0; i < 8; ++i) w[8 * h + i] = load(P.Wr + (size_t)(k + i) * E);
#pragma unroll
                for (int u = 0; u < TT; ++u) xv[u][h] = *reinterpret_cast<const uint4*>(xr[u] + k);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (k0 + h * 8 * rows >= P.d) break;
#pragma unroll
                for (int u = 0; u < TT; ++u) {
                    const uint32_t two[4] = {xv[u][h].x, xv[u][h].y, xv[u][h].z, xv[u][h].w};
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const float v = __uint_as_float(i & 1 ? two[i / 2] & 0xffff0000u : two[i / 2] << 16);
                        acc[u].x = fmaf(v, w[8 * h + i].x, acc[u].x);
                        acc[u].y = fmaf(v, w[8 * h + i].y, acc[u].y);
                        acc[u].z = fmaf(v, w[8 * h + i].z, acc[u].z);
                        acc[u].w = fmaf(v, w[8 * h + i].w, acc[u].w);
                    }
                }
            }
        }
    };
    if ((E & 3) == 0) {
        const int at = min(e0, E - 4);
        walk([&](const float* r) { return *reinterpret_cast<const float4*>(r + at); });
    } else {
        walk([&](const float* r) {
            return make_float4(r[min(e0, E - 1)], r[min(e0 + 1, E - 1)], r[min(e0 + 2, E - 1)], r[min(e0 + 3, E - 1)]);
        });
    }
#pragma unroll
    for (int u = 0; u < TT; ++u) {
        for (int o = 16; o >= quads; o >>= 1) {
            acc[u].x += __shfl_xor_sync(0xffffffffu, acc[u].x, o);
            acc[u].y += __shfl_xor_sync(0xffffffffu, acc[u].y, o);
            acc[u].z += __shfl_xor_sync(0xffffffffu, acc[u].z, o);
            acc[u].w += __shfl_xor_sync(0xffffffffu, acc[u].w, o);
        }
        if (lane < quads) *reinterpret_cast<float4*>(red[u][warp * quads + qd]) = acc[u];
    }
    __syncthreads();
    if (warp < n) {
        float l = 0.f;
        if (lane < E) {
            l = P.br ? P.br[lane] : 0.f;
#pragma unroll
            for (int w = 0; w < kDgWarps; ++w) l += red[warp][w * quads + (lane >> 2)][lane & 3];
        }
        softmax_select_store(l, 0.f, t0 + warp, P.sel, lane, P.scores, P.mask, P.k_t);
    }
}

__device__ __forceinline__ void store_sums(const DecodeGemmParams& P, bool f32, size_t at, float4 v) {
    if (f32) *reinterpret_cast<float4*>(static_cast<float*>(P.out) + at) = v;
    else *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(P.out) + at) = make_uint2(pack2(v.x, v.y), pack2(v.z, v.w));
}

template <int NT, bool QUERY>
__global__ void __launch_bounds__(kDgThreads, 1)
moa_decode_gemm_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX, const DecodeGemmParams P) {
    using G = DgGeo<NT>;
    constexpr int S = G::STAGES;
    extern __shared__ uint8_t dg_smem[];
    __shared__ DgShared<NT> sh;
    const uint32_t raw = ptx::smem_u32(dg_smem), base = (raw + 1023u) & ~1023u;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (QUERY && (int)blockIdx.x < P.routers) {
        chain_wait();
        chain_next();
        if (blockIdx.x == 0)
            for (int i = tid; i < P.n_zero; i += kDgThreads) P.zero[i] = 0;
        const int t0 = P.T * (int)blockIdx.x / P.routers;
        const int tokens = P.T * ((int)blockIdx.x + 1) / P.routers - t0;
        if (tokens > 1) decode_router<kDgRouterTokens>(P, sh.red, t0, tokens);
        else if (tokens == 1) decode_router<1>(P, sh.red, t0, tokens);       // (a cluster's CTAs may be more than the tokens)
        return;
    }
    const int C = P.cluster, cta = (int)blockIdx.x - (QUERY ? P.routers : 0), rank = cta % C, group = cta / C;
    const int b0 = P.blocks * rank / C, n = P.blocks * (rank + 1) / C - b0;      // this CTA's reduction blocks
    if (lane == 0) {
        for (int s = 0; s < S; ++s) ptx::mbar_init(ptx::smem_u32(&sh.full[warp][s]), 1);
        if (warp == 0) {
            sh.abort_flag = 0;
            ptx::prefetch_tensormap(&tmW);
            ptx::prefetch_tensormap(&tmX);
        }
        ptx::fence_barrier_init();
    }
    __syncwarp();                                             // the lane that is elected below need not be this one
    const uint32_t ring = base + (uint32_t)(warp * S * G::STAGE);
    const int row0 = group * kDgRows;                         // the rows lie in one expert (queries)
    const int w_row = QUERY ? row0 % P.rows_per_expert : row0, w_e = QUERY ? row0 / P.rows_per_expert : 0;
    // (an elected lane) block i of the CTA into stage s of the warp
    const auto load_w = [&](int i, int s) {
        const uint32_t bar = ptx::smem_u32(&sh.full[warp][s]), dst = ring + (uint32_t)(s * G::STAGE);
        ptx::mbar_expect_tx(bar, G::STAGE);
        const int b = b0 + i, kb = QUERY ? b : b % P.k_blocks;
        ptx::tma_load_3d(dst, &tmW, bar, 0, kb * P.rows_per_expert + w_row, QUERY ? w_e : b / P.k_blocks);
    };
    const auto load_x = [&](int i, int s) {
        ptx::tma_load_2d(ring + (uint32_t)(s * G::STAGE + G::W_BYTES), &tmX, ptx::smem_u32(&sh.full[warp][s]), (b0 + i) * 64, 0);
    };
    // the output projection's first weights do not wait for the attention step: nothing that the call writes
    if (!QUERY && ptx::elect_one())
        for (int s = 0; s < S; ++s)
            if (warp + s * kDgWarps < n) load_w(warp + s * kDgWarps, s);
    chain_wait();
    chain_next();
    if (ptx::elect_one())
        for (int s = 0; s < S; ++s)
            if (warp + s * kDgWarps < n) {
                if (QUERY) load_w(warp + s * kDgWarps, s);
                load_x(warp + s * kDgWarps, s);
            }
    if (!QUERY) {
        for (int i = tid; i < P.E * NT * 8; i += kDgThreads) {
            const int e = i / (NT * 8), t = i % (NT * 8);
            sh.gate[e][t] = t < P.T && ((P.mask[t] >> e) & 1ull) ? P.scores[(size_t)t * P.E + e] : -1.f;
        }
        if (blockIdx.x == 0 && P.counts_out && tid < P.E) {
            int c = 0;
            for (int t = 0; t < P.T; ++t) c += (int)((P.mask[t] >> tid) & 1ull);
            P.counts_out[tid] = c;
        }
    }
    __syncthreads();                                          // gates, abort flag

    float acc[2][NT][4], sum[2][NT][4];
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int t = 0; t < NT; ++t)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[m][t][c] = sum[m][t][c] = 0.f;
    const int q2 = (lane & 3) * 2;
    const auto flush = [&](int e) {
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            const float2 g = *reinterpret_cast<const float2*>(&sh.gate[e][t * 8 + q2]);
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                sum[m][t][0] += g.x < 0.f ? 0.f : g.x * acc[m][t][0];
                sum[m][t][1] += g.y < 0.f ? 0.f : g.y * acc[m][t][1];
                sum[m][t][2] += g.x < 0.f ? 0.f : g.x * acc[m][t][2];
                sum[m][t][3] += g.y < 0.f ? 0.f : g.y * acc[m][t][3];
                acc[m][t][0] = acc[m][t][1] = acc[m][t][2] = acc[m][t][3] = 0.f;
            }
        }
    };
    {
        // fragment addresses inside a block (128-byte rows, 16-byte pieces swizzled by the row): rows 16 m .. of the weights,
        // tokens 16 p .. of X
        const uint32_t wrow0 = (uint32_t)(((lane & 7) + ((lane >> 3) & 1) * 8) * 128), wc = (uint32_t)(lane >> 4);
        const uint32_t xrow0 = (uint32_t)(G::W_BYTES + ((lane & 7) + (lane >> 4) * 8) * 128), xc = (uint32_t)((lane >> 3) & 1);
        const uint32_t swz = (uint32_t)(lane & 7);
        int e = QUERY ? 0 : (b0 + warp) / P.k_blocks, left = QUERY ? 0 : (e + 1) * P.k_blocks - (b0 + warp);      // blocks up to the next expert
        uint32_t s = 0, parity = 0;
        for (int i = warp; i < n; i += kDgWarps) {
            if (!QUERY) {
                while (left <= 0) {
                    flush(e);
                    ++e;
                    left += P.k_blocks;
                }
                left -= kDgWarps;
            }
            if (__any_sync(0xffffffffu, !ptx::mbar_wait(ptx::smem_u32(&sh.full[warp][s]), parity, &sh.abort_flag))) break;
            const uint32_t at = ring + s * G::STAGE;
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) {
                uint32_t a[2][4];
#pragma unroll
                for (int m = 0; m < 2; ++m) ldsm_x4(a[m], at + (uint32_t)(m * 16 * 128) + wrow0 + ((((uint32_t)(ks * 2) + wc) ^ swz) << 4));
#pragma unroll
                for (int p = 0; p < NT / 2; ++p) {
                    uint32_t b[4];
                    ldsm_x4(b, at + xrow0 + (uint32_t)(p * 16 * 128) + ((((uint32_t)(ks * 2) + xc) ^ swz) << 4));
#pragma unroll
                    for (int m = 0; m < 2; ++m) {
                        mma_16816(acc[m][2 * p], a[m], b[0], b[1]);
                        mma_16816(acc[m][2 * p + 1], a[m], b[2], b[3]);
                    }
                }
            }
            __syncwarp();
            if (i + S * kDgWarps < n && ptx::elect_one()) {
                load_w(i + S * kDgWarps, (int)s);
                load_x(i + S * kDgWarps, (int)s);
            }
            if (++s == S) {
                s = 0;
                parity ^= 1u;
            }
        }
        if (!QUERY && e < P.E) flush(e);
    }
    __syncthreads();                                        // every block of the rings has been read (or the CTA gave up)
    const bool gave_up = sh.abort_flag != 0;
    if (gave_up && tid == 0) {                              // copies under way still land in this CTA's memory
        const uint64_t t0 = ptx::globaltimer_ns();
        while (ptx::globaltimer_ns() - t0 < 200000ull) {
        }
    }
    float* const part = reinterpret_cast<float*>(dg_smem + (base - raw));       // [warps][8 NT][kDgLd]
    if (!gave_up) {
        float* const to = part + (size_t)warp * (NT * 8 * kDgLd) + (lane >> 2);
#pragma unroll
        for (int t = 0; t < NT; ++t)
#pragma unroll
            for (int c = 0; c < 8; ++c)                       // column (token) q2 + (c & 1), row 8 (c >> 1)
                to[(t * 8 + q2 + (c & 1)) * kDgLd + 8 * (c >> 1)] =
                    QUERY ? acc[c >> 2][t][c & 3] : sum[c >> 2][t][c & 3];
    }
    __syncthreads();
    // four neighbouring rows of a token at a time
    const int T = P.T, ld = QUERY ? P.E * P.H : P.d;
    for (int i = tid; i < T * (kDgRows / 4); i += kDgThreads) {
        const int t = i / (kDgRows / 4), r = i % (kDgRows / 4) * 4;
        float* const at = part + t * kDgLd + r;
        float4 v = *reinterpret_cast<const float4*>(at);
#pragma unroll
        for (int m = 1; m < kDgWarps; ++m) {
            const float4 w = *reinterpret_cast<const float4*>(at + (size_t)m * (NT * 8 * kDgLd));
            v.x += w.x;
            v.y += w.y;
            v.z += w.z;
            v.w += w.w;
        }
        if (C > 1) *reinterpret_cast<float4*>(at) = v;
        else if (!gave_up) store_sums(P, !QUERY && P.out_f32, (size_t)t * ld + (size_t)row0 + r, v);
    }
    if (C > 1) {
        ptx::cluster_sync();
        for (int i = tid; i < T * (kDgRows / 4); i += kDgThreads) {
            const int t = i / (kDgRows / 4), r = i % (kDgRows / 4) * 4;
            if (t % C != rank) continue;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int c = 0; c < C; ++c) {
                const float4 w = ld_cluster4(ptx::map_to_cta(ptx::smem_u32(part + t * kDgLd + r), (uint32_t)c));
                v.x += w.x;
                v.y += w.y;
                v.z += w.z;
                v.w += w.w;
            }
            if (!gave_up) store_sums(P, !QUERY && P.out_f32, (size_t)t * ld + (size_t)row0 + r, v);
        }
        ptx::cluster_sync();                                 // nobody leaves while another CTA may read its sums
    }
    if (gave_up && tid == 0) report_status(P.dev_status, DSMOE_ERR_TIMEOUT);
}

// ---------------------------------------------------------------- attention
//
// The (token, head) pairs' visible keys, in units of 16, are one list, cut into equal runs, one per CTA; the CTA's 8 warps take
// every eighth unit of its run, each through a ring of its own (cp.async, two units and more under way).  A pair's 16 rows are the queries of
// the token's selected experts.  The warps' (maximum, sum, accumulator) of a pair meet in shared memory; a pair that several CTAs
// share leaves one such triple per CTA in memory, and the CTA that comes last adds them up in order of the CTAs.  Bound by the keys' and
// values' way out of memory: 24 KB under way a warp; a unit's two chains of MMAs take a third of the time that its bytes do.
constexpr int kDaWarps = 8, kDaUnit = 16;
constexpr int kDaMaxPairs = 1024;

template <int DH>
struct DaGeo {
    static constexpr int STRIDE = DH * 2 + 16;                     // bytes per key row in shared memory: 16 of padding
    static constexpr int UNIT = 2 * kDaUnit * STRIDE;              // K and V; also holds a warp's 16 x (DH + 8) accumulators
    static constexpr int BUFS = DH == 128 ? 3 : DH == 96 ? 4 : 5;
    static constexpr int SMEM = kDaWarps * BUFS * UNIT;
    static_assert(16 * (DH + 8) * 4 <= UNIT, "accumulators take a unit's place");
};

// The expert of a token's r-th row (its selected experts ascend); -1: the token has fewer
__device__ __forceinline__ int expert_of(uint64_t selected, int r, int rows) {
    for (int i = 0; i < r; ++i) selected &= selected - 1;
    return r < rows ? __ffsll((long long)selected) - 1 : -1;
}

struct DecodeAttnParams {
    const __nv_bfloat16* q;      // [T, E * H]
    __nv_bfloat16* o;            // [T, E * H]: selected experts' parts alone
    int T, E, H, n_head, W;
    const __nv_bfloat16 *Kc, *Vc;
    const int32_t *tok_seq, *pos;
    int n_seq, L;
    float scale_log2;
    const uint64_t* mask;
    float* parts;                // [CTAs + pairs][W][DH + 2]
    int* done;                   // [pairs], zero
    int32_t* dev_status;
};

}  // namespace

// Aligned runs over pairs of `units` units each: where CTA c's begins.  split: `per` CTAs to a pair, else `per` pairs to a CTA.  The
// product stays an int's as long as decode_runs_align allows such runs (asking for that here, or a quotient without it, cost 0.4 of 44.5 us).
__host__ __device__ int decode_run_start(int c, int units, int per, int pairs, bool split) {
    return split ? c / per * units + units * (c % per) / per : (c * per < pairs ? c * per : pairs) * units;
}
// Whether pairs of `units` units each are to be cut so, the longest run being `longest` of `total` units (see the kernel).  From 134 million
// keys a pair on never: 255 CTAs times their units would leave an int.
__host__ __device__ bool decode_runs_align(int units, int longest, int total) { return units < 1 << 23 && longest <= total / 100 + 64; }

namespace {

template <int DH>
__global__ void __launch_bounds__(32 * kDaWarps, 1) moa_decode_attention_kernel(const DecodeAttnParams P) {
    using G = DaGeo<DH>;
    constexpr int STRIDE = G::STRIDE, KS = DH / 16, DT = DH / 8, CH = DH / 8, LDO = DH + 8, BUFS = G::BUFS;
    extern __shared__ __align__(16) unsigned char da_smem[];
    __shared__ int seq_s[kDgMaxT], last_s[kDgMaxT], units_s[kDgMaxT], base_s[kDgMaxT + 1];
    __shared__ float ms[kDaWarps][16], ls[kDaWarps][16];
    __shared__ uint32_t at_s[kDaWarps];                 // where each warp's accumulators of the pair are
    __shared__ int last_cta_s, alike_s;
    __shared__ __align__(16) unsigned char q_s[kDgMaxE * STRIDE];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, q4 = lane & 3;
    const int nh = P.n_head, T = P.T;
    if (tid < T) {
        // (before the wait, as the keys are: past an L1 that may hold an earlier step's positions)
        const int sq = P.tok_seq ? __ldcg(P.tok_seq + tid) : 0, last = __ldcg(P.pos + tid);
        if (blockIdx.x == 0 && (sq < 0 || sq >= P.n_seq || last < 0 || last >= P.L)) report_status(P.dev_status, DSMOE_ERR_INVALID_ARG);
        seq_s[tid] = min(max(sq, 0), P.n_seq - 1);
        last_s[tid] = min(max(last, 0), P.L - 1);
        units_s[tid] = last_s[tid] / kDaUnit + 1;
    }
    __syncthreads();
    if (warp == 0) {                                    // units before token t's
        const int a = lane < T ? units_s[lane] : 0, b = lane + 32 < T ? units_s[lane + 32] : 0;
        int ia = a, ib = b;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int ua = __shfl_up_sync(0xffffffffu, ia, o), ub = __shfl_up_sync(0xffffffffu, ib, o);
            if (lane >= o) {
                ia += ua;
                ib += ub;
            }
        }
        ib += __shfl_sync(0xffffffffu, ia, 31);
        if (lane < T) base_s[lane + 1] = ia * nh;
        if (lane + 32 < T) base_s[lane + 33] = ib * nh;
        const int one = __shfl_sync(0xffffffffu, a, 0);
        const bool alike = __all_sync(0xffffffffu, (lane >= T || a == one) && (lane + 32 >= T || b == one));
        if (lane == 0) {
            base_s[0] = 0;
            alike_s = alike;
        }
    }
    __syncthreads();
    // Runs: `per` CTAs to a pair, or `per` pairs to a CTA, where the tokens see equally many keys; else the whole list in equal pieces,
    // which keeps every SM busy but leaves most CTAs with parts of two pairs to merge, some 8 us more (64 units' time on one SM).  The
    // longest aligned run, at the 66 KB/us that an SM was seen to read, is set against that and the list at the whole GPU's 6500.  The
    // layer with equal pieces and aligned, 4 heads of 128: 20 tokens of 700 keys 36.5, 28.4 us, of 3000 keys 49.0, 45.7; 48 tokens of 3000 keys
    // 83.5, 79.7; 40 tokens of 3000 keys, heads of 96: 58.0, 63.0.
    // Every CTA's run holds a unit at least: who adds up a pair's parts counts on it.
    const int total = base_s[T], pairs = T * nh, units0 = units_s[0], grid = (int)gridDim.x;
    const bool split = pairs <= grid;
    const int per = split ? min(grid / pairs, units0) : (pairs + grid - 1) / grid;
    const int whole_ctas = split ? pairs * per : (pairs + per - 1) / per;
    const int longest = split ? (units0 + per - 1) / per : per * units0;
    const bool aligned = alike_s && decode_runs_align(units0, longest, total);
    const int n_cta = aligned ? whole_ctas : min(grid, total);
    if ((int)blockIdx.x >= n_cta) return;
    const int share = total / n_cta, extra = total - share * n_cta;
    const auto run_start = [&](int c) {
        return aligned ? decode_run_start(c, units0, per, pairs, split) : c * share + min(c, extra);
    };
    const int u0 = run_start(blockIdx.x), u1 = run_start(blockIdx.x + 1);

    // Where a unit lies: token, head, key block of it
    struct Cursor {
        int t, j, k;
    };
    const auto settle = [&](Cursor& c) {                // k past the pair's units: on to the pair that holds it
        while (c.t < T && c.k >= units_s[c.t]) {
            c.k -= units_s[c.t];
            if (++c.j == nh) {
                c.j = 0;
                ++c.t;
            }
        }
    };
    // the first unit's token: as many as end before it
    Cursor seg{__popc(__ballot_sync(0xffffffffu, lane < T && base_s[min(lane, T - 1) + 1] <= u0)) +
                   __popc(__ballot_sync(0xffffffffu, lane + 32 < T && base_s[min(lane + 32, T - 1) + 1] <= u0)), 0, 0};
    seg.k = u0 - base_s[seg.t];
    seg.j = seg.k / units_s[seg.t];
    seg.k -= seg.j * units_s[seg.t];
    Cursor ahead = seg;                                 // the next unit to fetch
    ahead.k += warp;
    settle(ahead);
    int u_ahead = u0 + warp;
    unsigned char* const ring = da_smem + (size_t)warp * BUFS * G::UNIT;
    const uint32_t ring0 = (uint32_t)__cvta_generic_to_shared(ring);
    const auto fetch = [&](int buf) {
        if (u_ahead < u1) {
            const int last = last_s[ahead.t], key0 = ahead.k * kDaUnit, nk = min(kDaUnit, last + 1 - key0);
            const size_t head = (size_t)(seq_s[ahead.t] * nh + ahead.j) * P.L * DH + (size_t)key0 * DH;
            const uint32_t kd = ring0 + (uint32_t)(buf * G::UNIT), vd = kd + (uint32_t)(kDaUnit * STRIDE);
#pragma unroll
            for (int i = 0; i < CH * kDaUnit / 32; ++i) {
                const int idx = lane + 32 * i, row = idx / CH, ch = idx % CH;
                const size_t src = head + (size_t)(row < nk ? row : 0) * DH + ch * 8;
                const uint32_t nbytes = row < nk ? 16u : 0u, dst = (uint32_t)(row * STRIDE + ch * 16);      // past the last key: zeros
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(kd + dst), "l"(P.Kc + src), "r"(nbytes) : "memory");
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(vd + dst), "l"(P.Vc + src), "r"(nbytes) : "memory");
            }
            ahead.k += kDaWarps;
            settle(ahead);
            u_ahead += kDaWarps;
        }
        ptx::cp_async_commit();
    };
    for (int b = 0; b < BUFS - 1; ++b) fetch(b);
    chain_wait();
    chain_next();

    const uint32_t kfrag = (uint32_t)(((lane >> 4) * 8 + (lane & 7)) * STRIDE + ((lane >> 3) & 1) * 16);
    const uint32_t vfrag = (uint32_t)((((lane >> 3) & 1) * 8 + (lane & 7)) * STRIDE + (lane >> 4) * 16);
    int buf = 0, mine = u0 + warp;                      // this warp's next unit
    uint4 next_q = make_uint4(0u, 0u, 0u, 0u);          // a thread's piece of the next pair's queries, and its selection
    uint64_t next_sel = 0;
    const auto ask_queries = [&](const Cursor& c) {
        next_sel = P.mask[c.t];
        if (tid < P.E * CH)
            next_q = *reinterpret_cast<const uint4*>(P.q + ((size_t)c.t * P.E + tid / CH) * P.H + c.j * DH + tid % CH * 8);
    };
    ask_queries(seg);
    for (int at = u0; at < u1;) {
        const int units = units_s[seg.t], end = min(u1, at + units - seg.k), t = seg.t, j = seg.j, first_k = seg.k;
        const uint64_t sel = next_sel;
        const int rows = min(__popcll(sel), P.W);        // (under top-K more are set where a token's scores are no numbers: a part has W rows)
        // the queries of all experts: the selection comes with them, not before
        if (tid < P.E * CH) *reinterpret_cast<uint4*>(q_s + (tid / CH) * STRIDE + tid % CH * 16) = next_q;
        __syncthreads();
        // rows: the token's selected experts, in order
        const int e0 = expert_of(sel, lane & 15, rows);
        const uint32_t qrow = (uint32_t)__cvta_generic_to_shared(q_s) + (uint32_t)(max(e0, 0) * STRIDE + (lane >> 4) * 16);
        uint32_t qf[KS][4];
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) ldsm_x4(qf[ks], qrow + (uint32_t)(ks * 32));
        float m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;
        float o[DT][4];
#pragma unroll
        for (int i = 0; i < DT; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
        for (; mine < end; mine += kDaWarps) {
            __syncwarp();                               // every lane is past its reads of the buffer that is filled again now
            fetch((buf + BUFS - 1) % BUFS);
            ptx::cp_async_wait<BUFS - 1>();
            __syncwarp();
            const uint32_t kb = ring0 + (uint32_t)(buf * G::UNIT) + kfrag, vb = ring0 + (uint32_t)(buf * G::UNIT + kDaUnit * STRIDE) + vfrag;
            float sc[2][4];
#pragma unroll
            for (int i = 0; i < 2; ++i) sc[i][0] = sc[i][1] = sc[i][2] = sc[i][3] = 0.f;
#pragma unroll
            for (int ks = 0; ks < KS; ++ks) {
                uint32_t b[4];
                ldsm_x4(b, kb + (uint32_t)(ks * 32));
                mma_16816(sc[0], qf[ks], b[0], b[1]);
                mma_16816(sc[1], qf[ks], b[2], b[3]);
            }
            // to base 2; keys past the token's position are hidden (in its last unit)
            const int key0 = (first_k + mine - at) * kDaUnit + q4 * 2, last = last_s[t];
            float b0 = -INFINITY, b1 = -INFINITY;
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const bool seen = key0 + i * 8 + c <= last;
                    sc[i][c] = seen ? sc[i][c] * P.scale_log2 : -INFINITY;
                    sc[i][2 + c] = seen ? sc[i][2 + c] * P.scale_log2 : -INFINITY;
                    b0 = fmaxf(b0, sc[i][c]);
                    b1 = fmaxf(b1, sc[i][2 + c]);
                }
            b0 = fmaxf(b0, __shfl_xor_sync(0xffffffffu, b0, 1));
            b1 = fmaxf(b1, __shfl_xor_sync(0xffffffffu, b1, 1));
            b0 = fmaxf(b0, __shfl_xor_sync(0xffffffffu, b0, 2));
            b1 = fmaxf(b1, __shfl_xor_sync(0xffffffffu, b1, 2));
            if (__any_sync(0xffffffffu, b0 > m0 || b1 > m1)) {
                const float n0 = fmaxf(m0, b0), n1 = fmaxf(m1, b1);
                const float c0 = n0 == -INFINITY ? 1.f : exp2_fast(m0 - n0), c1 = n1 == -INFINITY ? 1.f : exp2_fast(m1 - n1);
                m0 = n0;
                m1 = n1;
                l0 *= c0;
                l1 *= c1;
#pragma unroll
                for (int i = 0; i < DT; ++i) {
                    o[i][0] *= c0;
                    o[i][1] *= c0;
                    o[i][2] *= c1;
                    o[i][3] *= c1;
                }
            }
            const float z0 = m0 == -INFINITY ? 0.f : m0, z1 = m1 == -INFINITY ? 0.f : m1;
            uint32_t pf[4];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const float p0 = exp2_fast(sc[i][0] - z0), p1 = exp2_fast(sc[i][1] - z0);
                const float p2 = exp2_fast(sc[i][2] - z1), p3 = exp2_fast(sc[i][3] - z1);
                l0 += p0 + p1;
                l1 += p2 + p3;
                pf[2 * i] = pack2(p0, p1);
                pf[2 * i + 1] = pack2(p2, p3);
            }
#pragma unroll
            for (int dp = 0; dp < DT / 2; ++dp) {
                uint32_t v[4];
                ldsm_x4_trans(v, vb + (uint32_t)(dp * 32));
                mma_16816(o[2 * dp], pf, v[0], v[1]);
                mma_16816(o[2 * dp + 1], pf, v[2], v[3]);
            }
            buf = buf + 1 == BUFS ? 0 : buf + 1;
        }
        Cursor next = seg;
        next.k += end - at;
        settle(next);
        if (end < u1) ask_queries(next);
        // ---- the warps' parts of the pair, through the buffer that each has just finished (the next fetch would fill it)
        l0 += __shfl_xor_sync(0xffffffffu, l0, 1);
        l1 += __shfl_xor_sync(0xffffffffu, l1, 1);
        l0 += __shfl_xor_sync(0xffffffffu, l0, 2);
        l1 += __shfl_xor_sync(0xffffffffu, l1, 2);
        const uint32_t free_at = (uint32_t)((warp * BUFS + (buf + BUFS - 1) % BUFS) * G::UNIT);
        __syncwarp();
        if (q4 == 0) {
            ms[warp][g] = m0;
            ms[warp][g + 8] = m1;
            ls[warp][g] = l0;
            ls[warp][g + 8] = l1;
            if (g == 0) at_s[warp] = free_at;
        }
        float* const acc = reinterpret_cast<float*>(da_smem + free_at);
#pragma unroll
        for (int dt = 0; dt < DT; ++dt) {
            *reinterpret_cast<float2*>(acc + g * LDO + dt * 8 + q4 * 2) = make_float2(o[dt][0], o[dt][1]);
            if (rows > 8) *reinterpret_cast<float2*>(acc + (g + 8) * LDO + dt * 8 + q4 * 2) = make_float2(o[dt][2], o[dt][3]);
        }
        __syncthreads();
        const bool whole = end - at == units;
        const int pair = t * nh + j;
        float* const slot = P.parts + (size_t)(blockIdx.x + pair) * P.W * (DH + 2);
        for (int idx = tid; idx < rows * (DH / 2); idx += 32 * kDaWarps) {
            const int row = idx / (DH / 2), col = idx % (DH / 2) * 2;
            float M = -INFINITY;
#pragma unroll
            for (int w = 0; w < kDaWarps; ++w) M = fmaxf(M, ms[w][row]);
            float nx = 0.f, ny = 0.f, den = 0.f;
#pragma unroll
            for (int w = 0; w < kDaWarps; ++w) {
                const float wgt = exp2_fast(ms[w][row] - M);              // 0 for a warp that saw no key
                const float2 v = *reinterpret_cast<const float2*>(reinterpret_cast<const float*>(da_smem + at_s[w]) + row * LDO + col);
                nx = fmaf(wgt, v.x, nx);
                ny = fmaf(wgt, v.y, ny);
                den = fmaf(wgt, ls[w][row], den);
            }
            if (whole) {
                const int e = expert_of(sel, row, rows);
                *reinterpret_cast<uint32_t*>(P.o + ((size_t)t * P.E + e) * P.H + j * DH + col) = pack2(nx / den, ny / den);
            } else {
                *reinterpret_cast<float2*>(slot + row * DH + col) = make_float2(nx, ny);
                if (col == 0) {
                    slot[P.W * DH + row * 2] = M;
                    slot[P.W * DH + row * 2 + 1] = den;
                }
            }
        }
        if (!whole) {
            // the CTA that comes last adds up the CTAs' parts, in their order
            __threadfence();
            __syncthreads();
            if (tid == 0) last_cta_s = atomicAdd(P.done + pair, end - at) + (end - at) == units;
            __syncthreads();
            if (last_cta_s && rows > 0) {
                __threadfence();
                // its first and last CTA
                const int p0 = base_s[t] + j * units, p1 = p0 + units - 1, cut = extra * (share + 1);
                const auto cta_of = [&](int u) { return u < cut ? u / (share + 1) : extra + (u - cut) / share; };
                const int c0 = aligned ? pair * per : cta_of(p0), c1 = aligned ? c0 + per - 1 : cta_of(p1);
                const size_t step = (size_t)P.W * (DH + 2);
                const float* const from = P.parts + (size_t)(c0 + pair) * step;
                const int nc = c1 - c0 + 1;
                for (int idx = tid; idx < rows * (DH / 2); idx += 32 * kDaWarps) {
                    const int row = idx / (DH / 2), col = idx % (DH / 2) * 2;
                    float M = -INFINITY;
#pragma unroll 4
                    for (int c = 0; c < nc; ++c) M = fmaxf(M, __ldcg(from + c * step + P.W * DH + row * 2));
                    float nx = 0.f, ny = 0.f, den = 0.f;
#pragma unroll 4
                    for (int c = 0; c < nc; ++c) {
                        const float2 ml = __ldcg(reinterpret_cast<const float2*>(from + c * step + P.W * DH + row * 2));
                        const float2 v = __ldcg(reinterpret_cast<const float2*>(from + c * step + row * DH + col));
                        const float wgt = exp2_fast(ml.x - M);
                        nx = fmaf(wgt, v.x, nx);
                        ny = fmaf(wgt, v.y, ny);
                        den = fmaf(wgt, ml.y, den);
                    }
                    const int e = expert_of(sel, row, rows);
                    *reinterpret_cast<uint32_t*>(P.o + ((size_t)t * P.E + e) * P.H + j * DH + col) = pack2(nx / den, ny / den);
                }
            }
        } else {
            __syncthreads();                            // the warps' parts are read before the next fetch overwrites them
        }
        seg = next;
        at = end;
    }
}

template <int NT, bool QUERY>
dsmoe_status launch_decode_gemm(const CUtensorMap& mW, const CUtensorMap& mX, const DecodeGemmParams& P, int ctas, cudaStream_t s) {
    static bool attr[kMaxDeviceSlots] = {};
    int dev = 0;
    DeviceState* st = nullptr;
    DSMOE_TRY(device_state(&st, &dev));
    auto* kernel = moa_decode_gemm_kernel<NT, QUERY>;
    if (!attr[dev]) {
        DSMOE_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, DgGeo<NT>::SMEM));
        attr[dev] = true;
    }
    int timed = -1;
    DSMOE_TRY(timing_begin(s, &timed));
    DSMOE_CUDA_TRY(launch_chained_clusters(kernel, (unsigned)ctas, kDgThreads, DgGeo<NT>::SMEM, s, P.cluster, true, mW, mX, P));
    return timing_end(s, timed);
}

// rows: weight rows in all
template <bool QUERY>
dsmoe_status launch_decode_gemm_sized(const CUtensorMap& mW, const CUtensorMap& mX, DecodeGemmParams P, int rows, cudaStream_t s) {
    // as many CTAs as SMs, at least one reduction block each; the router takes the SMs that are left over, or a few more
    const int groups = rows / kDgRows;
    P.cluster = 1;
    while (P.cluster < kDgMaxCluster && groups * P.cluster * 2 <= sm_count() && P.cluster * 2 <= P.blocks) P.cluster *= 2;
    const int most = std::max(kDgMaxT / kDgRouterTokens, sm_count() - groups * P.cluster);
    P.routers = !QUERY ? 0 : (std::min(P.T, most) + P.cluster - 1) / P.cluster * P.cluster;
    const int ctas = P.routers + groups * P.cluster;
    if (P.T <= 16) return launch_decode_gemm<2, QUERY>(mW, mX, P, ctas, s);
    if (P.T <= 32) return launch_decode_gemm<4, QUERY>(mW, mX, P, ctas, s);
    return launch_decode_gemm<8, QUERY>(mW, mX, P, ctas, s);
}

template <int DH>
dsmoe_status launch_decode_attention(const DecodeAttnParams& P, int ctas, cudaStream_t s) {
    static bool attr[kMaxDeviceSlots] = {};
    int dev = 0;
    DeviceState* st = nullptr;
    DSMOE_TRY(device_state(&st, &dev));
    if (!attr[dev]) {
        DSMOE_CUDA_TRY(cudaFuncSetAttribute(moa_decode_attention_kernel<DH>, cudaFuncAttributeMaxDynamicSharedMemorySize, DaGeo<DH>::SMEM));
        attr[dev] = true;
    }
    int timed = -1;
    DSMOE_TRY(timing_begin(s, &timed));
    DSMOE_CUDA_TRY(launch_chained(moa_decode_attention_kernel<DH>, (unsigned)ctas, 32 * kDaWarps, DaGeo<DH>::SMEM, s, P));
    return timing_end(s, timed);
}

size_t attention_part_bytes(const dsmoe_layer_desc& p, const MoaCore& c) { return (size_t)width_of(p) * (p.H / c.n_head + 2) * 4; }

// CTAs of the attention step: one per SM, as far as the parts that they may leave fit the small-T buffer, and no more than there
// are rounds of its warps over the cache
int attention_ctas(const dsmoe_layer_desc& p, const MoaCore& c) {
    const long long pairs = (long long)p.T * c.n_head;
    const long long room = (long long)((size_t)kSmallMaxCtas * 2 * p.T * 256 * 4 / attention_part_bytes(p, c)) - pairs;
    const long long rounds = pairs * ceil_div(c.L, kDaUnit * kDaWarps);
    return (int)std::min<long long>({(long long)sm_count(), room, rounds});
}

}  // namespace

// Taken for up to 64 tokens (the columns of the projections) of at most 16 experts (a tile of queries), when the library chooses where
// the sum is taken, heads of 64, 96 or 128, unless neighbouring tokens share their keys.  Experts that nobody selects are read all the
// same, so their weights may not outweigh the launches saved: 4096, 16 experts of 512, one token of one expert (126 MB read in vain)
// 40.9 -> 31.1 us; 8192, 16 experts of 1024, top-2, two tokens (403 MB) 94.2 -> 87.4, one token (470 MB) 84.3 -> 86.5.
bool moa_decode_supported(const dsmoe_layer_desc& p, const MoaCore& c) {
    const int dh = p.H / c.n_head;
    if (p.T > kDgMaxT || p.E > kDgMaxE || p.fuse_combine != 0 || p.mode == DSMOE_SELECT_THRESHOLD_TOPK) return false;
    if ((dh != 64 && dh != 96 && dh != 128) || getenv("DSMOE_MOA_PLAIN") || moa_shares_keys(p, c)) return false;
    const long long pairs = (long long)p.T * c.n_head;
    if (pairs > std::min(kDaMaxPairs, kMaxExperts * ceil_div(p.d, 256))) return false;          // (counters take tile_done's place)
    if (pairs * (c.L / kDaUnit + 1ll) > (1ll << 30)) return false;
    if ((long long)p.E * p.H > 2ll * width_of(p) * p.d) return false;                          // (queries take acc's place)
    const long long used = std::min<long long>(p.E, (long long)p.T * (p.mode == DSMOE_SELECT_THRESHOLD ? 1 : width_of(p)));
    if ((p.E - used) * p.H * p.d * 4 > 400000000ll) return false;
    return attention_ctas(p, c) >= 1;
}

dsmoe_status launch_moa_decode(const dsmoe_layer_desc& p, const MoaCore& c, const void* x, const float* Wr, const float* br, const void* packed,
                               float* scores, uint64_t* mask, int32_t* k_t, int32_t* counts_out, void* out, char* ws, const WsLayout& L,
                               int32_t* dev_status, cudaStream_t s) {
    const __nv_bfloat16* const wq = static_cast<const __nv_bfloat16*>(packed);
    const __nv_bfloat16* const wo = wq + (size_t)p.E * p.H * p.d;
    const uint64_t EH = (uint64_t)p.E * p.H;
    // the queries [T, E * H] take the place of the expert outputs, the attention outputs that of the hidden activations
    void* const q = ws + L.acc;
    void* const o = ws + L.h;
    const int box = p.T <= 16 ? 16 : p.T <= 32 ? 32 : 64;
    CUtensorMap mX, mO;
    BMaps mQ, mW;
    DSMOE_TRY(cached_map_2d(&mX, x, p.T, p.d, box));
    DSMOE_TRY(cached_map_2d(&mO, o, p.T, EH, box));
    DSMOE_TRY(cached_bmaps(&mQ, wq, p.E, p.H, p.d));
    DSMOE_TRY(cached_bmaps(&mW, wo, p.E, p.d, p.H));
    DecodeGemmParams P{};
    P.T = p.T; P.d = p.d; P.E = p.E; P.H = p.H;
    P.rows_per_expert = p.H; P.blocks = p.d / 64; P.k_blocks = p.d / 64;
    P.out = q;
    P.x = static_cast<const __nv_bfloat16*>(x);
    P.Wr = Wr;
    P.br = br;
    P.sel = SelParams{p.E, p.mode, p.eps, p.eps_normalized, p.K, p.min_k, nullptr};
    P.scores = scores;
    P.mask = mask;
    P.k_t = k_t;
    P.zero = reinterpret_cast<int*>(ws + L.tile_done);
    P.n_zero = p.T * c.n_head;
    P.counts_out = counts_out;
    P.dev_status = dev_status;
    DSMOE_TRY(launch_decode_gemm_sized<true>(mQ.m[1], mX, P, (int)EH, s));

    DecodeAttnParams A{};
    A.q = static_cast<const __nv_bfloat16*>(q);
    A.o = static_cast<__nv_bfloat16*>(o);
    A.T = p.T; A.E = p.E; A.H = p.H; A.n_head = c.n_head; A.W = width_of(p);
    A.Kc = static_cast<const __nv_bfloat16*>(c.Kc);
    A.Vc = static_cast<const __nv_bfloat16*>(c.Vc);
    A.tok_seq = c.tok_seq;
    A.pos = c.pos;
    A.n_seq = c.n_seq;
    A.L = c.L;
    A.scale_log2 = c.scale * 1.4426950408889634f;
    A.mask = mask;
    A.parts = reinterpret_cast<float*>(ws + L.partial);
    A.done = P.zero;
    A.dev_status = dev_status;
    const int ctas = attention_ctas(p, c), dh = p.H / c.n_head;
    if (dh == 64) DSMOE_TRY(launch_decode_attention<64>(A, ctas, s));
    else if (dh == 96) DSMOE_TRY(launch_decode_attention<96>(A, ctas, s));
    else DSMOE_TRY(launch_decode_attention<128>(A, ctas, s));

    P.rows_per_expert = p.d; P.blocks = (int)(EH / 64); P.k_blocks = p.H / 64;
    P.out = out;
    P.out_f32 = p.out_fp32 ? 1 : 0;
    return launch_decode_gemm_sized<false>(mW.m[1], mO, P, p.d, s);
}

}  // namespace dsmoe
