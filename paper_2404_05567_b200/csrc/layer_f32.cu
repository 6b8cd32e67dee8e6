// The fp32 layer where it is so small that the plain path is all latency: three chained launches instead of five.
//
//   router  a warp per token: logits, softmax, selection
//   up      h = GeLU(x . W1[e]): a CTA per (expert, 32 or 16 columns)
//   down    rows gate * (h . W2[e]) by tiles likewise; of the CTAs of a column range the one that comes last adds up every token's
//           rows, in ascending order of the experts
//
// A CTA finds its expert's tokens in the selection words itself, and a token's row for its i-th selected expert (i < W) is row t * W + i of h and of
// the outputs: no row indices, no launch that computes them.  A tile's weights (all of its reduction) are asked for before the CTA waits
// for its predecessor: nothing that the call itself writes.  Bound by the chain of short steps (router 2.3 us; tokens found, rows fetched,
// multiplied and stored 6 and, without the first, 5; the last CTA's sum 2; some 0.9 from a launch's end to the next one's start): 64 tokens of
// d 256, H 512, 8 experts by threshold 27.9 -> 17.2 us a layer.  As one cooperative launch with two grid barriers: 25.4.
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "router_device.cuh"

namespace dsmoe {

namespace {

constexpr int kLfThreads = 512, kLfWarps = kLfThreads / 32;
constexpr int kLfRows = 64, kLfOct = kLfRows / 8, kLfPiece = 256, kLfLda = kLfPiece + 4;
constexpr int kLfMaxT = kLfThreads, kLfMaxE = 32, kLfMaxK = 1024;
constexpr int kLfA = kLfRows * kLfLda;                     // floats of a piece of 64 rows, whose place the sums of the slices take
static_assert(kLfWarps * 16 * kLfRows <= kLfA, "16 slices of 16 columns, or 8 of 32");
constexpr int kLfRouterWarps = 4;

__device__ __forceinline__ float gelu_f32(float v) { return 0.5f * v * (1.f + erff(v * 0.70710678118654752440f)); }

__device__ __forceinline__ void copy16(float* dst, const float* src, bool ok) {      // !ok: zeros
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(ok ? 16u : 0u)
                 : "memory");
}
__device__ __forceinline__ void commit_copies() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void wait_copies() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

template <int EP>        // experts, padded
__global__ void __launch_bounds__(32 * kLfRouterWarps) layer_f32_router_kernel(const float* x, const float* Wr, const float* br,
                                                                              float* __restrict__ scores, uint64_t* __restrict__ mask,
                                                                              int32_t* __restrict__ k_t, int* __restrict__ done, int n_done, int T,
                                                                              int d, const SelParams q) {
    chain_wait();
    chain_next();            // (not before: the tiles' weights may be what came before this launch wrote)
    const int lane = threadIdx.x & 31, t = blockIdx.x * kLfRouterWarps + (threadIdx.x >> 5), E = q.E;
    if (blockIdx.x == 0)
        for (int i = threadIdx.x; i < n_done; i += 32 * kLfRouterWarps) done[i] = 0;
    if (t >= T) return;
    const float* const xr = x + (size_t)t * d;
    float a[EP];
#pragma unroll
    for (int e = 0; e < EP; ++e) a[e] = 0.f;
    if ((E & 3) == 0) {
#pragma unroll(EP == 8 ? 8 : 4)
        for (int k = lane; k < d; k += 32) {
            const float xv = xr[k];
            const float4* const w = reinterpret_cast<const float4*>(Wr + (size_t)k * E);
#pragma unroll
            for (int c = 0; c < EP / 4; ++c) {
                if (4 * c < E) {
                    const float4 v = w[c];
                    a[4 * c] = fmaf(xv, v.x, a[4 * c]);
                    a[4 * c + 1] = fmaf(xv, v.y, a[4 * c + 1]);
                    a[4 * c + 2] = fmaf(xv, v.z, a[4 * c + 2]);
                    a[4 * c + 3] = fmaf(xv, v.w, a[4 * c + 3]);
                }
            }
        }
    } else {
        for (int k = lane; k < d; k += 32) {
            const float xv = xr[k];
#pragma unroll
            for (int e = 0; e < EP; ++e)
                if (e < E) a[e] = fmaf(xv, Wr[(size_t)k * E + e], a[e]);
        }
    }
    // each exchange halves the experts that a lane still holds: expert e ends up in the lanes whose upper bits are e
    int o = 16;
#pragma unroll
    for (int n = EP / 2; n >= 1; n >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const float keep = up ? a[i + n] : a[i], give = up ? a[i] : a[i + n];
            a[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
        o >>= 1;
    }
    for (; o > 0; o >>= 1) a[0] += __shfl_xor_sync(0xffffffffu, a[0], o);
    float l = __shfl_sync(0xffffffffu, a[0], (lane % EP) * (32 / EP));
    if (br && lane < E) l += br[lane];
    softmax_select_store(l, 0.f, t, q, lane, scores, mask, k_t);
}

struct TileF32Params {
    int T, K, N, E, W;
    const float* A;              // up: x [T, K]; down: h [T * W, K]
    const float* B;              // [E, K, N]
    float* rows;                 // up: h; down: the gate-weighted outputs [T * W, N]
    const uint64_t* mask;
    const float* scores;
    int32_t* counts_out;         // up (nullable)
    float* out;                  // down
    int* done;                   // down: finished tiles of each column range, zero
};

// Rows are taken up to 64 at a time, in pieces of 256 of the reduction.  A warp owns 16 columns of all rows over one of 8 slices of the piece
// (32 columns a tile; 16 slices: 16 columns), a thread 4 columns of every eighth row.  The slices' sums meet in shared memory and are
// added in slice order.  Bound by latency: 22 rows x 32 columns x 256 take 2.7 us from the rows' arrival to the sums, with 8 x 8 outputs a
// thread in half as many threads (half of the reads of shared memory) 2.2, but 1.0 instead of 1.2 times the plain path's speed at d 512, H 1024.
template <bool UP, int TN>
__global__ void __launch_bounds__(kLfThreads, 2) layer_f32_tile_kernel(const TileF32Params P) {
    constexpr int HALVES = TN / 16, SLICES = kLfWarps / HALVES, SLICE = kLfPiece / SLICES;
    extern __shared__ __align__(16) float lf_smem[];
    __shared__ uint64_t mask_s[kLfMaxT];
    __shared__ int list_s[kLfMaxT], count_s[kLfWarps], row_s[kLfRows], last_s;
    __shared__ float gate_s[kLfRows];
    float* const As = lf_smem;                              // a piece of A; then the slices' sums
    float* const Bs = lf_smem + kLfA;                       // the tile's weights [K][TN]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int T = P.T, K = P.K, N = P.N, E = P.E, e = blockIdx.x % E, n0 = blockIdx.x / E * TN, cols = min(TN, N - n0);
    {
        const float* const src = P.B + (size_t)e * K * N + n0;
        for (int i = tid; i < K * (TN / 4); i += kLfThreads) {
            const int k = i / (TN / 4), n = i % (TN / 4) * 4;
            copy16(Bs + k * TN + n, src + (n < cols ? (size_t)k * N + n : 0), n < cols);
        }
        commit_copies();
    }
    // (the selection is not the up tiles' work: when a down tile starts, they have all seen the router's end, and its words lie in L2.  Nothing
    // but its own wait tells a CTA what its SM's L1 may still hold of them from an earlier call: they are read past it)
    if (UP) {
        chain_wait();
        chain_next();
    }
    // the expert's tokens, in order
    uint64_t m = tid < T ? __ldcg(reinterpret_cast<const unsigned long long*>(P.mask) + tid) : 0;
    if (UP && n0 == 0 && P.counts_out) {
        const int n = __syncthreads_count((m >> e) & 1ull);
        if (tid == 0) P.counts_out[e] = n;
    }
    // a token has W rows: one whose scores are no numbers is selected by all experts under top-K, and keeps the first W
    while (__popcll(m) > P.W) m ^= 1ull << (63 - __clzll((long long)m));
    mask_s[tid] = m;
    const bool mine = (m >> e) & 1ull;
    const unsigned hit = __ballot_sync(0xffffffffu, mine);
    if (lane == 0) count_s[warp] = __popc(hit);
    __syncthreads();
    int before = 0, n_rows = 0;
#pragma unroll
    for (int w = 0; w < kLfWarps; ++w) {
        before += w < warp ? count_s[w] : 0;
        n_rows += count_s[w];
    }
    if (mine) list_s[before + __popc(hit & ((1u << lane) - 1u))] = tid;
    if (!UP) {
        chain_wait();
        chain_next();
    }
    __syncthreads();

    const int g = lane >> 2, c4 = (warp % HALVES) * 16 + (lane & 3) * 4, slice = warp / HALVES;
    for (int r0 = 0; r0 < n_rows; r0 += kLfRows) {
        const int rows = min(kLfRows, n_rows - r0), octets = (rows + 7) / 8;
        if (tid < rows) {
            const int t = list_s[r0 + tid];
            row_s[tid] = t * P.W + __popcll(mask_s[t] & ((1ull << e) - 1ull));
            if (!UP) gate_s[tid] = P.scores[(size_t)t * E + e];
        }
        if (!UP) __syncthreads();
        float acc[kLfOct][4] = {};
        for (int p0 = 0; p0 < K; p0 += kLfPiece) {
            const int kn = min(kLfPiece, K - p0);            // (a multiple of 8)
            for (int i = tid; i < rows * (kLfPiece / 4); i += kLfThreads) {
                const int r = i / (kLfPiece / 4), k = i % (kLfPiece / 4) * 4;
                if (k < kn) copy16(As + r * kLfLda + k, P.A + (size_t)(UP ? list_s[r0 + r] : row_s[r]) * K + p0 + k, true);
            }
            commit_copies();
            wait_copies();
            __syncthreads();
            const float* const a0 = As + g * kLfLda;
            const float* const b0 = Bs + p0 * TN + c4;
            const int kend = min(slice * SLICE + SLICE, kn);
            const auto multiply = [&](auto oct) {
#pragma unroll 2
                for (int k = slice * SLICE; k < kend; k += 4) {
                    float4 b[4];
#pragma unroll
                    for (int v = 0; v < 4; ++v) b[v] = *reinterpret_cast<const float4*>(b0 + (k + v) * TN);
#pragma unroll
                    for (int i = 0; i < oct.value; ++i) {
                        const float4 a = *reinterpret_cast<const float4*>(a0 + 8 * i * kLfLda + k);
#pragma unroll
                        for (int v = 0; v < 4; ++v) {
                            const float av = v == 0 ? a.x : v == 1 ? a.y : v == 2 ? a.z : a.w;
                            acc[i][0] = fmaf(av, b[v].x, acc[i][0]);
                            acc[i][1] = fmaf(av, b[v].y, acc[i][1]);
                            acc[i][2] = fmaf(av, b[v].z, acc[i][2]);
                            acc[i][3] = fmaf(av, b[v].w, acc[i][3]);
                        }
                    }
                }
            };
            // (rows past the last are multiplied too, by whatever lies there: nobody reads their sums)
            if (octets <= 2) multiply(std::integral_constant<int, 2>{});
            else if (octets <= 4) multiply(std::integral_constant<int, 4>{});
            else multiply(std::integral_constant<int, kLfOct>{});
            __syncthreads();
        }
#pragma unroll
        for (int i = 0; i < kLfOct; ++i) {
            if (i >= octets) break;
            *reinterpret_cast<float4*>(As + (slice * kLfRows + g + 8 * i) * TN + c4) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
        }
        __syncthreads();
        for (int i = tid; i < rows * (TN / 4); i += kLfThreads) {
            const int r = i / (TN / 4), n = i % (TN / 4) * 4;
            float4 v = *reinterpret_cast<const float4*>(As + r * TN + n);
#pragma unroll
            for (int s = 1; s < SLICES; ++s) {
                const float4 u = *reinterpret_cast<const float4*>(As + (s * kLfRows + r) * TN + n);
                v.x += u.x;
                v.y += u.y;
                v.z += u.z;
                v.w += u.w;
            }
            if (n >= cols) continue;
            const float gt = UP ? 0.f : gate_s[r];
            *reinterpret_cast<float4*>(P.rows + (size_t)row_s[r] * N + n0 + n) =
                UP ? make_float4(gelu_f32(v.x), gelu_f32(v.y), gelu_f32(v.z), gelu_f32(v.w)) : make_float4(gt * v.x, gt * v.y, gt * v.z, gt * v.w);
        }
        __syncthreads();
    }
    if (n_rows == 0) wait_copies();                          // the weights are on their way all the same
    if (UP) return;
    // the last of a column range's CTAs adds up
    __threadfence();
    __syncthreads();
    if (tid == 0) last_s = atomicAdd(P.done + blockIdx.x / E, 1) == E - 1;
    __syncthreads();
    if (!last_s) return;
    __threadfence();
    const int quads = cols / 4;
    for (int i = tid; i < T * quads; i += kLfThreads) {
        const int t = i / quads, n = n0 + i % quads * 4, k = __popcll(mask_s[t]);
        const float* const from = P.rows + (size_t)t * P.W * N + n;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int s = 0; s < k; s += 4) {
            float4 r[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) r[j] = s + j < k ? __ldcg(reinterpret_cast<const float4*>(from + (size_t)(s + j) * N)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                v.x += r[j].x;
                v.y += r[j].y;
                v.z += r[j].z;
                v.w += r[j].w;
            }
        }
        *reinterpret_cast<float4*>(P.out + (size_t)t * N + n) = v;
    }
}

template <bool UP, int TN>
dsmoe_status launch_tiles_of(const TileF32Params& P, cudaStream_t s) {
    static bool attr[kMaxDeviceSlots] = {};
    int dev = 0;
    DeviceState* st = nullptr;
    DSMOE_TRY(device_state(&st, &dev));
    auto* kernel = layer_f32_tile_kernel<UP, TN>;
    if (!attr[dev]) {
        DSMOE_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)((kLfA + kLfMaxK * TN) * sizeof(float))));
        attr[dev] = true;
    }
    DSMOE_CUDA_TRY(launch_chained(kernel, (unsigned)(P.E * ceil_div(P.N, TN)), kLfThreads, (kLfA + (size_t)P.K * TN) * sizeof(float), s, P));
    return DSMOE_OK;
}

// 16 columns a tile where 32 would leave half of the SMs out
template <bool UP>
dsmoe_status launch_tiles(const TileF32Params& P, cudaStream_t s) {
    return 2 * P.E * ceil_div(P.N, 32) <= sm_count() ? launch_tiles_of<UP, 16>(P, s) : launch_tiles_of<UP, 32>(P, s);
}

}  // namespace

// Where the launches weigh more than the work: an expert's tokens are half a pass of 64 rows on average (how many a threshold selects the host
// does not know: a third of them is assumed), and the weights of experts without tokens, which are read all the same, are few.  us a
// layer, plain path and here:
//   64 tokens, d 256, H 512, 8 experts by threshold 28.1, 17.4; top-2 27.8, 16.9; d 512, H 1024, 16 experts 88.3, 73.4; 7 tokens of d 384, H 256 24.5, 15.8
//   more rows: 150 tokens, top-2 of 8 experts (37 rows) of d 384, H 256 28.7, 30.8, by threshold (52) 30.8, 36.1; 100 tokens of all of 32 experts 182, 203
//   one token, top-2 of 16 experts of d 512, H 1024 (58 MB in vain) 37.9, 40.6; reductions of 1024 leave room for one CTA an SM: 100
//   tokens top-2 of 8 experts of d 1024, H 1024 75.4, 82.3
bool layer_f32_supported(const dsmoe_layer_desc& p) {
    if (p.dtype != DSMOE_F32 || p.E > kLfMaxE || p.T > kLfMaxT || p.d > kLfMaxK / 2 || p.H > kLfMaxK) return false;
    if (p.mode == DSMOE_SELECT_THRESHOLD_TOPK) return false;
    const long long E = p.E, rows = (long long)p.T * width_of(p);
    if (rows > (p.mode == DSMOE_SELECT_THRESHOLD ? 3 : 1) * kLfRows / 2 * E) return false;
    const long long used = p.mode == DSMOE_SELECT_TOPK ? std::min(E, rows) : E;
    return (E - used) * p.d * p.H * 8 <= 24000000ll;
}

dsmoe_status launch_layer_f32(const dsmoe_layer_desc& p, const void* x, const float* Wr, const float* br, const void* W1, const void* W2,
                              float* scores, uint64_t* mask, int32_t* k_t, int32_t* counts_out, void* out, char* ws, const WsLayout& L,
                              cudaStream_t s) {
    int* const done = reinterpret_cast<int*>(ws + L.tile_done);
    const SelParams q{p.E, p.mode, p.eps, p.eps_normalized, p.K, p.min_k, nullptr};
    const float* const xf = static_cast<const float*>(x);
    const auto router = [&](auto kernel) {
        return launch_chained(kernel, (unsigned)ceil_div(p.T, kLfRouterWarps), 32 * kLfRouterWarps, 0, s, xf, Wr, br, scores, mask, k_t, done,
                              ceil_div(p.d, 16), p.T, p.d, q);
    };
    DSMOE_CUDA_TRY(p.E <= 8 ? router(layer_f32_router_kernel<8>) : p.E <= 16 ? router(layer_f32_router_kernel<16>) : router(layer_f32_router_kernel<32>));
    TileF32Params P{};
    P.T = p.T; P.K = p.d; P.N = p.H; P.E = p.E; P.W = width_of(p);
    P.A = xf;
    P.B = static_cast<const float*>(W1);
    P.rows = reinterpret_cast<float*>(ws + L.h_plain);
    P.mask = mask;
    P.scores = scores;
    P.counts_out = counts_out;
    P.done = done;
    DSMOE_TRY(launch_tiles<true>(P, s));
    P.K = p.H; P.N = p.d;
    P.A = P.rows;
    P.B = static_cast<const float*>(W2);
    P.rows = reinterpret_cast<float*>(ws + L.yp);
    P.out = static_cast<float*>(out);
    return launch_tiles<false>(P, s);
}

}  // namespace dsmoe
