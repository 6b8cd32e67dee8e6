// Router for some hundred tokens (bf16): a cluster of 8 CTAs takes 32 tokens and shares out the reduction over d, on warp-level MMAs.
//
// Between router_small_kernel, each of whose blocks reads all of Wr for four tokens, and router_umma_kernel, whose clusters take 128
// tokens each and leave most SMs without any, the launch is a chain of latencies: this form has one round of loads or two, one sum in
// shared memory and one across the cluster.  A lane's 16-byte load of 8 neighbouring elements of x serves two steps of m16n8k16, since the
// order of the reduction is free; the router's weights come straight out of memory into the fragments, as the exact sum of three bf16
// terms (3 x 8 significant bits = fp32's 24).  A step of 32 has its own accumulator, the rest is added in
// fp32 (the tensor core cuts its sums off): 1.4e-7 to 3.2e-7 from 64 bits, the two others 1.4e-7 to 2.7e-7 and 1.6e-7 to 9.2e-7.
//
// Top-4 layers of 32 experts, whole calls, before (router_small_kernel up to 256 tokens, router_umma_kernel above) and with this: d 2048,
// H 256: 64.0 -> 51.1 us at 150 tokens, 55.9 -> 53.2 at 300; d 4096, H 512: 102.8 -> 85.2 and 90.2 -> 86.6.  Asking the first weights
// into L2 from CTAs behind the router's made calls of few experts up to 11 % slower (the weights' own copies met the same lines).
#include "common.cuh"
#include "router_device.cuh"
#include "umma.cuh"

namespace dsmoe {

namespace {

constexpr int kRcTokens = 32, kRcCtas = 8, kRcWarps = 8, kRcThreads = 32 * kRcWarps, kRcStep = 32;

__device__ __forceinline__ void mma_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ float ld_cluster_f32(uint32_t addr) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}

template <int EP, int PER_SM>        // experts, padded; CTAs that an SM is to hold
__global__ void __launch_bounds__(kRcThreads, PER_SM) router_cluster_kernel(const __nv_bfloat16* x, const float* Wr, const float* br,
                                                                    float* __restrict__ scores, uint64_t* __restrict__ mask,
                                                                    int32_t* __restrict__ k_t, int32_t* __restrict__ chunk_counts, int T, int d,
                                                                    const SelParams q, const ZeroInts zero) {
    constexpr int NT = EP / 8, LD = EP + 8;              // floats between two tokens' sums: no bank conflicts
    extern __shared__ __align__(16) float rc_part[];     // [warps][tokens][LD]
    __shared__ uint64_t mask_s[kRcTokens];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, q4 = lane & 3, E = q.E;
    const int group = blockIdx.x / kRcCtas, rank = blockIdx.x % kRcCtas;
    chain_wait();
    zero_ints(zero);
    const int t0 = group * kRcTokens, steps = d / kRcStep;
    float acc[2][NT][4];
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int n = 0; n < NT; ++n) acc[m][n][0] = acc[m][n][1] = acc[m][n][2] = acc[m][n][3] = 0.f;
    const __nv_bfloat16* xr[4];                          // this lane's rows: 8 i + g of the group (past the last token: it again, unused)
#pragma unroll
    for (int i = 0; i < 4; ++i) xr[i] = x + (size_t)min(t0 + 8 * i + g, T - 1) * d + q4 * 8;
    const int end = steps * (rank + 1) / kRcCtas;
    for (int st = steps * rank / kRcCtas + warp; st < end; st += kRcWarps) {
        uint4 a[4];
        float w[NT][8];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const uint4*>(xr[i] + st * kRcStep);
        const float* const wr = Wr + (size_t)(st * kRcStep + q4 * 8) * E + g;
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int k = 0; k < 8; ++k) w[n][k] = 8 * n + g < E ? wr[(size_t)k * E + 8 * n] : 0.f;
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            // (cut off, not rounded: the terms are just as exact, and a mask and a subtraction each)
            uint32_t t[3][4];
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                uint32_t v1[2], v2[2], v3[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    v1[u] = __float_as_uint(w[n][2 * p + u]);
                    const float r1 = w[n][2 * p + u] - __uint_as_float(v1[u] & 0xffff0000u);
                    v2[u] = __float_as_uint(r1);
                    v3[u] = __float_as_uint(r1 - __uint_as_float(v2[u] & 0xffff0000u));
                }
                t[0][p] = __byte_perm(v1[0], v1[1], 0x7632);
                t[1][p] = __byte_perm(v2[0], v2[1], 0x7632);
                t[2][p] = __byte_perm(v3[0], v3[1], 0x7632);
            }
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                const uint32_t lo[4] = {a[2 * m].x, a[2 * m + 1].x, a[2 * m].y, a[2 * m + 1].y};
                const uint32_t hi[4] = {a[2 * m].z, a[2 * m + 1].z, a[2 * m].w, a[2 * m + 1].w};
                float sum[4] = {};
#pragma unroll
                for (int c = 2; c >= 0; --c) {           // the smallest terms first
                    mma_16816(sum, lo, t[c][0], t[c][1]);
                    mma_16816(sum, hi, t[c][2], t[c][3]);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[m][n][i] += sum[i];
            }
        }
    }
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            float* const to = rc_part + ((size_t)warp * kRcTokens + m * 16 + g) * LD + n * 8 + q4 * 2;
            *reinterpret_cast<float2*>(to) = make_float2(acc[m][n][0], acc[m][n][1]);
            *reinterpret_cast<float2*>(to + 8 * LD) = make_float2(acc[m][n][2], acc[m][n][3]);
        }
    __syncthreads();
    for (int i = tid; i < kRcTokens * EP; i += kRcThreads) {
        float* const at = rc_part + (i / EP) * LD + i % EP;
        float v = at[0];
#pragma unroll
        for (int w = 1; w < kRcWarps; ++w) v += at[(size_t)w * kRcTokens * LD];
        at[0] = v;
    }
    // (not at the start: what comes next then waits beside the reduction, and attention layers of d 4096 lost what this router gained:
    // 78.8 us with it here, 86.0 at the start, at 130 tokens)
    chain_next();
    ptx::cluster_sync();                                 // every rank's sums are in place
    constexpr int PER = kRcTokens / kRcCtas;
    if (warp < PER) {
        const int tl = rank * PER + warp, t = t0 + tl;
        const bool v_lo = lane < E, v_hi = lane + 32 < E;
        float l_lo = br && v_lo ? br[lane] : 0.f, l_hi = br && v_hi ? br[lane + 32] : 0.f;
        const uint32_t at = ptx::smem_u32(rc_part + tl * LD + lane);
        float lo[kRcCtas], hi[kRcCtas];
#pragma unroll
        for (int r = 0; r < kRcCtas; ++r) {
            const uint32_t from = ptx::map_to_cta(at, (uint32_t)r);
            lo[r] = v_lo ? ld_cluster_f32(from) : 0.f;
            hi[r] = EP > 32 && v_hi ? ld_cluster_f32(from + 128) : 0.f;
        }
#pragma unroll
        for (int r = 0; r < kRcCtas; ++r) {
            l_lo += lo[r];
            l_hi += hi[r];
        }
        uint64_t m = 0;
        if (t < T) m = softmax_select_store(l_lo, l_hi, t, q, lane, scores, mask, k_t);
        if (lane == 0)
            asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(ptx::map_to_cta(ptx::smem_u32(&mask_s[tl]), 0u)), "l"(m) : "memory");
    }
    ptx::cluster_sync();                                 // rank 0 has the selections; nobody leaves while another rank may read its sums
    if (chunk_counts && rank == 0 && warp == 0) {
        const uint64_t mt = mask_s[lane];
        int c_lo = 0, c_hi = 0;
        for (int e = 0; e < E; ++e) {
            const int n = __popc(__ballot_sync(0xffffffffu, (mt >> e) & 1));
            if (lane == (e & 31)) {
                if (e < 32) c_lo = n;
                else c_hi = n;
            }
        }
        if (lane < E) chunk_counts[(size_t)group * E + lane] = c_lo;
        if (lane + 32 < E) chunk_counts[(size_t)group * E + lane + 32] = c_hi;
    }
}
static_assert(kRcTokens == kChunk, "a cluster's tokens are a chunk");

template <int EP, int PER_SM = 1>
dsmoe_status launch_ep(const dsmoe_layer_desc& p, const void* x, const float* Wr, const float* br, float* scores, uint64_t* mask, int32_t* k_t,
                       cudaStream_t s, int32_t* chunk_counts, const ZeroInts& zero) {
    constexpr size_t smem = (size_t)kRcWarps * kRcTokens * (EP + 8) * sizeof(float);
    static bool attr[kMaxDeviceSlots] = {};
    int dev = 0;
    DeviceState* st = nullptr;
    DSMOE_TRY(device_state(&st, &dev));
    if (!attr[dev]) {
        DSMOE_CUDA_TRY(cudaFuncSetAttribute(router_cluster_kernel<EP, PER_SM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        attr[dev] = true;
    }
    DSMOE_CUDA_TRY(launch_chained_clusters(router_cluster_kernel<EP, PER_SM>, (unsigned)(ceil_div(p.T, kRcTokens) * kRcCtas), kRcThreads,
        smem, s, kRcCtas, true, static_cast<const __nv_bfloat16*>(x), Wr, br, scores, mask, k_t, chunk_counts, p.T, p.d,
        SelParams{p.E, p.mode, p.eps, p.eps_normalized, p.K, p.min_k, nullptr}, zero));
    return DSMOE_OK;
}

}  // namespace

// 384 tokens are 12 clusters of 8, and about as many have an SM for each of their CTAs; up to 32 experts two CTAs share an SM
// (up to 16 they do anyhow, and with that little to do a second wave costs less than router_umma_kernel's longer chain).  Just beyond
// each line: 33 experts and more 0.95 at 512 tokens (1.02 to 1.05 at 384), 17 to 32 experts 0.94 to 0.98 at 1000 (1.03 to 1.05 at 700); up
// to 16 experts still 1.025 to 1.07 at 1000.  One CTA on an SM is the faster of the two while all fit: 300 tokens 1.04 to 1.06 beside 1.03 to
// 1.05.  Below d 1024 (2048 up to 256 tokens of at most 16 experts, whose router_small_kernel reads little) most warps have no step to take:
// 0.98 to 1.00.  Up to 64 tokens the one-launch layers route for themselves.
bool router_cluster_supported(const dsmoe_layer_desc& p) {
    return umma_supported(p) && p.T > 64 && p.T <= (p.E <= 16 ? 1024 : p.E <= 32 ? 768 : 384) &&
           p.d >= (p.T > 256 ? 1024 : p.E <= 16 ? 2048 : kRcStep * kRcCtas);
}

dsmoe_status launch_router_cluster(const dsmoe_layer_desc& p, const void* x, const float* Wr, const float* br, float* scores, uint64_t* mask,
                                   int32_t* k_t, cudaStream_t s, int32_t* chunk_counts, const ZeroInts& zero) {
    return p.E <= 8 ? launch_ep<8>(p, x, Wr, br, scores, mask, k_t, s, chunk_counts, zero)
           : p.E <= 16 ? launch_ep<16>(p, x, Wr, br, scores, mask, k_t, s, chunk_counts, zero)
           : p.E <= 32 && p.T <= 384 ? launch_ep<32>(p, x, Wr, br, scores, mask, k_t, s, chunk_counts, zero)
           : p.E <= 32 ? launch_ep<32, 2>(p, x, Wr, br, scores, mask, k_t, s, chunk_counts, zero)
                       : launch_ep<64>(p, x, Wr, br, scores, mask, k_t, s, chunk_counts, zero);
}

}  // namespace dsmoe
