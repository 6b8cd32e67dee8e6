// Plain fp32-FMA grouped GEMMs for the expert MLPs (Eq. 1's e(X) = GeLU(X.W1).W2): the path for fp32
// layers and for bf16 layers whose weights have not been packed for the tensor-core kernels.
// Rows are grouped by expert (offsets[e] .. offsets[e+1]); a block computes one output tile of one expert's segment.
#include "common.cuh"

namespace dsmoe {

__device__ __forceinline__ float gelu_erf(float v) { return 0.5f * v * (1.f + erff(v * 0.70710678118654752440f)); }

// C[r, n] = act( sum_k A[row(r), k] * B[e, k, n] ),  r in segment e;  row(r) = gather[r] where given, else r.
// A [*,K], B [E,K,N], C [rows,N]; K and N are multiples of 8.
//
// The layers that come here are small (a tiny fp32 layer: 64 tokens, 8 experts, d 256, H 512), so the kernel is built for
// latency: a block computes a TM x TN tile, 32 x 32 or 64 x 64, from 256- or 128-wide pieces of the reduction that it
// copies to shared memory in one go (two buffers, both under way from the start: 512 elements of a reduction wait for memory
// once).
// A warp owns a 32 x 32 part of the tile over one of KSPLIT slices of the piece -- 8 warps, so 8 or 2 slices -- and a thread
// 4 rows x 8 columns of it: 12 16-byte reads of shared memory, none with a bank conflict, per 128 FMAs.  The slices' sums
// meet in shared memory and are added in slice order.  Measured on that layer: the two launches 10 + 9 us, 35 + 65 with
// 64 x 64 tiles in 16-wide steps with a barrier before and after each; 4096 tokens, d 1024, H 2048, top-2 of 8: the layer
// 3.23 -> 2.22 ms.
template <int TM, int TN>
struct FmaGeo {
    static constexpr int KC = TM * TN > 1024 ? 128 : 256;    // piece of the reduction; two of them fit shared memory
    static constexpr int LDA = KC + 4;                       // a row of A there: + 4 floats keep 8 rows' reads apart
    static constexpr int BUF = TM * LDA + KC * TN;           // floats of a buffer
};

// 4 consecutive elements to shared memory as floats; !ok = zeros
__device__ __forceinline__ void stage4(float* dst, const float* src, bool ok) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(ok ? 16u : 0u) : "memory");
}
__device__ __forceinline__ void stage4(float* dst, const __nv_bfloat16* src, bool ok) {
    const uint2 u = ok ? *reinterpret_cast<const uint2*>(src) : make_uint2(0u, 0u);
    *reinterpret_cast<float4*>(dst) = make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u),
                                                  __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xffff0000u));
}
__device__ __forceinline__ void st_out4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ void st_out4(__nv_bfloat16* p, float4 v) {
    __nv_bfloat162 h[2] = {__floats2bfloat162_rn(v.x, v.y), __floats2bfloat162_rn(v.z, v.w)};
    *reinterpret_cast<uint2*>(p) = *reinterpret_cast<uint2*>(h);
}

template <typename AT, typename BT, typename OT, bool GELU, int TM, int TN>
__global__ void __launch_bounds__(256) grouped_gemm_fma_kernel(const AT* A, const int32_t* gather,
                                                               int gather_rows, const BT* B, OT* __restrict__ C,
                                                               const int32_t* offsets, int E, int K, int N,
                                                               int64_t amax, int bufs) {
    chain_wait();
    using Geo = FmaGeo<TM, TN>;
    constexpr int SUB = (TM / 32) * (TN / 32), KSPLIT = 8 / SUB, KSLICE = Geo::KC / KSPLIT;
    extern __shared__ __align__(16) float fma_smem[];
    __shared__ int row_s[TM];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // which expert's segment, and which row tile of it: a lane holds the tile counts of experts lane and lane + 32
    int e = -1, seg0 = 0, seg1 = 0, tile = blockIdx.x;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int le = lane + 32 * h;
        if (e >= 0 || 32 * h >= E) break;
        const int s0 = le < E ? offsets[le] : 0, s1 = le < E ? offsets[le + 1] : 0;
        const bool bad = s0 < 0 || s1 < s0 || s1 > amax;        // a segment that cannot be: no rows
        const int n = bad ? 0 : (s1 - s0 + TM - 1) / TM;
        int incl = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += u;
        }
        const unsigned hit = __ballot_sync(0xffffffffu, tile < incl);
        if (hit) {
            const int l = __ffs(hit) - 1;
            tile -= __shfl_sync(0xffffffffu, incl - n, l);
            seg0 = __shfl_sync(0xffffffffu, s0, l);
            seg1 = __shfl_sync(0xffffffffu, s1, l);
            e = l + 32 * h;
        } else {
            tile -= __shfl_sync(0xffffffffu, incl, 31);
        }
    }
    if (e < 0) return;
    const int r0 = seg0 + tile * TM, rows = min(TM, seg1 - r0), n0 = blockIdx.y * TN;
    if (tid < TM) {
        const int r = r0 + min(tid, rows - 1);             // rows past the end: the last one again, not stored
        row_s[tid] = gather ? min(max(gather[r], 0), gather_rows - 1) : r;
    }
    __syncthreads();
    const BT* Be = B + (size_t)e * K * N + n0;
    const int cols = min(TN, N - n0);
    const auto fetch = [&](int k0, float* buf) {
        float* As = buf;
        float* Bs = buf + TM * Geo::LDA;
        for (int i = tid; i < TM * (Geo::KC / 4); i += 256) {
            const int m = i / (Geo::KC / 4), k = (i % (Geo::KC / 4)) * 4;
            const bool ok = k0 + k < K;
            stage4(As + m * Geo::LDA + k, A + (size_t)row_s[m] * K + (ok ? k0 + k : 0), ok);
        }
        for (int i = tid; i < Geo::KC * (TN / 4); i += 256) {
            const int k = i / (TN / 4), n = (i % (TN / 4)) * 4;
            const bool ok = k0 + k < K && n < cols;
            stage4(Bs + k * TN + n, Be + (ok ? (size_t)(k0 + k) * N + n : 0), ok);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    const int pieces = (K + Geo::KC - 1) / Geo::KC;
    for (int p = 0; p < bufs; ++p) fetch(p * Geo::KC, fma_smem + p * (size_t)Geo::BUF);
    // this thread's 4 x 8 outputs: rows g, g + 8, g + 16, g + 24 and columns 4c .. 4c + 3, 16 + 4c .. of its warp's part
    const int sub = warp % SUB, slice = warp / SUB, sm = (sub % (TM / 32)) * 32, sn = (sub / (TM / 32)) * 32;
    const int g = lane >> 2, c = lane & 3;
    float acc[4][8] = {};
    for (int p = 0; p < pieces; ++p) {
        const bool more = p + 1 < pieces;
        if (more && bufs > 1) asm volatile("cp.async.wait_group 1;" ::: "memory");
        else asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        float* buf = fma_smem + (p % bufs) * (size_t)Geo::BUF;
        const float* As = buf + (sm + g) * Geo::LDA;
        const float* Bs = buf + TM * Geo::LDA + sn + 4 * c;
        const int kend = min(slice * KSLICE + KSLICE, (K - p * Geo::KC + 3) & ~3);
#pragma unroll 2
        for (int k = slice * KSLICE; k < kend; k += 4) {
            float4 a[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const float4*>(As + 8 * i * Geo::LDA + k);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float4 b0 = *reinterpret_cast<const float4*>(Bs + (k + u) * TN);
                const float4 b1 = *reinterpret_cast<const float4*>(Bs + (k + u) * TN + 16);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float av = u == 0 ? a[i].x : u == 1 ? a[i].y : u == 2 ? a[i].z : a[i].w;
                    acc[i][0] = fmaf(av, b0.x, acc[i][0]);
                    acc[i][1] = fmaf(av, b0.y, acc[i][1]);
                    acc[i][2] = fmaf(av, b0.z, acc[i][2]);
                    acc[i][3] = fmaf(av, b0.w, acc[i][3]);
                    acc[i][4] = fmaf(av, b1.x, acc[i][4]);
                    acc[i][5] = fmaf(av, b1.y, acc[i][5]);
                    acc[i][6] = fmaf(av, b1.z, acc[i][6]);
                    acc[i][7] = fmaf(av, b1.w, acc[i][7]);
                }
            }
        }
        __syncthreads();
        if (p + bufs < pieces) fetch((p + bufs) * Geo::KC, buf);
    }
    chain_next();
    // the slices' sums: [slice][TM][TN], then every thread adds the slices of its outputs in order
    float* red = fma_smem;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float* dst = red + ((size_t)slice * TM + sm + g + 8 * i) * TN + sn + 4 * c;
        *reinterpret_cast<float4*>(dst) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
        *reinterpret_cast<float4*>(dst + 16) = make_float4(acc[i][4], acc[i][5], acc[i][6], acc[i][7]);
    }
    __syncthreads();
    for (int i = tid; i < TM * (TN / 4); i += 256) {
        const int m = i / (TN / 4), n = (i % (TN / 4)) * 4;
        if (m >= rows || n >= cols) continue;
        float4 v = *reinterpret_cast<const float4*>(red + m * TN + n);
#pragma unroll
        for (int sl = 1; sl < KSPLIT; ++sl) {
            const float4 w = *reinterpret_cast<const float4*>(red + ((size_t)sl * TM + m) * TN + n);
            v.x += w.x;
            v.y += w.y;
            v.z += w.z;
            v.w += w.w;
        }
        if (GELU) v = make_float4(gelu_erf(v.x), gelu_erf(v.y), gelu_erf(v.z), gelu_erf(v.w));
        st_out4(C + (size_t)(r0 + m) * N + n0 + n, v);
    }
}

template <typename AT, typename BT, typename OT, bool GELU, int TM, int TN>
static dsmoe_status launch_fma(const AT* A, const int32_t* gather, int gather_rows, const BT* B, OT* C, const int32_t* offsets,
                               int E, int K, int N, size_t amax, cudaStream_t s) {
    using Geo = FmaGeo<TM, TN>;
    const int bufs = K > Geo::KC ? 2 : 1;
    const size_t loop = bufs * (size_t)Geo::BUF, red = (size_t)(8 / ((TM / 32) * (TN / 32))) * TM * TN;
    const size_t smem = (loop > red ? loop : red) * sizeof(float);
    static bool attr[kMaxDeviceSlots] = {};
    int dev = 0;
    DeviceState* st = nullptr;
    DSMOE_TRY(device_state(&st, &dev));
    auto* kernel = grouped_gemm_fma_kernel<AT, BT, OT, GELU, TM, TN>;
    if (!attr[dev]) {
        const size_t most = 2 * (size_t)Geo::BUF * sizeof(float);
        DSMOE_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most));
        attr[dev] = true;
    }
    DSMOE_CUDA_TRY(launch_chained(kernel, dim3((unsigned)(amax / TM + E), ceil_div(N, TN)), 256, smem, s,
        A, gather, gather_rows, B, C, offsets, E, K, N, (int64_t)amax, bufs));
    return DSMOE_OK;
}

// 64 x 64 tiles read half as much of A and B per FMA; 32 x 32 ones give four times the blocks.  The larger ones where
// they still give every SM about two blocks.
template <typename AT, typename BT, typename OT, bool GELU>
static dsmoe_status launch_fma_sized(const AT* A, const int32_t* gather, int gather_rows, const BT* B, OT* C,
                                     const int32_t* offsets, int E, int K, int N, size_t amax, cudaStream_t s) {
    const size_t tiles64 = (amax / 64 + E) * ceil_div(N, 64);
    if (tiles64 >= 2 * (size_t)sm_count())
        return launch_fma<AT, BT, OT, GELU, 64, 64>(A, gather, gather_rows, B, C, offsets, E, K, N, amax, s);
    return launch_fma<AT, BT, OT, GELU, 32, 32>(A, gather, gather_rows, B, C, offsets, E, K, N, amax, s);
}

template <typename XT>
static dsmoe_status run(const dsmoe_layer_desc& p, const XT* x, const int32_t* row_token, const XT* W1, const XT* W2,
                        const int32_t* offsets, float* h, XT* yp, cudaStream_t s) {
    const size_t amax = amax_of(p);
    DSMOE_TRY((launch_fma_sized<XT, XT, float, true>(x, row_token, p.T, W1, h, offsets, p.E, p.d, p.H, amax, s)));
    return launch_fma_sized<float, XT, XT, false>(h, nullptr, 0, W2, yp, offsets, p.E, p.H, p.d, amax, s);
}

dsmoe_status launch_mlp_generic(const dsmoe_layer_desc& p, const void* x, const void* W1, const void* W2,
                                const int32_t* offsets, float* h, void* yp, cudaStream_t s, const int32_t* row_token) {
    if (p.T == 0) return DSMOE_OK;
    if (p.dtype == DSMOE_BF16)
        return run(p, static_cast<const __nv_bfloat16*>(x), row_token, static_cast<const __nv_bfloat16*>(W1),
                   static_cast<const __nv_bfloat16*>(W2), offsets, h, static_cast<__nv_bfloat16*>(yp), s);
    return run(p, static_cast<const float*>(x), row_token, static_cast<const float*>(W1), static_cast<const float*>(W2),
               offsets, h, static_cast<float*>(yp), s);
}

}  // namespace dsmoe
