// The router for many tokens (Eq. 1's S = softmax(x.Wr + b)) on the 5th-generation tensor cores, in one launch: logits,
// softmax, selection and the per-chunk counts that the grouping step needs.
//
// Wr (fp32) enters as the exact sum of three bf16 terms, w = w1 + w2 + w3: the upper, middle and lower 8 of its 24
// significant bits.  x is bf16, so every product x.w_i is exact in fp32 and
// the three sums accumulate in fp32, at tensor-core speed.  The terms sit side by side along the MMA's N: 3 * EP columns, EP = E
// rounded up to 32 or 64.  The tensor core cuts its running sums off instead of rounding them, an error that grows with the
// length of a sum, so a CTA spreads its part of the reduction over 5 (EP = 64: 2) accumulators, one run of blocks after the
// other, which are added in fp32.  Scores against 64 bits, relative 2-norm: 7001 tokens of 4096, 32 experts 3.7e-7 (one
// accumulator 2.0e-6, router_tile_kernel's FMAs 5.5e-7); 4096 tokens of 4096, 64 experts 4.9e-7 (1.0e-6, 5.9e-7); 0.3 us.
//
// A cluster of C CTAs (1, 2 or 4) owns 128 tokens and shares out the reduction over d, so that few row tiles still cover most
// SMs.  Each CTA:
//   warp 0      brings its 128 x 64 tiles of x by TMA                      (one lane)
//   warp 1      issues the MMAs (M = 128, N = 3 EP); owns the TMEM columns (one lane)
//   warps 2..17 split Wr: teams of four warps take every fourth 64-wide block of the reduction, an expert per lane, and write
//               the three terms in the 128-byte-swizzle order the MMA reads; then they finish the tokens
// The CTAs' partial logits meet through distributed shared memory: each CTA finishes 128 / C of the tokens, adding the
// ranks' sums in ascending order.
// At 7001 tokens of 4096 and 32 experts it takes 24.7 us (x once from HBM: 57 MB, 9 us); as three launches -- splitting Wr into a
// global buffer, a GEMM, the finish over its sums -- 3.2 + 24.5 + 9.5 us and two gaps; 300 tokens of 2048: 10.6 against
// 2.3 + 8.6 + 4.1 us and two gaps, the layer 97.2 -> 92.2 us.  What bounds it: shared memory (per 64-wide block 12 KB of terms
// and 16 KB of x are written and read by the MMAs) and, below 1000 tokens, the chain of first loads, sums and softmax.
#include "common.cuh"
#include "router_device.cuh"
#include "tensor_maps.cuh"
#include "umma.cuh"

namespace dsmoe {

namespace {

constexpr int kRuM = 128, kRuK = 64, kRuTeams = 4, kRuWarps = 16, kRuThreads = 64 + 32 * kRuWarps;

template <int EP>
struct RuGeo {
    static constexpr int N = 3 * EP;
    static constexpr int A_BYTES = kRuM * kRuK * 2, B_BYTES = N * kRuK * 2;
    static constexpr int STA = 6, STB = EP == 32 ? 8 : 4;           // slots of x and of Wr's terms
    static constexpr int RING = STA * A_BYTES + STB * B_BYTES;      // 192 KB
    static constexpr int LD = EP + 1;                              // floats per token of the partial logits (in the idle ring)
    static constexpr int ACCS = EP == 32 ? 5 : 2;                   // accumulators side by side in the 512 TMEM columns
    static constexpr uint32_t TMEM = 512;
    static_assert(kRuM * LD * 4 <= RING, "the partial logits take the ring's place");
};

struct RuShared {
    uint64_t full_a[6], empty_a[6], full_b[8], empty_b[8], done;
    uint32_t tmem_base;
    volatile int abort_flag;
    uint64_t mask_s[kRuM];
};

template <int EP>
constexpr size_t router_umma_smem() { return 1024 + (size_t)RuGeo<EP>::RING + sizeof(RuShared); }

__device__ __forceinline__ float ld_cluster(uint32_t addr) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}

template <int EP, int C>
__global__ void __launch_bounds__(kRuThreads, 1)
router_umma_kernel(const __grid_constant__ CUtensorMap tmX, const float* Wr, const float* br,
                   float* __restrict__ scores, uint64_t* __restrict__ mask, int32_t* __restrict__ k_t,
                   int32_t* __restrict__ chunk_counts, int T, int d, const SelParams q, int32_t* __restrict__ dev_status, const ZeroInts zero) {
    using G = RuGeo<EP>;
    extern __shared__ uint8_t ru_smem[];
    const uint32_t raw = ptx::smem_u32(ru_smem), base = (raw + 1023u) & ~1023u;
    RuShared& sh = *reinterpret_cast<RuShared*>(ru_smem + (base - raw) + G::RING);
    const uint32_t smA = base, smB = base + G::STA * G::A_BYTES;
    unsigned char* const pB = ru_smem + (base - raw) + G::STA * G::A_BYTES;
    float* const part = reinterpret_cast<float*>(ru_smem + (base - raw));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = (int)ptx::cluster_ctarank(), tile = (int)blockIdx.x / C;
    const int nk = d / kRuK / C, kb0 = rank * nk;
    const int run = (nk + G::ACCS - 1) / G::ACCS;        // blocks per accumulator

    if (threadIdx.x == 0) {
        for (int s = 0; s < G::STA; ++s) {
            ptx::mbar_init(ptx::smem_u32(&sh.full_a[s]), 1);
            ptx::mbar_init(ptx::smem_u32(&sh.empty_a[s]), 1);
        }
        for (int s = 0; s < G::STB; ++s) {
            ptx::mbar_init(ptx::smem_u32(&sh.full_b[s]), kRuWarps / kRuTeams);
            ptx::mbar_init(ptx::smem_u32(&sh.empty_b[s]), 1);
        }
        ptx::mbar_init(ptx::smem_u32(&sh.done), 1);
#ifdef DSMOE_TEST_GIVE_UP_RANK      // a build for the tests: this rank's CTAs behave as if a wait had run out
        sh.abort_flag = rank == DSMOE_TEST_GIVE_UP_RANK;
#else
        sh.abort_flag = 0;
#endif
        ptx::fence_barrier_init();
        ptx::prefetch_tensormap(&tmX);
    }
    if (warp == 1) {
        ptx::tmem_alloc(ptx::smem_u32(&sh.tmem_base), G::TMEM);
        ptx::tmem_relinquish();
    }
    chain_next();
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = sh.tmem_base;
    chain_wait();
    zero_ints(zero);

    if (warp == 0) {
        if (ptx::elect_one()) {
            for (int n = 0; n < nk; ++n) {
                const int s = n % G::STA;
                if (!ptx::mbar_wait(ptx::smem_u32(&sh.empty_a[s]), ((uint32_t)(n / G::STA) & 1u) ^ 1u, &sh.abort_flag)) break;
                const uint32_t bar = ptx::smem_u32(&sh.full_a[s]);
                ptx::mbar_expect_tx(bar, G::A_BYTES);
                ptx::tma_load_2d(smA + s * G::A_BYTES, &tmX, bar, (kb0 + n) * kRuK, tile * kRuM);
            }
        }
    } else if (warp == 1) {
        if (ptx::elect_one()) {
            const uint32_t idesc = ptx::make_idesc_bf16(kRuM, G::N);
            bool alive = true;
            uint32_t acc = tmem;
            for (int n = 0, in_run = 0; n < nk; ++n, ++in_run) {
                const int a = n % G::STA, b = n % G::STB;
                if (in_run == run) {                        // the next accumulator
                    in_run = 0;
                    acc += G::N;
                }
                if (!ptx::mbar_wait(ptx::smem_u32(&sh.full_b[b]), (uint32_t)(n / G::STB) & 1u, &sh.abort_flag) ||
                    !ptx::mbar_wait(ptx::smem_u32(&sh.full_a[a]), (uint32_t)(n / G::STA) & 1u, &sh.abort_flag)) {
                    alive = false;
                    break;
                }
                ptx::tc_fence_after();
#pragma unroll
                for (int k = 0; k < kRuK / 16; ++k)
                    ptx::umma_bf16(acc, ptx::make_desc_k_sw128(smA + a * G::A_BYTES + k * 32),
                                   ptx::make_desc_k_sw128(smB + b * G::B_BYTES + k * 32), idesc, (uint32_t)((in_run | k) != 0));
                ptx::umma_commit(ptx::smem_u32(&sh.empty_a[a]));
                ptx::umma_commit(ptx::smem_u32(&sh.empty_b[b]));
            }
            if (alive) ptx::umma_commit(ptx::smem_u32(&sh.done));
        }
    } else {
        constexpr int PC = 8 / (kRuWarps / kRuTeams);                     // 16-byte pieces of a row per warp
        const int w = warp - 2, team = w % kRuTeams, c0 = (w / kRuTeams) * PC;
        for (int n = team; n < nk; n += kRuTeams) {
            const int s = n % G::STB;
            bool alive = true;
#pragma unroll
            for (int h = 0; h < EP / 32; ++h) {
                const int e = lane + 32 * h;
                const float* src = Wr + (size_t)((kb0 + n) * kRuK + c0 * 8) * q.E + e;
                float v[8 * PC];
#pragma unroll
                for (int i = 0; i < 8 * PC; ++i) v[i] = e < q.E ? src[(size_t)i * q.E] : 0.f;
                if (h == 0 && !ptx::mbar_wait(ptx::smem_u32(&sh.empty_b[s]), ((uint32_t)(n / G::STB) & 1u) ^ 1u, &sh.abort_flag)) {
                    alive = false;
                    break;
                }
                unsigned char* const row0 = pB + s * G::B_BYTES + e * 128;
#pragma unroll
                for (int c = 0; c < PC; ++c) {
                    // (cut off, not rounded: the terms are just as exact, and a mask and a subtraction each)
                    uint32_t t1[4], t2[4], t3[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        uint32_t a[2], b[2], g[2];
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            a[u] = __float_as_uint(v[8 * c + 2 * i + u]);
                            const float r1 = v[8 * c + 2 * i + u] - __uint_as_float(a[u] & 0xffff0000u);
                            b[u] = __float_as_uint(r1);
                            g[u] = __float_as_uint(r1 - __uint_as_float(b[u] & 0xffff0000u));
                        }
                        t1[i] = __byte_perm(a[0], a[1], 0x7632);
                        t2[i] = __byte_perm(b[0], b[1], 0x7632);
                        t3[i] = __byte_perm(g[0], g[1], 0x7632);
                    }
                    const int at = ((c0 + c) ^ (e & 7)) * 16;           // EP is a multiple of 8: the same for all three terms
                    *reinterpret_cast<uint4*>(row0 + at) = make_uint4(t1[0], t1[1], t1[2], t1[3]);
                    *reinterpret_cast<uint4*>(row0 + EP * 128 + at) = make_uint4(t2[0], t2[1], t2[2], t2[3]);
                    *reinterpret_cast<uint4*>(row0 + 2 * EP * 128 + at) = make_uint4(t3[0], t3[1], t3[2], t3[3]);
                }
            }
            if (__any_sync(0xffffffffu, !alive)) break;
            ptx::fence_proxy_async();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&sh.full_b[s]));
        }
        // this CTA's sums, (s1 + s2) + s3 per expert and accumulator: four warps per TMEM lane quarter, a quarter of the experts each
        constexpr int EW = EP / (kRuWarps / 4);
        const int qd = warp & 3, row = qd * 32 + lane;
        const bool ok = !__any_sync(0xffffffffu, !ptx::mbar_wait(ptx::smem_u32(&sh.done), 0u, &sh.abort_flag));
        if (ok) {
            ptx::tc_fence_after();
#pragma unroll
            for (int e0 = (w >> 2) * EW, h = 0; h < EW / 8; ++h, e0 += 8) {
                float sum[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) sum[i] = 0.f;
#pragma unroll
                for (int a0 = 0; a0 < G::ACCS; a0 += 3) {        // three accumulators' reads at a time
                    uint32_t v[3][3][8];
#pragma unroll
                    for (int a = 0; a < 3; ++a)
#pragma unroll
                        for (int g = 0; g < 3; ++g)
                            if (a0 + a < G::ACCS)
                                ptx::tmem_ld8(tmem + ((uint32_t)(qd * 32) << 16) + (uint32_t)((a0 + a) * G::N + g * EP + e0), v[a][g]);
                    ptx::tmem_ld_wait();
#pragma unroll
                    for (int a = 0; a < 3; ++a)
                        if (a0 + a < G::ACCS && (a0 + a) * run < nk)
#pragma unroll
                            for (int i = 0; i < 8; ++i)
                                sum[i] += (__uint_as_float(v[a][0][i]) + __uint_as_float(v[a][1][i])) + __uint_as_float(v[a][2][i]);
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) part[row * G::LD + e0 + i] = sum[i];
            }
            ptx::tc_fence_before();
        }
    }
    ptx::cluster_sync();                               // every rank's partial logits are in place
    // A rank whose wait ran out has no sums to add: the tokens of its cluster then have no scores.  They become NaN, which
    // dsmoe_router's caller sees (it gets no status word), and select nothing.
    bool gave_up = false;
#pragma unroll
    for (int r = 0; r < C; ++r)
        gave_up |= __float_as_int(ld_cluster(ptx::map_to_cta(ptx::smem_u32(const_cast<int*>(&sh.abort_flag)), (uint32_t)r))) != 0;
    if (warp >= 2) {
        const int w = warp - 2, per = kRuM / C, first = rank * per;
        const bool v_lo = lane < q.E, v_hi = lane + 32 < q.E;
        const float b_lo = br && v_lo ? br[lane] : 0.f, b_hi = br && v_hi ? br[lane + 32] : 0.f;
        // a warp's 128 / 16 / C tokens: every rank's sums of all of them are asked for before the first is used
        constexpr int NT = kRuM / kRuWarps;
        float lo[NT], hi[NT];
#pragma unroll
        for (int j = 0; j < NT; ++j) {                 // j = token * C + rank
            const int tl = first + w + (j / C) * kRuWarps, r = j % C;
            const uint32_t at = ptx::map_to_cta(ptx::smem_u32(part + tl * G::LD + lane), (uint32_t)r);
            lo[j] = v_lo ? ld_cluster(at) : 0.f;
            hi[j] = EP > 32 && v_hi ? ld_cluster(at + 128) : 0.f;
        }
#pragma unroll 1
        for (int i = 0; i < NT / C; ++i) {
            const int t = tile * kRuM + first + w + i * kRuWarps;
            float l_lo = 0.f, l_hi = 0.f;
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                if (j / C == i) {
                    l_lo += lo[j];
                    l_hi += hi[j];
                }
            }
            if (br) {
                l_lo += b_lo;
                l_hi += b_hi;
            }
            uint64_t m = 0;
            if (t < T && !gave_up) m = softmax_select_store(l_lo, l_hi, t, q, lane, scores, mask, k_t);
            if (t < T && gave_up) {
                if (v_lo) scores[(size_t)t * q.E + lane] = __int_as_float(0x7fffffff);
                if (v_hi) scores[(size_t)t * q.E + lane + 32] = __int_as_float(0x7fffffff);
                if (lane == 0 && mask) mask[t] = 0;
                if (lane == 0 && k_t) k_t[t] = 0;
            }
            if (lane == 0) sh.mask_s[w + i * kRuWarps] = m;
        }
        if (chunk_counts) {
            asm volatile("bar.sync 1, %0;" ::"n"(32 * kRuWarps) : "memory");
            const int chunk = (tile * kRuM + first) / kChunk + w;
            if (w < per / kChunk && chunk * kChunk < T) {
                const uint64_t mt = sh.mask_s[w * kChunk + lane];
                int c_lo = 0, c_hi = 0;
                for (int e = 0; e < q.E; ++e) {
                    const int n = __popc(__ballot_sync(0xffffffffu, (mt >> e) & 1));
                    if (lane == (e & 31)) {
                        if (e < 32) c_lo = n; else c_hi = n;
                    }
                }
                if (v_lo) chunk_counts[(size_t)chunk * q.E + lane] = c_lo;
                if (v_hi) chunk_counts[(size_t)chunk * q.E + lane + 32] = c_hi;
            }
        }
    }
    if (gave_up && threadIdx.x == 0) {                 // copies and MMAs already issued still land in this CTA's memory
        const uint64_t t0 = ptx::globaltimer_ns();
        while (ptx::globaltimer_ns() - t0 < 200000ull) {
        }
    }
    ptx::tc_fence_before();
    ptx::cluster_sync();                               // nobody leaves while another rank may read its sums
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem, G::TMEM);
    }
    if (threadIdx.x == 0 && gave_up) report_status(dev_status, DSMOE_ERR_TIMEOUT);
}

template <int EP, int C>
dsmoe_status launch_clusters(const dsmoe_layer_desc& p, const CUtensorMap& mX, const float* Wr, const float* br, float* scores,
                             uint64_t* mask, int32_t* k_t, int32_t* chunk_counts, int32_t* dev_status, cudaStream_t s, const ZeroInts& zero) {
    static bool attr[kMaxDeviceSlots] = {};
    int dev = 0;
    DeviceState* st = nullptr;
    DSMOE_TRY(device_state(&st, &dev));
    if (!attr[dev]) {
        DSMOE_CUDA_TRY(cudaFuncSetAttribute(router_umma_kernel<EP, C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)router_umma_smem<EP>()));
        attr[dev] = true;
    }
    DSMOE_CUDA_TRY(launch_chained_clusters(router_umma_kernel<EP, C>, ceil_div(p.T, kRuM) * C, kRuThreads, router_umma_smem<EP>(), s, C, true,
        mX, Wr, br, scores, mask, k_t, chunk_counts, p.T, p.d, SelParams{p.E, p.mode, p.eps, p.eps_normalized, p.K, p.min_k, nullptr},
        dev_status, zero));
    return DSMOE_OK;
}

// How many CTAs share out a row tile's reduction over d.  With few row tiles 2 or 4, so that the launch covers most SMs;
// `max_run` > 0 also keeps an accumulator's run of 64-wide blocks that short.  0: no such number.
template <int EP>
int clusters_of(const dsmoe_layer_desc& p, int max_run) {
    const int row_tiles = ceil_div(p.T, kRuM), blocks = p.d / kRuK;
    int C = 4;
    while (C > 1 && (row_tiles * C > sm_count() || blocks % C)) C /= 2;
    while (max_run > 0 && ceil_div(blocks / C, RuGeo<EP>::ACCS) > max_run) {
        C *= 2;
        if (C > 4 || blocks % C) return 0;
    }
    return C;
}

template <int EP>
dsmoe_status launch_ep(const dsmoe_layer_desc& p, int max_run, const CUtensorMap& mX, const float* Wr, const float* br, float* scores,
                       uint64_t* mask, int32_t* k_t, int32_t* chunk_counts, int32_t* dev_status, cudaStream_t s, const ZeroInts& zero) {
    switch (clusters_of<EP>(p, max_run)) {
        case 4: return launch_clusters<EP, 4>(p, mX, Wr, br, scores, mask, k_t, chunk_counts, dev_status, s, zero);
        case 2: return launch_clusters<EP, 2>(p, mX, Wr, br, scores, mask, k_t, chunk_counts, dev_status, s, zero);
        case 1: return launch_clusters<EP, 1>(p, mX, Wr, br, scores, mask, k_t, chunk_counts, dev_status, s, zero);
        default: return DSMOE_ERR_UNSUPPORTED;
    }
}

}  // namespace

bool router_umma_supported(const dsmoe_layer_desc& p, int max_run) {
    return umma_supported(p) && p.T > 256 && (p.E <= 32 ? clusters_of<32>(p, max_run) : clusters_of<64>(p, max_run)) > 0;
}

dsmoe_status launch_router_umma(const dsmoe_layer_desc& p, const void* x, const float* Wr, const float* br, float* scores,
                                uint64_t* mask, int32_t* k_t, int32_t* dev_status, cudaStream_t s, int32_t* chunk_counts,
                                int max_run, const ZeroInts& zero) {
    CUtensorMap mX;
    DSMOE_TRY(cached_map_2d(&mX, x, p.T, p.d, kRuM));
    return p.E <= 32 ? launch_ep<32>(p, max_run, mX, Wr, br, scores, mask, k_t, chunk_counts, dev_status, s, zero)
                     : launch_ep<64>(p, max_run, mX, Wr, br, scores, mask, k_t, chunk_counts, dev_status, s, zero);
}

}  // namespace dsmoe
