// What the tensor-core kernels of the expert MLPs share: tile sizes, the operand ring, GeLU, the weight tiles' copies and the
// bounded wait on a flag in global memory.
#pragma once

#include "common.cuh"
#include "tensor_maps.cuh"
#include "umma.cuh"

namespace dsmoe {

constexpr int BM = 128, BK = 64, BN = 256, STAGES = 4;
constexpr int A_STAGE_BYTES = BM * BK * 2;
constexpr int B_STAGE_BYTES = BN * BK * 2;
constexpr int NUM_THREADS = 192;      // producer, MMA issuer, four epilogue warps
constexpr int GATHER_WARPS = 8;
constexpr int GATHER_THREADS = NUM_THREADS + 32 * GATHER_WARPS;   // ... and more warps that gather the rows of A
constexpr int TMEM_COLS = 512;
constexpr int RING_BYTES = STAGES * (A_STAGE_BYTES + B_STAGE_BYTES);   // operand ring: 4 x 48 KB, or more, smaller slots

// GeLU(v) = v Phi(v) with the exact Phi (the erf form, not the tanh form).  Phi comes from Abramowitz & Stegun's
// rational approximation 7.1.28, erfc(z) = (1 + a1 z + ... + a6 z^6)^-16 with |error| <= 3e-7 for z >= 0 -- three
// orders below the bf16 rounding of the result: Phi(v) = erfc(|v| / sqrt 2) / 2 for v < 0 and 1 minus that for
// v >= 0, so the negative tail has no cancellation.  Six FMAs, one reciprocal, four squarings: about half the
// instructions of erff, which matters because the GeLU epilogue of a tile costs the CUDA cores nearly as many issue
// slots as its mainloop costs the tensor core.
__device__ __forceinline__ float gelu_erf(float v) {
    const float z = fabsf(v) * 0.70710678118654752440f;
    float p = fmaf(z, 0.0000430638f, 0.0002765672f);
    p = fmaf(z, p, 0.0001520143f);
    p = fmaf(z, p, 0.0092705272f);
    p = fmaf(z, p, 0.0422820123f);
    p = fmaf(z, p, 0.0705230784f);
    p = fmaf(z, p, 1.f);
    float q;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(q) : "f"(p));   // p >= 1: one unit in the last place is plenty
    q *= q;
    q *= q;
    q *= q;
    q *= q;
    const float tail = 0.5f * q;                    // Phi(-|v|)
    return v * (v < 0.f ? tail : 1.f - tail);
}

// The packed weights are block-major along the reduction: [E][k / 64][n][64], so the tile (64 k, rows n0..) of
// reduction block kb is the `rows` consecutive 128-byte rows starting at wrow(kb, n0, N) of a [E][(K/64)*N][64]
// tensor: one contiguous piece of memory.
__device__ __forceinline__ int wrow(int kb, int n0, int N) { return kb * N + n0; }

// Weight rows [row0, row0 + rows) of expert e (see wrow): power-of-two boxes, largest first.
template <bool PAIR = false>
__device__ __forceinline__ void load_weight_rows(const BMaps* maps, uint32_t dst, uint32_t bar, int row0, int rows,
                                                 int e, int x0 = 0) {
    int done = 0;
#pragma unroll
    for (int lvl = 4; lvl >= 0; --lvl) {
        if ((rows - done) >= (16 << lvl)) {
            if (PAIR) ptx::tma_load_3d_pair(dst + done * (BK * 2), &maps->m[lvl], bar, x0, row0 + done, e);
            else ptx::tma_load_3d(dst + done * (BK * 2), &maps->m[lvl], bar, x0, row0 + done, e);
            done += 16 << lvl;
        }
    }
}

// Bounded wait until the int at `flag` (written by other CTAs with a release fence before it) is at least
// `target`.  false = gave up (limit reached, or another thread of the CTA already had).
__device__ __forceinline__ bool flag_wait_ge(const int* flag, int target, volatile int* abort_flag) {
    uint64_t t0 = 0;
    for (uint32_t spin = 1;; ++spin) {
        int v;
        asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(flag) : "memory");
        if (v >= target) return true;
        if ((spin & 0x3f) == 0) {
            if (*abort_flag) return false;
            const uint64_t now = ptx::globaltimer_ns();
            if (t0 == 0) t0 = now;
            if (now - t0 > ptx::kWaitLimitNs) {
                *abort_flag = 1;
                return false;
            }
        }
    }
}

}  // namespace dsmoe
