// Mixture-of-attention-heads layer (Eq. 7-8): the attention step between the two grouped projections.
//
// The layer is the feed-forward layer's pipeline with another middle: router, selection and grouping as there; the
// "up-projection" is the experts' query projection (no activation), the "down-projection" their output projection
// with the router-weighted sum of Eq. 8; in between every grouped row -- one (token, expert) pair, n_head query
// vectors of d_head -- attends to the keys and values of its token's sequence, head j to key/value head j
// (the keys and values are shared by all experts).  This file holds that middle step.
#include <climits>
#include <cstdlib>

#include "common.cuh"
#include "tensor_maps.cuh"
#include "umma.cuh"

namespace dsmoe {

namespace {

constexpr int kMoaWarps = 4;

__device__ __forceinline__ float bf16_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t u) { return __uint_as_float(u & 0xffff0000u); }

// One warp per (grouped row, head).  Pass 1: the lanes share out the visible keys, each key's logit is a full dot
// product of the query (fp32, in shared memory) with the key's row (read in 16-byte pieces); logits go to shared
// memory.  Then max, exponentials and their sum.  Pass 2: the lanes share out the d_head dimensions (lane l owns
// l, l + 32, ...) and walk the keys, so a value row is read by the whole warp at once.  The result replaces the
// query in place (the warp has read all of it before it writes).
template <int DPL>   // d_head / 32
__global__ void __launch_bounds__(32 * kMoaWarps)
moa_attention_kernel(__nv_bfloat16* __restrict__ qa, const int32_t* row_token, const int32_t* offsets,
                     int E, int n_head, int H, int T, const __nv_bfloat16* Kc, const __nv_bfloat16* Vc,
                     const int32_t* tok_seq, const int32_t* pos, int n_seq, int L, float scale,
                     int* __restrict__ dev_status) {
    chain_wait();
    constexpr int DH = 32 * DPL;
    extern __shared__ float moa_smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float* qs = moa_smem + warp * (DH + ((L + 3) & ~3));     // the query, then the logits / probabilities
    float* ws = qs + DH;
    const long long A = offsets[E];
    const long long pair = (long long)blockIdx.x * kMoaWarps + warp;
    if (pair >= A * n_head) return;
    const long long r = pair / n_head;
    const int j = (int)(pair % n_head);
    int t = row_token[r];
    bool bad = t < 0 || t >= T;
    t = min(max(t, 0), T - 1);
    int sq = tok_seq ? tok_seq[t] : 0, last = pos[t];
    bad = bad || sq < 0 || sq >= n_seq || last < 0 || last >= L;
    if (bad) {                                        // report, and stay inside the cache
        if (lane == 0) report_status(dev_status, DSMOE_ERR_INVALID_ARG);
        sq = min(max(sq, 0), n_seq - 1);
        last = min(max(last, 0), L - 1);
    }
    __nv_bfloat16* qrow = qa + r * H + j * DH;
#pragma unroll
    for (int i = 0; i < DPL; ++i) qs[lane + 32 * i] = __bfloat162float(qrow[lane + 32 * i]);
    __syncwarp();
    const __nv_bfloat16* Kh = Kc + ((size_t)(sq * n_head + j) * L) * DH;
    const __nv_bfloat16* Vh = Vc + ((size_t)(sq * n_head + j) * L) * DH;
    float mx = -INFINITY;
    for (int k = lane; k <= last; k += 32) {
        const uint4* kr = reinterpret_cast<const uint4*>(Kh + (size_t)k * DH);
        float dot = 0.f;
#pragma unroll
        for (int c = 0; c < DH / 8; ++c) {
            const uint4 u = kr[c];
            const float4 q0 = *reinterpret_cast<const float4*>(qs + 8 * c), q1 = *reinterpret_cast<const float4*>(qs + 8 * c + 4);
            dot = fmaf(q0.x, bf16_lo(u.x), dot);
            dot = fmaf(q0.y, bf16_hi(u.x), dot);
            dot = fmaf(q0.z, bf16_lo(u.y), dot);
            dot = fmaf(q0.w, bf16_hi(u.y), dot);
            dot = fmaf(q1.x, bf16_lo(u.z), dot);
            dot = fmaf(q1.y, bf16_hi(u.z), dot);
            dot = fmaf(q1.z, bf16_lo(u.w), dot);
            dot = fmaf(q1.w, bf16_hi(u.w), dot);
        }
        dot *= scale;
        ws[k] = dot;
        mx = fmaxf(mx, dot);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    float den = 0.f;
    for (int k = lane; k <= last; k += 32) {
        const float p = expf(ws[k] - mx);
        ws[k] = p;
        den += p;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) den += __shfl_xor_sync(0xffffffffu, den, o);
    __syncwarp();
    float acc[DPL];
#pragma unroll
    for (int i = 0; i < DPL; ++i) acc[i] = 0.f;
    for (int k = 0; k <= last; ++k) {
        const float p = ws[k];
        const __nv_bfloat16* vr = Vh + (size_t)k * DH + lane;
#pragma unroll
        for (int i = 0; i < DPL; ++i) acc[i] = fmaf(p, __bfloat162float(vr[32 * i]), acc[i]);
    }
    chain_next();
    const float inv = 1.f / den;
#pragma unroll
    for (int i = 0; i < DPL; ++i) qrow[lane + 32 * i] = __float2bfloat16_rn(acc[i] * inv);
}

// ---------------------------------------------------------------- the same step on the warp-level tensor-core path
//
// One CTA per (token, head, tile of up to 16 of the token's grouped rows): the rows of a token share its keys and
// values, and 16 rows are exactly the M of an m16n8k16 MMA.  The 8 warps share out the visible keys in blocks of 32:
// a warp copies its block of K and V into (padded, conflict-free) shared memory, forms S = Q.K^T (Q fragments stay
// in registers for the whole kernel), updates the running row maxima and sums, rescales its accumulators and adds
// P.V with P taken straight from S's registers -- the usual streaming-softmax order.  The warps' partial results
// (maximum, sum, accumulator per row) are merged through shared memory at the end, in warp order.  Exponentials are
// the fast ones (ex2.approx of the argument times log2 e): the weights are rounded to bf16 before P.V anyway.
constexpr int kKeyBlock = 32;
#ifndef DSMOE_MOA_MINBLOCKS
#define DSMOE_MOA_MINBLOCKS 6
#endif

__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

constexpr int kTileMaxKeys = 512;  // caches up to this many positions: a warp walks all keys of its tile; longer ones: 8 warps share them out
constexpr int kShWarps = 4;        // tiles of a CTA that share their copies of the keys (moa_attention_shared_kernel)

struct AttnArgs {
    __nv_bfloat16* qa;
    const int32_t* token_rows;
    int W, row_tiles, tpt;      // rows of a token, 16-row tiles they take, tokens of a tile
    int group_tpt;              // ... of the shared-key kernel's tiles, whatever this launch's are
    long long amax;
    int n_head, H, T;
    const __nv_bfloat16 *Kc, *Vc;
    const int32_t *tok_seq, *pos;
    int n_seq, L;
    float scale;
    int* dev_status;
    bool leave_mixed;           // mixed groups are another launch's
    // With `dense`, the outputs go to dense[T][E * H] instead: expert e's columns e * H .. of token t hold its gate times its
    // attention output, zeros where the token did not select e (these zeros are the shared-key kernel's)
    __nv_bfloat16* dense;
    int E;
    const uint64_t* mask;
    const float* row_gate;
};

// The expert of a token's slot-th grouped row (its selected experts ascend); -1: the token has fewer
__device__ __forceinline__ int expert_of_slot(uint64_t selected, int slot) {
    for (; slot > 0; --slot) selected &= selected - 1;
    return __ffsll((long long)selected) - 1;
}

// Four neighbouring tiles are a mixed group if some token's sequence is neither the first token's nor the last one's: decoding
// sequences side by side, or tokens in no order of sequences.  They share no keys.
__device__ __forceinline__ void group_tokens(const AttnArgs& P, int group, int& t0, int& t1) {
    t0 = (group * kShWarps / P.row_tiles) * P.group_tpt;
    t1 = min(P.T, ((group * kShWarps + kShWarps - 1) / P.row_tiles) * P.group_tpt + P.group_tpt);
}
// Whether token u makes tokens a .. b - 1 mixed.  Every kernel asks here: a group is attended by exactly one launch, which puts its outputs
// where the queries were.
template <typename Seq>
__device__ __forceinline__ bool mixes(const Seq& seq, int a, int b, int u) {
    const int sq = seq(u);
    return sq != seq(a) && sq != seq(b - 1);
}
__device__ __forceinline__ int seq_of(const AttnArgs& P, int t) { return P.tok_seq ? min(max(P.tok_seq[t], 0), P.n_seq - 1) : 0; }

template <int DH, int kMmaWarps, bool MIXED>      // long caches: 8 warps share out the keys; short ones: 2, and several CTAs fit an SM
__global__ void __launch_bounds__(32 * kMmaWarps, kMmaWarps == 2 ? DSMOE_MOA_MINBLOCKS : 1)
moa_attention_mma_kernel(__nv_bfloat16* __restrict__ qa, const int32_t* token_rows, int W, int row_tiles,
                         int tpt, long long amax, int n_head, int H, int T, const __nv_bfloat16* Kc,
                         const __nv_bfloat16* Vc, const int32_t* tok_seq,
                         const int32_t* pos, int n_seq, int L, float scale, long long n_tiles,
                         int* __restrict__ dev_status, const AttnArgs P /* MIXED only */) {
    chain_wait();
    constexpr int STRIDE = DH * 2 + 16;                 // bytes per key row in shared memory: 16 of padding
    constexpr int KS = DH / 16, DT = DH / 8, CH = DH / 8;
    extern __shared__ __align__(16) unsigned char moa_mma_smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, q4 = lane & 3;
    // The tile's 16 rows: with tpt == 1, slots 16 rt .. of token t0; with tpt > 1 (rows per token W <= 8, one row
    // tile), all W slots of the tpt tokens t0, t0 + 1, ...: neighbouring tokens of one sequence see nearly the same
    // keys, so their rows share the copies of K and V.
    // The CTAs are persistent (as many as fit the GPU at once) and walk the tiles: a tile is short, and starting a CTA per
    // tile cost more than the tile's work.
    // With 8 warps (long caches, few tiles) the warps of a CTA share out the KEYS of one tile and merge their partial
    // results at the end; with 2 warps (short caches, many tiles) each warp takes a tile of its OWN, walks all its
    // keys and writes its result straight from registers: no merge, no CTA-wide barrier.
    constexpr bool SPLIT = kMmaWarps > 2;
    constexpr int TW = SPLIT ? 1 : kMmaWarps;           // tiles a CTA works on at a time
    static_assert(SPLIT || !MIXED, "the tile loop must be the same for the whole CTA");
    __shared__ int found_s;
    // MIXED: the tiles of mixed groups alone; every thread looks at one of the CTA's next tiles
    const auto next_tile = [&](long long from) {
        if (!MIXED) return from;
        for (; from < n_tiles; from += (long long)gridDim.x * blockDim.x) {
            const long long mine = from + (long long)gridDim.x * threadIdx.x;
            bool mixed = false;
            if (mine < n_tiles) {
                int a, b;
                const int tt = (int)(mine / ((long long)row_tiles * n_head)) * tpt;
                group_tokens(P, (tt / P.group_tpt * row_tiles + (int)(mine % row_tiles)) / kShWarps, a, b);
                const auto seq = [&](int t) { return seq_of(P, t); };
                for (int u = a + 1; u + 1 < b; ++u) mixed = mixed || mixes(seq, a, b, u);
            }
            if (threadIdx.x == 0) found_s = INT_MAX;
            __syncthreads();
            if (mixed) atomicMin(&found_s, (int)threadIdx.x);
            __syncthreads();
            const int found = found_s;
            __syncthreads();
            if (found != INT_MAX) return from + (long long)gridDim.x * found;
        }
        return from;
    };
    for (long long tile = next_tile((long long)blockIdx.x * TW + (SPLIT ? 0 : warp)); tile < n_tiles;
         tile = next_tile(tile + (long long)gridDim.x * TW)) {
    if (SPLIT) __syncthreads();                         // the previous tile's merge has read shared memory
    const int rt = (int)(tile % row_tiles);
    const int j = (int)((tile / row_tiles) % n_head);
    const int t0 = (int)(tile / ((long long)row_tiles * n_head)) * tpt;
    const auto row_token_slot = [&](int i, int& tok, int& slot) {
        if (tpt == 1) {
            tok = t0;
            slot = rt * 16 + i;
        } else {
            tok = t0 + i / W;
            slot = i % W;
            if (i >= tpt * W) tok = T;
        }
    };
    // this thread's two rows of the tile (g and g + 8): grouped row (-1 = none), token, last visible key
    int r0 = -1, r1 = -1, tk0, tk1, sl0, sl1, last0 = 0, last1 = 0;
    row_token_slot(g, tk0, sl0);
    row_token_slot(g + 8, tk1, sl1);
    if (tk0 < T && sl0 < W) r0 = token_rows[(size_t)tk0 * W + sl0];
    if (tk1 < T && sl1 < W) r1 = token_rows[(size_t)tk1 * W + sl1];
    if (r0 >= amax) r0 = -1;
    if (r1 >= amax) r1 = -1;
    if ((SPLIT ? __syncthreads_or(r0 >= 0 || r1 >= 0) : (int)__any_sync(0xffffffffu, r0 >= 0 || r1 >= 0)) == 0) continue;   // no rows in this tile
    bool bad = false;
    if (r0 >= 0) {
        last0 = pos[tk0];
        bad = bad || last0 < 0 || last0 >= L;
        last0 = min(max(last0, 0), L - 1);
    }
    if (r1 >= 0) {
        last1 = pos[tk1];
        bad = bad || last1 < 0 || last1 >= L;
        last1 = min(max(last1, 0), L - 1);
    }
    // the tokens of the tile: one pass over the keys if they all belong to one sequence, else one pass per token
    const int ntok = min(tpt, T - t0);
    int seq_first = tok_seq ? tok_seq[t0] : 0;
    bool same = true;
    for (int u = 1; u < ntok; ++u) same = same && (tok_seq ? tok_seq[t0 + u] : 0) == seq_first;
    const int npass = same ? 1 : ntok;
    // Q fragments (the A operand of S = Q.K^T)
    uint32_t qf[KS][4];
#pragma unroll
    for (int ks = 0; ks < KS; ++ks) {
        const int c = j * DH + ks * 16 + q4 * 2;
        qf[ks][0] = r0 >= 0 ? *reinterpret_cast<const uint32_t*>(qa + (size_t)r0 * H + c) : 0u;
        qf[ks][1] = r1 >= 0 ? *reinterpret_cast<const uint32_t*>(qa + (size_t)r1 * H + c) : 0u;
        qf[ks][2] = r0 >= 0 ? *reinterpret_cast<const uint32_t*>(qa + (size_t)r0 * H + c + 8) : 0u;
        qf[ks][3] = r1 >= 0 ? *reinterpret_cast<const uint32_t*>(qa + (size_t)r1 * H + c + 8) : 0u;
    }
    constexpr int KB = SPLIT ? kKeyBlock / 2 : kKeyBlock;     // keys per block (SPLIT: two buffers of half a block each)
    unsigned char* const Ks0 = moa_mma_smem + (size_t)warp * 2 * kKeyBlock * STRIDE;
    float m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;
    float o[DT][4];
#pragma unroll
    for (int i = 0; i < DT; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
    for (int ps = 0; ps < npass; ++ps) {
    // this pass: the sequence whose keys are walked, the rows that take part, the last key any of them sees
    int sq = same ? seq_first : (tok_seq ? tok_seq[t0 + ps] : 0);
    bad = bad || sq < 0 || sq >= n_seq;
    sq = min(max(sq, 0), n_seq - 1);
    const bool act0 = r0 >= 0 && (same || tk0 == t0 + ps), act1 = r1 >= 0 && (same || tk1 == t0 + ps);
    int last = 0;
    for (int u = same ? 0 : ps; u < (same ? ntok : ps + 1); ++u) last = max(last, min(max(pos[t0 + u], 0), L - 1));
    const __nv_bfloat16* Kh = Kc + ((size_t)(sq * n_head + j) * L) * DH;
    const __nv_bfloat16* Vh = Vc + ((size_t)(sq * n_head + j) * L) * DH;
    // Sharing out one tile's keys (SPLIT), a warp walks blocks of KB = 16 keys through two buffers: the copies of its
    // next block are under way while it works on this one (with one buffer of 32 keys and a wait right behind the
    // copies, the decode shape's step took 35 us for 134 MB of keys and values).  A tile per warp: one buffer of 32.
    const int nblocks = last / KB + 1;
    const auto fetch = [&](int b, unsigned char* Kb, unsigned char* Vb) {
        const int key0 = b * KB, nk = min(KB, last + 1 - key0);
#pragma unroll
        for (int i = 0; i < CH * KB / 32; ++i) {        // KB rows x CH 16-byte pieces, a piece per lane and step
            const int idx = lane + 32 * i, row = idx / CH, ch = idx % CH;
            // asynchronous 16-byte copies, all in flight at once; rows past the last visible key are filled with zeros
            const int rr = row < nk ? row : 0;
            const uint32_t nbytes = row < nk ? 16u : 0u;
            const uint32_t kd = (uint32_t)__cvta_generic_to_shared(Kb + row * STRIDE + ch * 16);
            const uint32_t vd = (uint32_t)__cvta_generic_to_shared(Vb + row * STRIDE + ch * 16);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(kd), "l"(Kh + (size_t)(key0 + rr) * DH + ch * 8), "r"(nbytes) : "memory");
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(vd), "l"(Vh + (size_t)(key0 + rr) * DH + ch * 8), "r"(nbytes) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    int buf = 0;
    if (SPLIT && warp < nblocks) {
        __syncwarp();
        fetch(warp, Ks0, Ks0 + KB * STRIDE);
    }
    for (int b = SPLIT ? warp : 0; b < nblocks; b += SPLIT ? kMmaWarps : 1) {
        const int key0 = b * KB;
        unsigned char* Ks = Ks0 + buf * 2 * KB * STRIDE;
        unsigned char* Vs = Ks + KB * STRIDE;
        if (SPLIT) {
            __syncwarp();              // the other buffer was last read an iteration ago: every lane is past those reads
            if (b + kMmaWarps < nblocks) {
                unsigned char* Kn = Ks0 + (buf ^ 1) * 2 * KB * STRIDE;
                fetch(b + kMmaWarps, Kn, Kn + KB * STRIDE);
                asm volatile("cp.async.wait_group 1;" ::: "memory");
            } else {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
            }
            buf ^= 1;
        } else {
            const int nk = min(KB, last + 1 - key0);
            __syncwarp();
#pragma unroll
            for (int i = 0; i < CH; ++i) {                  // 32 rows x CH 16-byte pieces, a piece per lane and step
                const int idx = lane + 32 * i, row = idx / CH, ch = idx % CH;
                const int rr = row < nk ? row : 0;
                const uint32_t nbytes = row < nk ? 16u : 0u;
                const uint32_t kd = (uint32_t)__cvta_generic_to_shared(Ks + row * STRIDE + ch * 16);
                const uint32_t vd = (uint32_t)__cvta_generic_to_shared(Vs + row * STRIDE + ch * 16);
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(kd), "l"(Kh + (size_t)(key0 + rr) * DH + ch * 8), "r"(nbytes) : "memory");
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(vd), "l"(Vh + (size_t)(key0 + rr) * DH + ch * 8), "r"(nbytes) : "memory");
            }
            asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
        }
        __syncwarp();
        float sc[KB / 8][4];
#pragma unroll
        for (int nt = 0; nt < KB / 8; ++nt) sc[nt][0] = sc[nt][1] = sc[nt][2] = sc[nt][3] = 0.f;
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) {
#pragma unroll
            for (int nt = 0; nt < KB / 8; ++nt) {
                const unsigned char* kp = Ks + (nt * 8 + g) * STRIDE + (ks * 16 + q4 * 2) * 2;
                mma_bf16_16816(sc[nt], qf[ks], *reinterpret_cast<const uint32_t*>(kp), *reinterpret_cast<const uint32_t*>(kp + 16));
            }
        }
        // scale, hide the keys past each row's position (and everything from rows not in this pass), new row maxima
        float bm0 = -INFINITY, bm1 = -INFINITY;
#pragma unroll
        for (int nt = 0; nt < KB / 8; ++nt) {
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int key = key0 + nt * 8 + q4 * 2 + c;
                sc[nt][c] = (act0 && key <= last0) ? sc[nt][c] * scale : -INFINITY;
                sc[nt][2 + c] = (act1 && key <= last1) ? sc[nt][2 + c] * scale : -INFINITY;
                bm0 = fmaxf(bm0, sc[nt][c]);
                bm1 = fmaxf(bm1, sc[nt][2 + c]);
            }
        }
        bm0 = fmaxf(bm0, __shfl_xor_sync(0xffffffffu, bm0, 1));
        bm0 = fmaxf(bm0, __shfl_xor_sync(0xffffffffu, bm0, 2));
        bm1 = fmaxf(bm1, __shfl_xor_sync(0xffffffffu, bm1, 1));
        bm1 = fmaxf(bm1, __shfl_xor_sync(0xffffffffu, bm1, 2));
        // a row that has seen no key yet (and sees none here) keeps m = -inf: nothing to rescale, nothing to add
        const float n0 = fmaxf(m0, bm0), n1 = fmaxf(m1, bm1);
        const float c0 = n0 == -INFINITY ? 1.f : __expf(m0 - n0), c1 = n1 == -INFINITY ? 1.f : __expf(m1 - n1);
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
        uint32_t pf[KB / 16][4];
#pragma unroll
        for (int nt = 0; nt < KB / 8; ++nt) {
            const float p0 = sc[nt][0] > -INFINITY ? __expf(sc[nt][0] - m0) : 0.f, p1 = sc[nt][1] > -INFINITY ? __expf(sc[nt][1] - m0) : 0.f;
            const float p2 = sc[nt][2] > -INFINITY ? __expf(sc[nt][2] - m1) : 0.f, p3 = sc[nt][3] > -INFINITY ? __expf(sc[nt][3] - m1) : 0.f;
            l0 += p0 + p1;
            l1 += p2 + p3;
            pf[nt / 2][(nt & 1) * 2] = pack_bf16(p0, p1);
            pf[nt / 2][(nt & 1) * 2 + 1] = pack_bf16(p2, p3);
        }
#pragma unroll
        for (int kk = 0; kk < KB / 16; ++kk) {
#pragma unroll
            for (int dt = 0; dt < DT; ++dt) {
                uint32_t b0, b1;
                const uint32_t addr = (uint32_t)__cvta_generic_to_shared(Vs + (kk * 16 + (lane & 15)) * STRIDE + dt * 16);
                asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0, %1}, [%2];" : "=r"(b0), "=r"(b1) : "r"(addr));
                mma_bf16_16816(o[dt], pf[kk], b0, b1);
            }
        }
    }
    }
    if (bad && lane == 0) report_status(dev_status, DSMOE_ERR_INVALID_ARG);             // clamped above: nothing left the cache
    l0 += __shfl_xor_sync(0xffffffffu, l0, 1);
    l0 += __shfl_xor_sync(0xffffffffu, l0, 2);
    l1 += __shfl_xor_sync(0xffffffffu, l1, 1);
    l1 += __shfl_xor_sync(0xffffffffu, l1, 2);
    if (!SPLIT) {
        // the warp has seen every key of its rows: normalise and write (the queries it replaces are in its registers)
        const float i0 = 1.f / l0, i1 = 1.f / l1;
#pragma unroll
        for (int dt = 0; dt < DT; ++dt) {
            const int c = j * DH + dt * 8 + q4 * 2;
            if (r0 >= 0) *reinterpret_cast<uint32_t*>(qa + (size_t)r0 * H + c) = pack_bf16(o[dt][0] * i0, o[dt][1] * i0);
            if (r1 >= 0) *reinterpret_cast<uint32_t*>(qa + (size_t)r1 * H + c) = pack_bf16(o[dt][2] * i1, o[dt][3] * i1);
        }
        continue;
    }
    // ---- merge the warps' partial results: per warp 16 maxima, 16 sums, 16 x DH accumulators
    __syncthreads();
    float* ms = reinterpret_cast<float*>(moa_mma_smem);                 // [warps][16]
    float* ls = ms + kMmaWarps * 16;                                    // [warps][16]
    float* os = ls + kMmaWarps * 16;                                    // [warps][16][DH]
    if (q4 == 0) {
        ms[warp * 16 + g] = m0;
        ms[warp * 16 + g + 8] = m1;
        ls[warp * 16 + g] = l0;
        ls[warp * 16 + g + 8] = l1;
    }
#pragma unroll
    for (int dt = 0; dt < DT; ++dt) {
        float* o0 = os + ((size_t)warp * 16 + g) * DH + dt * 8 + q4 * 2;
        float* o1 = os + ((size_t)warp * 16 + g + 8) * DH + dt * 8 + q4 * 2;
        o0[0] = o[dt][0];
        o0[1] = o[dt][1];
        o1[0] = o[dt][2];
        o1[1] = o[dt][3];
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < 16 * DH; idx += 32 * kMmaWarps) {
        const int row = idx / DH, dcol = idx % DH;
        int tok, slot;
        row_token_slot(row, tok, slot);
        if (tok >= T || slot >= W) continue;
        const int r = token_rows[(size_t)tok * W + slot];
        if (r < 0 || r >= amax) continue;
        float M = -INFINITY;
#pragma unroll
        for (int w = 0; w < kMmaWarps; ++w) M = fmaxf(M, ms[w * 16 + row]);
        float num = 0.f, den = 0.f;
#pragma unroll
        for (int w = 0; w < kMmaWarps; ++w) {
            const float wgt = __expf(ms[w * 16 + row] - M);               // 0 for a warp that saw no key
            num = fmaf(wgt, os[((size_t)w * 16 + row) * DH + dcol], num);
            den = fmaf(wgt, ls[w * 16 + row], den);
        }
        if (!MIXED || !P.dense) {
            qa[(size_t)r * H + j * DH + dcol] = __float2bfloat16_rn(num / den);
        } else if (const int e = expert_of_slot(P.mask[tok], slot); e >= 0) {
            P.dense[((size_t)tok * P.E + e) * H + j * DH + dcol] = __float2bfloat16_rn(num / den * P.row_gate[r]);
        }
    }
    }
    chain_next();
}

// ---------------------------------------------------------------- prompts: neighbouring tokens share the copies of their keys
//
// One CTA per (head, four 16-row tiles of neighbouring tokens); a warp owns a tile (its rows, queries, sums), and all four walk
// the same keys: blocks of 64 keys and values come by cp.async into two buffers, one under way while the other is worked on.
// Tokens of a prompt see nearly the same keys, so a block is read once for 12 tokens (5 rows each) instead of once per tile,
// and no warp waits behind its own copies.  A group whose tokens belong to two sequences walks first the one's keys, then the
// other's.  In a mixed group nothing is shared: with caches of up to kTileMaxKeys positions each warp walks its own tile's
// sequences by itself, through its quarter of the buffers; with longer ones the group is left to moa_attention_mma_kernel, whose
// CTAs share out a tile's keys (31 sequences decoding at 2048 positions beside a prompt of 512: the layer 693 us with shared
// blocks of one active warp each, 157 so).  Both operands' fragments come by ldmatrix.x4; exponents are base 2 with the scale folded in; a block that every row of the warp
// sees in full is not masked, and sums are rescaled only where a maximum moved.  Three CTAs of 70 KB and 168 registers a
// thread fill an SM.  Bound by the instruction issue of the warp-level tensor path and the exponentials.
// 32 prompts of 256 tokens, 4 heads of 128, 8 experts top-5: 133 us with a tile per warp and its own copies, 83 with shared ones
// (tensor pipe 31 % busy, 0.38 instructions a cycle and scheduler; the layer 702 -> 653 us; with the dense output projection's
// rows to write, under a profiler with cold caches: 101 us, 23 %, 0.34).
constexpr int kShKeys = 64, kShTokens = kShWarps * 16;

__device__ __forceinline__ float ex2(float v) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}

int shared_tile_tokens(int W) { return W <= 8 ? 16 / W : 1; }
long long shared_groups(const dsmoe_layer_desc& p) {
    const int W = width_of(p), tpt = shared_tile_tokens(W);
    return ((long long)((p.T + tpt - 1) / tpt) * ((W + 15) / 16) + kShWarps - 1) / kShWarps;
}

template <int DH>
constexpr size_t shared_attention_smem() { return (size_t)2 * 2 * kShKeys * (DH * 2 + 16); }

// This lane's two rows of tile (t0, rt), g and g + 8: grouped row (-1 = none), token
__device__ __forceinline__ void tile_rows(const AttnArgs& P, int t0, int rt, int g, int (&r)[2], int (&tk)[2]) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int i = g + 8 * h;
        int slot;
        if (P.tpt == 1) {
            tk[h] = t0;
            slot = rt * 16 + i;
        } else {
            tk[h] = i < P.tpt * P.W ? t0 + i / P.W : P.T;
            slot = i % P.W;
        }
        r[h] = tk[h] < P.T && slot < P.W ? P.token_rows[(size_t)tk[h] * P.W + slot] : -1;
        if (r[h] >= P.amax) r[h] = -1;
    }
}

// Attends with this warp's tile (t0, rt) of head j and writes its rows.  The keys of tokens first_u .. end_u - 1 of the group (tokens
// tg0 ..) are walked by the CTA together, or (ALONE) by the warp by itself.
template <int DH, bool ALONE>
__device__ __forceinline__ void attend(const AttnArgs& P, unsigned char* const smem, const int* const seq_s, const int* const last_s,
                                       const int j, const int t0, const int rt, const int tg0, const int first_u, const int end_u,
                                       int (&r)[2], int (&tk)[2]) {
    constexpr int STRIDE = DH * 2 + 16;                 // bytes per key row in shared memory: 16 of padding, no bank conflicts
    constexpr int KS = DH / 16, DT = DH / 8, CH = DH / 8;
    constexpr int keys = ALONE ? kShKeys / 2 : kShKeys, workers = ALONE ? 32 : 32 * kShWarps;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, q4 = lane & 3;
    const int worker = ALONE ? lane : threadIdx.x;
    int last[2], sq_of[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        last[h] = r[h] >= 0 ? last_s[tk[h] - tg0] : 0;
        sq_of[h] = r[h] >= 0 ? seq_s[tk[h] - tg0] : -1;
    }
    // Q fragments (the A operand of S = Q.K^T)
    uint32_t qf[KS][4];
#pragma unroll
    for (int ks = 0; ks < KS; ++ks) {
        const int c = j * DH + ks * 16 + q4 * 2;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const __nv_bfloat16* q = P.qa + (size_t)max(r[h], 0) * P.H + c;
            qf[ks][h] = r[h] >= 0 ? *reinterpret_cast<const uint32_t*>(q) : 0u;
            qf[ks][2 + h] = r[h] >= 0 ? *reinterpret_cast<const uint32_t*>(q + 8) : 0u;
        }
    }
    const float sl2 = P.scale * 1.4426950408889634f;
    float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};
    float o[DT][4];
#pragma unroll
    for (int i = 0; i < DT; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;

    const uint32_t smem0 = (uint32_t)__cvta_generic_to_shared(smem);
    // fragment addresses inside a block: K (rows = keys, two 8-key tiles x two 8-wide halves of k) and V (transposed)
    const uint32_t kfrag = (uint32_t)(((lane >> 4) * 8 + (lane & 7)) * STRIDE + ((lane >> 3) & 1) * 16);
    const uint32_t vfrag = (uint32_t)((((lane >> 3) & 1) * 8 + (lane & 7)) * STRIDE + (lane >> 4) * 16);

    const uint32_t own = ALONE ? (uint32_t)(warp * kShKeys * STRIDE) : 0u;
    for (int u = first_u; u < end_u; ++u) {
        // one pass per sequence among them (a prompt's tokens: one)
        const int sq = seq_s[u];
        bool again = false;
        for (int v = first_u; v < u && !again; ++v) again = seq_s[v] == sq;
        if (again) continue;
        int last_key = 0;
        for (int v = u; v < end_u; ++v)
            if (seq_s[v] == sq) last_key = max(last_key, last_s[v]);
        // this pass: which rows take part, the last key any of the warp's rows sees, the last one they all see
        const bool act0 = sq_of[0] == sq, act1 = sq_of[1] == sq;
        const int wlast = (int)__reduce_max_sync(0xffffffffu, max(act0 ? last[0] : -1, act1 ? last[1] : -1));
        const int wfull = (int)__reduce_min_sync(0xffffffffu, min(act0 ? last[0] : r[0] >= 0 ? -1 : INT_MAX,
                                                                  act1 ? last[1] : r[1] >= 0 ? -1 : INT_MAX));
        const __nv_bfloat16* Kh = P.Kc + ((size_t)(sq * P.n_head + j) * P.L) * DH;
        const __nv_bfloat16* Vh = P.Vc + ((size_t)(sq * P.n_head + j) * P.L) * DH;
        const int nblocks = last_key / keys + 1;
        const auto fetch = [&](int b, int buf) {
            const int key0 = b * keys, nk = min(keys, last_key + 1 - key0);
            const uint32_t kd = smem0 + own + (uint32_t)(buf * 2 * kShKeys * STRIDE), vd = kd + (uint32_t)(keys * STRIDE);
#pragma unroll(ALONE ? 4 : CH * keys / workers)          // (ALONE in full: the kernel spills)
            for (int i = 0; i < CH * keys / workers; ++i) {
                const int idx = worker + workers * i, row = idx / CH, ch = idx % CH;
                // rows past the last visible key are filled with zeros
                const size_t src = (size_t)(key0 + (row < nk ? row : 0)) * DH + ch * 8;
                const uint32_t nbytes = row < nk ? 16u : 0u, dst = (uint32_t)(row * STRIDE + ch * 16);
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(kd + dst), "l"(Kh + src), "r"(nbytes) : "memory");
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(vd + dst), "l"(Vh + src), "r"(nbytes) : "memory");
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        if (!ALONE) fetch(0, 0);
        for (int b = 0; b < nblocks; ++b) {
            const int buf = ALONE ? 0 : b & 1;
            if (ALONE) fetch(b, 0);
            if (!ALONE && b + 1 < nblocks) {
                fetch(b + 1, buf ^ 1);
                asm volatile("cp.async.wait_group 1;" ::: "memory");
            } else {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
            }
            if (ALONE) __syncwarp();
            else __syncthreads();
            const uint32_t kblock = smem0 + own + (uint32_t)(buf * 2 * kShKeys * STRIDE), vblock = kblock + (uint32_t)(keys * STRIDE);
#pragma unroll 1
            for (int half = 0; half < keys / 32; ++half) {
                const int key0 = b * keys + 32 * half;
                if (key0 > wlast) break;                // (uniform in the warp) nothing more for this warp's rows
                const uint32_t ka = kblock + (uint32_t)(32 * half * STRIDE) + kfrag;
                const uint32_t va = vblock + (uint32_t)(32 * half * STRIDE) + vfrag;
                float sc[4][4];
#pragma unroll
                for (int nt = 0; nt < 4; ++nt) sc[nt][0] = sc[nt][1] = sc[nt][2] = sc[nt][3] = 0.f;
#pragma unroll
                for (int ks = 0; ks < KS; ++ks) {
#pragma unroll
                    for (int np = 0; np < 2; ++np) {
                        uint32_t kb[4];
                        ldsm4(kb, ka + (uint32_t)(np * 16 * STRIDE + ks * 32));
                        mma_bf16_16816(sc[2 * np], qf[ks], kb[0], kb[1]);
                        mma_bf16_16816(sc[2 * np + 1], qf[ks], kb[2], kb[3]);
                    }
                }
                // scale (to base 2), hide the keys past each row's position and everything from rows not in this pass
                float bm0 = -INFINITY, bm1 = -INFINITY;
                if (key0 + 31 <= wfull) {
#pragma unroll
                    for (int nt = 0; nt < 4; ++nt) {
#pragma unroll
                        for (int c = 0; c < 4; ++c) sc[nt][c] *= sl2;
                        bm0 = fmaxf(bm0, fmaxf(sc[nt][0], sc[nt][1]));
                        bm1 = fmaxf(bm1, fmaxf(sc[nt][2], sc[nt][3]));
                    }
                } else {
                    const int e0 = act0 ? last[0] : -1, e1 = act1 ? last[1] : -1;
#pragma unroll
                    for (int nt = 0; nt < 4; ++nt) {
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
                            const int key = key0 + nt * 8 + q4 * 2 + c;
                            sc[nt][c] = key <= e0 ? sc[nt][c] * sl2 : -INFINITY;
                            sc[nt][2 + c] = key <= e1 ? sc[nt][2 + c] * sl2 : -INFINITY;
                        }
                        bm0 = fmaxf(bm0, fmaxf(sc[nt][0], sc[nt][1]));
                        bm1 = fmaxf(bm1, fmaxf(sc[nt][2], sc[nt][3]));
                    }
                }
                bm0 = fmaxf(bm0, __shfl_xor_sync(0xffffffffu, bm0, 1));
                bm1 = fmaxf(bm1, __shfl_xor_sync(0xffffffffu, bm1, 1));
                bm0 = fmaxf(bm0, __shfl_xor_sync(0xffffffffu, bm0, 2));
                bm1 = fmaxf(bm1, __shfl_xor_sync(0xffffffffu, bm1, 2));
                if (__any_sync(0xffffffffu, bm0 > m[0] || bm1 > m[1])) {
                    const float n0 = fmaxf(m[0], bm0), n1 = fmaxf(m[1], bm1);
                    // a row that has seen no key yet (and sees none here) keeps m = -inf: nothing to rescale
                    const float c0 = n0 == -INFINITY ? 1.f : ex2(m[0] - n0), c1 = n1 == -INFINITY ? 1.f : ex2(m[1] - n1);
                    m[0] = n0;
                    m[1] = n1;
                    l[0] *= c0;
                    l[1] *= c1;
#pragma unroll
                    for (int i = 0; i < DT; ++i) {
                        o[i][0] *= c0;
                        o[i][1] *= c0;
                        o[i][2] *= c1;
                        o[i][3] *= c1;
                    }
                }
                const float z0 = m[0] == -INFINITY ? 0.f : m[0], z1 = m[1] == -INFINITY ? 0.f : m[1];
                uint32_t pf[2][4];
#pragma unroll
                for (int nt = 0; nt < 4; ++nt) {
                    const float p0 = ex2(sc[nt][0] - z0), p1 = ex2(sc[nt][1] - z0);
                    const float p2 = ex2(sc[nt][2] - z1), p3 = ex2(sc[nt][3] - z1);
                    l[0] += p0 + p1;
                    l[1] += p2 + p3;
                    pf[nt / 2][(nt & 1) * 2] = pack_bf16(p0, p1);
                    pf[nt / 2][(nt & 1) * 2 + 1] = pack_bf16(p2, p3);
                }
#pragma unroll
                for (int kk = 0; kk < 2; ++kk) {
#pragma unroll
                    for (int dp = 0; dp < DT / 2; ++dp) {
                        uint32_t vb[4];
                        ldsm4t(vb, va + (uint32_t)(kk * 16 * STRIDE + dp * 32));
                        mma_bf16_16816(o[2 * dp], pf[kk], vb[0], vb[1]);
                        mma_bf16_16816(o[2 * dp + 1], pf[kk], vb[2], vb[3]);
                    }
                }
            }
            if (ALONE) __syncwarp();
            else __syncthreads();
        }
    }
    chain_next();
    // normalise (and weigh); the rows go out through shared memory (the buffers are free), whole rows per store
    float inv[2];
    __nv_bfloat16* dst[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        l[h] += __shfl_xor_sync(0xffffffffu, l[h], 1);
        l[h] += __shfl_xor_sync(0xffffffffu, l[h], 2);
        inv[h] = 1.f / l[h];
        dst[h] = r[h] >= 0 ? P.qa + (size_t)r[h] * P.H + j * DH : nullptr;
        if (P.dense && r[h] >= 0) {
            const int i = g + 8 * h, e = expert_of_slot(P.mask[tk[h]], P.tpt == 1 ? rt * 16 + i : i % P.W);
            dst[h] = e >= 0 ? P.dense + ((size_t)tk[h] * P.E + e) * P.H + j * DH : nullptr;
            inv[h] *= P.row_gate[r[h]];
        }
    }
    unsigned char* const st = smem + warp * kShKeys * STRIDE;      // (where only this warp may still have been reading)
#pragma unroll
    for (int dt = 0; dt < DT; ++dt) {
        *reinterpret_cast<uint32_t*>(st + g * STRIDE + (dt * 8 + q4 * 2) * 2) = pack_bf16(o[dt][0] * inv[0], o[dt][1] * inv[0]);
        *reinterpret_cast<uint32_t*>(st + (g + 8) * STRIDE + (dt * 8 + q4 * 2) * 2) = pack_bf16(o[dt][2] * inv[1], o[dt][3] * inv[1]);
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 16 * CH / 32; ++i) {
        const int idx = lane + 32 * i, row = idx / CH, ch = idx % CH;
        __nv_bfloat16* const da = reinterpret_cast<__nv_bfloat16*>(__shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(dst[0]), (row & 7) * 4));
        __nv_bfloat16* const db = reinterpret_cast<__nv_bfloat16*>(__shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(dst[1]), (row & 7) * 4));
        __nv_bfloat16* const to = row < 8 ? da : db;
        if (to) *reinterpret_cast<uint4*>(to + ch * 8) = *reinterpret_cast<const uint4*>(st + row * STRIDE + ch * 16);
    }
}

// Four tiles of neighbouring tokens, by the whole CTA: its smem of shared_attention_smem<DH>() bytes, room for kShTokens tokens
template <int DH>
__device__ __forceinline__ void attend_group(const AttnArgs& P, unsigned char* const smem, int* const seq_s, int* const last_s, const int j,
                                             const int group) {
    constexpr int CH = DH / 8;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // this CTA's tokens: their sequences and last visible keys, clamped into the cache (and reported)
    int tg0, tg1;
    group_tokens(P, group, tg0, tg1);
    const int ng = tg1 - tg0;
    if (threadIdx.x < ng) {
        const int t = tg0 + threadIdx.x;
        const int sq = P.tok_seq ? P.tok_seq[t] : 0, last = P.pos[t];
        if (sq < 0 || sq >= P.n_seq || last < 0 || last >= P.L) report_status(P.dev_status, DSMOE_ERR_INVALID_ARG);
        seq_s[threadIdx.x] = min(max(sq, 0), P.n_seq - 1);
        last_s[threadIdx.x] = min(max(last, 0), P.L - 1);
    }
    const int wt = group * kShWarps + warp, t0 = (wt / P.row_tiles) * P.tpt, rt = wt % P.row_tiles;
    int r[2], tk[2];
    tile_rows(P, t0, rt, lane >> 2, r, tk);
    __syncthreads();
    bool mixed = false;
    const auto seq = [&](int i) { return seq_s[i]; };
    for (int i = lane; i < ng; i += 32) mixed = mixed || mixes(seq, 0, ng, i);
    mixed = __any_sync(0xffffffffu, mixed);
    if (P.dense && rt == 0) {
        for (int t = t0; t < min(P.T, t0 + P.tpt); ++t) {
            const uint64_t sel = P.mask[t];
            for (int idx = lane; idx < P.E * CH; idx += 32) {
                const int e = idx / CH, ch = idx % CH;
                if (!((sel >> e) & 1ull))
                    *reinterpret_cast<uint4*>(P.dense + ((size_t)t * P.E + e) * P.H + j * DH + ch * 8) = make_uint4(0u, 0u, 0u, 0u);
            }
        }
    }
    if (!mixed) attend<DH, false>(P, smem, seq_s, last_s, j, t0, rt, tg0, 0, ng, r, tk);
    else if (!P.leave_mixed) {
        tile_rows(P, t0, rt, lane >> 2, r, tk);         // (again: kept over the branch, they cost registers that the common path lacks)
        attend<DH, true>(P, smem, seq_s, last_s, j, t0, rt, tg0, t0 - tg0, min(t0 - tg0 + P.tpt, ng), r, tk);
    }
}

template <int DH>
__global__ void __launch_bounds__(32 * kShWarps, 3) moa_attention_shared_kernel(const __grid_constant__ AttnArgs P) {
    chain_wait();
    extern __shared__ __align__(16) unsigned char moa_sh_smem[];
    __shared__ int seq_s[kShTokens], last_s[kShTokens];
    attend_group<DH>(P, moa_sh_smem, seq_s, last_s, (int)(blockIdx.x % P.n_head), (int)(blockIdx.x / P.n_head));
}

// ---------------------------------------------------------------- the same for a tile of up to 128 rows on the 5th-generation tensor cores
// One CTA per (head, tile of neighbouring tokens: 24 of 5 rows each); a thread owns a row.  Per 64 keys: S = Q.K^T into TMEM, each thread its
// row's maximum, weights and sum without a word from its neighbours, P (bf16) into the 128-byte swizzle where the keys lay, P.V into TMEM,
// and the running values in the thread's registers (fp32; nothing is rescaled in TMEM).  Keys and values lie as in memory; V is an N-major
// operand.  A block of both is copied while the one before is worked on, two CTAs fill an SM (255 registers a thread, 97 KB each).
// 32 prompts of 256 tokens, 4 heads of 128, 8 experts top-5: 102 us with the warp-level path, 81 to 84 so (cold caches; the layer 482 -> 452).
// Bound by the instruction issue of the weights and of the copies' addresses (0.34 a cycle and scheduler with two warps each; the
// tensor pipe 9 % busy).  Asking for the next block's S before this one's weights, and adding P.V a block later: 85 us (registers).
// The sums are of the rounded weights, which P.V is made of: whole layers of 4 heads of 128 and of 96 and 2 of 64 are 1.970e-3, 2.017e-3 and
// 2.030e-3 from 64 bits (1.988e-3, 2.031e-3, 2.041e-3 before; 1.995e-3, 2.040e-3, 2.044e-3 with sums of the unrounded ones).
// What it does not take -- tiles of tokens of three sequences and more, tiles with a mixed group that is the key-splitting kernel's, keys
// or values that are not finite -- it does in the other form.
constexpr int kUaRows = 128, kUaKeys = 64;

// Groups of four 16-row tiles that one 128-row tile takes (0: not this kernel's)
int umma_attention_groups(int W) { return W <= 16 ? kUaRows / (W * kShWarps * shared_tile_tokens(W)) : 0; }

// Where it is the faster one: with an SM's worth of CTAs each, which are half as many as the shared-key kernel's (8 experts of 4 heads of 128,
// top-5, us a layer, that kernel and this one: 400 tokens, 68 CTAs, 83, 86; 1024, 172 CTAs, 119, 117; 8192 482, 452; one prompt of 2048
// 243, 215; 16 of 2 heads of 64, top-6: 800 tokens, 100 CTAs, 63, 65; 2048, 256 CTAs, 101, 98), and with prompts long enough that few tiles walk two
// (16 of 2 heads of 64: 30 prompts of 100 tokens 86, 88, of 128 159, 156; 8 of 4 heads of 128: 60 of 64 234, 237, 30 of 100 192, 181).
// Tokens of several sequences in no order, which the host does not see, are slower here (8 of 4 heads of 128, that kernel alone and this one: 2500 tokens of
// 5 sequences at random, 300 positions, 262, 302; 4096 of 16, 256 positions, 355, 397; 1250 of 2, 400 positions, 169, 183; in rounds of two 160, 140): their
// groups take the other form with 8 warps an SM for its 12.  Left to a launch of their own they were no faster and prompts in order 2 to 9 % slower.
bool umma_attention_fits(const dsmoe_layer_desc& p, const MoaCore& c) {
    const int W = width_of(p);
    const long long span = (long long)umma_attention_groups(W) * kShWarps * shared_tile_tokens(W), n_seq = c.tok_seq ? c.n_seq : 1;
    return span > 0 && (p.T + span - 1) / span * c.n_head >= sm_count() && p.T >= n_seq * (p.H / c.n_head == 64 ? 128 : 96);
}

template <int DH>
struct UaShape {
    static constexpr int HALVES = (DH + 63) / 64;                 // a row's 128-byte pieces
    static constexpr uint32_t QB = HALVES * kUaRows * 128, KB = HALVES * kUaKeys * 128;
    static constexpr uint32_t TMEM = DH <= 64 ? 128 : 256;        // 64 columns of logits, DH of weighted values
    // the weights lie where the block's keys did, if they fit there: two CTAs on an SM
    static constexpr bool P_ON_K = KB >= kUaRows * 128;
    static constexpr size_t smem = 1024 + QB + 4 * KB + (P_ON_K ? 0 : kUaRows * 128);
    static_assert(smem - 1024 >= (size_t)2 * 2 * kShKeys * (DH * 2 + 16), "room for attend_group");
};

// Operand B = V as it lies in memory, [keys][64 columns] in the 128-byte swizzle: N-major.  Eight keys are 1024 bytes, the next 64 columns
// begin kUaKeys rows further on.
__device__ __forceinline__ uint64_t make_desc_mn_sw128(uint32_t smem_addr) {
    uint64_t d = 0;
    d |= (uint64_t)((smem_addr & 0x3FFFF) >> 4);
    d |= (uint64_t)((kUaKeys * 128) >> 4) << 16;                  // leading byte offset: between 64-column groups
    d |= (uint64_t)(1024 >> 4) << 32;                             // stride byte offset: between groups of 8 keys
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

template <int DH>
__global__ void __launch_bounds__(kUaRows, 2) moa_attention_umma_kernel(const __grid_constant__ AttnArgs P, const int groups) {
    using S = UaShape<DH>;
    constexpr int CH = DH / 8;
    extern __shared__ unsigned char moa_ua_smem[];
    __shared__ int seq_s[kUaRows], last_s[kUaRows];
    __shared__ uint64_t bar[2];
    __shared__ uint32_t tmem_s;
    __shared__ volatile int abort_flag;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t raw = ptx::smem_u32(moa_ua_smem), base = (raw + 1023u) & ~1023u;
    unsigned char* const smem = moa_ua_smem + (base - raw);
    const uint32_t sQ = base, sK = sQ + S::QB, sV = sK + 2 * S::KB;
    const int j = (int)(blockIdx.x % P.n_head), tile = (int)(blockIdx.x / P.n_head);
    const int span = groups * kShWarps * P.group_tpt;             // tokens of a tile
    const int tg0 = tile * span, ng = min(P.T - tg0, span);
    if (tid == 0) {
        ptx::mbar_init(ptx::smem_u32(&bar[0]), 1);
        ptx::mbar_init(ptx::smem_u32(&bar[1]), 1);
        abort_flag = 0;
        ptx::fence_barrier_init();
    }
    chain_wait();
    if (warp == 0) {
        ptx::tmem_alloc(ptx::smem_u32(&tmem_s), S::TMEM);
        ptx::tmem_relinquish();
    }
    if (tid < ng) {
        const int t = tg0 + tid;
        const int sq = P.tok_seq ? P.tok_seq[t] : 0, last = P.pos[t];
        if (sq < 0 || sq >= P.n_seq || last < 0 || last >= P.L) report_status(P.dev_status, DSMOE_ERR_INVALID_ARG);
        seq_s[tid] = min(max(sq, 0), P.n_seq - 1);
        last_s[tid] = min(max(last, 0), P.L - 1);
    }
    // this thread's row of the tile: grouped row (-1: none), token of the tile
    const int tl = tid / P.W, slot = tid % P.W;
    int r = -1;
    if (tl < ng) {
        r = P.token_rows[(size_t)(tg0 + tl) * P.W + slot];
        if (r >= P.amax) r = -1;
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = tmem_s;
    // a tile of three sequences and more, or with a group that is left to another launch, goes the other way, group by group
    bool mixed = false;
    const auto seq = [&](int i) { return seq_s[i]; };
    const int per_group = kShWarps * P.group_tpt;
    for (int i = lane; i < ng; i += 32) {
        const int a = i / per_group * per_group;
        mixed = mixed || mixes(seq, 0, ng, i) || (P.leave_mixed && mixes(seq, a, min(a + per_group, ng), i));
    }
    bool redo = __any_sync(0xffffffffu, mixed);                   // (the same for all warps)

    if (!redo) {
        // queries: a warp's 32 rows, DH / 8 pieces of 16 bytes each, in the swizzle's order; rows that are none are zeros
        for (int i = lane; i < 32 * CH; i += 32) {
            const int row = i / CH, ch = i % CH, rr = __shfl_sync(0xffffffffu, r, row), at = warp * 32 + row;
            const __nv_bfloat16* q = P.qa + (size_t)max(rr, 0) * P.H + j * DH + ch * 8;
            const uint32_t dst = sQ + (uint32_t)((ch >> 3) * kUaRows * 128 + at * 128 + (((ch & 7) ^ (at & 7)) << 4)), nbytes = rr >= 0 ? 16u : 0u;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(q), "r"(nbytes) : "memory");
        }
        const auto zeros = [&]() {                                // where a token did not select an expert
            for (int t = tg0 + warp; t < tg0 + ng; t += kUaRows / 32) {
                const uint64_t sel = P.mask[t];
                for (int idx = lane; idx < P.E * CH; idx += 32) {
                    const int e = idx / CH, ch = idx % CH;
                    if (!((sel >> e) & 1ull))
                        *reinterpret_cast<uint4*>(P.dense + ((size_t)t * P.E + e) * P.H + j * DH + ch * 8) = make_uint4(0u, 0u, 0u, 0u);
                }
            }
        };
        const float sl2 = P.scale * 1.4426950408889634f;
        const int last = r >= 0 ? last_s[tl] : -1, sq_of = r >= 0 ? seq_s[tl] : -1;
        float m = -INFINITY, l = 0.f, o[DH];
#pragma unroll
        for (int i = 0; i < DH; ++i) o[i] = 0.f;
        uint32_t phase = 0;
        bool alive = true;
        const int passes = seq_s[0] == seq_s[ng - 1] ? 1 : 2;
        for (int pass = 0; pass < passes && alive; ++pass) {
            const int sq = pass == 0 ? seq_s[0] : seq_s[ng - 1];
            int mine = -1;
            for (int i = lane; i < ng; i += 32)
                if (seq_s[i] == sq) mine = max(mine, last_s[i]);
            const int last_key = __reduce_max_sync(0xffffffffu, mine);
            const int elast = sq_of == sq ? last : -1;
            const __nv_bfloat16* Kh = P.Kc + ((size_t)(sq * P.n_head + j) * P.L) * DH;
            const __nv_bfloat16* Vh = P.Vc + ((size_t)(sq * P.n_head + j) * P.L) * DH;
            const int nblocks = last_key / kUaKeys + 1;
            const auto fetch = [&](int b) {
                const int key0 = b * kUaKeys, nk = min(kUaKeys, last_key + 1 - key0);
                const uint32_t kd = sK + (b & 1) * S::KB, vd = sV + (b & 1) * S::KB;
#pragma unroll
                for (int i = 0; i < kUaKeys * CH / kUaRows; ++i) {
                    const int idx = tid + kUaRows * i, row = idx / CH, ch = idx % CH;
                    // rows past the last visible key are filled with zeros
                    const size_t src = (size_t)(key0 + (row < nk ? row : 0)) * DH + ch * 8;
                    const uint32_t nbytes = row < nk ? 16u : 0u;
                    const uint32_t dst = (uint32_t)((ch >> 3) * kUaKeys * 128 + row * 128 + (((ch & 7) ^ (row & 7)) << 4));
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(kd + dst), "l"(Kh + src), "r"(nbytes) : "memory");
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(vd + dst), "l"(Vh + src), "r"(nbytes) : "memory");
                }
                ptx::cp_async_commit();
            };
            fetch(0);
            if (P.dense && pass == 0) zeros();                    // (while the copies are on their way)
            for (int b = 0; b < nblocks; ++b) {
                if (b + 1 < nblocks) {
                    fetch(b + 1);
                    ptx::cp_async_wait<1>();
                } else {
                    ptx::cp_async_wait<0>();
                }
                ptx::fence_proxy_async();
                ptx::tc_fence_before();
                __syncthreads();
                if (warp == 0 && ptx::elect_one()) {
                    ptx::tc_fence_after();
                    const uint32_t k0 = sK + (b & 1) * S::KB, idesc = ptx::make_idesc_bf16(kUaRows, kUaKeys);
#pragma unroll
                    for (int k = 0; k < DH / 16; ++k)
                        ptx::umma_bf16(tmem, ptx::make_desc_k_sw128(sQ + (k >> 2) * kUaRows * 128 + (k & 3) * 32),
                                       ptx::make_desc_k_sw128(k0 + (k >> 2) * kUaKeys * 128 + (k & 3) * 32), idesc, (uint32_t)(k != 0));
                    ptx::umma_commit(ptx::smem_u32(&bar[0]));
                }
                __syncwarp();
                alive = ptx::mbar_wait(ptx::smem_u32(&bar[0]), phase, &abort_flag);
                alive = __syncthreads_and(alive);
                if (!alive) break;
                ptx::tc_fence_after();
                const uint32_t row0 = tmem + ((uint32_t)(warp * 32) << 16);
                uint32_t v[2][32];
                ptx::tmem_ld32(row0, v[0]);
                ptx::tmem_ld32(row0 + 32, v[1]);
                ptx::tmem_ld_wait();
                const uint32_t sP = S::P_ON_K ? sK + (b & 1) * S::KB : sV + 2 * S::KB;
                const int seen = elast - b * kUaKeys;             // keys 0 .. seen of the block are this row's
                float bm = -INFINITY, alpha;
                const auto weigh = [&](float scale) {             // v -> weights, in base 2, relative to the running maximum
                    const float n = fmaxf(m, bm), z = n == -INFINITY ? 0.f : n;
                    alpha = n == -INFINITY ? 1.f : ex2(m - n);
                    m = n;
                    l *= alpha;
#pragma unroll
                    for (int c = 0; c < kUaKeys / 8; ++c) {
                        uint32_t pk[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const int at = c * 8 + 2 * i;
                            const float p0 = ex2(fmaf(__uint_as_float(v[at / 32][at % 32]), scale, -z));
                            const float p1 = ex2(fmaf(__uint_as_float(v[at / 32][at % 32 + 1]), scale, -z));
                            pk[i] = pack_bf16(p0, p1);
                            l += bf16_lo(pk[i]) + bf16_hi(pk[i]);     // (what is multiplied is what is divided by)
                        }
                        *reinterpret_cast<uint4*>(smem + (sP - base) + tid * 128 + ((c ^ (tid & 7)) << 4)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                    }
                };
                if (__all_sync(0xffffffffu, seen >= kUaKeys - 1) && sl2 > 0.f) {       // nothing to hide from this warp's rows
#pragma unroll
                    for (int i = 0; i < kUaKeys; ++i) bm = fmaxf(bm, __uint_as_float(v[i / 32][i % 32]));
                    bm *= sl2;
                    weigh(sl2);
                } else {
#pragma unroll
                    for (int i = 0; i < kUaKeys; ++i) {
                        const float x = i <= seen ? __uint_as_float(v[i / 32][i % 32]) * sl2 : -INFINITY;
                        v[i / 32][i % 32] = __float_as_uint(x);
                        bm = fmaxf(bm, x);
                    }
                    weigh(1.f);
                }
                ptx::fence_proxy_async();
                ptx::tc_fence_before();
                __syncthreads();
                if (warp == 0 && ptx::elect_one()) {
                    ptx::tc_fence_after();
                    const uint32_t v0 = sV + (b & 1) * S::KB, idesc = ptx::make_idesc_bf16(kUaRows, DH) | (1u << 16);      // B is N-major
#pragma unroll
                    for (int k = 0; k < kUaKeys / 16; ++k)
                        ptx::umma_bf16(tmem + kUaKeys, ptx::make_desc_k_sw128(sP + k * 32), make_desc_mn_sw128(v0 + k * 2048), idesc, (uint32_t)(k != 0));
                    ptx::umma_commit(ptx::smem_u32(&bar[1]));
                }
                __syncwarp();
                alive = ptx::mbar_wait(ptx::smem_u32(&bar[1]), phase, &abort_flag);
                phase ^= 1u;
                alive = __syncthreads_and(alive);
                if (!alive) break;
                ptx::tc_fence_after();
#pragma unroll
                for (int c = 0; c < DH / 32; ++c) {
                    uint32_t w[32];
                    ptx::tmem_ld32(row0 + kUaKeys + c * 32, w);
                    ptx::tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 32; ++i) o[c * 32 + i] = fmaf(o[c * 32 + i], alpha, __uint_as_float(w[i]));
                }
            }
        }
        ptx::cp_async_wait<0>();
        if (!alive && tid == 0) report_status(P.dev_status, DSMOE_ERR_TIMEOUT);
        // A key or value that is not finite reaches all rows of the tile here, also those that do not see it: such a tile is done again
        // the other way, whose tiles are 16 rows.
        float sum = l * 0.f;
#pragma unroll
        for (int i = 0; i < DH; ++i) sum = fmaf(o[i], 0.f, sum);
        redo = __syncthreads_or(!(sum == 0.f)) != 0;
        if (!redo) {
            chain_next();
            // normalise (and weigh); the rows go out through shared memory (the queries' place), whole rows per store
            float inv = 1.f / l;
            __nv_bfloat16* dst = r >= 0 ? P.qa + (size_t)r * P.H + j * DH : nullptr;
            if (P.dense && r >= 0) {
                const int e = expert_of_slot(P.mask[tg0 + tl], slot);
                dst = e >= 0 ? P.dense + ((size_t)(tg0 + tl) * P.E + e) * P.H + j * DH : nullptr;
                inv *= P.row_gate[r];
            }
            unsigned char* const st = smem + warp * 32 * (DH * 2 + 16);
#pragma unroll
            for (int c = 0; c < CH; ++c)
                *reinterpret_cast<uint4*>(st + lane * (DH * 2 + 16) + c * 16) =
                    make_uint4(pack_bf16(o[c * 8] * inv, o[c * 8 + 1] * inv), pack_bf16(o[c * 8 + 2] * inv, o[c * 8 + 3] * inv),
                               pack_bf16(o[c * 8 + 4] * inv, o[c * 8 + 5] * inv), pack_bf16(o[c * 8 + 6] * inv, o[c * 8 + 7] * inv));
            __syncwarp();
            for (int i = lane; i < 32 * CH; i += 32) {
                const int row = i / CH, ch = i % CH;
                __nv_bfloat16* const to = reinterpret_cast<__nv_bfloat16*>(__shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(dst), row));
                if (to) *reinterpret_cast<uint4*>(to + ch * 8) = *reinterpret_cast<const uint4*>(st + row * (DH * 2 + 16) + ch * 16);
            }
        }
    }
    if (redo) {
        for (int g = 0; g < groups; ++g) {
            const int group = tile * groups + g;
            if (group * kShWarps * P.group_tpt >= P.T) break;
            __syncthreads();
            attend_group<DH>(P, smem, seq_s, last_s, j, group);
        }
    }
    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem, S::TMEM);
    }
}

// Whether the groups that share no keys go to the key-splitting kernel
bool leaves_mixed(const dsmoe_layer_desc& p, const MoaCore& c) {
    return c.tok_seq && c.n_seq > 1 && c.L > kTileMaxKeys;
}

// tpt: tokens of a tile in this launch
AttnArgs attn_args(const dsmoe_layer_desc& p, const MoaCore& c, __nv_bfloat16* q, const int32_t* token_rows, int tpt,
                   int32_t* dev_status) {
    const int W = width_of(p);
    return AttnArgs{q, token_rows, W, (W + 15) / 16, tpt, shared_tile_tokens(W), (long long)amax_of(p), c.n_head, p.H, p.T,
                    static_cast<const __nv_bfloat16*>(c.Kc), static_cast<const __nv_bfloat16*>(c.Vc), c.tok_seq, c.pos,
                    c.n_seq, c.L, c.scale, dev_status, leaves_mixed(p, c), static_cast<__nv_bfloat16*>(c.dense), p.E, c.mask, c.row_gate};
}

template <int DH>
dsmoe_status launch_umma_attention(const dsmoe_layer_desc& p, const MoaCore& c, __nv_bfloat16* q, const int32_t* token_rows,
                                   int32_t* dev_status, cudaStream_t s) {
    static bool attr[kMaxDeviceSlots] = {};
    int dev = 0;
    DeviceState* st = nullptr;
    DSMOE_TRY(device_state(&st, &dev));
    if (!attr[dev]) {
        DSMOE_CUDA_TRY(cudaFuncSetAttribute(moa_attention_umma_kernel<DH>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)UaShape<DH>::smem));
        attr[dev] = true;
    }
    const int W = width_of(p), groups = umma_attention_groups(W);
    const long long span = (long long)groups * kShWarps * shared_tile_tokens(W), ctas = (p.T + span - 1) / span * c.n_head;
    if (ctas > 0x7fffffffll) return DSMOE_ERR_UNSUPPORTED;
    DSMOE_CUDA_TRY(launch_chained(moa_attention_umma_kernel<DH>, (unsigned)ctas, kUaRows, UaShape<DH>::smem, s,
        attn_args(p, c, q, token_rows, shared_tile_tokens(W), dev_status), groups));
    return DSMOE_OK;
}

template <int DH>
dsmoe_status launch_shared_attention(const dsmoe_layer_desc& p, const MoaCore& c, __nv_bfloat16* q, const int32_t* token_rows,
                                     int32_t* dev_status, cudaStream_t s) {
    static bool attr[kMaxDeviceSlots] = {};
    int dev = 0;
    DeviceState* st = nullptr;
    DSMOE_TRY(device_state(&st, &dev));
    if (!attr[dev]) {
        DSMOE_CUDA_TRY(cudaFuncSetAttribute(moa_attention_shared_kernel<DH>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)shared_attention_smem<DH>()));
        attr[dev] = true;
    }
    const long long ctas = shared_groups(p) * c.n_head;
    if (ctas > 0x7fffffffll) return DSMOE_ERR_UNSUPPORTED;
    DSMOE_CUDA_TRY(launch_chained(moa_attention_shared_kernel<DH>, (unsigned)ctas, 32 * kShWarps, shared_attention_smem<DH>(), s,
        attn_args(p, c, q, token_rows, shared_tile_tokens(width_of(p)), dev_status)));
    return DSMOE_OK;
}

// MIXED: the groups that moa_attention_shared_kernel leaves, a token per tile (their tokens share no keys)
template <int DH, int kMmaWarps, bool MIXED = false>
dsmoe_status launch_mma_attention_nw(const dsmoe_layer_desc& p, const MoaCore& c, __nv_bfloat16* q, const int32_t* token_rows,
                                  int32_t* dev_status, cudaStream_t s) {
    constexpr size_t stride = DH * 2 + 16;
    const size_t loop_bytes = (size_t)kMmaWarps * 2 * kKeyBlock * stride;
    const size_t merge_bytes = (size_t)kMmaWarps * (32 + 16 * DH) * 4;
    const size_t smem = loop_bytes > merge_bytes ? loop_bytes : merge_bytes;
    static bool attr[kMaxDeviceSlots] = {};
    int dev = 0;
    DeviceState* st = nullptr;
    DSMOE_TRY(device_state(&st, &dev));
    if (!attr[dev]) {
        DSMOE_CUDA_TRY(cudaFuncSetAttribute(moa_attention_mma_kernel<DH, kMmaWarps, MIXED>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        attr[dev] = true;
    }
    const int W = width_of(p), row_tiles = (W + 15) / 16;
    // several tokens per tile where a token has few rows and there are tokens enough to fill the GPU without
    const int tpt = (W <= 8 && (long long)p.T * c.n_head >= (MIXED ? 64ll : 8ll) * st->sm_count) ? 16 / W : 1;
    const long long n_tiles = (long long)((p.T + tpt - 1) / tpt) * c.n_head * row_tiles;
    static int per_sm_of[kMaxDeviceSlots] = {};      // CTAs of this kernel that fit an SM, asked once per device
    if (!per_sm_of[dev])
        DSMOE_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_of[dev], moa_attention_mma_kernel<DH, kMmaWarps, MIXED>,
                                                                     32 * kMmaWarps, smem));
    const int per_sm = per_sm_of[dev];
    const long long resident = (long long)st->sm_count * (per_sm > 0 ? per_sm : 1);
    const long long want = kMmaWarps > 2 ? n_tiles : (n_tiles + kMmaWarps - 1) / kMmaWarps;     // 2 warps: a tile per warp
    const long long ctas = want < resident ? want : resident;
    DSMOE_CUDA_TRY(launch_chained(moa_attention_mma_kernel<DH, kMmaWarps, MIXED>, (unsigned)ctas, 32 * kMmaWarps, smem, s,
        q, token_rows, W, row_tiles, tpt, (long long)amax_of(p), c.n_head, p.H, p.T, static_cast<const __nv_bfloat16*>(c.Kc),
        static_cast<const __nv_bfloat16*>(c.Vc), c.tok_seq, c.pos, c.n_seq, c.L, c.scale, n_tiles, dev_status,
        attn_args(p, c, q, token_rows, tpt, dev_status)));
    return DSMOE_OK;
}

template <int DH>
dsmoe_status launch_mma_attention(const dsmoe_layer_desc& p, const MoaCore& c, __nv_bfloat16* q, const int32_t* token_rows,
                                  int32_t* dev_status, cudaStream_t s) {
    if (moa_shares_keys(p, c)) {
        DSMOE_TRY(umma_attention_fits(p, c) ? launch_umma_attention<DH>(p, c, q, token_rows, dev_status, s)
                                                         : launch_shared_attention<DH>(p, c, q, token_rows, dev_status, s));
        return leaves_mixed(p, c) ? launch_mma_attention_nw<DH, 8, true>(p, c, q, token_rows, dev_status, s) : DSMOE_OK;
    }
    if (c.L <= kTileMaxKeys) return launch_mma_attention_nw<DH, 2>(p, c, q, token_rows, dev_status, s);
    return launch_mma_attention_nw<DH, 8>(p, c, q, token_rows, dev_status, s);
}

}  // namespace

bool moa_supported(const dsmoe_layer_desc& p, int n_head, int L) {
    if (!umma_supported(p) || n_head <= 0 || p.H % n_head) return false;
    const int dh = p.H / n_head;
    if (L <= 0 || dh % 32 || dh > 256) return false;
    if (dh == 64 || dh == 96 || dh == 128) return true;                       // tensor-core kernel: any cache length
    return (size_t)(dh + L + 3) * 4 * kMoaWarps <= 200 * 1024;                // plain kernel: a warp's logits sit in shared memory
}

// Prompts and chunks of them.  The host knows neither how much of a cache is visible nor the tokens' order, so the rule sees to
// it that no length and no order of sequences makes the shared-key kernel the much slower one (layer times key-splitting, shared
// for 8 experts of 4 heads of 128, top-5; 16 of 2 heads of 64, top-6, are alike):
//   long caches: its CTAs walk all keys by themselves, where the other kernel's warps share them out.  One sequence, 2048
//   positions: 64 tokens (24 CTAs) 103, 155 us; 128 (44) 154, 156; 256 (88) 236, 169; 2048 534, 254; 16384 positions, 256
//   tokens 1215, 842.  Of several sequences some CTAs walk two: 16384 positions, 12 sequences of 40 tokens (160 CTAs) 1083, 1294;
//   44 of 18 (264) 1465, 1388; 11 of 72 (264) 1465, 888; 2048 positions, 32 prompts of 256 1280, 469; 31 sequences decoding
//   beside a prompt of 768, their groups left to the other kernel, 271, 202.
//   short caches: the other kernel walks a tile per warp as well, of one token while T * n_head < 8 SMs; mixed groups then have
//   longer chains here, and groups of two sequences are walked twice.  4 sequences of 64 tokens, 256 positions: 96, 93; of 8
//   tokens 73, 76; 31 sequences decoding beside a prompt of 512, 512 positions: 201, 188, with 2 heads of 64 98, 112; 32 prompts
//   of 256: 633, 458; their tokens round-robin over the sequences 781, 619.
bool moa_shares_keys(const dsmoe_layer_desc& p, const MoaCore& c) {
    const int dh = p.H / c.n_head, n_seq = c.tok_seq ? c.n_seq : 1;
    if ((dh != 64 && dh != 96 && dh != 128) || getenv("DSMOE_MOA_PLAIN")) return false;
    const int W = width_of(p), group = kShWarps * shared_tile_tokens(W) / ((W + 15) / 16);       // tokens of a group
    const bool longer = c.L > kTileMaxKeys;
    const int least = longer ? 8 : (long long)p.T * c.n_head < 8ll * sm_count() ? 32 : group + group / 2;
    if (p.T < 8 || (n_seq > 1 && p.T < (long long)(least > 8 ? least : 8) * n_seq)) return false;
    return !longer || shared_groups(p) * c.n_head >= (n_seq > 1 ? 256 : 64);
}

dsmoe_status launch_moa_attention(const dsmoe_layer_desc& p, const MoaCore& c, void* qa, const int32_t* row_token,
                                  const int32_t* token_rows, const int32_t* offsets, int32_t* dev_status, cudaStream_t s) {
    const int dh = p.H / c.n_head;
    // DSMOE_MOA_PLAIN in the environment sends every head width to the plain kernel (a testing aid)
    if (token_rows && (dh == 64 || dh == 96 || dh == 128) && !getenv("DSMOE_MOA_PLAIN")) {
        // head widths of the paper's models: the tensor-core kernel, a CTA per (token, head)
        int timed = -1;
        DSMOE_TRY(timing_begin(s, &timed));
        auto* qb = static_cast<__nv_bfloat16*>(qa);
        if (dh == 64) DSMOE_TRY(launch_mma_attention<64>(p, c, qb, token_rows, dev_status, s));
        else if (dh == 96) DSMOE_TRY(launch_mma_attention<96>(p, c, qb, token_rows, dev_status, s));
        else DSMOE_TRY(launch_mma_attention<128>(p, c, qb, token_rows, dev_status, s));
        return timing_end(s, timed);
    }
    int warps = kMoaWarps;
    const size_t per_warp = (size_t)(dh + ((c.L + 3) & ~3)) * 4;
    const size_t smem = per_warp * warps;
    if (smem > 200 * 1024) return DSMOE_ERR_UNSUPPORTED;
    const long long pairs = (long long)amax_of(p) * c.n_head;
    const unsigned grid = (unsigned)((pairs + warps - 1) / warps);
    auto* q = static_cast<__nv_bfloat16*>(qa);
    auto* K = static_cast<const __nv_bfloat16*>(c.Kc);
    auto* V = static_cast<const __nv_bfloat16*>(c.Vc);
    int timed = -1;
    DSMOE_TRY(timing_begin(s, &timed));
#define MOA_LAUNCH(DPL)                                                                                                   \
    do {                                                                                                                  \
        if (smem > 48 * 1024)                                                                                             \
            DSMOE_CUDA_TRY(cudaFuncSetAttribute(moa_attention_kernel<DPL>, cudaFuncAttributeMaxDynamicSharedMemorySize,  \
                                                (int)smem));                                                              \
        DSMOE_CUDA_TRY(launch_chained(moa_attention_kernel<DPL>, grid, 32 * kMoaWarps, smem, s,                         \
            q, row_token, offsets, p.E, c.n_head, p.H, p.T, K, V, c.tok_seq, c.pos, c.n_seq, c.L, c.scale,              \
            dev_status));                                                                                               \
    } while (0)
    switch (dh / 32) {
        case 1: MOA_LAUNCH(1); break;
        case 2: MOA_LAUNCH(2); break;
        case 3: MOA_LAUNCH(3); break;
        case 4: MOA_LAUNCH(4); break;
        case 5: MOA_LAUNCH(5); break;
        case 6: MOA_LAUNCH(6); break;
        case 7: MOA_LAUNCH(7); break;
        case 8: MOA_LAUNCH(8); break;
        default: return DSMOE_ERR_UNSUPPORTED;
    }
#undef MOA_LAUNCH
    DSMOE_TRY(timing_end(s, timed));
    return DSMOE_OK;
}

}  // namespace dsmoe
