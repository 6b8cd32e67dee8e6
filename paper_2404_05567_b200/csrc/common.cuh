// Shared declarations of the dsmoe CUDA library: argument checks, the workspace layout and the
// internal launchers that the C entry points in api.cu call.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "dsmoe.h"

namespace dsmoe {

constexpr int kMaxExperts = 64;
constexpr int kChunk = 32;   // tokens per ballot chunk in the grouping kernels
constexpr int kSmallMaxT = 128;      // the small-T (decode) path keeps all tokens in one 128-row MMA tile
constexpr int kSmallMaxCtas = 192;   // upper bound on that path's grid (sizes its partial-sum buffer)

#define DSMOE_CUDA_TRY(expr)                                  \
    do {                                                      \
        cudaError_t err__ = (expr);                           \
        if (err__ != cudaSuccess) return DSMOE_ERR_CUDA;      \
    } while (0)

#define DSMOE_TRY(expr)                                       \
    do {                                                      \
        dsmoe_status st__ = (expr);                           \
        if (st__ != DSMOE_OK) return st__;                    \
    } while (0)

static inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }
__host__ __device__ static inline int ceil_div(int a, int b) { return (a + b - 1) / b; }

static inline size_t elem_size(int dtype) { return dtype == DSMOE_BF16 ? 2 : 4; }
static inline int width_of(const dsmoe_layer_desc& p) {
    return p.mode == DSMOE_SELECT_TOPK ? (p.K < p.E ? p.K : p.E) : p.E;
}
static inline size_t amax_of(const dsmoe_layer_desc& p) { return (size_t)p.T * (size_t)width_of(p); }

// Launches chained on one stream.  A layer call is up to eight dependent launches, and 2 to 3 us passed between one
// kernel's end and the next one's first instruction.  launch_chained lets the next kernel of the stream be set up
// (blocks placed, barriers and tensor memory prepared) while its predecessor still runs: every kernel launched this
// way calls chain_wait() before it touches global memory that a predecessor may write or read -- it returns once all
// kernels before it have completed and their writes are visible -- and chain_next() to let its own successor be set up: short kernels at
// once, long ones when their last loads are under way (blocks that wait beside a long kernel slow it down: with
// chain_next() at its start the gradients of dense training took 2067 instead of 1989 us).
// Such a kernel runs while its inputs are still being written, so it reads them with ordinary loads only: ld.global.nc (__ldg,
// or what the compiler makes of a `const T* __restrict__` parameter) is for data that nothing writes during the whole kernel,
// and as such may be served from a stale line or be moved above the wait.  No parameter that is only read is __restrict__.
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Every entry point's dev_status is optional: the only place that stores to it.
__device__ __forceinline__ void report_status(int32_t* dev_status, int32_t code) {
    if (dev_status) *dev_status = code;
}

int sm_count();
// Grids of more threads than the SMs hold are launched the ordinary way: most of their blocks would pay for a chain_wait() that
// has nothing left to wait for.  (Threads are all that is looked at: kernels that fill an SM with shared memory or registers
// stay chained over several waves.)
template <typename... KArgs, typename... Args>
static inline cudaError_t launch_chained_clusters(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                                  int cluster, bool chain, Args... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    unsigned n = 0;
    if (cluster > 1) {
        at[n].id = cudaLaunchAttributeClusterDimension;
        at[n].val.clusterDim.x = cluster; at[n].val.clusterDim.y = 1; at[n].val.clusterDim.z = 1;
        ++n;
    }
    if (chain && (size_t)grid.x * grid.y * grid.z * block.x <= (size_t)sm_count() * 2048) {
        at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[n].val.programmaticStreamSerializationAllowed = 1;
        ++n;
    }
    cfg.attrs = at;
    cfg.numAttrs = n;
    const cudaError_t err = cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
    if (err != cudaSuccess) cudaGetLastError();      // reported by the caller's status, not left behind for others
    return err;
}
template <typename... KArgs, typename... Args>
static inline cudaError_t launch_chained(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                         Args... args) {
    return launch_chained_clusters(kernel, grid, block, smem, s, 1, true, args...);
}
// chain == false: the ordinary launch of a kernel that can be chained (its chain_wait() then returns at once)
template <typename... KArgs, typename... Args>
static inline cudaError_t launch_chained_if(bool chain, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                            Args... args) {
    return launch_chained_clusters(kernel, grid, block, smem, s, 1, chain, args...);
}

dsmoe_status check_desc(const dsmoe_layer_desc* desc);
static inline bool aligned16(const void* p) { return ((uintptr_t)p & 15u) == 0; }

// Byte offsets of every internal buffer inside the caller's workspace.  The small per-token and per-assignment
// index buffers come first (`stage_total` bytes: all that dsmoe_select and dsmoe_permute touch); the large
// activation buffers follow and overlap between the execution paths, of which a call takes exactly one:
//   plain (fp32-FMA GEMMs)     h (fp32), yp
//   tensor-core paths          h (bf16: grouped [Amax,H]; dense and small-T [T,E*H]), acc (grouped: fp32 [T,d] running
//                              sum of the expert outputs), partial (small-T)
// total_packed = bytes a call with packed weights needs; total = the maximum over both kinds of call.
struct WsLayout {
    size_t scores, mask, k_t, counts, offsets, chunk_prefix, batch_k, sync, tile_done, mi, row_token, row_gate, token_rows;
    size_t stage_total;
    size_t h_plain, yp;                     // plain path
    size_t h, acc, partial, bwd;            // tensor-core paths
    size_t total_plain, total_packed, total;
};
WsLayout ws_layout(const dsmoe_layer_desc& p);
// The layout of a call with packed weights and ws_bytes of workspace.  A workspace too small for the outputs' rows that the second
// kernel adds up, but large enough for the tokens' running sums, has the sum taken inside the down-projection (*p changes).
WsLayout ws_layout_within(dsmoe_layer_desc* p, size_t ws_bytes);

// What the library keeps per device (attributes that must be set once per device, the SM count).  Entry points
// are not thread-safe: one host thread at a time may call into the library.
constexpr int kMaxDeviceSlots = 64;
struct DeviceState {
    int sm_count = 0;
    bool attr_gemm = false, attr_small = false, attr_grouped = false, attr_few = false;
    int max_pairs = -1;   // CTA pairs of umma_gemm_kernel that can be resident at once; -1 not asked yet, 0 pairs unavailable
};
dsmoe_status device_state(DeviceState** out, int* device = nullptr);   // of the current device

// Counters of a later launch that an earlier kernel of the call sets to zero on its way
struct ZeroInts {
    int* at = nullptr;
    long long n = 0;
};

// ---- router.cu
dsmoe_status launch_router(const dsmoe_layer_desc& p, const void* x, const float* Wr, const float* br,
                           float* scores, uint64_t* mask, int32_t* k_t, cudaStream_t s, const ZeroInts& zero = ZeroInts{});
// k_scratch: one int of device memory, needed by DSMOE_SELECT_THRESHOLD_TOPK only (the batch's K)
dsmoe_status launch_select(const dsmoe_layer_desc& p, const float* scores, uint64_t* mask, int32_t* k_t,
                           cudaStream_t s, int* k_scratch = nullptr);
// launch_finalize = launch_chunk_counts (per chunk of 32 tokens, how many selected each expert) + launch_chunk_scan
// (prefixes over the chunks, counts, offsets)
dsmoe_status launch_chunk_counts(const dsmoe_layer_desc& p, const uint64_t* mask, int32_t* chunk_prefix, cudaStream_t s);
dsmoe_status launch_chunk_scan(const dsmoe_layer_desc& p, int32_t* counts, int32_t* offsets, int32_t* chunk_prefix,
                               int32_t* counts_out, cudaStream_t s);
dsmoe_status launch_finalize(const dsmoe_layer_desc& p, const uint64_t* mask, int32_t* counts,
                             int32_t* offsets, int32_t* chunk_prefix, int32_t* counts_out, cudaStream_t s);

// ---- permute.cu
// zero_out (optional): the layer output [T,d]; rows of tokens that selected no expert are set to zero
dsmoe_status launch_permute(const dsmoe_layer_desc& p, const void* x, const float* scores,
                            const uint64_t* mask, const int32_t* offsets, const int32_t* chunk_prefix,
                            int32_t* row_token, float* row_gate, int32_t* token_rows, void* xp,
                            cudaStream_t s, void* zero_out = nullptr, const ZeroInts& zero = ZeroInts{});
// Grouping for the fused layers: counts, offsets and the row indices of launch_finalize + launch_permute (without a
// grouped copy of x).  chunk_counts_ready: chunk_prefix already holds the chunks' counts (the router wrote them).
dsmoe_status launch_group(const dsmoe_layer_desc& p, const float* scores, const uint64_t* mask, int32_t* counts,
                          int32_t* offsets, int32_t* chunk_prefix, int32_t* counts_out, int32_t* row_token,
                          float* row_gate, int32_t* token_rows, cudaStream_t s, void* zero_out, bool chunk_counts_ready,
                          const ZeroInts& zero = ZeroInts{});
// Selection statistics (see dsmoe_stats)
dsmoe_status launch_stats(const dsmoe_layer_desc& p, const float* scores, const uint64_t* mask,
                          dsmoe_selection_stats* stats, cudaStream_t s);
// yp_f32: the rows are fp32 whatever p.dtype says; row_gate == NULL: the rows are gate-weighted already
dsmoe_status launch_combine(const dsmoe_layer_desc& p, const void* yp, const float* row_gate,
                            const int32_t* token_rows, const int32_t* k_t, void* out, cudaStream_t s,
                            bool yp_f32 = false);
// Whether dsmoe_layer_forward's tensor-core grouped path aggregates inside the down-projection (see dsmoe.h).  The library's own choice
// (fuse_combine == 0) is the second kernel, both projections then being one launch, except for wide experts of very many rows.  us a layer of
// 32 experts, inside and beside: 8192 tokens of d 2048, H 1024 top-4 610, 333, top-12 (3072 rows an expert) 1018, 925; of d 3072, H 1536 top-4
// 910, 673, top-6 1105, 988, top-12 1906, 1962; 5000 tokens top-12 (1875 rows) 1230, 1210; 3333 tokens 959, 774.
static inline bool fuses_combine(const dsmoe_layer_desc& p) {
    if (p.fuse_combine != 0) return p.fuse_combine == 1;
    return p.mode == DSMOE_SELECT_TOPK && p.H >= 1536 && (long long)p.T * width_of(p) >= 2560ll * p.E;
}
dsmoe_status launch_pack(const dsmoe_layer_desc& p, const void* W1, const void* W2, void* packed,
                         cudaStream_t s);

// ---- mlp_generic.cu : plain fp32-FMA grouped GEMMs (any dtype, no packed weights needed)
// x: the grouped rows; with row_token, the tokens, of which grouped row r is row_token[r]
dsmoe_status launch_mlp_generic(const dsmoe_layer_desc& p, const void* x, const void* W1, const void* W2,
                                const int32_t* offsets, float* h, void* yp, cudaStream_t s,
                                const int32_t* row_token = nullptr);


// ---- layer_f32.cu : the whole layer for small fp32 layers, three launches
bool layer_f32_supported(const dsmoe_layer_desc& p);
dsmoe_status launch_layer_f32(const dsmoe_layer_desc& p, const void* x, const float* Wr, const float* br, const void* W1, const void* W2,
                              float* scores, uint64_t* mask, int32_t* k_t, int32_t* counts_out, void* out, char* ws, const WsLayout& L,
                              cudaStream_t s);

// ---- mlp_umma.cu : tcgen05 / TMEM / TMA kernels on packed bf16 weights
dsmoe_status timing_enable(int n_pairs);
dsmoe_status timing_read(float* ms, int n_max, int* n);
bool umma_supported(const dsmoe_layer_desc& p);   // bf16, d and H multiples of 64
// Router for many tokens (router_umma.cu): logits on the tensor cores (bf16 x; Wr split exactly into three bf16 terms, fp32
// accumulation), softmax, selection; mask, k_t and chunk_counts (see launch_group) optional.
// max_run > 0: no accumulator sums over more 64-wide blocks of d than this (kRouterExactRun: the scores are then closer to 64
// bits than router_tile_kernel's, measured at d 2048 to 6144, 8 to 64 experts, 300 to 16384 tokens).
constexpr int kRouterExactRun = 7;
bool router_umma_supported(const dsmoe_layer_desc& p, int max_run = 0);
dsmoe_status launch_router_umma(const dsmoe_layer_desc& p, const void* x, const float* Wr, const float* br,
                                float* scores, uint64_t* mask, int32_t* k_t, int32_t* dev_status, cudaStream_t s,
                                int32_t* chunk_counts = nullptr, int max_run = 0, const ZeroInts& zero = ZeroInts{});
// Router for some hundred tokens (router_cluster.cu), as launch_router_umma otherwise.
bool router_cluster_supported(const dsmoe_layer_desc& p);
dsmoe_status launch_router_cluster(const dsmoe_layer_desc& p, const void* x, const float* Wr, const float* br, float* scores, uint64_t* mask,
                                   int32_t* k_t, cudaStream_t s, int32_t* chunk_counts, const ZeroInts& zero = ZeroInts{});
// Grouped expert MLPs on expert-sorted rows: h = GeLU(xp.W1[e]) (bf16, in `hbuf`), yp = h.W2[e].
// With row_token (and x), the up-projection gathers its rows from x by index and xp is not read.
// With cmb->out, the down-projection's epilogue also aggregates (Eq. 1's weighted sum, ascending expert order per
// token): it writes the layer output cmb->out [T,d] and yp is not touched.  With cmb->out == NULL only the gate
// multiply moves into the epilogue: yp[r,:] = row_gate[r] * e(x)[r,:], stored as fp32.
struct CombineArgs {
    const int32_t* row_token;
    const float* row_gate;
    const uint64_t* mask;
    float* acc;          // fp32 [T,d] running sums (unused when the output itself is fp32)
    int* tile_done;      // E * ceil(d / 256) ints
    void* out;
};
// With moa, the layer is the mixture of attention heads (Eq. 7-8): the up-projection is the experts' query projection
// (no activation) and every grouped row attends to its sequence's keys and values before the down-projection.
struct MoaCore {
    int n_head, n_seq, L;
    float scale;
    const void* Kc;
    const void* Vc;          // [n_seq][n_head][L][d_head]
    const int32_t* tok_seq;  // [T] or NULL (one sequence)
    const int32_t* pos;      // [T]: token t sees keys 0..pos[t]
    const int32_t* token_rows;   // [T, W]: the grouped rows of each token (from the permute step)
    // the dense form of the output projection (moa_dense_down): gate-weighted attention outputs go to dense[T][E*H]
    void* dense;
    const uint64_t* mask;
    const float* row_gate;
};
// Whether launch_moa_attention takes the kernel whose tiles share their copies of the keys (`dense` needs it)
bool moa_shares_keys(const dsmoe_layer_desc& p, const MoaCore& c);
// Output projection and the weighted sum of Eq. 8 as ONE dense GEMM over the experts side by side, out = dense . Wo[E*H, d], as
// in the dense forward: E / K times the multiplications of the grouped form, but at the rate of a long reduction (E * H
// instead of H) and without expert outputs written to and read back from memory as fp32 rows (8 bytes per row and column).
// By the measured costs of both -- dense 1.43 fs per expert, hidden unit, token and column, grouped 1.6 ps plus 2 fs per hidden
// unit for each selected expert -- the dense form wins while E * H < K * (H + 640) or so.  6B prompts (8 experts of 512, top-5,
// 8192 tokens): 203 + 122 us grouped, 174 us dense.  Needs row tiles enough to cover the SMs, and the scratch of the
// grouped form's fp32 rows for the [T, E*H] buffer.
static inline bool moa_dense_down(const dsmoe_layer_desc& p, int sms) {
    if (p.fuse_combine != 0 || (p.mode != DSMOE_SELECT_TOPK && p.mode != DSMOE_SELECT_ALL)) return false;
    const long long K = width_of(p);
    return (long long)p.E * p.H < K * (p.H + 640ll) && (long long)p.E * p.H <= (fuses_combine(p) ? 2ll : 2ll * K) * p.d &&
           (long long)ceil_div(p.T, 128) * ceil_div(p.d, 256) >= sms;
}

dsmoe_status launch_mlp_umma(const dsmoe_layer_desc& p, const void* xp, const void* packed, const int32_t* offsets,
                             void* hbuf, void* yp, int32_t* dev_status, cudaStream_t s, const void* x = nullptr,
                             const int32_t* row_token = nullptr, const CombineArgs* cmb = nullptr,
                             const MoaCore* moa = nullptr);

// ---- mlp_grouped.cu : both projections of the sparse expert MLPs in one launch
// Where its counters lie in the workspace (zeroed beforehand: ZeroInts); fits: there is room for them
struct GroupedScratch {
    size_t sync, sync_ints;
    bool fits;
};
GroupedScratch grouped_scratch(const dsmoe_layer_desc& p, const WsLayout& L);
// Whether the launch finds its rows in the selection words itself, without a row-index kernel before it
constexpr int kGroupedFoldWords = 64 * 33;
static inline bool grouped_folds(const dsmoe_layer_desc& p) { return p.T <= (p.E <= 32 ? 2048 : 1024); }
struct GroupedFold {
    const uint64_t* mask;
    const float* scores;
    int32_t *token_rows, *counts, *offsets;      // written: what the row-index kernel would have
    int32_t* counts_out;                         // nullable, written
};
// rows [Amax, d] fp32: the gate-weighted expert outputs.  With `fold`, offsets, row_token and row_gate are not read
dsmoe_status launch_grouped_layer(const dsmoe_layer_desc& p, const void* x, const void* packed, const int32_t* offsets,
                                  const int32_t* row_token, const float* row_gate, const GroupedFold* fold, float* rows, char* ws,
                                  const WsLayout& L, int32_t* dev_status, cudaStream_t s);

// ---- moa.cu : the attention step of the mixture-of-attention-heads layer
bool moa_supported(const dsmoe_layer_desc& p, int n_head, int L);
// qa [Amax, H] bf16: the grouped rows' queries on entry, their attention outputs on return
dsmoe_status launch_moa_attention(const dsmoe_layer_desc& p, const MoaCore& c, void* qa, const int32_t* row_token,
                                  const int32_t* token_rows, const int32_t* offsets, int32_t* dev_status, cudaStream_t s);
// ---- moa_decode.cu : the whole layer of attention heads for a few decoding tokens, three launches
bool moa_decode_supported(const dsmoe_layer_desc& p, const MoaCore& c);
dsmoe_status launch_moa_decode(const dsmoe_layer_desc& p, const MoaCore& c, const void* x, const float* Wr, const float* br, const void* packed,
                               float* scores, uint64_t* mask, int32_t* k_t, int32_t* counts_out, void* out, char* ws, const WsLayout& L,
                               int32_t* dev_status, cudaStream_t s);
// ---- few_tokens.cu : the whole layer for a handful of tokens, one cooperative launch
bool few_fits(const dsmoe_layer_desc& p, int ctas);
bool few_supported(const dsmoe_layer_desc& p, const void* packed);
dsmoe_status launch_layer_few(const dsmoe_layer_desc& p, const void* x, const float* Wr, const float* br, const void* packed,
                              float* scores, uint64_t* mask, int32_t* k_t, int32_t* counts_out, void* out, char* ws, const WsLayout& L,
                              int32_t* dev_status, cudaStream_t s);
// Whole-layer paths that need no grouping (all experts selected, or few tokens).  *done = false
// means "not taken": the caller continues with the grouped path.
// Whole layer for few tokens (T <= 128) in one cooperative launch, router included.
bool small_supported(const dsmoe_layer_desc& p);
dsmoe_status launch_layer_small(const dsmoe_layer_desc& p, const void* x, const float* Wr, const float* br,
                                const void* packed, float* scores, uint64_t* mask, int32_t* k_t, int32_t* counts_out,
                                void* out, char* ws, const WsLayout& L, int32_t* dev_status, cudaStream_t s);
dsmoe_status launch_layer_umma(const dsmoe_layer_desc& p, const void* x, const void* packed, const float* scores,
                               int32_t* counts_out, void* out, char* ws, const WsLayout& L, int32_t* dev_status, cudaStream_t s,
                               bool* done);

// ---- training.cu / mlp_umma.cu : the training side (Eq. 2-6)
size_t mi_scratch_bytes();
dsmoe_status launch_mi_loss(const dsmoe_layer_desc& p, const float* scores, float* out3, float* grad, char* scratch,
                            cudaStream_t s);
dsmoe_status launch_dense_backward_plain(const dsmoe_layer_desc& p, const void* x, const void* W1, const void* W2,
                                         const float* scores, const uint64_t* mask, const void* dO, float* dS, void* dA,
                                         cudaStream_t s);
// out[T,d] = hg[T, E*H] . W2 over the experts side by side (the dense forward's down-projection)
dsmoe_status launch_dense_down(const dsmoe_layer_desc& p, const void* hg, const void* packed, void* out, int32_t* dev_status,
                               cudaStream_t s);
dsmoe_status launch_dense_backward(const dsmoe_layer_desc& p, const void* x, const void* W2, const void* packed,
                                   const float* scores, const uint64_t* mask, const void* dO, float* dS, void* dA,
                                   void* act, float* dot_part, int32_t* dev_status, cudaStream_t s);

}  // namespace dsmoe
