// Shared device/host helpers of the RADAR hot-path library (sm_100a).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math_constants.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>

#include "../../include/radar.h"

// kernels the library launches (index into the profiling tables)
enum radar_kernel_id {
    RADAR_K_VOCAB_EXPAND = 0,   // expansion: top-k and log-normaliser of every row
    RADAR_K_SELECT_GATE,        // frontier selection + prediction model
    RADAR_K_TREE_BUILD,
    RADAR_K_ATTN,               // tree attention main kernel
    RADAR_K_ATTN_COMBINE,
    RADAR_K_VOCAB_ACCEPT,       // row-argmax pass of greedy acceptance
    RADAR_K_GREEDY_WALK,
    RADAR_K_STOCH_WALK,
    RADAR_K_ACCLEN_NODES,       // per-row conditional acceptance probabilities (Eq. 13)
    RADAR_K_ACCLEN_DIST,        // path products and the length distribution (Eq. 11-12)
    RADAR_K_GATE_FEATURES,      // input-side products of the hidden-state policy (Table 3)
    RADAR_K_TRAIN_ROLLOUT,      // REINFORCE step: rollout + backpropagation through time per data point
    RADAR_K_TRAIN_OUTER,        // REINFORCE step: parameter gradients
    RADAR_K_TRAIN_ADAM,         // REINFORCE step: batch loss + Adam update
    RADAR_K_ROW_MERGE,          // expansion: the merge of a long pass's rows
    RADAR_K_EXPAND_CALLS,       // radar_expand_calls: the calls of a sequence in one kernel
    RADAR_K_COUNT
};

// kernels whose blocks may take more than 48 KB of shared memory: one slot per instantiation
enum radar_smem_slot {
    RADAR_SMEM_SELECT_GATE = 0,
    RADAR_SMEM_SELECT_GATE_CLUSTER,   // the instantiation with helper blocks
    RADAR_SMEM_EXPAND_CALLS,
    RADAR_SMEM_EXPAND_CALLS_PLAIN,    // the instantiation without helper blocks
    RADAR_SMEM_TREE_BUILD,
    RADAR_SMEM_TRAIN_ROLLOUT,   // + log2 of the points a block
    RADAR_SMEM_WALK = RADAR_SMEM_TRAIN_ROLLOUT + 3,            // + 2 * (bf16) + CTAs per SM - 1
    RADAR_SMEM_ACCLEN = RADAR_SMEM_WALK + 4,        // the same
    RADAR_SMEM_ATTN_FMA = RADAR_SMEM_ACCLEN + 4,        // + 4 * (bf16) + 2 * (d == 128) + (clusters)
    RADAR_SMEM_ATTN_TC = RADAR_SMEM_ATTN_FMA + 8,   // + 8 * fine + 4 * (d == 128) + 2 * two + paged
    RADAR_SMEM_COUNT = RADAR_SMEM_ATTN_TC + 16
};

struct radar_ctx {
    int device;
    int sm_count;
    // dynamic shared memory opted in to, per kernel, ON THIS CONTEXT'S DEVICE (the attribute is per device: a second device
    // in the same process needs its own opt-in); 0: not yet
    size_t smem_room[RADAR_SMEM_COUNT];
    int* d_status;          // sticky device status word
    int acclen_clusters[4][4];   // clusters of 1, 2, 4, 8 of each per-row kernel of Eq. 11-13 that are resident at once (0: not asked yet)
    // launch accounting (host side)
    long long launches[RADAR_K_COUNT];
    // optional per-kernel CUDA-event timing
    bool profiling;
    cudaEvent_t* ev;        // 2 * ev_cap events
    int* ev_kernel;         // kernel id of record i
    int ev_cap, ev_used;
    double prof_ms[RADAR_K_COUNT];
    long long prof_n[RADAR_K_COUNT];
};

// Brackets one kernel launch: counts it and, while profiling, records an event pair on its stream.
struct radar_launch_scope {
    radar_ctx* c;
    cudaStream_t s;
    int slot;
    radar_launch_scope(radar_ctx* ctx, int kernel, cudaStream_t stream) : c(ctx), s(stream), slot(-1) {
        c->launches[kernel]++;
        if (c->profiling && c->ev_used < c->ev_cap) {
            slot = c->ev_used++;
            c->ev_kernel[slot] = kernel;
            cudaEventRecord(c->ev[2 * slot], s);
        }
    }
    ~radar_launch_scope() {
        if (slot >= 0) cudaEventRecord(c->ev[2 * slot + 1], s);
    }
};

// Every kernel of the library is launched with programmatic stream serialization, and most begin with
// chain_wait(): the next kernel's launch and block scheduling overlap the tail of the previous one, and
// nothing of such a kernel touches memory before its predecessor (and, transitively, every earlier kernel
// of the stream) has completed and flushed.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_chained(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                                  Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}
__device__ __forceinline__ void chain_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
// The two halves, for kernels that do work that cannot depend on the predecessor before they wait for
// it.  Rules that keep the chain sound: (1) every block runs chain_sync() in at least one thread
// before it exits, so "kernel N complete" always implies "kernel N-1 complete"; (2) nothing written by
// the immediate predecessor is read, and nothing it reads is written, before chain_sync() (or a block
// barrier behind a thread that ran it); (3) what kernels ahead of the predecessor wrote may be read before
// chain_sync() only if that is complete when the block starts: the predecessor triggers behind its own wait,
// or its own predecessor does and all that is read is older than that one.
// Ahead of their own wait trigger: row_merge_kernel, expand_select_gate_kernel (but not where it is launched on
// its own) and the tensor-core attention.  Read before their wait: row_merge_kernel, nothing but L2 prefetches;
// expand_select_gate_kernel (again not on its own) and expand_calls_kernel, the weights and the state that earlier
// calls have left: both always stand behind row_topk_kernel, which triggers behind its wait, or behind
// row_merge_kernel, whose predecessor row_pass_kernel does.  Whatever follows one of the early triggers waits first.
__device__ __forceinline__ void chain_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_sync() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Raises a kernel's dynamic shared-memory limit on the context's device, once, to all that its static arrays leave of a
// block's shared memory.  (The 48 KB that need no opt-in count the static arrays too, so a limit that looks at the dynamic
// bytes alone refuses launches; and the limit belongs to the kernel, not to the context: every context has to set the
// same one, or a small launch of one would take the room from another.)  Not a stream operation.
template <typename K>
inline cudaError_t radar_opt_in_smem(radar_ctx* ctx, int slot, K kernel, size_t bytes) {
    size_t& room = ctx->smem_room[slot];
    if (room == 0) {
        cudaFuncAttributes fa;
        int block = 0;
        cudaError_t e = cudaFuncGetAttributes(&fa, kernel);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&block, cudaDevAttrMaxSharedMemoryPerBlockOptin, ctx->device);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, block - (int)fa.sharedSizeBytes);
        if (e != cudaSuccess) return e;
        room = (size_t)block - fa.sharedSizeBytes;
    }
    return bytes <= room ? cudaSuccess : cudaErrorInvalidValue;
}

// A failing runtime call becomes RADAR_ERR_CUDA; with RADAR_DEBUG set in the environment the call and the
// runtime's message are also written to stderr.
#define RADAR_CUDA_CHECK(expr)                                                                     \
    do {                                                                                           \
        cudaError_t _e = (expr);                                                                   \
        if (_e != cudaSuccess) {                                                                   \
            if (getenv("RADAR_DEBUG")) fprintf(stderr, "radar: %s -> %s\n", #expr, cudaGetErrorString(_e)); \
            return RADAR_ERR_CUDA;                                                                 \
        }                                                                                          \
    } while (0)

namespace radar {

constexpr int kMaxNodes = RADAR_MAX_NODES;
constexpr int kHidden = RADAR_GATE_HIDDEN;
constexpr unsigned kFull = 0xffffffffu;

// first error wins
__device__ __forceinline__ void set_status(int* status, int code) { atomicCAS(status, 0, code); }

__device__ __forceinline__ float to_float(float x) { return x; }
__device__ __forceinline__ float to_float(__nv_bfloat16 x) { return __bfloat162float(x); }

// (value desc, index asc) ordering: true if a precedes b
__device__ __forceinline__ bool precedes(float va, int ia, float vb, int ib) {
    return va > vb || (va == vb && ia < ib);
}

template <typename T>
__device__ __forceinline__ T warp_max(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(kFull, v, o));
    return v;
}
template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

// Sums of N values over the warp's 32 lanes, N a power of two: lane l returns the sum of value l / (32 / N).  Halving the
// values with every exchange costs N - 1 + log2(32 / N) shuffles; N butterflies would cost 5 N, and an SM passes one
// warp's shuffle a clock.
template <int N>
__device__ __forceinline__ float transposed_sum(float (&v)[N]) {
    const int lane = threadIdx.x & 31;
    int o = 16;
#pragma unroll
    for (int m = N / 2; m > 0; m >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < m; ++i) {
            const float give = up ? v[i] : v[i + m], keep = up ? v[i + m] : v[i];
            v[i] = keep + __shfl_xor_sync(kFull, give, o);
        }
    }
    float t = v[0];
    for (; o > 0; o >>= 1) t += __shfl_xor_sync(kFull, t, o);
    return t;
}

// best (value desc, index asc) pair over the warp, in every lane
__device__ __forceinline__ void warp_best(float& v, int& i) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(kFull, v, o);
        const int oi = __shfl_xor_sync(kFull, i, o);
        if (precedes(ov, oi, v, i)) { v = ov; i = oi; }
    }
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// where another block of the cluster has this block's shared variable *p
__device__ __forceinline__ uint32_t cluster_addr(const void* p, uint32_t rank) {
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_addr(p)), "r"(rank));
    return a;
}

// --- best logit of every row (vocab_pass.cu) ----------------------------------------------
// One launch reduces every (row, chunk) of a [rows][V] logits matrix to its best (logit, token).
// rows are addressed as base + seq * seq_stride + f * row_stride with row = seq * F + f; rows whose
// index within the sequence is >= nrows[seq] are not read.
struct VocabPassParams {
    const void* logits;
    int dtype;
    int64_t row_stride, seq_stride;
    int n_seq, F, V;
    int n_chunks, chunk;             // chunk = elements per chunk (multiple of 8)
    const int32_t* seq_rows;         // rows to process per sequence
    float* part_v;                   // [rows][n_chunks]
    int32_t* part_i;                 // [rows][n_chunks]
    int* status;
};
int vocab_pass_plan_chunks(int sm_count, int rows, int V, int* chunk_out);   // returns n_chunks
size_t vocab_pass_partial_bytes(int rows, int n_chunks);
size_t vocab_pass_workspace_bytes(int sm_count, int rows, int V);       // for up to `rows` rows
void vocab_pass_carve(void* ws, int rows, int n_chunks, VocabPassParams* p);
cudaError_t vocab_pass_launch(radar_ctx* ctx, const VocabPassParams& p, cudaStream_t stream);
cudaError_t vocab_pass_preload_argbest();

// --- top-k and log-normaliser of rows (row_topk.cu) ------------------------------------------
// Rows as above; those of sequences with seq_active[seq] == 0 (if not NULL) are not read.
struct RowTopkParams {
    const void* logits;
    int dtype;
    int64_t row_stride, seq_stride;
    int n_seq, F, V, k;
    const uint8_t* seq_active;
    int32_t* tok;                    // [rows][k] in the workspace: tokens in order (kNanRow set where the row has a NaN),
    double* logp;                    // [rows][k] and their log-probabilities
    int spans, n_slots, lines;       // shares of a row, warps that go through them, and how many a warp has at most
    int live, per;                   // the merge's bound: warps that have maxima, and how many of each it looks at
    float* gmax;                     // [rows][n_slots][32]: largest logit of every group of a warp's
    float2* part;                    // [rows][n_slots]: (max, sum exp(logit - max)); max is NaN if there is one
    int* status;
};
constexpr int32_t kNanRow = INT32_MIN;
size_t row_topk_workspace_bytes(int rows, int V, int k);
void row_topk_carve(RowTopkParams& p, void* ws);      // sets what follows seq_active, from the rest
cudaError_t row_topk_launch(radar_ctx* ctx, RowTopkParams p, cudaStream_t stream);

// --- hidden-state policy (expand.cu) -----------------------------------------------------------
// Input-side products of the a.B rows of a.features: pre [B][4H] = W_ih f, and behind it [B][H] = W_1[:, H:] f.
cudaError_t gate_features_launch(radar_ctx* ctx, const radar_expand_args& a, float* pre, cudaStream_t stream);

// --- workspace-free greedy acceptance (verify_accept.cu) --------------------------------------
// Resolves the device address of the library's scratch array on the current device and loads the two kernels of
// that path, so that nothing is left for the driver to allocate at the first call.  Called by radar_create.
int noalloc_prepare_device(int device);

// --- tensor-core tree attention (tree_attention_tc.cu) --------------------------------------
constexpr int kTcMaxRatio = 128;         // query heads per KV head: a row block holds whole nodes
bool tree_attn_tc_supported(const radar_attn_args* a);
size_t tree_attn_tc_workspace_bytes(const radar_ctx* ctx, int B, int Hq, int Hkv, int d, int max_prefix_len);
int tree_attn_tc_launch(radar_ctx* ctx, const radar_attn_args* a, cudaStream_t stream);

static inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

}  // namespace radar
