// Arg-best pass of greedy acceptance: one coalesced, vectorised read of every live logits row produces, per (row, chunk),
// the chunk's best (logit, token).  It is HBM-bound: each logit is read exactly once, with 16-byte streaming loads, and a
// block keeps its whole chunk (16 or 32 values per thread) in registers, so every load of the chunk is in flight at once.
#include <algorithm>

#include "common.cuh"

namespace radar {

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kEmptyIdx = 0x40000000;          // empty slots sort after every real token id

template <typename T> struct Vec;
template <> struct Vec<float> {
    static constexpr int N = 4;
    __device__ static __forceinline__ void load(const float* p, float (&out)[4]) {
        const float4 v = __ldcs(reinterpret_cast<const float4*>(p));
        out[0] = v.x; out[1] = v.y; out[2] = v.z; out[3] = v.w;
    }
};
template <> struct Vec<__nv_bfloat16> {
    static constexpr int N = 8;
    __device__ static __forceinline__ void load(const __nv_bfloat16* p, float (&out)[8]) {
        const uint4 v = __ldcs(reinterpret_cast<const uint4*>(p));
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            out[2 * j] = __uint_as_float(w[j] << 16);
            out[2 * j + 1] = __uint_as_float(w[j] & 0xffff0000u);
        }
    }
};

__device__ __forceinline__ float max_nan(float a, float b) {
    float y;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(y) : "f"(a), "f"(b));
    return y;
}

// EPT = values per thread kept in registers (a multiple of the vector width), chunk = kThreads * EPT
template <typename T, int EPT>
__global__ void __launch_bounds__(kThreads, 5) vocab_pass_kernel(const VocabPassParams p) {
    chain_wait();
    using VT = Vec<T>;
    constexpr int N = VT::N;
    constexpr int NV = EPT / N;
    // grid = (chunks, rows of a sequence, sequences): no division on the way to the block's data
    const int chunk_id = blockIdx.x, f = blockIdx.y, seq = blockIdx.z;
    const int row = seq * p.F + f;
    if (f >= p.seq_rows[seq]) return;

    const T* base = reinterpret_cast<const T*>(p.logits) + (int64_t)seq * p.seq_stride + (int64_t)f * p.row_stride;
    const int e0 = min(chunk_id * p.chunk, p.V);
    const int e1 = min(e0 + p.chunk, p.V);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    // scalar head up to the first 16-byte boundary, vector body, scalar tail
    const uintptr_t addr = reinterpret_cast<uintptr_t>(base + e0);
    int head = (int)(((16 - (addr & 15)) & 15) / sizeof(T));
    head = min(head, e1 - e0);
    const int body0 = e0 + head;
    const int nvec = (e1 - body0) / N;             // <= kThreads * NV because chunk == kThreads * EPT
    const int tail0 = body0 + nvec * N;
    const int ntail = e1 - tail0;

    // ---- every load of the chunk in flight ----
    float x[NV][N];
    const T* vbase = base + body0;
    if (head == 0 && nvec == kThreads * NV) {        // a whole, aligned chunk (all but a row's last one): nothing to check
        const T* vp = vbase + (int64_t)tid * N;
#pragma unroll
        for (int u = 0; u < NV; ++u) VT::load(vp + (int64_t)u * (kThreads * N), x[u]);
    } else {
#pragma unroll
        for (int u = 0; u < NV; ++u) {
            const int j = tid + u * kThreads;
            if (j < nvec) {
                VT::load(vbase + (int64_t)j * N, x[u]);
            } else {
#pragma unroll
                for (int e = 0; e < N; ++e) x[u][e] = -CUDART_INF_F;
            }
        }
    }
    // head and tail (each shorter than one vector): one value for threads 0..N-1 and N..2N-1
    float xs = -CUDART_INF_F;
    int xs_idx = -1;
    if (tid < head) xs_idx = e0 + tid;
    else if (tid >= N && tid - N < ntail) xs_idx = tail0 + tid - N;
    if (xs_idx >= 0) xs = to_float(base[xs_idx]);

    // ---- per-thread max (NaN-propagating) ----
    float mxa[4] = {xs, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F};
#pragma unroll
    for (int u = 0; u < NV; ++u)
#pragma unroll
        for (int e = 0; e < N; ++e) mxa[e & 3] = max_nan(mxa[e & 3], x[u][e]);
    const float bv = max_nan(max_nan(mxa[0], mxa[1]), max_nan(mxa[2], mxa[3]));
    const bool nan = bv != bv;

    __shared__ float sh_tv[kWarps];
    __shared__ int sh_ti[kWarps];
    __shared__ int sh_nan;
    if (tid == 0) sh_nan = 0;

    const size_t rec = (size_t)row * p.n_chunks + chunk_id;
    // lowest index that holds the thread's max (index order: head scalar < vector elements < tail scalar)
    int bi = kEmptyIdx + tid;
    if (xs_idx >= 0 && tid >= N && xs == bv) bi = xs_idx;
#pragma unroll
    for (int u = NV - 1; u >= 0; --u) {
        const int idx0 = body0 + (tid + u * kThreads) * N;
        if (tid + u * kThreads < nvec) {
#pragma unroll
            for (int e = N - 1; e >= 0; --e)
                if (x[u][e] == bv) bi = idx0 + e;
        }
    }
    if (xs_idx >= 0 && tid < N && xs == bv) bi = xs_idx;
    float wv = bv;
    int wi = bi;
    warp_best(wv, wi);
    if (lane == 0) { sh_tv[warp] = wv; sh_ti[warp] = wi; }
    __syncthreads();
    if (nan) atomicOr(&sh_nan, 1);
    __syncthreads();
    if (warp == 0) {
        float v = lane < kWarps ? sh_tv[lane] : -CUDART_INF_F;
        int i = lane < kWarps ? sh_ti[lane] : 0x7fffffff;
        warp_best(v, i);
        if (lane == 0) {
            p.part_v[rec] = v;
            p.part_i[rec] = i >= kEmptyIdx ? 0x7fffffff : i;
        }
    }
    if (tid == 0 && sh_nan) set_status(p.status, RADAR_ERR_NUMERIC);
}

template <typename T>
cudaError_t launch_ept(const VocabPassParams& p, dim3 grid, cudaStream_t stream) {
    if (p.chunk / kThreads == 16) return launch_chained(vocab_pass_kernel<T, 16>, grid, dim3(kThreads), 0, stream, p);
    return launch_chained(vocab_pass_kernel<T, 32>, grid, dim3(kThreads), 0, stream, p);
}

}  // namespace

// chunk is 8192 values (32 per thread), or 4096 (16 per thread) when the larger one would leave less than two blocks an SM: a
// block's time is its chain of steps, hardly the size of its chunk, and half as many records are merged behind it.
int vocab_pass_plan_chunks(int sm_count, int rows, int V, int* chunk_out) {
    int chunk = 8192;
    if ((long long)rows * ((V + chunk - 1) / chunk) < 2LL * sm_count) chunk = 4096;
    *chunk_out = chunk;
    return (V + chunk - 1) / chunk;
}

size_t vocab_pass_partial_bytes(int rows, int n_chunks) { return align_up((size_t)rows * n_chunks * 4, 256) * 2; }

// The records of `rows` rows or fewer: below the line of vocab_pass_plan_chunks a row has twice the chunks, so a smaller
// launch may need more than a larger one.
size_t vocab_pass_workspace_bytes(int sm_count, int rows, int V) {
    int chunk;
    const int n = vocab_pass_plan_chunks(sm_count, rows, V, &chunk);
    size_t need = vocab_pass_partial_bytes(rows, n);
    const int c8 = (V + 8191) / 8192, below = std::min(rows, (2 * sm_count - 1) / c8);      // most rows below the line
    if (below > 0) need = std::max(need, vocab_pass_partial_bytes(below, vocab_pass_plan_chunks(sm_count, below, V, &chunk)));
    return need;
}

void vocab_pass_carve(void* ws, int rows, int n_chunks, VocabPassParams* p) {
    p->part_v = reinterpret_cast<float*>(ws);
    p->part_i = reinterpret_cast<int32_t*>(reinterpret_cast<char*>(ws) + align_up((size_t)rows * n_chunks * 4, 256));
}

// Makes the driver load the arg-best instantiations on the current device (kernel images are loaded lazily, at
// first use, and loading allocates): a caller that must not allocate later can have it done at set-up.
cudaError_t vocab_pass_preload_argbest() {
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, vocab_pass_kernel<float, 16>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, vocab_pass_kernel<float, 32>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, vocab_pass_kernel<__nv_bfloat16, 16>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, vocab_pass_kernel<__nv_bfloat16, 32>);
    return e;
}

cudaError_t vocab_pass_launch(radar_ctx* ctx, const VocabPassParams& p, cudaStream_t stream) {
    if (p.n_seq > 65535 || p.F > 65535) return cudaErrorInvalidValue;
    const dim3 grid((unsigned)p.n_chunks, (unsigned)p.F, (unsigned)p.n_seq);
    radar_launch_scope scope(ctx, RADAR_K_VOCAB_ACCEPT, stream);
    return p.dtype == RADAR_F32 ? launch_ept<float>(p, grid, stream) : launch_ept<__nv_bfloat16>(p, grid, stream);
}

}  // namespace radar
