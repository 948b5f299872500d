// Expansion's vocabulary pass: every logits row is read once and leaves its k best (logit, token) pairs, sorted by
// (logit desc, token asc), and its log-sum-exp.
//
// One thread-block cluster per row, each CTA owning a slice of the vocabulary.  A CTA fetches its slice into shared
// memory with bulk copies (all of them in flight at once, three CTAs per SM: 190 KB on the way per SM) and reduces each
// piece as it lands to a running (max, sum of exponentials) per thread.  Selection works on the whole ROW, not on
// chunks of it: the maxima of 32 groups of the row's elements are exchanged through distributed shared memory, and the
// k-th largest of them is a lower bound of the row's k-th best value that only about k + 2 of the row's elements
// reach (k = 10 of 32 groups: 12 expected).  Those few are re-read from shared memory, sent to CTA 0 as 64-bit order
// keys, ranked there by counting and written as the row's final list, so no later kernel merges anything.
// If ties push more elements over the bound than a CTA's list holds, that CTA finds its k best by k rounds of a
// block-wide arg-best and sends those: the same result.
#include "common.cuh"

namespace radar {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kMaxCluster = 8;               // portable cluster size limit
constexpr int kVecs = 4;                     // 16-byte vectors per thread and piece
constexpr int kPieceVecs = kThreads * kVecs;
constexpr int kPieceBytes = kPieceVecs * 16; // 16 KB per bulk copy
constexpr int kSliceBytes = 64 * 1024;       // slice of a CTA while three CTAs fit an SM
constexpr int kMaxSlots = 12;                // pieces in shared memory at most (one CTA per SM)
constexpr int kSeg = 128;                    // candidates a CTA may send
constexpr float kLog2e = 1.4426950408889634f;

template <typename T> struct Vec;
template <> struct Vec<float> {
    static constexpr int N = 4;
    __device__ static __forceinline__ void unpack(const uint4 v, float (&out)[4]) {
        out[0] = __uint_as_float(v.x); out[1] = __uint_as_float(v.y); out[2] = __uint_as_float(v.z); out[3] = __uint_as_float(v.w);
    }
};
template <> struct Vec<__nv_bfloat16> {
    static constexpr int N = 8;
    __device__ static __forceinline__ void unpack(const uint4 v, float (&out)[8]) {
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            out[2 * j] = __uint_as_float(w[j] << 16);
            out[2 * j + 1] = __uint_as_float(w[j] & 0xffff0000u);
        }
    }
};

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float max_nan(float a, float b) {
    float y;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(y) : "f"(a), "f"(b));
    return y;
}
__device__ __forceinline__ float max3_nan(float a, float b, float c) {
    float y;
    asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
    return y;
}
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t map_to(const void* local, uint32_t rank) {
    uint32_t ra;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(smem_addr(local)), "r"(rank));
    return ra;
}

template <typename T>
__global__ void __launch_bounds__(kThreads) row_topk_kernel(const RowTopkParams p) {
    using VT = Vec<T>;
    constexpr int N = VT::N;
    extern __shared__ __align__(128) unsigned char s_data[];          // this CTA's slice (or a ring of its pieces)
    __shared__ __align__(8) uint64_t s_full[kMaxSlots];
    __shared__ __align__(16) float4 s_gm[kMaxCluster * kWarps];       // maxima of the quarters of every warp of the cluster
    __shared__ float s_ws[kMaxCluster * kWarps];                      // ... and its sum of exp(x - warp max)
    __shared__ unsigned long long s_list[kSeg];                       // this CTA's candidates
    __shared__ unsigned long long s_all[kMaxCluster][kSeg];           // CTA 0: everybody's
    __shared__ int s_all_n[kMaxCluster];
    __shared__ int s_cnt;
    __shared__ unsigned long long s_best[kWarps];

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t rank = blockIdx.x, cs = gridDim.x;                 // the cluster spans the grid's x dimension
    const int f = blockIdx.y, seq = blockIdx.z;
    const int k = p.k;
    if (tid == 0) {
        for (int i = 0; i < kMaxSlots; ++i)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&s_full[i])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_cnt = 0;
    }
    __syncthreads();
    cluster_arrive();                                                 // (waited for before the first remote store)
    chain_wait();
    if (p.seq_active != nullptr && p.seq_active[seq] == 0) {          // the same answer in every CTA of the cluster
        cluster_wait();
        return;
    }

    // ---- the row: scalars up to the first 16-byte boundary, vectors, scalars behind the last one ----
    const int64_t row = (int64_t)seq * p.F + f;
    const T* base = reinterpret_cast<const T*>(p.logits) + (int64_t)seq * p.seq_stride + (int64_t)f * p.row_stride;
    const int head = min((int)(((16 - (reinterpret_cast<uintptr_t>(base) & 15)) & 15) / sizeof(T)), p.V);
    const int nvec = (p.V - head) / N;
    const int tail0 = head + nvec * N;
    const int v0 = (int)((long long)nvec * rank / cs), v1 = (int)((long long)nvec * (rank + 1) / cs);
    const int nv = v1 - v0;                                           // vectors of this CTA
    const uint4* gsrc = reinterpret_cast<const uint4*>(base + head) + v0;
    const int n_pieces = (nv + kPieceVecs - 1) / kPieceVecs;
    const bool resident = n_pieces <= p.n_slots;                      // the whole slice stays in shared memory
    auto fetch = [&](int piece) {
        const int slot = piece % p.n_slots;
        const uint32_t bytes = (uint32_t)min(nv - piece * kPieceVecs, kPieceVecs) * 16u;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(&s_full[slot])), "r"(bytes) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                         smem_addr(s_data + (size_t)slot * kPieceBytes)), "l"(gsrc + (int64_t)piece * kPieceVecs), "r"(bytes), "r"(smem_addr(&s_full[slot]))
                     : "memory");
    };
    if (tid == 0)
        for (int q = 0; q < min(n_pieces, p.n_slots); ++q) fetch(q);
    // head and tail (each shorter than a vector) belong to CTA 0: one value for threads 0..N-1 and N..2N-1
    float xs = -CUDART_INF_F;
    int xs_idx = -1;
    if (rank == 0) {
        if (tid < head) xs_idx = tid;
        else if (tid >= N && tid - N < p.V - tail0) xs_idx = tail0 + tid - N;
        if (xs_idx >= 0) xs = to_float(base[xs_idx]);
    }

    // ---- running (max, sum of exponentials) of this thread's values, piece by piece as they land ----
    float m = xs, s = xs > -CUDART_INF_F ? 1.f : 0.f;
    for (int q = 0; q < n_pieces; ++q) {
        const int slot = q % p.n_slots;
        bool ok = false;
        for (uint32_t it = 0; it < (1u << 22) && !ok; ++it) {
            uint32_t done;
            asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                         : "=r"(done) : "r"(smem_addr(&s_full[slot])), "r"((uint32_t)(q / p.n_slots) & 1u) : "memory");
            ok = done != 0;
        }
        if (!ok) set_status(p.status, RADAR_ERR_TIMEOUT);
        const uint4* sv = reinterpret_cast<const uint4*>(s_data + (size_t)slot * kPieceBytes);
        const int here = min(nv - q * kPieceVecs, kPieceVecs);
        float x[kVecs][N];
#pragma unroll
        for (int u = 0; u < kVecs; ++u) {
            const int j = tid + u * kThreads;
            if (j < here) {
                VT::unpack(sv[j], x[u]);
            } else {
#pragma unroll
                for (int e = 0; e < N; ++e) x[u][e] = -CUDART_INF_F;
            }
        }
        float mx[2] = {m, -CUDART_INF_F};
#pragma unroll
        for (int u = 0; u < kVecs; ++u)
#pragma unroll
            for (int e = 0; e < N; e += 2) mx[(e >> 1) & 1] = max3_nan(mx[(e >> 1) & 1], x[u][e], x[u][e + 1]);
        const float mn = max_nan(mx[0], mx[1]);
        if (mn > -CUDART_INF_F) {
            const float nb = -mn * kLog2e;
            float acc[2] = {s * ex2(fmaf(m, kLog2e, nb)), 0.f};       // (m = -inf on the first piece: factor 0)
#pragma unroll
            for (int u = 0; u < kVecs; ++u)
#pragma unroll
                for (int e = 0; e < N; ++e) acc[e & 1] += ex2(fmaf(x[u][e], kLog2e, nb));
            s = acc[0] + acc[1];
        }
        m = mn;
        if (!resident) {                                              // the slot is free once every thread has read it
            __syncthreads();
            if (tid == 0 && q + p.n_slots < n_pieces) fetch(q + p.n_slots);
        }
    }
    if (m != m) set_status(p.status, RADAR_ERR_NUMERIC);

    // ---- quarter-warp maxima and the warp's sum, to every CTA of the cluster ----
    {
        float qm = m;
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) qm = fmaxf(qm, __shfl_xor_sync(kFull, qm, o));
        const float4 g = make_float4(__shfl_sync(kFull, qm, 0), __shfl_sync(kFull, qm, 8), __shfl_sync(kFull, qm, 16), __shfl_sync(kFull, qm, 24));
        const float wm = fmaxf(fmaxf(g.x, g.y), fmaxf(g.z, g.w));
        const float ws = warp_sum(m > -CUDART_INF_F ? s * ex2((m - wm) * kLog2e) : 0.f);
        cluster_wait();                                               // every CTA of the cluster has started
        if (lane < cs) {
            const int at = rank * kWarps + warp;
            asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(map_to(&s_gm[at], lane)), "f"(g.x), "f"(g.y), "f"(g.z), "f"(g.w) : "memory");
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(map_to(&s_ws[at], lane)), "f"(ws) : "memory");
        }
        __syncwarp();
        cluster_arrive();
        cluster_wait();
    }

    // ---- the bound: lane l holds the maximum of group l (quarter l of every CTA's warps); k-th largest of 32 groups ----
    float gv = -CUDART_INF_F;
    for (uint32_t r = 0; r < cs; ++r) gv = fmaxf(gv, reinterpret_cast<const float*>(&s_gm[r * kWarps])[lane]);
    int grank = 0;
#pragma unroll
    for (int o = 0; o < 32; ++o) {
        const float ov = __shfl_sync(kFull, gv, o);
        grank += (ov > gv || (ov == gv && o < lane)) ? 1 : 0;
    }
    const float thr = __shfl_sync(kFull, gv, __ffs(__ballot_sync(kFull, grank == k - 1)) - 1);

    // ---- candidates: this thread's elements at or above the bound ----
    auto for_each = [&](auto&& fn) {                                  // fn(value, token) over this thread's elements
        if (xs_idx >= 0) fn(xs, xs_idx);
        for (int j = tid; j < nv; j += kThreads) {
            float x[N];
            VT::unpack(resident ? *(reinterpret_cast<const uint4*>(s_data) + j) : __ldg(gsrc + j), x);
            const int idx = head + (v0 + j) * N;
#pragma unroll
            for (int e = 0; e < N; ++e) fn(x[e], idx + e);
        }
    };
    if (m >= thr)
        for_each([&](float v, int idx) {
            if (v >= thr) {
                const int at = atomicAdd(&s_cnt, 1);
                if (at < kSeg) s_list[at] = order_key(v, idx);
            }
        });
    __syncthreads();
    int n_mine = s_cnt;
    if (n_mine > kSeg) {
        // more than the list holds: this CTA's k best, one per round
        unsigned long long last = ~0ull;
        for (n_mine = 0; n_mine < k; ++n_mine) {
            unsigned long long best = 0ull;
            for_each([&](float v, int idx) {
                const unsigned long long key = order_key(v, idx);
                if (key < last && key > best) best = key;
            });
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) best = max(best, __shfl_xor_sync(kFull, best, o));
            __syncthreads();                                          // (last round's readers are done)
            if (lane == 0) s_best[warp] = best;
            __syncthreads();
            best = s_best[0];
#pragma unroll
            for (int w = 1; w < kWarps; ++w) best = max(best, s_best[w]);
            if (best == 0ull) break;                                  // fewer than k elements
            if (tid == 0) s_list[n_mine] = best;
            last = best;
        }
        __syncthreads();
    }
    if (tid < n_mine) asm volatile("st.shared::cluster.b64 [%0], %1;" ::"r"(map_to(&s_all[rank][tid], 0)), "l"(s_list[tid]) : "memory");
    if (tid == 0) asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(map_to(&s_all_n[rank], 0)), "r"(n_mine) : "memory");
    __syncwarp();
    cluster_arrive();
    if (rank != 0) return;                                            // (nothing is written to this CTA any more)

    // ---- CTA 0: log-sum-exp of the row in fp64, and the ranks of the candidates ----
    if (warp == kWarps - 1) {
        const int n = (int)cs * kWarps;
        float wm[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const float4 g = s_gm[min(lane + 32 * i, n - 1)];
            wm[i] = lane + 32 * i < n ? fmaxf(fmaxf(g.x, g.y), fmaxf(g.z, g.w)) : -CUDART_INF_F;
        }
        const float M = warp_max(fmaxf(wm[0], wm[1]));
        double S = 0.0;
#pragma unroll
        for (int i = 0; i < 2; ++i)
            if (wm[i] > -CUDART_INF_F) S += (double)s_ws[lane + 32 * i] * exp((double)wm[i] - (double)M);
        S = warp_sum(S);
        if (lane == 0) p.rec_lse[row] = (double)M + log(S);
    }
    __syncwarp();
    cluster_wait();
    int total = 0;
    for (uint32_t r = 0; r < cs; ++r) total += s_all_n[r];
    float* out_v = p.rec_v + row * k;
    int32_t* out_i = p.rec_i + row * k;
    for (int c = tid; c < total; c += kThreads) {
        int at = c;
        uint32_t r = 0;
        while (at >= s_all_n[r]) at -= s_all_n[r++];
        const unsigned long long key = s_all[r][at];
        int rk = 0;
        for (uint32_t o = 0; o < cs; ++o)
            for (int j = 0; j < s_all_n[o]; ++j) rk += s_all[o][j] > key ? 1 : 0;
        if (rk < k) { out_v[rk] = key_value(key); out_i[rk] = key_index(key); }
    }
    for (int c = total + tid; c < k; c += kThreads) { out_v[c] = -CUDART_INF_F; out_i[c] = 0x7fffffff; }
}

}  // namespace

size_t row_topk_record_bytes(int rows, int k) { return align_up((size_t)rows * 8, 256) + 2 * align_up((size_t)rows * k * 4, 256); }

void row_topk_carve(void* ws, int rows, int k, RowTopkParams* p) {
    char* c = reinterpret_cast<char*>(ws);
    p->rec_lse = reinterpret_cast<double*>(c); c += align_up((size_t)rows * 8, 256);
    p->rec_v = reinterpret_cast<float*>(c); c += align_up((size_t)rows * k * 4, 256);
    p->rec_i = reinterpret_cast<int32_t*>(c);
}

cudaError_t row_topk_launch(radar_ctx* ctx, RowTopkParams p, cudaStream_t stream) {
    if (p.n_seq > 65535 || p.F > 65535) return cudaErrorInvalidValue;
    // CTAs per row: as few as keep a slice within 64 KB (three CTAs per SM), and more, down to 8 KB a slice, while
    // the launch leaves SMs without work.  Rows longer than eight such slices take more shared memory per CTA, and
    // beyond what a CTA can have the slice goes through it as a ring.
    const long long bytes = (long long)p.V * (p.dtype == RADAR_F32 ? 4 : 2);
    const long long rows = (long long)p.n_seq * p.F;
    int cs = 1;
    while (cs < kMaxCluster && bytes > (long long)cs * kSliceBytes) cs *= 2;
    while (cs < kMaxCluster && rows * cs * 2 <= ctx->sm_count && bytes >= 2LL * cs * 8192) cs *= 2;
    const long long slice_pieces = ((bytes + cs - 1) / cs + kPieceBytes - 1) / kPieceBytes;
    p.n_slots = (int)(slice_pieces < 1 ? 1 : slice_pieces < kMaxSlots ? slice_pieces : kMaxSlots);
    const size_t smem = (size_t)p.n_slots * kPieceBytes;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)cs, (unsigned)p.F, (unsigned)p.n_seq);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)cs;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    radar_launch_scope scope(ctx, RADAR_K_VOCAB_EXPAND, stream);
    if (p.dtype == RADAR_F32) {
        const cudaError_t e = radar_opt_in_smem(ctx, RADAR_SMEM_ROW_TOPK, row_topk_kernel<float>, smem);
        return e != cudaSuccess ? e : cudaLaunchKernelEx(&cfg, row_topk_kernel<float>, p);
    }
    const cudaError_t e = radar_opt_in_smem(ctx, RADAR_SMEM_ROW_TOPK + 1, row_topk_kernel<__nv_bfloat16>, smem);
    return e != cudaSuccess ? e : cudaLaunchKernelEx(&cfg, row_topk_kernel<__nv_bfloat16>, p);
}

}  // namespace radar
