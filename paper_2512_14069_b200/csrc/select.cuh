// Pieces shared by the kernels that follow a vocabulary pass (expand.cu, expand_calls.cu): the merge of a row's chunk
// records, and the cluster helpers of the recurrent product.
#pragma once
#include "common.cuh"

namespace radar {
namespace {

constexpr int kSelThreads = 1024;
constexpr int kSelWarps = kSelThreads / 32;
constexpr int kMaxF = 32;
constexpr int kSurvCap = 256;                        // per-row survivor list of the parallel merge (even: read in pairs)
constexpr int kSelCluster = 4;                       // blocks per sequence when the recurrent product is shared out,
constexpr long long kShortPassLogits = 4 << 20;      // ... which is done while a call's vocabulary pass reads at most this many logits

__device__ __forceinline__ float sigmoidf_(float x) { return 1.f / (1.f + expf(-x)); }

__device__ __forceinline__ void group_barrier(int id) { asm volatile("bar.sync %0, 512;" ::"r"(id) : "memory"); }
__device__ __forceinline__ void cp_async4(void* smem, const void* gmem) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Thread-block cluster pieces of the select + gate block: stores and barrier arrivals into block 0's shared memory.
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ void st_cluster_f32(const float* local, uint32_t rank, float v) {
    asm volatile("{\n\t.reg .b32 ra;\n\tmapa.shared::cluster.u32 ra, %0, %1;\n\tst.shared::cluster.f32 [ra], %2;\n\t}" ::"r"(
                     smem_addr(local)), "r"(rank), "f"(v) : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(const uint64_t* local, uint32_t rank) {
    asm volatile("{\n\t.reg .b32 ra;\n\tmapa.shared::cluster.u32 ra, %0, %1;\n\t"
                 "mbarrier.arrive.release.cluster.shared::cluster.b64 _, [ra];\n\t}" ::"r"(smem_addr(local)), "r"(rank) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait_cluster(const uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}" : "=r"(ok) : "r"(smem_addr(bar)), "r"(parity) : "memory");
    return ok != 0;
}
constexpr int kHelperRows(int n_help) { return (4 * kHidden + n_help - 1) / n_help; }

// (value, index) as one 64-bit word whose unsigned order is the merge's order: a precedes b (larger value, then
// smaller index) exactly if key(a) > key(b).  -0 is folded into +0 first, as the comparison of values does.
__device__ __forceinline__ unsigned long long order_key(float v, int i) {
    uint32_t u = __float_as_uint(v + 0.f);
    u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
    return ((unsigned long long)u << 32) | (uint32_t)(0x7fffffff - i);
}
__device__ __forceinline__ float key_value(unsigned long long key) {
    const uint32_t u = (uint32_t)(key >> 32);
    return __uint_as_float((u & 0x80000000u) ? (u ^ 0x80000000u) : ~u);
}
__device__ __forceinline__ int key_index(unsigned long long key) { return 0x7fffffff - (int)(uint32_t)key; }

// smallest of the lanes' values (redux on a monotone unsigned image of the floats)
__device__ __forceinline__ float warp_min_value(float v) {
    uint32_t u = __float_as_uint(v + 0.f);
    u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
    u = __reduce_min_sync(kFull, u);
    return __uint_as_float((u & 0x80000000u) ? (u ^ 0x80000000u) : ~u);
}

// Log-sum-exp over a row's chunks in fp64, by one warp.
__device__ __forceinline__ double row_normaliser(const VocabPassParams& vp, size_t row) {
    const int lane = threadIdx.x & 31, n_chunks = vp.n_chunks;
    const float pm0 = lane < n_chunks ? vp.part_m[row * n_chunks + lane] : -CUDART_INF_F;
    const float ps0 = lane < n_chunks ? vp.part_s[row * n_chunks + lane] : 0.f;
    float mloc = pm0;
    for (int c = lane + 32; c < n_chunks; c += 32) mloc = fmaxf(mloc, vp.part_m[row * n_chunks + c]);
    const float M = warp_max(mloc);
    double sloc = pm0 > -CUDART_INF_F ? (double)ps0 * exp((double)pm0 - (double)M) : 0.0;
    for (int c = lane + 32; c < n_chunks; c += 32) {
        const float mc = vp.part_m[row * n_chunks + c];
        if (mc > -CUDART_INF_F) sloc += (double)vp.part_s[row * n_chunks + c] * exp((double)mc - (double)M);
    }
    const double S = warp_sum(sloc);
    return (double)M + log(S);
}

// One warp merges a row's chunk records into its top-k and hands candidate `rank` to put(rank, logit, token); meanwhile() runs
// while the records are on their way.  pv_s / pi_s: the warp's copy of the records (staged), lk: kSurvCap keys.
// A warp works on its row alone, and on its own its time is the number of instructions it
// issues one after the other plus what its shuffles wait for the ones of the other rows (an SM passes one
// warp's shuffle a clock).  So the chunk heads and the survivors are ranked from shared memory, four and two
// to a broadcast load, the records are filtered flat (a lane takes every 32nd entry, whatever its chunk), and
// the only shuffles left are those of the log-normaliser.
template <typename Meanwhile, typename Put>
__device__ __forceinline__ void merge_row(const VocabPassParams& vp, size_t row, bool staged, float* pv_s, int* pi_s, unsigned long long* lk, Meanwhile meanwhile, Put put) {
    const int lane = threadIdx.x & 31, k = vp.k, n_chunks = vp.n_chunks, per_row = n_chunks * k;
    const float* gv = vp.part_v + row * per_row;
    const int* gi = vp.part_i + row * per_row;
    float* s_heads = reinterpret_cast<float*>(lk);              // (done with before the first survivor is written)
    __syncwarp();                                            // the previous row's lists have been read
    if (staged) {
        if ((per_row & 3) == 0) {                            // rows of records are 16-byte aligned then
            for (int e = lane; e < per_row / 4; e += 32) { cp_async16(pv_s + 4 * e, gv + 4 * e); cp_async16(pi_s + 4 * e, gi + 4 * e); }
        } else {
            for (int e = lane; e < per_row; e += 32) { cp_async4(pv_s + e, gv + e); cp_async4(pi_s + e, gi + e); }
        }
    }
    const int lists = min(n_chunks, 32), depth = lane / lists, first = (lane - depth * lists) * k + depth;
    meanwhile();
    bool merged = false;
    if (staged) {
        cp_async_wait_all();
        __syncwarp();
        // The k-th best of 32 entries bounds the row's k-th best value from below: the first 32 / n_chunks entries of every list,
        // or the chunk heads (the best head of every 32nd chunk, if there are more than 32).  A bound from the lists'
        // j-th entries let twice as many through where there are fewer lists than k (41 rows of 70000 in 9 lists: 59.2 -> 55.5 us a step).
        float hv = depth < k ? pv_s[first] : -CUDART_INF_F;
        for (int c = lane + 32; c < n_chunks; c += 32) hv = fmaxf(hv, pv_s[c * k]);
        s_heads[lane] = hv;
        __syncwarp();
        int above = 0;
#pragma unroll
        for (int o = 0; o < 32; o += 4) {
            const float4 h4 = *reinterpret_cast<const float4*>(s_heads + o);
            above += (h4.x > hv ? 1 : 0) + (h4.y > hv ? 1 : 0) + (h4.z > hv ? 1 : 0) + (h4.w > hv ? 1 : 0);
        }
        const float tv = warp_min_value(depth < k && above < k ? hv : CUDART_INF_F);
        __syncwarp();
        int total = 0;
#pragma unroll 4
        for (int e0 = 0; e0 < per_row; e0 += 32) {
            const int e = e0 + lane;
            const float v = e < per_row ? pv_s[e] : 0.f;
            const bool keep = e < per_row && v >= tv;
            const unsigned m = __ballot_sync(kFull, keep);
            const int at = total + __popc(m & ((1u << lane) - 1u));
            if (keep && at < kSurvCap) lk[at] = order_key(v, pi_s[e]);
            total += __popc(m);
        }
        if (total <= kSurvCap) {
            if (lane == 0 && (total & 1)) lk[total] = 0ull;   // read in pairs: a key that precedes nothing
            __syncwarp();
            for (int e = lane; e < total; e += 32) {
                const unsigned long long ck = lk[e];
                int rank = 0;
#pragma unroll 4
                for (int j = 0; j < total; j += 2) {
                    const ulonglong2 kk = *reinterpret_cast<const ulonglong2*>(lk + j);
                    rank += (kk.x > ck ? 1 : 0) + (kk.y > ck ? 1 : 0);
                }
                if (rank < k) put(rank, key_value(ck), key_index(ck));
            }
            for (int e = total + lane; e < k; e += 32) put(e, -CUDART_INF_F, 0x7fffffff);   // (only with NaN logits)
            merged = true;
        }
        __syncwarp();
    }
    if (!merged) {
        // serial merge (records too large to stage, or a survivor list that overflowed)
        const float* pv = staged ? pv_s : gv;
        const int* pi = staged ? pi_s : gi;
        WarpTopList<float> top;
        top.reset();
        float thr = -CUDART_INF_F;
        int thr_i = 0x7fffffff;
        for (int c = 0; c < n_chunks; ++c) {
            for (int e = 0; e < k; ++e) {
                const float cv = pv[c * k + e];
                const int ci = pi[c * k + e];
                if (!precedes(cv, ci, thr, thr_i)) break;          // each chunk's list is sorted
                top.insert(cv, ci);
                thr = top.value_at(k - 1);
                thr_i = top.index_at(k - 1);
            }
        }
        if (lane < k) put(lane, top.v, top.i);
    }
}

}  // namespace
}  // namespace radar
