// Pieces shared by the kernels of the expansion (row_topk.cu, expand.cu, expand_calls.cu): order keys, and the blocks of a
// cluster that share out the recurrent product.
#pragma once
#include "common.cuh"

namespace radar {
namespace {

constexpr int kSelThreads = 1024;
constexpr int kSelWarps = kSelThreads / 32;
constexpr int kMaxF = 32;
constexpr int kSelCluster = 4;                       // blocks per sequence when the recurrent product is shared out,
constexpr long long kShortPassLogits = 4 << 20;      // ... which is done while a call's vocabulary pass reads at most this many logits

__device__ __forceinline__ float sigmoidf_(float x) { return 1.f / (1.f + expf(-x)); }

__device__ __forceinline__ void cp_async4(void* smem, const void* gmem) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(smem)), "l"(gmem) : "memory");
}
// [rows][k] into shared memory at the odd stride k | 1, by the block; kSelThreads a multiple of rows.  Several threads to a row: an
// index over all elements would be divided by k for each, 2400 cycles of a block's instructions in front of every call.
__device__ __forceinline__ void copy_rows(float* smem, const float* gmem, int rows, int k) {
    const int per = kSelThreads / rows, r = (int)threadIdx.x / per;
    for (int j = (int)threadIdx.x % per; j < k; j += per) cp_async4(smem + r * (k | 1) + j, gmem + r * k + j);
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ bool mbar_try_wait_cluster(const uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}" : "=r"(ok) : "r"(smem_addr(bar)), "r"(parity) : "memory");
    return ok != 0;
}

// Monotone image of a float in the unsigned numbers, and back.  -0 is folded into +0 first, as the comparison of values does.
__device__ __forceinline__ uint32_t order_bits(float v) {
    const uint32_t u = __float_as_uint(v + 0.f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float bits_value(uint32_t u) { return __uint_as_float((u & 0x80000000u) ? (u ^ 0x80000000u) : ~u); }
// (value, index) as one 64-bit word whose unsigned order is the rows': a precedes b (larger value, then smaller index) exactly
// if key(a) > key(b).
__device__ __forceinline__ unsigned long long order_key(float v, int i) { return ((unsigned long long)order_bits(v) << 32) | (uint32_t)(0x7fffffff - i); }
__device__ __forceinline__ float key_value(unsigned long long key) { return bits_value((uint32_t)(key >> 32)); }
__device__ __forceinline__ int key_index(unsigned long long key) { return 0x7fffffff - (int)(uint32_t)key; }

// smallest of the lanes' values
__device__ __forceinline__ float warp_min_value(float v) { return bits_value(__reduce_min_sync(kFull, order_bits(v))); }

// bounded wait for a phase of a barrier that other blocks of the cluster complete
__device__ __forceinline__ bool cluster_wait(const uint64_t* bar, uint32_t parity) {
    bool ok = false;
    for (uint32_t it = 0; it < (1u << 22) && !(ok = mbar_try_wait_cluster(bar, parity)); ++it) {}
    return ok;
}
// a word into another block's shared memory, counted by a barrier there: the message needs no release of what came before it
__device__ __forceinline__ void send_f32(uint32_t addr, uint32_t bar, float v) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(addr), "r"(__float_as_uint(v)), "r"(bar) : "memory");
}
__device__ __forceinline__ void send_f32x2(uint32_t addr, uint32_t bar, float x, float y) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];"
                 ::"r"(addr), "r"(__float_as_uint(x)), "r"(__float_as_uint(y)), "r"(bar) : "memory");
}
__device__ __forceinline__ void expect_bytes(const uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void init_message_barrier(const uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    expect_bytes(bar, bytes);
}
// monotone image of a double (-0 folded into +0 first, as the comparison of values does)
__device__ __forceinline__ unsigned long long order_key64(double v) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(v + 0.0);
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}

// Ranks of two candidates (key, index) among n of them (key desc, index asc), by one warp.
__device__ __forceinline__ int2 ranks_of(const unsigned long long* keys, const short* index, int n, unsigned long long key0, int idx0, unsigned long long key1, int idx1) {
    int2 rank = make_int2(0, 0);
#pragma unroll 1
    for (int j0 = 0; j0 < n; j0 += 32) {
        const int j = j0 + (threadIdx.x & 31), jj = min(j, n - 1);
        const unsigned long long kj = keys[jj];
        const int ij = index[jj];
        rank.x += __popc(__ballot_sync(kFull, j < n && (kj > key0 || (kj == key0 && ij < idx0))));
        rank.y += __popc(__ballot_sync(kFull, j < n && (kj > key1 || (kj == key1 && ij < idx1))));
    }
    return rank;
}

// A helper block's share of the recurrent product: rows [r0, r1) of W_hh, six rows to a warp, four weights of each to a lane, in
// registers.  W_hh is 256 KB: one block would stream it through its SM for every call (2 us at 64 bytes a clock).
struct HelperRows {
    static constexpr int kRows = (4 * kHidden + kSelCluster - 2) / (kSelCluster - 1);
    static constexpr int kPer = (kRows + kSelWarps - 1) / kSelWarps;
    static_assert(kPer <= 8 && kRows >= kSelWarps, "every warp has rows, at most eight");
    float4 w[kPer];
    float bi, bh;
    int row;                                           // the row whose sum ends up in this lane
    bool sender;
    // bytes of W_hh h + biases from all helpers
    static constexpr uint32_t kProductBytes = 4 * kHidden * 4;

    __device__ __forceinline__ HelperRows(const radar_expand_args& a, int rank) {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        const int r0 = (rank - 1) * kRows, r1 = min(4 * kHidden, r0 + kRows);
#pragma unroll
        for (int i = 0; i < kPer; ++i) w[i] = *reinterpret_cast<const float4*>(a.w_hh + (size_t)min(r0 + warp + i * kSelWarps, r1 - 1) * kHidden + 4 * lane);
        row = r0 + warp + (lane >> 2) * kSelWarps;
        sender = (lane & 3) == 0 && (lane >> 2) < kPer && row < r1;
        bi = sender ? a.b_ih[row] : 0.f;
        bh = sender ? a.b_hh[row] : 0.f;
    }
    // h4: h[4 * lane ..]; the sum is valid in senders
    __device__ __forceinline__ float product(float4 h4) const {
        float acc[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            acc[i] = 0.f;
            if (i < kPer) {
                acc[i] = w[i].x * h4.x;
                acc[i] = fmaf(w[i].y, h4.y, acc[i]);
                acc[i] = fmaf(w[i].z, h4.z, acc[i]);
                acc[i] = fmaf(w[i].w, h4.w, acc[i]);
            }
        }
        return transposed_sum<8>(acc) + bi + bh;
    }
};

}  // namespace
}  // namespace radar
