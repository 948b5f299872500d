// Top-k and log-normaliser of logits rows: every row is read once, by as many warps as it has spans, and merged by 288 threads.
//
// A warp takes a span of 256 vectors of 16 bytes (every n-th one of a row longer than 128 spans) and leaves 34 numbers: the
// largest logit of each of its 32 groups of 128 bytes, and the span's (max, sum exp).  In the merge the k-th largest of the
// groups' maxima bounds the row's k-th largest logit from below, so only the few groups whose maximum reaches it are read again;
// their values are ranked exactly by (logit desc, token asc), beside them one warp adds up the spans in fp64.
//
// The read is bound by HBM as long as nothing but loads and exponentials is in it: no selection, and no barrier behind the
// loads.  (With a selection of each chunk's k best in the pass, four block barriers and a ranking behind every 32 KB, its blocks
// spent as long on those as on their loads, whatever their number: the reads of 320 rows of 128256 took 39 us, now 25.)  The merge
// is a chain of dependent steps, which other rows hide.  Two forms:
//
//   row_topk_kernel     a row to a cluster, whose warps send what they leave into the first CTA's shared memory; that CTA merges.
//                       For launches of up to two CTAs per SM, so that all clusters are resident at once or nearly (a cluster
//                       needs its SMs in one GPC): no second kernel, which costs a call 1.6 us from one kernel's last store to
//                       the next one's first load, and the reads of what the pass has left.
//   row_pass_kernel,    all warps of all rows, then a block per row.  Once clusters queue for SMs, a merging CTA keeps the
//   row_merge_kernel    reads of the next ones waiting (both kernels 12.9 us for 80 rows of 128256, 31.8 for 320; clusters
//                       16.3 and 47.4).  The pass lets the merge start at its end: earlier, the waiting blocks gather on the
//                       SMs that are free first, four to one, and merge there one beside the other (71 rows: 34.9 -> 31.1 us).
#include <algorithm>
#include <cfloat>

#include "select.cuh"

namespace radar {
namespace {

constexpr int kWarps = 16, kThreads = kWarps * 32;   // of a cluster's CTA
constexpr int kMaxCluster = 8;
constexpr int kMaxSlots = kMaxCluster * kWarps;      // warps that share a row
constexpr int kPassWarps = 8;                        // of a block of the pass by itself
constexpr int kSpanVecs = 256;                       // vectors of a warp's span
constexpr int kLaneVecs = kSpanVecs / 32;            // ... of a lane
constexpr int kSelThreadsRow = 256;                  // of the merge's selection; one more warp forms the normaliser
constexpr int kSelWarpsRow = kSelThreadsRow / 32, kMergeThreads = kSelThreadsRow + 32;
constexpr int kHeld = kMaxSlots * 32 / kSelThreadsRow;       // maxima a thread of the merge holds
constexpr int kBoundSlots = 64;                      // maxima that the bound is chosen from
constexpr int kGroupCap = 512, kCandCap = 2048;      // groups and values that the merge lists; beyond, it scans the row
constexpr int kRankAll = 128;                        // values that it ranks as they are; more are thinned out first
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kNear = 128.f;                       // span maxima up to which the second product of 2^(x log2 e - max log2 e) is
                                                     // rounded by less than 8e-6

__device__ __forceinline__ float fast_exp2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// e^(x - top), mb = top * kLog2e
template <bool kFar>
__device__ __forceinline__ float power(float x, float top, float mb) {
    return fast_exp2(kFar ? (x - top) * kLog2e : fmaf(x, kLog2e, -mb));
}
// largest of the warp's values, in every lane (NaN loses)
__device__ __forceinline__ float warp_max_value(float v) {
    float y;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(y) : "f"(v));
    return y;
}

// A vector's values, from the 16 bytes that were loaded.
template <typename T> struct Unpack;
template <> struct Unpack<float> {
    static constexpr int N = 4;
    __device__ static __forceinline__ float at(const uint4& v, int e) {
        return __uint_as_float(e == 0 ? v.x : e == 1 ? v.y : e == 2 ? v.z : v.w);
    }
    // largest value of a vector (NaN loses; -inf if there is nothing else)
    __device__ static __forceinline__ float largest(const uint4& v) { return fmaxf(fmaxf(fmaxf(at(v, 0), at(v, 1)), fmaxf(at(v, 2), at(v, 3))), -CUDART_INF_F); }
};
template <> struct Unpack<__nv_bfloat16> {
    static constexpr int N = 8;
    __device__ static __forceinline__ float at(const uint4& v, int e) {
        const uint32_t w = e < 2 ? v.x : e < 4 ? v.y : e < 6 ? v.z : v.w;
        return __uint_as_float((e & 1) ? (w & 0xffff0000u) : (w << 16));
    }
    // (on pairs: unpacked, 64 values would have to be held for the exponentials, or unpacked twice)
    __device__ static __forceinline__ float largest(const uint4& v) {
        auto pair = [](uint32_t x) { return *reinterpret_cast<const __nv_bfloat162*>(&x); };
        const __nv_bfloat162 m = __hmax2(__hmax2(pair(v.x), pair(v.y)), __hmax2(pair(v.z), pair(v.w)));
        return fmaxf(fmaxf(__low2float(m), __high2float(m)), -CUDART_INF_F);
    }
};

// A row: up to N - 1 values in front of the first 16-byte boundary, whole vectors, up to N - 1 values behind them.
template <typename T>
struct Row {
    const T* x;
    int head, nvec, tail0, ntail;
    __device__ __forceinline__ Row(const RowTopkParams& p, int seq, int f) {
        constexpr int N = Unpack<T>::N;
        x = reinterpret_cast<const T*>(p.logits) + (int64_t)seq * p.seq_stride + (int64_t)f * p.row_stride;
        head = min((int)(((16 - (reinterpret_cast<uintptr_t>(x) & 15)) & 15) / sizeof(T)), p.V);
        nvec = (p.V - head) / N;
        tail0 = head + nvec * N;
        ntail = p.V - tail0;
    }
    // index of scalar value i (head first, then tail), i < head + ntail
    __device__ __forceinline__ int scalar(int i) const { return i < head ? i : tail0 + i - head; }
};

// A warp's vectors of one span.
template <typename T>
struct Span {
    using U = Unpack<T>;
    uint4 w[kLaneVecs];
    __device__ __forceinline__ void load(const Row<T>& r, int span) {
        constexpr uint32_t kMinusInf = sizeof(T) == 4 ? 0xff800000u : 0xff80ff80u;
        const int v0 = span * kSpanVecs + (threadIdx.x & 31);
        const uint4* vec = reinterpret_cast<const uint4*>(r.x + r.head) + v0;
        if ((span + 1) * kSpanVecs <= r.nvec) {
#pragma unroll
            for (int u = 0; u < kLaneVecs; ++u) w[u] = __ldcs(vec + 32 * u);
        } else {
#pragma unroll
            for (int u = 0; u < kLaneVecs; ++u) w[u] = v0 + 32 * u < r.nvec ? __ldcs(vec + 32 * u) : make_uint4(kMinusInf, kMinusInf, kMinusInf, kMinusInf);
        }
    }
    // The largest of every group of eight lanes' vectors (128 bytes in a row), one group to a lane: octet lane / 8, vector
    // lane % 8.  Each exchange halves the vectors a lane still has a maximum of.
    __device__ __forceinline__ float group_max() const {
        const int lane = threadIdx.x & 31;
        float g[kLaneVecs];
#pragma unroll
        for (int u = 0; u < kLaneVecs; ++u) g[u] = U::largest(w[u]);
#pragma unroll
        for (int o = kLaneVecs / 2; o > 0; o >>= 1) {
            const bool up = (lane & o) != 0;
#pragma unroll
            for (int i = 0; i < o; ++i) {
                const float give = up ? g[i] : g[i + o], keep = up ? g[i + o] : g[i];
                g[i] = fmaxf(keep, __shfl_xor_sync(kFull, give, o));
            }
        }
        return g[0];
    }
    // of this lane, relative to e^top.  kFar: for maxima so far from zero that the rounding of top log2 e counts (a span that is
    // masked as a whole; at -1e10 the rounding alone is up to 512, and such a span's infinite sum would make its row NaN).
    template <bool kFar>
    __device__ __forceinline__ float exp_sum(float top) const {
        float s[4] = {0.f, 0.f, 0.f, 0.f};
        const float mb = top * kLog2e;
#pragma unroll
        for (int u = 0; u < kLaneVecs; ++u)
#pragma unroll
            for (int e = 0; e < U::N; ++e) s[e & 3] += power<kFar>(U::at(w[u], e), top, mb);
        return (s[0] + s[1]) + (s[2] + s[3]);
    }
    __device__ __forceinline__ bool has_nan() const {
        bool nan = false;
#pragma unroll
        for (int u = 0; u < kLaneVecs; ++u)
#pragma unroll
            for (int e = 0; e < U::N; ++e) { const float x = U::at(w[u], e); nan |= x != x; }
        return nan;
    }
};

// barriers of the merge: its 256 selecting threads, and with the normaliser's warp
__device__ __forceinline__ void selection_barrier() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
__device__ __forceinline__ void merge_barrier() { asm volatile("bar.sync 2, 288;" ::: "memory"); }

struct __align__(16) MergeShared {
    unsigned long long key[kCandCap];
    unsigned long long best[kSelWarpsRow][32], best_slots[kBoundSlots], best_bound[2];       // (two: 16-byte boundaries)
    int group[kGroupCap];
    uint32_t lanes[kSelWarpsRow][32], slots[kBoundSlots];
    uint32_t bound;
    float kth[kSelWarpsRow];
    float best_v[kSelWarpsRow];
    int best_i[kSelWarpsRow];
    int n_groups, n_cand, n_kept;
    float v[RADAR_MAX_K];
    int t[RADAR_MAX_K];
    double lse;
    int mark;
};

// Log-sum-exp over the n warps of a row in fp64, by one warp; whether one of them has seen a NaN.
__device__ __forceinline__ double row_normaliser(const float2* part, int n, bool& nan) {
    const int lane = threadIdx.x & 31;
    constexpr int kHold = kMaxSlots / 32;
    float2 p[kHold];
    float top = -CUDART_INF_F;
    nan = false;
#pragma unroll
    for (int i = 0; i < kHold; ++i) {
        p[i] = lane + 32 * i < n ? part[lane + 32 * i] : make_float2(-CUDART_INF_F, 0.f);
        top = fmaxf(top, p[i].x);
        nan |= p[i].x != p[i].x;
    }
    nan = __any_sync(kFull, nan);
    top = warp_max_value(top);
    double sum = 0.0;
#pragma unroll
    for (int i = 0; i < kHold; ++i)
        if (p[i].x > -CUDART_INF_F) sum += (double)p[i].y * exp((double)p[i].x - (double)top);
    return (double)top + log(warp_sum(sum));
}

// Ties beyond the lists' room: a tournament over the row.  A thread holds the best of every 256th value; the owner of a
// winner gets its next one from its warp.
template <typename T>
__device__ __noinline__ void select_by_scan(const T* x, int V, int k, MergeShared& S) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float bv = -CUDART_INF_F;
    int bi = 0x7fffffff;
#pragma unroll 8
    for (int i = tid; i < V; i += kSelThreadsRow) {
        const float v = to_float(x[i]);
        if (precedes(v, i, bv, bi)) { bv = v; bi = i; }
    }
    for (int r = 0; r < k; ++r) {
        float v = bv;
        int i = bi;
        warp_best(v, i);
        selection_barrier();                          // the previous round's readers are done
        if (lane == 0) { S.best_v[warp] = v; S.best_i[warp] = i; }
        selection_barrier();
        v = S.best_v[0];
        i = S.best_i[0];
#pragma unroll
        for (int w = 1; w < kSelWarpsRow; ++w)
            if (precedes(S.best_v[w], S.best_i[w], v, i)) { v = S.best_v[w]; i = S.best_i[w]; }
        if (tid == 0) { S.v[r] = v; S.t[r] = i; }
        const int owner = i & (kSelThreadsRow - 1);
        if (i != 0x7fffffff && owner >> 5 == warp) {
            float nv = -CUDART_INF_F;
            int ni = 0x7fffffff;
#pragma unroll 4
            for (int c = owner + kSelThreadsRow * lane; c < V; c += kSelThreadsRow * 32) {
                const float y = to_float(x[c]);
                if (precedes(v, i, y, c) && precedes(y, c, nv, ni)) { nv = y; ni = c; }
            }
            warp_best(nv, ni);
            if (tid == owner) { bv = nv; bi = ni; }
        }
    }
}

// Many values are listed where fewer than about 2 k groups have any (short rows with a large k, masked rows).  A better bound, the
// k-th largest of 64 of them, the eight best of every warp's, thins out more than kRankAll: ranks take n^2 comparisons.  Us for the
// calls of a step without this / with it, bf16: t_max = 5, V = 1000, k = 32, one sequence that makes the first call 153 / 35, eight
// that make all 550 / 84; V = 600, k = 16 135 / 33.  Returns how many are left.
__device__ __noinline__ int thin_out(MergeShared& S, int n, int k) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int kEach = kCandCap / kSelThreadsRow, kPer = kBoundSlots / kSelWarpsRow;
    unsigned long long key[kEach], best = 31 - lane;   // (of none: distinct, and less than any listed value's)
#pragma unroll
    for (int i = 0; i < kEach; ++i) {
        const int at = tid + kSelThreadsRow * i;
        key[i] = at < n ? S.key[at] : 0ull;
        best = max(best, key[i]);
    }
    S.best[warp][lane] = best;
    __syncwarp();
    int rank = 0;
#pragma unroll 4
    for (int o = 0; o < 32; o += 2) {
        const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(&S.best[warp][o]);
        rank += (q.x > best ? 1 : 0) + (q.y > best ? 1 : 0);
    }
    if (rank < kPer) S.best_slots[warp * kPer + rank] = best;
    selection_barrier();
    const unsigned long long mine = S.best_slots[tid >> 2];
    rank = 0;
#pragma unroll 4
    for (int o = 0; o < kBoundSlots / 4; o += 2) {
        const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(&S.best_slots[(tid & 3) * (kBoundSlots / 4) + o]);
        rank += (q.x > mine ? 1 : 0) + (q.y > mine ? 1 : 0);
    }
    rank += __shfl_xor_sync(kFull, rank, 1);
    rank += __shfl_xor_sync(kFull, rank, 2);
    if (rank == k - 1) S.best_bound[0] = mine;
    selection_barrier();
    const unsigned long long bound = S.best_bound[0];
#pragma unroll
    for (int i = 0; i < kEach; ++i)
        if (key[i] >= bound) S.key[atomicAdd(&S.n_kept, 1)] = key[i];
    selection_barrier();
    return S.n_kept;
}

// What the warps of a row have left, where it is.
struct InShared {
    const float* gmax;                                // [n_slots][32]
    const float2* part;                               // [n_slots]
    __device__ __forceinline__ float one(int i) const { return gmax[i]; }
    __device__ __forceinline__ float4 four(int i) const { return *reinterpret_cast<const float4*>(gmax + i); }
};
struct InGlobal {                                     // (read once: the compiler would rather read again than hold it)
    const float* gmax;
    const float2* part;
    __device__ __forceinline__ float one(int i) const {
        float v;
        asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(gmax + i));
        return v;
    }
    __device__ __forceinline__ float4 four(int i) const {
        float4 v;
        asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(gmax + i));
        return v;
    }
};

// One row's k best into S, by threads 0 .. 255.
template <typename T, typename Left>
__device__ __forceinline__ void select_row(const RowTopkParams& p, const Row<T>& r, const Left& left, MergeShared& S) {
    constexpr int N = Unpack<T>::N;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, k = p.k, n_slots = p.n_slots;
    if (tid == 0) { S.n_groups = 0; S.n_cand = 0; S.n_kept = 0; }
    // Thread tid holds 16 groups: four in a row of every 1024 (a request for 512 bytes takes the SM hardly longer than one for
    // 128: 16 KB in fours 0.6 us, one by one 1.3), or, where there are at most 1024, every 256th, so that every
    // warp has some.
    const bool fours = n_slots >= 32;
    auto group_id = [&](int i) { return fours ? 4 * tid + (i & 3) + 4 * kSelThreadsRow * (i >> 2) : tid + kSelThreadsRow * i; };
    float g[kHeld], mine = -CUDART_INF_F;
    if (fours) {
#pragma unroll
        for (int i = 0; i < kHeld / 4; ++i) {
            float4 q = make_float4(-CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F);
            if (group_id(4 * i) < n_slots * 32) q = left.four(group_id(4 * i));
            g[4 * i] = q.x; g[4 * i + 1] = q.y; g[4 * i + 2] = q.z; g[4 * i + 3] = q.w;
        }
    } else {
#pragma unroll
        for (int i = 0; i < kHeld; ++i) g[i] = i < 4 && group_id(i) < n_slots * 32 ? left.one(group_id(i)) : -CUDART_INF_F;
    }
#pragma unroll
    for (int i = 0; i < kHeld; ++i) mine = fmaxf(mine, g[i]);

    // The bound: the k-th largest of 64 maxima, the best ones of every warp that has groups.  Where that is -inf (the finite
    // values sit in few spans), the best of the warps' k-th largest.  Maxima are ranked as integers, made distinct by
    // their lowest bits; either bound is the integer it was ranked by without those bits (not the maximum itself, which
    // may lie above some that were ranked ahead of it), so that the k ranked first are all at or above it.
    const int live = p.live, per = p.per;
    {
        const uint32_t key = (order_bits(mine) & ~31u) | (31u - lane);
        S.lanes[warp][lane] = key;
        __syncwarp();
        int rank = 0;
#pragma unroll 2
        for (int o = 0; o < 32; o += 4) {
            const uint4 q = *reinterpret_cast<const uint4*>(&S.lanes[warp][o]);
            rank += (q.x > key ? 1 : 0) + (q.y > key ? 1 : 0) + (q.z > key ? 1 : 0) + (q.w > key ? 1 : 0);
        }
        const int slot = warp * per + rank;
        if (warp < live && rank < per) S.slots[slot] = (order_bits(mine) & ~63u) | (63u - slot);
        if (rank == k - 1) S.kth[warp] = fmaxf(bits_value(key & ~31u), -FLT_MAX);      // (of -inf: NaN, which loses)
        if (tid >= live * per && tid < kBoundSlots) S.slots[tid] = 63u - tid;
    }
    selection_barrier();
    {   // four lanes to a slot
        const uint32_t key = S.slots[tid >> 2];
        int rank = 0;
#pragma unroll 2
        for (int o = 0; o < kBoundSlots / 4; o += 4) {
            const uint4 q = *reinterpret_cast<const uint4*>(&S.slots[(tid & 3) * (kBoundSlots / 4) + o]);
            rank += (q.x > key ? 1 : 0) + (q.y > key ? 1 : 0) + (q.z > key ? 1 : 0) + (q.w > key ? 1 : 0);
        }
        rank += __shfl_xor_sync(kFull, rank, 1);
        rank += __shfl_xor_sync(kFull, rank, 2);
        if (rank == k - 1) S.bound = key & ~63u;
    }
    selection_barrier();
    float tv = -FLT_MAX;                              // (values at -inf are never listed)
    if (S.bound > order_bits(-CUDART_INF_F)) tv = bits_value(S.bound);
    else
        for (int w = 0; w < live; ++w) tv = fmaxf(tv, S.kth[w]);
    if (mine >= tv) {
        unsigned reach = 0;                           // which of the held groups reach the bound
#pragma unroll
        for (int i = 0; i < kHeld; ++i) reach |= (g[i] >= tv ? 1u : 0u) << i;
        int at = atomicAdd(&S.n_groups, __popc(reach));
        for (; reach != 0 && at < kGroupCap; reach &= reach - 1) S.group[at++] = group_id(__ffs(reach) - 1);
    }
    selection_barrier();

    // ---- the listed groups' values, and the row's scalar ones: what reaches the bound is listed ----
    const int lines = p.lines, ng = min(S.n_groups, kGroupCap) * lines;
    constexpr int kBatch = 2, kEach = N / 4;          // lines at a time; values of a line per lane
    for (int q0 = warp; q0 < ng; q0 += kBatch * kSelWarpsRow) {
        float v[kBatch * kEach];
        int at[kBatch];
#pragma unroll
        for (int q = 0; q < kBatch; ++q) {
            const int gi = q0 + q * kSelWarpsRow, which = lines == 1 ? gi : gi / lines;
            const int id = gi < ng ? S.group[which] : 0, span = (id >> 5) + (gi - which * lines) * n_slots;
            const int vec = span * kSpanVecs + (id & 7) * 32 + ((id >> 3) & 3) * 8 + (lane >> 2);
            at[q] = gi < ng && vec < r.nvec ? r.head + vec * N + (lane & 3) * kEach : -1;
#pragma unroll
            for (int e = 0; e < kEach; ++e) v[q * kEach + e] = at[q] >= 0 ? to_float(r.x[at[q] + e]) : -CUDART_INF_F;
        }
#pragma unroll
        for (int x = 0; x < kBatch * kEach; ++x)
            if (v[x] >= tv) {
                const int to = atomicAdd(&S.n_cand, 1);
                if (to < kCandCap) S.key[to] = order_key(v[x], at[x / kEach] + x % kEach);
            }
    }
    if (warp == kSelWarpsRow - 1 && lane < r.head + r.ntail) {
        const int i = r.scalar(lane);
        const float v = to_float(r.x[i]);
        if (v >= tv) {
            const int to = atomicAdd(&S.n_cand, 1);
            if (to < kCandCap) S.key[to] = order_key(v, i);
        }
    }
    selection_barrier();

    // ---- ranks: a warp to a value ----
    int nc = S.n_cand;
    if (S.n_groups <= kGroupCap && nc <= kCandCap) {
        if (nc > kRankAll) nc = thin_out(S, nc, k);
        const unsigned long long k0 = lane < nc ? S.key[lane] : 0ull;
        for (int c = warp; c < nc; c += kSelWarpsRow) {
            const unsigned long long key = S.key[c];
            int rank = __popc(__ballot_sync(kFull, k0 > key));
            for (int j = 32; j < nc; j += 32) rank += __popc(__ballot_sync(kFull, j + lane < nc && S.key[j + lane] > key));
            if (lane == 0 && rank < k) { S.v[rank] = key_value(key); S.t[rank] = key_index(key); }
        }
        if (nc < k && warp == 0) {                    // fewer finite values than k: the first tokens at -inf
            int have = nc;
#pragma unroll 8
            for (int i0 = 0; i0 < p.V; i0 += 32) {
                const bool is = i0 + lane < p.V && to_float(r.x[i0 + lane]) == -CUDART_INF_F;
                const unsigned who = __ballot_sync(kFull, is);
                const int rank = have + __popc(who & ((1u << lane) - 1u));
                if (is && rank < k) { S.v[rank] = -CUDART_INF_F; S.t[rank] = i0 + lane; }
                have += __popc(who);
                if (have >= k) break;
            }
            for (int i = have + lane; i < k; i += 32) { S.v[i] = -CUDART_INF_F; S.t[i] = 0x7fffffff; }    // (only with NaN logits)
        }
    } else {
        select_by_scan(r.x, p.V, k, S);
    }
}

// A warp's share of a row, spans slot, slot + n_slots, ...: this lane's group maximum and the warp's (max, sum exp), max NaN if it
// has seen one.  x holds the first span.
template <typename T>
__device__ __forceinline__ void pass_row(const RowTopkParams& p, const Row<T>& r, int slot, Span<T>& x, float& gmax, float& m, float& s) {
    const int lane = threadIdx.x & 31;
    gmax = m = -CUDART_INF_F;
    s = 0.f;
    for (int span = slot; span < p.spans; span += p.n_slots) {
        if (span != slot) x.load(r, span);
        float xs = -CUDART_INF_F;                     // the row's scalar values go with its last span
        if (span == p.spans - 1 && lane < r.head + r.ntail) xs = to_float(r.x[r.scalar(lane)]);
        const float g = x.group_max(), top = warp_max_value(fmaxf(g, xs));
        float sum = 0.f;
        if (fabsf(top) <= kNear) sum = warp_sum(x.template exp_sum<false>(top) + power<false>(xs, top, top * kLog2e));
        else if (top > -CUDART_INF_F) sum = warp_sum(x.template exp_sum<true>(top) + power<true>(xs, top, 0.f));
        float seen = top;
        if (sum != sum || top == -CUDART_INF_F) {     // +inf, or a NaN (the maxima pass it by): the merge reports it
            if (__any_sync(kFull, xs != xs || x.has_nan())) seen = CUDART_NAN_F;
        }
        gmax = fmaxf(gmax, g);
        if (span == slot) {
            m = seen;
            s = sum;
        } else if (m == m) {                          // (a NaN stays)
            const float both = fmaxf(m, top);
            if (both > -CUDART_INF_F) s = s * fast_exp2((m - both) * kLog2e) + sum * fast_exp2((top - both) * kLog2e);
            m = seen == seen ? both : seen;
        }
    }
}

// By threads 0 .. 287.
template <typename T, typename Left>
__device__ __forceinline__ void merge_row(const RowTopkParams& p, const Row<T>& r, size_t row, const Left& left, MergeShared& S) {
    const int tid = threadIdx.x;
    if (tid >= kSelThreadsRow) {
        bool nan;
        const double lse = row_normaliser(left.part, p.n_slots, nan);
        if (tid == kSelThreadsRow) { S.lse = lse; S.mark = nan ? kNanRow : 0; }
    } else {
        select_row<T>(p, r, left, S);
    }
    merge_barrier();
    if (tid < p.k) {
        p.tok[row * p.k + tid] = S.t[tid] | S.mark;
        p.logp[row * p.k + tid] = (double)S.v[tid] - S.lse;
    }
}

// The mask may be written while this runs (a sequence that stops meanwhile is read in vain): the first CTA's look at it decides
// for the cluster, whose blocks would else wait for messages of blocks that have left, or send to one.  It sends the others
// what it saw; a thread's own look only decides whether its span is asked for ahead of that.
template <typename T>
__global__ void __launch_bounds__(kThreads, 2) row_topk_kernel(const RowTopkParams p) {
    __shared__ MergeShared S;
    __shared__ __align__(16) float s_gmax[kMaxSlots * 32];           // the first CTA's: what all warps of the cluster leave
    __shared__ __align__(16) float2 s_part[kMaxSlots];
    __shared__ __align__(8) uint64_t s_bar;                          // the first CTA's completes when they have sent it,
    __shared__ uint32_t s_live;                                      // the others' with what the first CTA saw in the mask
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n = gridDim.x, rank = blockIdx.x, f = blockIdx.y, seq = blockIdx.z;
    if (threadIdx.x == 0) init_message_barrier(&s_bar, rank == 0 ? (uint32_t)(n * kWarps * (32 * sizeof(float) + sizeof(float2))) : (uint32_t)sizeof(s_live));
    if (n > 1) cluster_barrier();                     // every CTA has started and its barrier word is initialised
    else __syncthreads();
    chain_wait();
    const bool ahead = p.seq_active == nullptr || p.seq_active[seq] != 0;
    const Row<T> r(p, seq, f);
    const int slot = rank * kWarps + warp;
    Span<T> x;
    if (ahead) x.load(r, slot);                       // (past the row's end: -inf, nothing is read)
    if (p.seq_active != nullptr) {
        if (rank == 0) {
            if (warp == 0) {
                const uint32_t look = __shfl_sync(kFull, ahead ? 1u : 0u, 0);
                if (lane == 0) s_live = look;
                else if (lane < n) send_f32(cluster_addr(&s_live, lane), cluster_addr(&s_bar, lane), __uint_as_float(look));
            }
            __syncthreads();
        } else if (!cluster_wait(&s_bar, 0)) {
            set_status(p.status, RADAR_ERR_TIMEOUT);
            return;
        }
        if (s_live == 0) return;
        if (!ahead) x.load(r, slot);
    }
    float gmax, m, s;
    pass_row<T>(p, r, slot, x, gmax, m, s);
    const uint32_t bar = cluster_addr(&s_bar, 0);
    send_f32(cluster_addr(&s_gmax[slot * 32 + lane], 0), bar, gmax);
    if (lane == 0) send_f32x2(cluster_addr(&s_part[slot], 0), bar, m, s);
    if (rank != 0 || threadIdx.x >= kMergeThreads) return;
    if (!cluster_wait(&s_bar, 0)) set_status(p.status, RADAR_ERR_TIMEOUT);
    merge_row<T>(p, r, (size_t)seq * p.F + f, InShared{s_gmax, s_part}, S);
}

template <typename T>
__global__ void __launch_bounds__(kPassWarps * 32, 4) row_pass_kernel(const RowTopkParams p) {
    chain_sync();
    const int lane = threadIdx.x & 31, slot = blockIdx.x * kPassWarps + (threadIdx.x >> 5), f = blockIdx.y, seq = blockIdx.z;
    if (slot >= p.n_slots || (p.seq_active != nullptr && p.seq_active[seq] == 0)) return;
    const Row<T> r(p, seq, f);
    Span<T> x;
    x.load(r, slot);
    float gmax, m, s;
    pass_row<T>(p, r, slot, x, gmax, m, s);
    const size_t at = ((size_t)seq * p.F + f) * p.n_slots + slot;
    p.gmax[at * 32 + lane] = gmax;
    if (lane == 0) p.part[at] = make_float2(m, s);
    chain_trigger();
}

// Lets its successor start before it waits itself: the pass's blocks start it behind their own wait, so all that came before
// the pass is complete then.
template <typename T>
__global__ void __launch_bounds__(kMergeThreads) row_merge_kernel(const RowTopkParams p) {
    chain_trigger();
    __shared__ MergeShared S;
    const int row = blockIdx.x, seq = row / p.F, f = row - seq * p.F;
    const float* gmax = p.gmax + (size_t)row * p.n_slots * 32;
    const Row<T> r(p, seq, f);
    if (threadIdx.x < 32) {
        // the row and what the pass leaves were last touched from other SMs: asking for a line of each (L2 only, nothing is
        // read) brings the address translations in
        asm volatile("prefetch.global.L2 [%0];" ::"l"(r.x + (size_t)p.V * threadIdx.x / 32));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(gmax));
    }
    chain_sync();
    if (p.seq_active != nullptr && p.seq_active[seq] == 0) return;
    merge_row<T>(p, r, row, InGlobal{gmax, p.part + (size_t)row * p.n_slots}, S);
}

}  // namespace

static int spans_of(int V, int dtype) {
    const int per = kSpanVecs * (dtype == RADAR_F32 ? Unpack<float>::N : Unpack<__nv_bfloat16>::N);
    return (V + per - 1) / per;
}

size_t row_topk_workspace_bytes(int rows, int V, int k) {
    const size_t slots = (size_t)rows * std::min(spans_of(V, RADAR_F32), kMaxSlots);
    return align_up((size_t)rows * k * sizeof(double), 256) + align_up((size_t)rows * k * sizeof(int32_t), 256) +
           align_up(slots * sizeof(float2), 256) + align_up(slots * 32 * sizeof(float), 256);
}

void row_topk_carve(RowTopkParams& p, void* ws) {
    p.spans = spans_of(p.V, p.dtype);
    p.n_slots = std::min(p.spans, kMaxSlots);
    const size_t rows = (size_t)p.n_seq * p.F;
    char* c = static_cast<char*>(ws);
    p.logp = reinterpret_cast<double*>(c); c += align_up(rows * p.k * sizeof(double), 256);
    p.tok = reinterpret_cast<int32_t*>(c); c += align_up(rows * p.k * sizeof(int32_t), 256);
    p.part = reinterpret_cast<float2*>(c); c += align_up(rows * p.n_slots * sizeof(float2), 256);
    p.gmax = reinterpret_cast<float*>(c);
}

cudaError_t row_topk_launch(radar_ctx* ctx, RowTopkParams p, cudaStream_t stream) {
    if (p.n_seq > 65535 || p.F > 65535) return cudaErrorInvalidValue;
    p.status = ctx->d_status;
    p.live = std::min(kSelWarpsRow, p.spans);
    p.per = std::min(32, kBoundSlots / p.live);
    const bool f32 = p.dtype == RADAR_F32;
    int cluster = 1;                                  // a span to a warp, up to the cluster sizes that every device has
    while (cluster < kMaxCluster && cluster * kWarps < p.spans) cluster *= 2;
    if ((long long)p.n_seq * p.F * cluster <= 2 * ctx->sm_count) {
        p.n_slots = cluster * kWarps;
        p.lines = (p.spans + p.n_slots - 1) / p.n_slots;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)cluster, (unsigned)p.F, (unsigned)p.n_seq);
        cfg.blockDim = dim3(kThreads);
        cfg.stream = stream;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = (unsigned)cluster;
        attr[1].val.clusterDim.y = 1;
        attr[1].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 2;
        radar_launch_scope scope(ctx, RADAR_K_VOCAB_EXPAND, stream);
        return f32 ? cudaLaunchKernelEx(&cfg, row_topk_kernel<float>, p) : cudaLaunchKernelEx(&cfg, row_topk_kernel<__nv_bfloat16>, p);
    }
    p.lines = (p.spans + p.n_slots - 1) / p.n_slots;
    {
        const dim3 grid((unsigned)((p.n_slots + kPassWarps - 1) / kPassWarps), (unsigned)p.F, (unsigned)p.n_seq), block(kPassWarps * 32);
        radar_launch_scope scope(ctx, RADAR_K_VOCAB_EXPAND, stream);
        const cudaError_t e = f32 ? launch_chained(row_pass_kernel<float>, grid, block, 0, stream, p)
                                  : launch_chained(row_pass_kernel<__nv_bfloat16>, grid, block, 0, stream, p);
        if (e != cudaSuccess) return e;
    }
    const dim3 grid((unsigned)(p.n_seq * p.F)), block(kMergeThreads);
    radar_launch_scope scope(ctx, RADAR_K_ROW_MERGE, stream);
    return f32 ? launch_chained(row_merge_kernel<float>, grid, block, 0, stream, p) : launch_chained(row_merge_kernel<__nv_bfloat16>, grid, block, 0, stream, p);
}

}  // namespace radar
