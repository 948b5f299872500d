// radar_verify_accept: acceptance of the verified tree.
//   greedy     - vocabulary pass with k = 1 (row argmax, no exponentials) over the target logits of
//                the live tree rows, then one warp per sequence walks the tree with ballots.
//   stochastic - one thread-block cluster per sequence walks the tree lazily: only rows on the accepted
//                path are read, and each CTA of the cluster owns a slice of the vocabulary in every pass.
//                Probabilities are fp64.  exp((z - reference) / T) of the current node's target and draft rows
//                is cached on chip and, what has no room there, in the workspace (p, q = cached value / row sum); after j rejections the residual pair is, for every token v that has
//                not been proposed yet,  p_j(v) = max(0, p(v) - a_j q(v)) / W_j,  q_j(v) = c_j q(v),
//                and for the token proposed at trial i <= j,  p_j(x_i) = max(0, p(x_i) - a_i q(x_i)) / W_j,
//                q_j(x_i) = 0, with a_{j+1} = a_j + c_j W_j,  c_{j+1} = c_j / (1 - q_j(x_{j+1})) and
//                W_{j+1} = sum_v max(0, p(v) - a(v) q(v)).  This is the rectify / remove / renormalise
//                recursion of Eq. 2 unrolled, so each rejection costs one read-only pass.
#include <algorithm>
#include <cfloat>
#include <cmath>

#include "common.cuh"

namespace radar {
namespace {

// ------------------------------------------------------------------------------------------
// greedy walk
// ------------------------------------------------------------------------------------------
struct GreedyParams {
    radar_accept_args a;
    VocabPassParams vp;
};

// Latency is all there is to it: eight threads share a row's chunk records, and what the end needs (leaf count, retrieve
// rows) is asked for at the start.
constexpr int kGreedyThreads = 8 * kMaxNodes;
__global__ void __launch_bounds__(kGreedyThreads) greedy_walk_kernel(const GreedyParams P) {
    chain_wait();
    const radar_accept_args& a = P.a;
    const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
    __shared__ int s_arg[kMaxNodes], s_tok[kMaxNodes], s_par[kMaxNodes];
    const int M = min(max(a.n_nodes[b], 1), kMaxNodes);
    const int nl = a.n_leaves[b];
    const int nc = P.vp.n_chunks;
    const int retr = a.N * (a.t_max + 1);
    if (tid * 32 < retr) asm volatile("prefetch.global.L1 [%0];" ::"l"(a.retrieve + (size_t)b * retr + tid * 32));
    {   // argmax of row tid / 8: best chunk record by (value desc, token asc)
        const int r = tid >> 3;
        int best_i = 0x7fffffff;
        float best_v = -CUDART_INF_F;
        if (r < M) {
            const size_t rec0 = ((size_t)b * kMaxNodes + r) * nc;
#pragma unroll 4
            for (int c = tid & 7; c < nc; c += 8) {
                const float v = P.vp.part_v[rec0 + c];
                const int i = P.vp.part_i[rec0 + c];
                if (precedes(v, i, best_v, best_i)) { best_v = v; best_i = i; }
            }
        }
        if (tid < kMaxNodes) {
            const size_t o = (size_t)b * kMaxNodes + tid;
            const int tok = a.tree_tok[o], par = a.tree_parent[o];
            s_tok[tid] = tid < M ? tok : -1;
            s_par[tid] = tid < M ? par : -2;
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            const float ov = __shfl_xor_sync(kFull, best_v, o);
            const int oi = __shfl_xor_sync(kFull, best_i, o);
            if (precedes(ov, oi, best_v, best_i)) { best_v = ov; best_i = oi; }
        }
        if ((tid & 7) == 0) s_arg[r] = best_i;
    }
    __syncthreads();
    if (tid >= 32) return;
    const int W = a.t_max + 1;
    int32_t* pn = a.path_nodes + (size_t)b * W;
    int32_t* pt = a.path_tokens + (size_t)b * W;
    int cur = 0, len = 0;
    if (lane == 0) { pn[0] = 0; pt[0] = s_tok[0]; }
    while (len < a.t_max) {
        const int want = s_arg[cur];
        const unsigned lo = __ballot_sync(kFull, s_par[lane] == cur && s_tok[lane] == want && lane > 0);
        const unsigned hi = __ballot_sync(kFull, s_par[lane + 32] == cur && s_tok[lane + 32] == want);
        const int nxt = lo ? __ffs(lo) - 1 : (hi ? 32 + __ffs(hi) - 1 : -1);
        if (nxt < 0) break;
        cur = nxt;
        ++len;
        if (lane == 0) { pn[len] = cur; pt[len] = s_tok[cur]; }
    }
    for (int dd = len + 1 + lane; dd < W; dd += 32) { pn[dd] = -1; pt[dd] = -1; }
    int best = 0x7fffffff;
    for (int r = lane; r < nl; r += 32)
        if (a.retrieve[((size_t)b * a.N + r) * W + len] == cur) best = min(best, r);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) best = min(best, __shfl_xor_sync(kFull, best, o));
    if (lane == 0) {
        a.accept_len[b] = len;
        a.next_token[b] = s_arg[cur];
        a.best_retrieve_row[b] = best == 0x7fffffff ? -1 : best;
    }
}

// ------------------------------------------------------------------------------------------
// stochastic walk
// ------------------------------------------------------------------------------------------
// Few warps: all of them carry the walk's scalars, so its steps between two passes wait for what every warp issues, and
// the exponentials get their overlap from eight chains a thread (512 threads: 40 us for four sequences of 32000
// tokens, 256: 31).  kernels<1>: one CTA per SM, 255 registers a thread, for launches that leave room; kernels<2>: two, so
// that one's passes run while the other exchanges.
constexpr int kSThreads = 256;
constexpr int kSWarps = kSThreads / 32;
constexpr int kMaxCluster = 8;           // portable cluster size limit
constexpr int kMinSlice = 1024;          // tokens of a CTA's slice below which a larger cluster is not worth its exchanges
constexpr int kAccMinSlice = 4096;       // ... where there are rows enough to fill the device anyway

// A CTA's slice of the vocabulary is worked on in tiles of 128 tokens, a contiguous run of tiles to each warp, a quad of
// tokens to a lane: a warp's partial sum is the mass of a run of tokens, and the partial sums of the pass that settles the
// last weights are all that the final draw needs to find the warp that owns the sampled point.
// The exponentials of both rows are cached tile by tile (128 of the target row, 128 of the draft row): the first tiles of every
// warp's run in shared memory, what has no room there in the workspace (all warps wait for L2 then, a third as long; with the
// slice's first tiles on chip, the last warps' runs lay in the workspace as a whole: walk, one sequence of 128256 tokens 43.5 -> 37.4 us,
// 32 of them 99 -> 95; acceptance lengths, one tree of 151001 51 -> 44).  Inside a tile come the first pairs of its
// quads, then their second pairs, so that a warp's two 16-byte accesses each cover 512 bytes without gaps.  A slice's
// last tile may be only partly real (its padding holds zeros); in the workspace CTA r's tiles start 128 r tokens
// behind its first one's index, which keeps the slices apart.
constexpr int kTileTokens = 128;
constexpr int kTileDoubles = 2 * kTileTokens;
constexpr size_t kTileBytes = kTileDoubles * sizeof(double);
// shared memory left for cached tiles when `per_sm` CTAs with `fixed` bytes of static arrays share an SM's 228 KB (1 KB of each
// is the system's)
constexpr size_t cache_room(int per_sm, size_t fixed) { return ((228 * 1024 / per_sm - 1024 - fixed) / kTileBytes) * kTileBytes; }
__host__ __device__ inline size_t cache_stride(int V) { return (((size_t)V + 3) & ~(size_t)3) + kTileTokens * 8; }
extern __shared__ __align__(16) double s_cache[];
struct Tiles { int t0, t1; };            // a warp's run
__device__ __forceinline__ Tiles warp_tiles(int n, int warp) {       // n: tokens of the slice
    const int T = (n + kTileTokens - 1) / kTileTokens;
    return {T * warp / kSWarps, T * (warp + 1) / kSWarps};
}
// A warp's tiles (no other warp touches them): the first of its run, as many as are its share, in shared memory.
struct Cache {
    double* g;                           // this CTA's tiles in the workspace
    double* s;                           // where its first tile would lie in shared memory, if this warp's run went on to it
    int end;                             // tiles [t0, end) are there
    __device__ __forceinline__ Cache(double* g_, int smem_tiles, int n) : g(g_) {
        const int warp = threadIdx.x >> 5, first = smem_tiles * warp / kSWarps;
        const Tiles w = warp_tiles(n, warp);
        end = w.t0 + smem_tiles * (warp + 1) / kSWarps - first;
        s = s_cache + (first - w.t0) * kTileDoubles;
    }
    __device__ __forceinline__ double* tile(int t) const { return (t < end ? s : g) + (ptrdiff_t)t * kTileDoubles; }
    __device__ __forceinline__ double& token(int o, int which) const {       // o: offset in the slice
        return tile(o / kTileTokens)[which * kTileTokens + 2 * ((o >> 2) & 31) + 32 * (o & 2) + (o & 1)];
    }
};

struct ExpTable { double t[64]; };       // 2^(j/64)
// 64 / ln 2; ln 2 / 64 and what its rounding left; 1/5!, 1/4!, 1/3!: instructions take them from the constant bank
__constant__ double c_exp[6] = {92.33248261689366, 0.010830424696249145, 3.623510646634843e-19, 1.0 / 120.0, 1.0 / 24.0, 1.0 / 6.0};
// The table in shared memory, sixteen copies side by side: lane l reads the one in its own pair of banks, so that a
// warp's 32 look-ups never conflict (one copy: 3 of 16 lanes on the same banks on average).
struct ExpShared {
    double t[64][16];
    __device__ __forceinline__ void fill(const ExpTable& T) {
        for (int i = threadIdx.x; i < 64 * 16; i += blockDim.x) t[i >> 4][i & 15] = T.t[i >> 4];
    }
    __device__ __forceinline__ const double* mine() const { return &t[0][threadIdx.x & 15]; }
};

struct StochParams {
    radar_accept_args a;
    double* cache;       // [B][2 * cache_stride] exponentials of the current node's target and draft rows that have no room on chip
    int smem_tiles;      // tiles of a slice whose exponentials are kept in shared memory
    int* status;
    ExpTable tab;
};

// exp(x) in fp64 by table look-up (P. T. P. Tang, "Table-driven implementation of the exponential function in IEEE
// floating-point arithmetic", ACM TOMS 15(2), 1989): x = (64 m + j) ln2/64 + r with |r| <= ln2/128, so
// exp(x) = 2^m 2^(j/64) exp(r), and the Taylor series of exp(r) is exact to 4e-17 after its r^5 term.  Ten fp64
// instructions and a shared-memory read; the results are within 1.1 ulp.  tab: ExpShared::mine()
// exp_split: the factor 2^(j/64) exp(r), and m.
__device__ __forceinline__ double exp_split(double x, const double* tab, int& m) {
    constexpr double kShift = 6755399441055744.0;                 // 1.5 * 2^52: the sum's low word is the rounded integer
    const double t = fma(x, c_exp[0], kShift);
    const int n = __double2loint(t);
    const double nd = t - kShift;
    const double r = fma(-nd, c_exp[2], fma(-nd, c_exp[1], x));
    double s = fma(r, c_exp[3], c_exp[4]);
    s = fma(s, r, c_exp[5]);
    s = fma(s, r, 0.5);
    s = fma(s * r, r, r);
    const double tj = tab[(n & 63) * 16];
    m = n >> 6;
    return fma(tj, s, tj);
}
__device__ __forceinline__ double times_2_to(double y, int m) { return __hiloint2double(__double2hiint(y) + (m << 20), __double2loint(y)); }
// ... over the whole range: 2 ulp below -700, where 2^m leaves the normal numbers; infinite above 700
__device__ __forceinline__ double exp64(double x, const double* tab) {
    int m;
    const double y = exp_split(x, tab, m);
    if (fabs(x) > 700.0) return x > 0.0 ? CUDART_INF : x < -760.0 ? 0.0 : times_2_to(y, m + 512) * 7.458340731200207e-155;   // 2^-512
    return times_2_to(y, m);
}
__device__ __forceinline__ float max_nan(float a, float b) {
    float y;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(y) : "f"(a), "f"(b));
    return y;
}
__device__ __forceinline__ float min_nan(float a, float b) {
    float y;
    asm("min.NaN.f32 %0, %1, %2;" : "=f"(y) : "f"(a), "f"(b));
    return y;
}
// exp(z[i] / T + shift) for 4 Q logits, with one fp32 test and one branch for the rare ranges and NaN (an fp64 comparison behind each
// exponential costs the pipe that bounds this, and a branch behind each keeps the chains from overlapping)
// kBits: the logit becomes a double by integer operations.  A conversion is an fp64 instruction at a fraction of the others' rate,
// which two blocks per SM are bound by (walk, 32 sequences of 50256 tokens 41.6 -> 37.0 us, 16 33.7 -> 30.6; lengths, eight trees 67.4 ->
// 64.4); a block by itself waits for its chains, which the three operations lengthen (4 of 32000 22.4 -> 24.0: not there).
struct ExpRange {
    double invT, scaled, shift;          // scaled: 2^896 / T
    float lo, hi;                        // finite logits between which |z / T + shift| stays below 700
    // Around the logit `ref`.  Both bounds are rounded towards it: with a small T an ulp of the logits is many units of z / T,
    // and a bound rounded away from it would let such a logit through.
    __device__ __forceinline__ ExpRange(double invT_, float ref) : invT(invT_), scaled(invT_ * 0x1p896), shift(-((double)ref * invT_)) {
        const double reach = 690.0 / invT_;
        // (2^896 / T overflows for T up to 2^-128: no logit is in the range then)
        lo = scaled < CUDART_INF ? fmaxf(__double2float_ru((double)ref - reach), -FLT_MAX) : CUDART_INF_F;
        hi = fminf(__double2float_rd((double)ref + reach), FLT_MAX);
    }
    __device__ __forceinline__ double arg(float z) const { return fma((double)z, invT, shift); }
    // ... of a finite one: its fields moved to where a double has them are z 2^-896, also for zeros and below fp32's normal range
    __device__ __forceinline__ double arg_by_bits(float z) const {
        const int u = __float_as_int(z);
        return fma(__hiloint2double((u >> 3) & 0x8fffffff, u << 29), scaled, shift);
    }
    // of any logit (-inf: 0, also where 1 / T has become 0)
    __device__ __forceinline__ double exp_of(float z, const double* tab) const { return z == -CUDART_INF_F ? 0.0 : exp64(arg(z), tab); }
};
// quad q: of range range(q)
template <int Q, bool kBits, typename F>
__device__ __forceinline__ void exp64_quads(const float (&z)[Q][4], F&& range, const double* tab, double (&e)[Q][4]) {
    bool usual = true;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const ExpRange& X = range(q);
        float lo = z[q][0], hi = z[q][0];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            int m;
            const double y = exp_split(kBits ? X.arg_by_bits(z[q][i]) : X.arg(z[q][i]), tab, m);
            e[q][i] = times_2_to(y, m);
            lo = min_nan(lo, z[q][i]);
            hi = max_nan(hi, z[q][i]);
        }
        usual = usual && lo >= X.lo && hi <= X.hi;
    }
    if (!usual) {
#pragma unroll
        for (int q = 0; q < Q; ++q)
#pragma unroll
            for (int i = 0; i < 4; ++i) e[q][i] = range(q).exp_of(z[q][i], tab);
    }
}

// logits v .. v + 3 of a row; -inf from v1 on.  `wide`: the row starts on a boundary of four
__device__ __forceinline__ void load_quad(const float* row, int v, int v1, bool wide, float (&o)[4]) {
    if (wide && v + 4 <= v1) {
        const float4 x = *reinterpret_cast<const float4*>(row + v);
        o[0] = x.x; o[1] = x.y; o[2] = x.z; o[3] = x.w;
    } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) o[e] = v + e < v1 ? row[v + e] : -CUDART_INF_F;
    }
}
__device__ __forceinline__ void load_quad(const __nv_bfloat16* row, int v, int v1, bool wide, float (&o)[4]) {
    if (wide && v + 4 <= v1) {
        const uint2 x = *reinterpret_cast<const uint2*>(row + v);
        o[0] = __uint_as_float(x.x << 16); o[1] = __uint_as_float(x.x & 0xffff0000u);
        o[2] = __uint_as_float(x.y << 16); o[3] = __uint_as_float(x.y & 0xffff0000u);
    } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) o[e] = v + e < v1 ? to_float(row[v + e]) : -CUDART_INF_F;
    }
}
template <typename T>
__device__ __forceinline__ bool row_is_wide(const T* row) { return (reinterpret_cast<uintptr_t>(row) & (4 * sizeof(T) - 1)) == 0; }
// this lane's quad of a cached tile
__device__ __forceinline__ void store_quad(double* tile, const double (&e)[4]) {
    const int lane = threadIdx.x & 31;
    reinterpret_cast<double2*>(tile)[lane] = make_double2(e[0], e[1]);
    reinterpret_cast<double2*>(tile)[lane + 32] = make_double2(e[2], e[3]);
}
__device__ __forceinline__ void load_quad(const double* tile, double (&e)[4]) {
    const int lane = threadIdx.x & 31;
    const double2 x = reinterpret_cast<const double2*>(tile)[lane], y = reinterpret_cast<const double2*>(tile)[lane + 32];
    e[0] = x.x; e[1] = x.y; e[2] = y.x; e[3] = y.y;
}

// Asks for this CTA's slice of a row to be brought into L2 (one instruction of one thread; the 16-byte granules that lie
// wholly inside the slice).
template <typename T>
__device__ __forceinline__ void prefetch_slice(const T* row, int v0, int v1) {
    const uintptr_t lo = (reinterpret_cast<uintptr_t>(row + v0) + 15) & ~(uintptr_t)15, hi = reinterpret_cast<uintptr_t>(row + v1) & ~(uintptr_t)15;
    if (hi > lo) asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(lo), "r"((uint32_t)(hi - lo)) : "memory");
}

// The walk of one sequence (and the evaluation of one tree row) is shared by the CTAs of a thread-block cluster: CTA r
// owns a slice of whole quads of tokens in every full-vocabulary pass.  Every scalar that steers the walk is reduced
// over the cluster into every CTA in a fixed order, so all CTAs take identical decisions and make the same exchanges.
// What a pass over a small slice costs is its exchange.  Every warp sends its partial pair into every CTA's slots with
// asynchronous stores that complete on the receiver's mbarrier, and every warp adds all of them up by itself: one way
// across the cluster, and no barrier whose release would first wait for the pass's stores to global memory (a cluster
// barrier in its place: 2000 cycles an exchange, at one CTA as at eight).
// Use k of a half of the slots follows use k - 2 safely: whoever sends in use k has waited for everyone's use k - 1,
// and a warp sends there only after it has read its use k - 2.
struct RedShared {
    double2 slots[2][kMaxCluster * kSWarps];
    uint64_t bar[2];                         // kSWarps local arrivals and the bytes of all warps of the cluster
};
struct ClusterRed {
    RedShared& R;
    int* status;
    unsigned rank, n, phase;

    __device__ static void cluster_sync() {
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
    // by all threads, before the first exchange
    __device__ void start() {
        if (threadIdx.x == 0) {
            for (int h = 0; h < 2; ++h)
                asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"((uint32_t)__cvta_generic_to_shared(&R.bar[h])), "r"(kSWarps) : "memory");
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        __syncthreads();
        cluster_sync();
    }
    // this warp's pair (the same in every lane) to slot (rank, warp) of every CTA.  What the warp has written to shared or
    // global memory before is visible to this CTA's other warps once they have received.
    __device__ __forceinline__ void send(double a, double b) {
        const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5, h = phase & 1;
        const uint32_t bar = (uint32_t)__cvta_generic_to_shared(&R.bar[h]);
        if (n == 1) {
            if (lane == 0) R.slots[h][warp] = make_double2(a, b);
        } else if (lane < n) {
            asm volatile(
                "{\n\t.reg .u32 ra, rb;\n\t"
                "mapa.shared::cluster.u32 ra, %0, %2;\n\t"
                "mapa.shared::cluster.u32 rb, %1, %2;\n\t"
                "st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f64 [ra], {%3, %4}, [rb];\n\t}"
                ::"r"((uint32_t)__cvta_generic_to_shared(&R.slots[h][rank * kSWarps + warp])), "r"(bar), "r"(lane), "d"(a), "d"(b)
                : "memory");
        }
        __syncwarp();
        if (lane == 0) {
            if (warp == 0 && n > 1) asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(n * kSWarps * 16) : "memory");
            else asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
        }
    }
    // the slots, filled (rank-major: token order of the slices)
    __device__ __forceinline__ const double2* receive() {
        const unsigned h = phase & 1, parity = (phase >> 1) & 1;
        const uint32_t bar = (uint32_t)__cvta_generic_to_shared(&R.bar[h]);
        uint32_t ok = 0;
        // (test_wait: a thread that try_wait has put to sleep takes longer to come back than the partials take to arrive)
        for (uint32_t it = 0; it < (1u << 24) && !ok; ++it)
            asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                         : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
        if (!ok) set_status(status, RADAR_ERR_TIMEOUT);
        __syncwarp();
        ++phase;
        return R.slots[h];
    }
    // the slots of the last exchange received (until the next but one is sent)
    __device__ __forceinline__ const double2* last() const { return R.slots[(phase - 1) & 1]; }
    __device__ double2 receive_sum2() {
        const double2* all = receive();
        double2 t = make_double2(0.0, 0.0);
        for (unsigned i = threadIdx.x & 31; i < n * kSWarps; i += 32) { t.x += all[i].x; t.y += all[i].y; }
        return make_double2(warp_sum(t.x), warp_sum(t.y));
    }
    __device__ double receive_sum() {
        const double2* all = receive();
        double t = 0.0;
        for (unsigned i = threadIdx.x & 31; i < n * kSWarps; i += 32) t += all[i].x;
        return warp_sum(t);
    }
    __device__ float2 max(float a, float b) {
        send((double)warp_max(a), (double)warp_max(b));
        const double2* all = receive();
        float2 t = make_float2(-CUDART_INF_F, -CUDART_INF_F);
        for (unsigned i = threadIdx.x & 31; i < n * kSWarps; i += 32) { t.x = fmaxf(t.x, (float)all[i].x); t.y = fmaxf(t.y, (float)all[i].y); }
        return make_float2(warp_max(t.x), warp_max(t.y));
    }
};

struct NodeShared {
    ExpShared exps;
    RedShared red;
    int tok[kMaxNodes], par[kMaxNodes], drow[kMaxNodes];
    double pe[kMaxNodes], qe[kMaxNodes];     // exponentials of the node's children, by tree row
};

// children of row c as a 64-bit set, in every thread
__device__ __forceinline__ unsigned long long children_of(const NodeShared& S, int c) {
    const int lane = threadIdx.x & 31;
    const unsigned lo = __ballot_sync(kFull, S.par[lane] == c && lane > c), hi = __ballot_sync(kFull, S.par[lane + 32] == c && lane + 32 > c);
    return (unsigned long long)hi << 32 | lo;
}

// this CTA's slice of one row: this thread's maximum (NaN if it has seen one)
template <typename T>
__device__ __forceinline__ float slice_max(const T* row, int v0, int v1) {
    const bool wide = row_is_wide(row);
    const Tiles w = warp_tiles(v1 - v0, threadIdx.x >> 5);
    float m = -CUDART_INF_F;
#pragma unroll 1
    for (int t = w.t0; t < w.t1; ++t) {
        float z[4];
        load_quad(row, v0 + t * kTileTokens + 4 * (threadIdx.x & 31), v1, wide, z);
        m = max_nan(max_nan(m, max_nan(z[0], z[1])), max_nan(z[2], z[3]));
    }
    return m;
}

// This CTA's slice of one row into the cache (which: 0 target, 1 draft): exp(z / T + shift); returns this thread's sum.
// Q tiles at a time, four chains of exponentials each, the next quads on their way meanwhile.  Two where the SM is full (walk of
// 32 sequences of 128256 tokens 88 us, one at a time 94), one in a block by itself, which goes through few tiles and waits for the
// loop's instructions (four of 32000 21.0, two at a time 22.4, four 26.2).  first: the thread's first quad.
template <typename T, bool kBits>
__device__ __forceinline__ double slice_exp(const T* row, int v0, int v1, const ExpRange& X, const double* tab, const Cache C, int which, float4 first) {
    constexpr int Q = kBits ? 2 : 1;
    const auto range = [&](int) -> const ExpRange& { return X; };
    const bool wide = row_is_wide(row);
    const Tiles w = warp_tiles(v1 - v0, threadIdx.x >> 5);
    const int mine = v0 + 4 * (threadIdx.x & 31);
    double s[Q] = {};
    float z[Q][4] = {{first.x, first.y, first.z, first.w}};
    auto load = [&](int t, float (&o)[4]) { load_quad(row, t < w.t1 ? mine + t * kTileTokens : v1, v1, wide, o); };
    if (Q == 2) load(w.t0 + 1, z[Q - 1]);
    int t = w.t0;
#pragma unroll 1
    for (; t + Q <= w.t1; t += Q) {
        float zn[Q][4];
#pragma unroll
        for (int q = 0; q < Q; ++q) load(t + Q + q, zn[q]);
        double e[Q][4];
        exp64_quads<Q, kBits>(z, range, tab, e);
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            store_quad(C.tile(t + q) + which * kTileTokens, e[q]);
            s[q] += (e[q][0] + e[q][1]) + (e[q][2] + e[q][3]);
#pragma unroll
            for (int i = 0; i < 4; ++i) z[q][i] = zn[q][i];
        }
    }
    if (Q == 2 && t < w.t1) {
        const float zl[1][4] = {{z[0][0], z[0][1], z[0][2], z[0][3]}};
        double e[1][4];
        exp64_quads<1, kBits>(zl, range, tab, e);
        store_quad(C.tile(t) + which * kTileTokens, e[0]);
        s[0] += (e[0][0] + e[0][1]) + (e[0][2] + e[0][3]);
    }
    return Q == 2 ? s[0] + s[Q - 1] : s[0];
}
// ... of both rows in one loop, a tile of each at a time; both sums.  Eight chains as well, and half the code: a warp goes through a
// few tiles of a row only, and its first pass over a loop waits for the instructions.  us in one loop / two: acceptance lengths of
// eight trees 124 / 133 (V = 128256), 62.7 / 64.3 (50256), of four of 32000 23.9 / 25.2, of one of 151001 43.5 / 43.7.  (In the
// walk, whose last node has no draft row, 94 / 90.5 for 32 sequences of 128256, 33.5 / 31.6 for 6 of 50257: not there.)
template <typename T, bool kBits>
__device__ __forceinline__ double2 slice_exp_both(const T* target, const T* draft, int v0, int v1, const ExpRange (&X)[2], const double* tab,
                                                  const Cache C, float4 first_t, float4 first_d) {
    const T* const row[2] = {target, draft};
    const bool wide[2] = {row_is_wide(target), row_is_wide(draft)};
    const Tiles w = warp_tiles(v1 - v0, threadIdx.x >> 5);
    const int mine = v0 + 4 * (threadIdx.x & 31);
    double s[2] = {0.0, 0.0};
    float z[2][4] = {{first_t.x, first_t.y, first_t.z, first_t.w}, {first_d.x, first_d.y, first_d.z, first_d.w}};
#pragma unroll 1
    for (int t = w.t0; t < w.t1; ++t) {
        float zn[2][4];
#pragma unroll
        for (int q = 0; q < 2; ++q) load_quad(row[q], t + 1 < w.t1 ? mine + (t + 1) * kTileTokens : v1, v1, wide[q], zn[q]);
        double e[2][4];
        exp64_quads<2, kBits>(z, [&](int q) -> const ExpRange& { return X[q]; }, tab, e);
        double* const tile = C.tile(t);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            store_quad(tile + q * kTileTokens, e[q]);
            s[q] += (e[q][0] + e[q][1]) + (e[q][2] + e[q][3]);
#pragma unroll
            for (int i = 0; i < 4; ++i) z[q][i] = zn[q][i];
        }
    }
    return make_double2(s[0], s[1]);
}
template <typename T>
__device__ __forceinline__ float4 first_quad(const T* row, int v0, int v1) {
    const Tiles w = warp_tiles(v1 - v0, threadIdx.x >> 5);
    float z[4] = {0.f, 0.f, 0.f, 0.f};
    if (w.t0 < w.t1) load_quad(row, v0 + w.t0 * kTileTokens + 4 * (threadIdx.x & 31), v1, row_is_wide(row), z);
    return make_float4(z[0], z[1], z[2], z[3]);
}

// this CTA's slice of the two rows (draft may be NULL): this thread's maxima, NaN if it has seen one
template <typename T>
__device__ __forceinline__ float2 slice_maxima(const T* target, const T* draft, int v0, int v1) {
    return make_float2(slice_max(target, v0, v1), draft != nullptr ? slice_max(draft, v0, v1) : 0.f);
}

// One tree node's rows: cache[v] = exp((z[v] - ref) / T) of the target row and, unless `draft` is NULL, of the draft
// row, over this CTA's slice [v0, v1); the exponentials at the node's children into S.pe / S.qe.  Returns the
// two row sums (1 for a missing draft row).  `meanwhile` runs while the sums are on their way.
// The reference of a row need not be its maximum: fp64 has room for exp(700), and relative precision does not depend on
// the scale.  It is the largest of 32 of the row's logits, the same ones in every warp, so a row is read once
// and its two rows take one exchange.  Only if a sum shows that some logit lies so far above (or that the sample held
// nothing finite) the pass is repeated from the exact maxima.  kBoth: `draft` is not NULL.
template <typename T, bool kBits, bool kBoth, typename F>
__device__ double2 softmax_rows(NodeShared& S, ClusterRed& red, const T* target, const T* draft, int V, int v0, int v1,
                                double invT, const Cache C, unsigned long long children, bool* nan_seen,
                                F&& meanwhile) {
    const int tid = threadIdx.x;
    const bool two = kBoth || draft != nullptr;
    const int x = tid < kMaxNodes && ((children >> tid) & 1) ? S.tok[tid] : -1;
    const bool child = x >= 0 && x < V;
    const float xt = child ? to_float(target[x]) : 0.f, xd = child && two ? to_float(draft[x]) : 0.f;
    const int at = (int)((long long)(V - 1) * (tid & 31) / 31);
    float rt = to_float(target[at]), rd = two ? to_float(draft[at]) : 0.f;
    const float4 ft = first_quad(target, v0, v1), fd = two ? first_quad(draft, v0, v1) : make_float4(0.f, 0.f, 0.f, 0.f);
    rt = warp_max(rt);
    rd = warp_max(rd);
    const double* tab = S.exps.mine();
    for (int pass = 0;; ++pass) {
        const ExpRange X[2] = {ExpRange(invT, rt), ExpRange(invT, rd)};
        double2 sum;
        if constexpr (kBoth) {
            sum = slice_exp_both<T, kBits>(target, draft, v0, v1, X, tab, C, ft, fd);
        } else {
            sum.x = slice_exp<T, kBits>(target, v0, v1, X[0], tab, C, 0, ft);
            sum.y = two ? slice_exp<T, kBits>(draft, v0, v1, X[1], tab, C, 1, fd) : 1.0 / (kMaxCluster * kSThreads);
        }
        if (child) {
            S.pe[tid] = X[0].exp_of(xt, tab);
            S.qe[tid] = two ? X[1].exp_of(xd, tab) : 0.0;
        }
        red.send(warp_sum(sum.x), warp_sum(sum.y));
        if (pass == 0) meanwhile();
        const double2 s = red.receive_sum2();                      // ... and S.pe and S.qe
        if ((s.x > 0.0 && s.x < 1e250 && s.y > 0.0 && s.y < 1e250) || pass == 1) return make_double2(s.x, two ? s.y : 1.0);
        const float2 mine = slice_maxima(target, draft, v0, v1);
        if (mine.x != mine.x || mine.y != mine.y) *nan_seen = true;
        const float2 m = red.max(mine.x, mine.y);
        rt = m.x;
        rd = m.y;
    }
}

// this thread's share of the sum over the slice (n tokens) of max(0, e_p - rho e_q), the exponentials from the caches (U tiles'
// loads side by side: four in the workspace; with more, or with the first of them ahead of the tiles on chip, kernels<2> spill: 3 to 13 % slower)
template <int U>
__device__ __forceinline__ double residual_of_tiles(const double* base, int t0, int t1, double rho) {
    double g0 = 0.0, g1 = 0.0;
#pragma unroll U
    for (int t = t0; t < t1; ++t) {
        double p[4], q[4];
        load_quad(base + (size_t)t * kTileDoubles, p);
        load_quad(base + (size_t)t * kTileDoubles + kTileTokens, q);
        const double d0 = fma(-rho, q[0], p[0]), d1 = fma(-rho, q[1], p[1]), d2 = fma(-rho, q[2], p[2]), d3 = fma(-rho, q[3], p[3]);
        if (d0 > 0.0) g0 += d0;                              // (a compare and a predicated add: fewer instructions than fmax)
        if (d1 > 0.0) g1 += d1;
        if (d2 > 0.0) g0 += d2;
        if (d3 > 0.0) g1 += d3;
    }
    return g0 + g1;
}
__device__ __forceinline__ double slice_residual(const Cache C, int n, double rho) {
    const Tiles w = warp_tiles(n, threadIdx.x >> 5);
    const int mid = min(C.end, w.t1);
    return residual_of_tiles<2>(C.s, w.t0, mid, rho) + residual_of_tiles<4>(C.g, mid, w.t1, rho);
}

// The residual pair of a node while its children are tried in order (file header), in units of the target row's sum:
// with the row sums s_p and s_q, rho = a s_p / s_q and G = W s_p, the residual of a token is max(0, e_p - rho e_q) / G
// and rho grows by c G / s_q.  Every thread carries it.
struct Residual {
    double rho = 0.0, G, c = 1.0, inv_sq;
    bool any = false;                    // some child has been rejected
    bool settled = true;                 // the last exchange carried the masses of the present weights
    __device__ Residual(double sp, double sq) : G(sp), inv_sq(1.0 / sq) {}
    __device__ double left(double ep, double eq) const { return fmax(0.0, fma(-rho, eq, ep)); }    // a token's residual (over G: its probability)
    __device__ double draft(double eq) const { return c * (eq * inv_sq); }                         // its probability under the draft left
    // reject the child with token x, of probability qj under the draft left; false once the draft's mass is used up.
    // `meanwhile` runs while the partial sums are on their way.
    template <typename F>
    __device__ bool reject(ClusterRed& red, const Cache C, int v0, int v1, int x, double ep, double eq, double qj, F&& meanwhile) {
        const double rho_new = fma(c * inv_sq, G, rho);
        red.send(warp_sum(slice_residual(C, v1 - v0, rho_new)), 0.0);
        meanwhile();
        const double rest = 1.0 - qj;                        // draft mass left after removing x
        c = c / rest;
        const double g = red.receive_sum();
        settled = g > 0.0;
        if (settled) { rho = rho_new; G = g; }               // else: residual empty, p stays as it is
        any = true;
        // From here on x keeps its own coefficient: its cached pair becomes (residual, 0), which every later pass takes as
        // it is.  The thread that writes it is the one that reads it in them.
        const int o = x - v0, t = o / kTileTokens;
        const Tiles w = warp_tiles(v1 - v0, threadIdx.x >> 5);
        if (o >= 0 && x < v1 && t >= w.t0 && t < w.t1 && ((o >> 2) & 31) == (int)(threadIdx.x & 31)) {
            C.token(o, 0) = left(ep, eq);
            C.token(o, 1) = 0.0;
        }
        return rest > 0.0;
    }
};

struct WalkShared {                      // all static shared memory of the kernel: cache_room counts on it
    NodeShared node;
    float ua[kMaxNodes];
};

template <typename T, int kPerSm>
__global__ void __launch_bounds__(kSThreads, kPerSm) stochastic_walk_kernel(const __grid_constant__ StochParams P) {
    const radar_accept_args& a = P.a;
    unsigned crank, csize;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(crank));
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(csize));
    const int b = blockIdx.x / csize, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int V = a.V, W = a.t_max + 1;
    __shared__ WalkShared sh;
    NodeShared& S = sh.node;
    float (&s_ua)[kMaxNodes] = sh.ua;
    S.exps.fill(P.tab);
    ClusterRed red{S.red, P.status, crank, csize, 0};
    red.start();
    chain_wait();
    const int nq = (V + 3) / 4;
    const int v0 = 4 * (int)((long long)nq * crank / csize), v1 = min(V, 4 * (int)((long long)nq * (crank + 1) / csize));
    const bool lead = crank == 0;                 // writes the per-sequence outputs

    const int nl = a.n_leaves[b];
    const int retr = a.N * W;                     // the retrieve rows, needed at the very end: into L1 by then
    if (lead && tid >= 64 && (tid - 64) * 32 < retr) asm volatile("prefetch.global.L1 [%0];" ::"l"(a.retrieve + (size_t)b * retr + (tid - 64) * 32));
    if (tid < kMaxNodes) {
        const size_t o = (size_t)b * kMaxNodes + tid;
        const int M = min(max(a.n_nodes[b], 1), kMaxNodes);
        const int tok = a.tree_tok[o], par = a.tree_parent[o], dr = a.tree_draft_row[o];
        s_ua[tid] = a.u_accept[o];
        S.tok[tid] = tid < M ? tok : -1;
        S.par[tid] = tid < M ? par : -2;
        S.drow[tid] = tid < M ? dr : -1;
    }
    const T* target = reinterpret_cast<const T*>(a.target_logits) + (size_t)b * kMaxNodes * V;
    const T* draft = reinterpret_cast<const T*>(a.draft_logits) + (size_t)b * a.R * V;
    const Cache C(P.cache + 2 * ((size_t)b * cache_stride(V) + v0 + kTileTokens * crank), P.smem_tiles, v1 - v0);
    if (tid == 0) prefetch_slice(target, v0, v1);                 // the root's rows
    if (tid == 0) prefetch_slice(draft, v0, v1);
    __syncthreads();
    const double invT = 1.0 / (double)a.temperature;
    bool nan_seen = false, bad_tree = false;

    int32_t* pn = a.path_nodes + (size_t)b * W;
    int32_t* pt = a.path_tokens + (size_t)b * W;
    int cur = 0, len = 0;
    if (lead && tid == 0) { pn[0] = 0; pt[0] = S.tok[0]; }

    Residual res(1.0, 1.0);
    for (;;) {
        unsigned long long kids = len >= a.t_max ? 0ull : children_of(S, cur);
        const int drow = S.drow[cur];
        if (kids != 0 && (drow < 0 || drow >= a.R)) { bad_tree = true; kids = 0; }
        // The rows of the child that is tried next are asked for ahead: if it is accepted they are the next node's, and a
        // row's first access otherwise waits for memory and address translation (2500 cycles).
        auto fetch_ahead = [&](unsigned long long next) {
            if (tid == 0 && next != 0) {
                const int j = __ffsll(next) - 1, dr = S.drow[j];
                prefetch_slice(target + (size_t)j * V, v0, v1);
                if (dr >= 0 && dr < a.R) prefetch_slice(draft + (size_t)dr * V, v0, v1);
            }
        };
        const double2 sums = softmax_rows<T, kPerSm == 2, false>(S, red, target + (size_t)cur * V, kids != 0 ? draft + (size_t)drow * V : nullptr, V, v0, v1, invT,
                                             C, kids, &nan_seen, [&] { fetch_ahead(kids); });
        res = Residual(sums.x, sums.y);
        int accepted = -1;
        for (; kids != 0; kids &= kids - 1) {
            const int j = __ffsll(kids) - 1;
            const int x = S.tok[j];
            if (x < 0 || x >= V) { bad_tree = true; break; }
            const double ep = S.pe[j], eq = S.qe[j];
            const double pj = res.left(ep, eq);                      // x has not been proposed before
            const double qj = res.draft(eq);
            // u < min(1, (pj / G) / qj) without the divisions; u is below 1
            if (qj <= 0.0 ? pj > 0.0 : (double)s_ua[j] * (qj * res.G) < pj) { accepted = j; break; }
            if (!res.reject(red, C, v0, v1, x, ep, eq, qj, [&] { fetch_ahead(kids & (kids - 1)); })) break;
        }
        if (bad_tree || accepted < 0) break;
        cur = accepted;
        ++len;
        if (lead && tid == 0) { pn[len] = cur; pt[len] = S.tok[cur]; }
    }

    // ---- final draw: inverse CDF over w(v) = max(0, p(v) - a(v) q(v)) (or p(v) when nothing was rejected) ----
    // The warps' masses, in token order, tell every warp which one holds the point; that warp then goes through its tiles.
    // The last exchange has carried them: the sums of the exponentials if nothing was rejected, else those of the last
    // residual (unless that was empty, and the weights are still the ones before it).
    auto weights = [&](int t, double (&w)[4]) {   // (of a tile's quad, in units of G)
        load_quad(C.tile(t), w);
        if (res.any) {
            double q[4];
            load_quad(C.tile(t) + kTileTokens, q);
#pragma unroll
            for (int i = 0; i < 4; ++i) w[i] = res.left(w[i], q[i]);
        }
    };
    const Tiles mine_t = warp_tiles(v1 - v0, warp);
    if (!res.settled) {
        double mass = 0.0;
        for (int t = mine_t.t0; t < mine_t.t1; ++t) {
            double w[4];
            weights(t, w);
            mass += (w[0] + w[1]) + (w[2] + w[3]);
        }
        red.send(warp_sum(mass), 0.0);
        red.receive();
    }
    const double2* all = red.last();
    // running sums over all warps of the cluster, four consecutive ones to a lane
    const int nw = (int)csize * kSWarps;
    double m4[4], own = 0.0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        m4[i] = 4 * lane + i < nw ? all[4 * lane + i].x : 0.0;
        own += m4[i];
    }
    double incl = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double t = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += t;
    }
    const double total = __shfl_sync(kFull, incl, 31);
    const double tgt = (double)a.u_sample[b] * total;
    // owner: the first warp whose end exceeds the point; if rounding leaves none, the last one with mass
    int first = 0x7fffffff, last_live = -1;
    double start = 0.0, run = incl - own;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const double before = run;
        run += m4[i];
        if (m4[i] > 0.0) last_live = 4 * lane + i;
        if (first == 0x7fffffff && tgt < run && m4[i] > 0.0) { first = 4 * lane + i; start = before; }
    }
    const int who = __reduce_min_sync(kFull, first);
    const int live = __reduce_max_sync(kFull, last_live);
    start = __shfl_sync(kFull, start, who != 0x7fffffff ? who >> 2 : 0);
    const int owner = who != 0x7fffffff ? who : max(live, 0);
    if (owner == (int)crank * kSWarps + warp) {
        double at = start;
        int pick = -1, last_pos = -1;
        for (int t = mine_t.t0; t < mine_t.t1; ++t) {
            const int v = v0 + t * kTileTokens + 4 * lane;
            double w[4];
            weights(t, w);
            const double mine = (w[0] + w[1]) + (w[2] + w[3]);
            double in = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const double u = __shfl_up_sync(kFull, in, o);
                if (lane >= o) in += u;
            }
            double c = at + (in - mine);
            int hit = 0x7fffffff, pos = -1;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                c += w[i];
                if (w[i] > 0.0) {
                    pos = v + i;
                    if (hit == 0x7fffffff && c > tgt) hit = v + i;
                }
            }
            hit = __reduce_min_sync(kFull, hit);
            last_pos = max(last_pos, __reduce_max_sync(kFull, pos));
            if (who != 0x7fffffff && hit != 0x7fffffff) { pick = hit; break; }
            at += __shfl_sync(kFull, in, 31);
        }
        if (lane == 0) a.next_token[b] = pick >= 0 ? pick : last_pos;     // (rounding guard: the crossing is in this run)
    }
    if (lead && tid == 0) {
        a.accept_len[b] = len;
        if (bad_tree) set_status(P.status, RADAR_ERR_TREE);
    }
    if (nan_seen) set_status(P.status, RADAR_ERR_NUMERIC);
    if (lead) {
        for (int dd = len + 1 + tid; dd < W; dd += kSThreads) { pn[dd] = -1; pt[dd] = -1; }
        if (tid < 32) {
            int best = 0x7fffffff;
            for (int r = tid; r < nl; r += 32)
                if (a.retrieve[((size_t)b * a.N + r) * W + len] == cur) best = min(best, r);
            best = __reduce_min_sync(kFull, best);
            if (tid == 0) a.best_retrieve_row[b] = best == 0x7fffffff ? -1 : best;
        }
    }
    // (every CTA has received all that was sent to it: none leaves before a store into its shared memory has landed)
}

// ------------------------------------------------------------------------------------------
// acceptance-length distribution (Eq. 11-13)
// ------------------------------------------------------------------------------------------
struct AccLenParams {
    radar_acclen_args a;
    double* cache;       // [clusters][2 * cache_stride]
    int smem_tiles;
    double* cond;        // [B][64]: P_acc(row | its parent), in the workspace
    int* status;
    ExpTable tab;
};

constexpr int kAccBatch = 8, kAccRows = kAccBatch * kMaxNodes;     // sequences whose trees are looked at together, their rows
struct AccLenShared {                    // all static shared memory of the kernel
    NodeShared node;
    __align__(16) int count[kAccRows + 4];      // children of each of their rows, then the order's keys
    int group[kAccRows / 32];
    int tok[kAccRows], par[kAccRows], drow[kAccRows];      // the batch's trees
    short order[kAccRows];
};

// One item = one tree row with children of one sequence, evaluated by a cluster of CTAs (slices of the vocabulary, as in
// the walk above).  The resident clusters take the items in turn; a row's children are tried in order with the same
// closed-form residual recursion, but every rejection branch is followed: child j gets reach_j a_j with
// reach_j = prod_{i<j} (1 - a_i).  Clusters of 8 at V = 128256 keep at most 36 pairs of cached rows alive (74 MB,
// inside L2; one CTA per row had 300 MB of them and went to HBM with every pass).
template <typename T, int kPerSm>
__global__ void __launch_bounds__(kSThreads, kPerSm) accept_length_nodes_kernel(const __grid_constant__ AccLenParams P) {
    const radar_acclen_args& a = P.a;
    unsigned crank, csize;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(crank));
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(csize));
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, V = a.V;
    constexpr int kBatch = kAccBatch, kRows = kAccRows, kEach = kRows / kSThreads;
    __shared__ AccLenShared sh;
    NodeShared& S = sh.node;
    int (&s_count)[kRows + 4] = sh.count;
    int (&s_group)[kRows / 32] = sh.group;
    short (&s_order)[kRows] = sh.order;
    int (&s_tok)[kRows] = sh.tok, (&s_par)[kRows] = sh.par, (&s_drow)[kRows] = sh.drow;
    S.exps.fill(P.tab);
    ClusterRed red{S.red, P.status, crank, csize, 0};
    red.start();
    chain_wait();
    const int cluster = blockIdx.x / csize, n_clusters = gridDim.x / csize;
    const int nq = (V + 3) / 4;
    const int v0 = 4 * (int)((long long)nq * crank / csize), v1 = min(V, 4 * (int)((long long)nq * (crank + 1) / csize));
    const Cache C(P.cache + 2 * ((size_t)cluster * cache_stride(V) + v0 + kTileTokens * crank), P.smem_tiles, v1 - v0);
    const double invT = 1.0 / (double)a.temperature;
    bool nan_seen = false, bad_tree = false;

    for (int b0 = 0; b0 < a.B; b0 += kBatch) {
        int n_items;
        // Rows with children of up to eight sequences, those with the most children first (a row's time is two passes
        // over its logits and one per child but the last), dealt out over the clusters back and forth: thread (b, c)
        // counts row c's children and finds its own place in that order.
        {
            // (every thread does kEach rows: row e = tid + i * kSThreads of the batch)
            int tok[kEach], up[kEach], dr[kEach], M[kEach];
#pragma unroll
            for (int i = 0; i < kEach; ++i) {
                const int e = tid + i * kSThreads, b = b0 + e / kMaxNodes;
                const size_t o = (size_t)(b < a.B ? b : 0) * kMaxNodes + e % kMaxNodes;
                tok[i] = a.tree_tok[o]; up[i] = a.tree_parent[o]; dr[i] = a.tree_draft_row[o];
                M[i] = b < a.B ? min(max(a.n_nodes[b], 1), kMaxNodes) : 0;
            }
            __syncthreads();                                 // the previous batch's readers are done
#pragma unroll
            for (int i = 0; i < kEach; ++i) {
                const int e = tid + i * kSThreads, c = e % kMaxNodes;
                s_count[e] = 0;
                s_tok[e] = c < M[i] ? tok[i] : -1;
                s_par[e] = c < M[i] ? up[i] : -2;
                s_drow[e] = dr[i];
            }
            __syncthreads();
#pragma unroll
            for (int i = 0; i < kEach; ++i) {
                const int e = tid + i * kSThreads, c = e % kMaxNodes;
                if (c > 0 && c < M[i] && up[i] >= 0 && up[i] < c) atomicAdd(&s_count[e - c + up[i]], 1);
            }
            __syncthreads();
            int mine[kEach];
            unsigned has[kEach];
#pragma unroll
            for (int i = 0; i < kEach; ++i) {
                mine[i] = s_count[tid + i * kSThreads];
                has[i] = __ballot_sync(kFull, mine[i] > 0);
                if (lane == 0) s_group[warp + i * kSWarps] = __popc(has[i]);
            }
            __syncthreads();
            n_items = 0;
            int before[kEach];
#pragma unroll
            for (int g = 0; g < kRows / 32; ++g) {           // groups of 32 rows, in order
#pragma unroll
                for (int i = 0; i < kEach; ++i)
                    if (g == warp + i * kSWarps) before[i] = n_items;
                n_items += s_group[g];
            }
#pragma unroll
            for (int i = 0; i < kEach; ++i)                  // (all counts have been read)
                if (mine[i] > 0) s_count[before[i] + __popc(has[i] & ((1u << lane) - 1u))] = (kMaxNodes - mine[i]) * kRows + tid + i * kSThreads;
            if (tid < 3) s_count[n_items + tid] = 0x7fffffff;
            __syncthreads();
            for (int x = tid; x < n_items; x += kSThreads) {
                const int key = s_count[x];
                int place = 0;
                for (int o = 0; o < n_items; o += 4) {
                    const int4 k4 = *reinterpret_cast<const int4*>(s_count + o);
                    place += (k4.x < key ? 1 : 0) + (k4.y < key ? 1 : 0) + (k4.z < key ? 1 : 0) + (k4.w < key ? 1 : 0);
                }
                s_order[place] = (short)(key % kRows);
            }
            __syncthreads();
        }
        for (int round = 0; round * n_clusters < n_items; ++round) {
            const int place = round * n_clusters + ((round & 1) ? n_clusters - 1 - cluster : cluster);
            if (place < n_items) {
                const int item = s_order[place], first = item & ~(kMaxNodes - 1);
                const int b = b0 + item / kMaxNodes, c = item % kMaxNodes;
                const int drow = s_drow[item];
                __syncthreads();                             // the previous item's readers are done with S
                if (tid < kMaxNodes) {
                    S.tok[tid] = s_tok[first + tid];
                    S.par[tid] = s_par[first + tid];
                }
                __syncthreads();
                if (drow < 0 || drow >= a.R) { bad_tree = true; continue; }
                unsigned long long kids = children_of(S, c);
                const T* target = reinterpret_cast<const T*>(a.target_logits) + ((size_t)b * kMaxNodes + c) * V;
                const T* draft = reinterpret_cast<const T*>(a.draft_logits) + ((size_t)b * a.R + drow) * V;
                // the rows of this cluster's next item are asked for while this one's are worked on
                const int next = (round + 1) * n_clusters + ((round & 1) ? cluster : n_clusters - 1 - cluster);
                const double2 sums = softmax_rows<T, kPerSm == 2, true>(S, red, target, draft, V, v0, v1, invT, C, kids, &nan_seen, [&] {
                    if (tid == 0 && next < n_items) {
                        const size_t bn = b0 + s_order[next] / kMaxNodes, cn = s_order[next] % kMaxNodes;
                        const int dn = s_drow[s_order[next]];
                        prefetch_slice(reinterpret_cast<const T*>(a.target_logits) + (bn * kMaxNodes + cn) * V, v0, v1);
                        if (dn >= 0 && dn < a.R) prefetch_slice(reinterpret_cast<const T*>(a.draft_logits) + (bn * a.R + dn) * V, v0, v1);
                    }
                });
                Residual res(sums.x, sums.y);
                double reach = 1.0;
                bool exhausted = false;
                for (; kids != 0; kids &= kids - 1) {
                    const int j = __ffsll(kids) - 1;
                    if (exhausted) {
                        if (crank == 0 && tid == 0) P.cond[(size_t)b * kMaxNodes + j] = 0.0;
                        continue;
                    }
                    const int x = S.tok[j];
                    if (x < 0 || x >= V) { bad_tree = true; break; }
                    const double ep = S.pe[j], eq = S.qe[j];
                    const double pj = res.left(ep, eq), qj = res.draft(eq);
                    auto book = [&] {
                        double acc;
                        if (qj <= 0.0) acc = pj > 0.0 ? 1.0 : 0.0;
                        else { acc = pj / (qj * res.G); if (acc > 1.0) acc = 1.0; }
                        if (crank == 0 && tid == 0) P.cond[(size_t)b * kMaxNodes + j] = reach * acc;
                        reach *= 1.0 - acc;
                    };
                    // the rejection branch: new residual, x leaves the draft distribution (nobody is left to see the last one's)
                    if ((kids & (kids - 1)) != 0) exhausted = !res.reject(red, C, v0, v1, x, ep, eq, qj, book);
                    else book();
                }
            }
        }
    }
    // (every CTA has received all that was sent to it: none leaves before a store into its shared memory has landed)
    if (nan_seen) set_status(P.status, RADAR_ERR_NUMERIC);
    if (bad_tree && tid == 0) set_status(P.status, RADAR_ERR_TREE);
}

// one warp per sequence: P_acc along the paths, P_stop, p_i.  Lane l owns rows l and l + 32 (and length l).
__global__ void __launch_bounds__(32) accept_length_dist_kernel(const AccLenParams P) {
    chain_wait();
    const radar_acclen_args& a = P.a;
    const int b = blockIdx.x, lane = threadIdx.x;
    const int M = min(max(a.n_nodes[b], 1), kMaxNodes);
    __shared__ double s_cond[kMaxNodes], s_stop[kMaxNodes];
    __shared__ int s_par[kMaxNodes], s_dep[kMaxNodes];
#pragma unroll
    for (int j = lane; j < kMaxNodes; j += 32) {
        const size_t o = (size_t)b * kMaxNodes + j;
        const int par = j > 0 && j < M ? a.tree_parent[o] : -1;
        s_par[j] = par < j ? par : -1;
        s_dep[j] = j < M ? a.tree_depth[o] : -1;
        s_cond[j] = s_par[j] >= 0 ? P.cond[o] : (j == 0 ? 1.0 : 0.0);       // the root is always "accepted"
    }
    __syncwarp();
#pragma unroll
    for (int c = lane; c < kMaxNodes; c += 32) {
        double p = s_cond[c];
        for (int q = s_par[c]; q > 0; q = s_par[q]) p *= s_cond[q];
        double acc = 0.0;                                                   // children in row order
        for (int j = c + 1; j < M; ++j) acc += s_par[j] == c ? s_cond[j] : 0.0;
        if (c >= M) p = 0.0;
        a.p_acc_node[(size_t)b * kMaxNodes + c] = p;
        s_stop[c] = p * (1.0 - acc);
    }
    __syncwarp();
    for (int i = lane; i <= a.t_max; i += 32) {
        double d = 0.0;
        for (int c = 0; c < M; ++c) d += s_dep[c] == i ? s_stop[c] : 0.0;
        a.dist[(size_t)b * (a.t_max + 1) + i] = d;
    }
}

// correctly rounded from 64-bit mantissas
ExpTable exp_table() {
    static const ExpTable t = [] {
        ExpTable x;
        for (int j = 0; j < 64; ++j) x.t[j] = (double)exp2l((long double)j / 64.0L);
        return x;
    }();
    return t;
}

}  // namespace
}  // namespace radar

using namespace radar;

// shared memory for the cached tiles of a slice, all of them or as many as fit
static size_t cache_smem(int V, int cs, size_t room) {
    const int slice = 4 * (((V + 3) / 4 + cs - 1) / cs);
    return std::min(room, (size_t)(slice + kTileTokens - 1) / kTileTokens * kTileBytes);
}

// launch configuration of the cluster kernels (attr: two attributes that outlive it)
static cudaLaunchConfig_t cluster_config(int ctas, int cs, size_t smem, cudaStream_t stream, cudaLaunchAttribute* attr) {
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3(kSThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cfg;
}

template <typename T, int kPerSm>
static cudaError_t launch_walk(radar_ctx* ctx, StochParams& sp, int cs, cudaStream_t stream) {
    constexpr size_t kRoom = cache_room(kPerSm, sizeof(WalkShared));
    const size_t smem = cache_smem(sp.a.V, cs, kRoom);
    sp.smem_tiles = (int)(smem / kTileBytes);
    cudaError_t e = radar_opt_in_smem(ctx, RADAR_SMEM_WALK + 2 * (sizeof(T) == 2) + kPerSm - 1, stochastic_walk_kernel<T, kPerSm>, kRoom);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = cluster_config(sp.a.B * cs, cs, smem, stream, attr);
    radar_launch_scope scope(ctx, RADAR_K_STOCH_WALK, stream);
    return cudaLaunchKernelEx(&cfg, stochastic_walk_kernel<T, kPerSm>, sp);
}

extern "C" size_t radar_accept_workspace_bytes(const radar_ctx* ctx, int B, int V, int mode) {
    if (!ctx || B <= 0 || V <= 0) return 0;
    if (mode == RADAR_GREEDY) return vocab_pass_workspace_bytes(ctx->sm_count, B * kMaxNodes, V);
    return align_up((size_t)B * cache_stride(V) * sizeof(double), 256) * 2;
}

extern "C" int radar_verify_accept(radar_ctx* ctx, const radar_accept_args* a, void* stream_) {
    if (!ctx || !a) return RADAR_ERR_INVALID_ARG;
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
    if (a->B <= 0 || a->V <= 0 || a->t_max < 1 || a->N < 1) return RADAR_ERR_INVALID_ARG;
    if (a->mode != RADAR_GREEDY && a->mode != RADAR_STOCHASTIC) return RADAR_ERR_INVALID_ARG;
    if (a->logits_dtype != RADAR_F32 && a->logits_dtype != RADAR_BF16) return RADAR_ERR_UNSUPPORTED;
    if (!a->target_logits || !a->tree_tok || !a->tree_parent || !a->n_nodes || !a->retrieve || !a->n_leaves ||
        !a->accept_len || !a->path_nodes || !a->path_tokens || !a->next_token || !a->best_retrieve_row ||
        !a->workspace)
        return RADAR_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(a->workspace) & 255) != 0) return RADAR_ERR_WORKSPACE;
    if (a->mode == RADAR_STOCHASTIC && radar_accept_workspace_bytes(ctx, a->B, a->V, a->mode) > a->workspace_bytes) return RADAR_ERR_WORKSPACE;

    if (a->mode == RADAR_GREEDY) {
        GreedyParams gp;
        gp.a = *a;
        VocabPassParams& vp = gp.vp;
        vp.logits = a->target_logits;
        vp.dtype = a->logits_dtype;
        vp.row_stride = a->V;
        vp.seq_stride = (int64_t)kMaxNodes * a->V;
        vp.n_seq = a->B;
        vp.F = kMaxNodes;
        vp.V = a->V;
        vp.n_chunks = vocab_pass_plan_chunks(ctx->sm_count, a->B * kMaxNodes, a->V, &vp.chunk);
        vp.seq_rows = a->n_nodes;
        vp.status = ctx->d_status;
        if (vocab_pass_partial_bytes(a->B * kMaxNodes, vp.n_chunks) > a->workspace_bytes) return RADAR_ERR_WORKSPACE;
        vocab_pass_carve(a->workspace, a->B * kMaxNodes, vp.n_chunks, &vp);
        RADAR_CUDA_CHECK(vocab_pass_launch(ctx, vp, stream));
        {
            radar_launch_scope scope(ctx, RADAR_K_GREEDY_WALK, stream);
            RADAR_CUDA_CHECK(launch_chained(greedy_walk_kernel, dim3(a->B), dim3(kGreedyThreads), 0, stream, gp));
        }
        RADAR_CUDA_CHECK(cudaGetLastError());
        return RADAR_OK;
    }
    if (!a->tree_draft_row || !a->draft_logits || !a->u_accept || !a->u_sample || a->R < 1) return RADAR_ERR_INVALID_ARG;
    if (!(a->temperature > 0.f)) return RADAR_ERR_INVALID_ARG;
    StochParams sp;
    sp.a = *a;
    sp.cache = reinterpret_cast<double*>(a->workspace);
    sp.status = ctx->d_status;
    sp.tab = exp_table();
    // Cluster size: as many CTAs per sequence as keep the whole batch resident at once, two to an SM, while a CTA's slice
    // of the vocabulary is worth an exchange between them.  One CTA per SM where that still leaves SMs over (clusters need
    // their SMs in one GPC, so not all SMs can be used that way).  us for one / two at clusters of eight: B = 4, V = 32000 21.2 /
    // 27.5; 8, 128256 45.6 / 57.4; 14, 128256 60.4 / 66.9; 16, 17000 25.0 / 25.4; 16, 50256 41.9 / 37.9; 16, 128256 80.4 / 77.9;
    // B = 32, V = 128256 157 (clusters of four, one) / 106.  (Off the rule: B = 24, V = 32000 38 with clusters of four, one per SM, 41 so.)
    int cs = 1;
    while (cs < kMaxCluster && (long long)a->B * cs * 2 <= 2 * ctx->sm_count && a->V >= cs * 2 * kMinSlice) cs *= 2;
    const bool one = 4ll * a->B * cs <= 3ll * ctx->sm_count;
    if (a->logits_dtype == RADAR_F32) RADAR_CUDA_CHECK((one ? launch_walk<float, 1>(ctx, sp, cs, stream) : launch_walk<float, 2>(ctx, sp, cs, stream)));
    else RADAR_CUDA_CHECK((one ? launch_walk<__nv_bfloat16, 1>(ctx, sp, cs, stream) : launch_walk<__nv_bfloat16, 2>(ctx, sp, cs, stream)));
    RADAR_CUDA_CHECK(cudaGetLastError());
    return RADAR_OK;
}

// CTAs per tree row: a slice of at least kAccMinSlice tokens each
static int acclen_cluster(int V) {
    int cs = 1;
    while (cs < kMaxCluster && V >= cs * 2 * kAccMinSlice) cs *= 2;
    return cs;
}
static int acclen_max_clusters(const radar_ctx* ctx, int B, int cs) { return std::min(B * kMaxNodes, std::max(1, 2 * ctx->sm_count / cs)); }

extern "C" size_t radar_acclen_workspace_bytes(const radar_ctx* ctx, int B, int V) {
    if (!ctx || B <= 0 || V <= 0) return 0;
    return 2 * align_up((size_t)acclen_max_clusters(ctx, B, acclen_cluster(V)) * cache_stride(V) * sizeof(double), 256) +
           align_up((size_t)B * kMaxNodes * sizeof(double), 256);
}

template <typename T, int kPerSm>
static cudaError_t launch_acclen(radar_ctx* ctx, AccLenParams& P, int cs, int max_clusters, cudaStream_t stream) {
    constexpr int kind = 2 * (sizeof(T) == 2) + kPerSm - 1;
    constexpr size_t kRoom = cache_room(kPerSm, sizeof(AccLenShared));
    cudaError_t e = radar_opt_in_smem(ctx, RADAR_SMEM_ACCLEN + kind, accept_length_nodes_kernel<T, kPerSm>, kRoom);
    if (e != cudaSuccess) return e;
    // As many clusters as are resident at once: the rows are dealt out over them in advance.  How many that is, is a
    // property of the kernel and the device, asked for once per cluster size (with the most shared memory it may get).
    int log_cs = 0;
    while ((1 << log_cs) < cs) ++log_cs;
    cudaLaunchAttribute attr[2];
    int& resident = ctx->acclen_clusters[kind][log_cs];
    if (resident == 0) {
        cudaLaunchConfig_t q = cluster_config(2 * ctx->sm_count / cs * cs, cs, kRoom, stream, attr);
        q.numAttrs = 1;
        int n = 0;
        e = cudaOccupancyMaxActiveClusters(&n, accept_length_nodes_kernel<T, kPerSm>, &q);
        if (e != cudaSuccess) return e;
        resident = n > 0 ? n : 1;
    }
    const size_t smem = cache_smem(P.a.V, cs, kRoom);
    P.smem_tiles = (int)(smem / kTileBytes);
    const cudaLaunchConfig_t cfg = cluster_config(std::min(max_clusters, resident) * cs, cs, smem, stream, attr);
    radar_launch_scope scope(ctx, RADAR_K_ACCLEN_NODES, stream);
    return cudaLaunchKernelEx(&cfg, accept_length_nodes_kernel<T, kPerSm>, P);
}

extern "C" int radar_accept_length_distribution(radar_ctx* ctx, const radar_acclen_args* a, void* stream_) {
    if (!ctx || !a) return RADAR_ERR_INVALID_ARG;
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
    if (a->B <= 0 || a->V <= 0 || a->t_max < 1 || a->R < 1 || !(a->temperature > 0.f)) return RADAR_ERR_INVALID_ARG;
    if (a->t_max >= 64) return RADAR_ERR_UNSUPPORTED;
    if (a->logits_dtype != RADAR_F32 && a->logits_dtype != RADAR_BF16) return RADAR_ERR_UNSUPPORTED;
    if (!a->target_logits || !a->draft_logits || !a->tree_tok || !a->tree_parent || !a->tree_depth || !a->tree_draft_row ||
        !a->n_nodes || !a->dist || !a->p_acc_node || !a->workspace)
        return RADAR_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(a->workspace) & 255) != 0) return RADAR_ERR_WORKSPACE;
    if (radar_acclen_workspace_bytes(ctx, a->B, a->V) > a->workspace_bytes) return RADAR_ERR_WORKSPACE;
    const int cs = acclen_cluster(a->V), max_clusters = acclen_max_clusters(ctx, a->B, cs);
    AccLenParams P;
    P.a = *a;
    char* w = reinterpret_cast<char*>(a->workspace);
    const size_t cache = align_up((size_t)max_clusters * cache_stride(a->V) * sizeof(double), 256);
    P.cache = reinterpret_cast<double*>(w);
    P.cond = reinterpret_cast<double*>(w + 2 * cache);
    P.status = ctx->d_status;
    P.tab = exp_table();
    // One CTA per SM while the rows (about twenty with children to a tree) are few waves, two when their passes are what
    // takes the time.  us for one / two, by trees times CTAs a row: 8 (1 tree, V = 128256) 34 / 41; 16 (4, 32000) 24 / 31, (8, 16000)
    // 24 / 31, (2, 128256) 35 / 45; 20 (5, 32000) 30 / 31; 24 (6, 32000) 35 / 32, (3, 70000) 37 / 33, (3, 128256) 55 / 48; 32 (4, 70000)
    // 42 / 35; 64 (16, 32000) 76 / 61, (8, 128256) 126 / 101.  (Short vocabularies cross later: 16 trees, V = 16000 44 / 57.)
    const bool one = a->B * cs <= 16;
    if (a->logits_dtype == RADAR_F32) RADAR_CUDA_CHECK((one ? launch_acclen<float, 1>(ctx, P, cs, max_clusters, stream) : launch_acclen<float, 2>(ctx, P, cs, max_clusters, stream)));
    else RADAR_CUDA_CHECK((one ? launch_acclen<__nv_bfloat16, 1>(ctx, P, cs, max_clusters, stream) : launch_acclen<__nv_bfloat16, 2>(ctx, P, cs, max_clusters, stream)));
    RADAR_CUDA_CHECK(cudaGetLastError());
    {
        radar_launch_scope scope(ctx, RADAR_K_ACCLEN_DIST, stream);
        RADAR_CUDA_CHECK(launch_chained(accept_length_dist_kernel, dim3(a->B), dim3(32), 0, stream, P));
    }
    RADAR_CUDA_CHECK(cudaGetLastError());
    return RADAR_OK;
}

// ------------------------------------------------------------------------------------------
// Greedy acceptance for callers that cannot hand over a workspace.
//
// Who needs this: code that runs after its host application has frozen device memory.  A serving
// engine typically gives every free byte of the GPU to its own KV-cache pool at start-up; from
// then on a cudaMalloc either fails or has to be carved out of that pool by hand, and cudaMalloc /
// cudaFree also synchronise the whole device, which a decode loop cannot afford per step.  Such a
// caller has inputs and outputs (they are part of its own pre-planned buffers) but no spare
// scratch to lend.  For it the scratch lives in this library's image: one fixed array per GPU.
// The driver loads a library's device image lazily and allocates the array (and the kernels'
// code) when it does, so radar_create makes that happen for its device - it resolves the array's
// address and loads the two kernels of this path - and the array then stays until the process
// exits.  Create the context BEFORE the host freezes device memory; the calls themselves then
// allocate nothing.
//
// Consequences of that choice, all of which the caller must know:
//   * the array has a fixed size (RADAR_NOALLOC_SCRATCH_BYTES = 1 MiB); a batch / vocabulary whose
//     chunk records do not fit is refused with RADAR_ERR_UNSUPPORTED before anything is launched;
//   * all calls on a device share it.  Two calls whose kernels may overlap on the GPU (different
//     streams, or graphs replayed concurrently) race on it and give undefined results; calls on
//     one stream are safe;
//   * it keeps whatever the previous call left.  Nothing in this path needs zeroed scratch: every
//     record that is read has been written earlier in the same call, so no clearing is done;
//   * in host code the array's name is only a handle.  radar_create looks up the real device
//     address with cudaGetSymbolAddress (with its device current) and caches it per device; a call
//     that finds no cached address (a context made by other means) does the look-up itself, so
//     make the first call outside any stream capture.
// ------------------------------------------------------------------------------------------
#include <mutex>

namespace {
constexpr size_t kNoAllocScratchBytes = 1u << 20;
constexpr int kNoAllocMaxDevices = 64;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];
std::mutex g_noalloc_mutex;
void* g_noalloc_addr[kNoAllocMaxDevices] = {nullptr};      // per device: device address of g_noalloc_scratch
}  // namespace

namespace radar {
int noalloc_prepare_device(int device) {
    if (device < 0 || device >= kNoAllocMaxDevices) return RADAR_OK;       // beyond the table: resolved per call
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (g_noalloc_addr[device] == nullptr) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || p == nullptr) return RADAR_ERR_CUDA;
        g_noalloc_addr[device] = p;
    }
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, greedy_walk_kernel) != cudaSuccess || vocab_pass_preload_argbest() != cudaSuccess)
        return RADAR_ERR_CUDA;
    return RADAR_OK;
}
}  // namespace radar

extern "C" size_t radar_noalloc_scratch_bytes(void) { return kNoAllocScratchBytes; }

extern "C" int radar_verify_accept_greedy_noalloc(radar_ctx* ctx, const radar_accept_args* a, void* stream_) {
    if (!ctx || !a) return RADAR_ERR_INVALID_ARG;
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
    if (a->B <= 0 || a->V <= 0 || a->t_max < 1 || a->N < 1) return RADAR_ERR_INVALID_ARG;
    if (a->mode != RADAR_GREEDY) return RADAR_ERR_UNSUPPORTED;        // the stochastic walk needs 16 * B * V bytes
    if (a->logits_dtype != RADAR_F32 && a->logits_dtype != RADAR_BF16) return RADAR_ERR_UNSUPPORTED;
    // size first: a request that cannot fit is refused whatever else it carries
    int chunk = 0;
    const int n_chunks = vocab_pass_plan_chunks(ctx->sm_count, a->B * kMaxNodes, a->V, &chunk);
    if ((long long)a->B * kMaxNodes > 0x7fffffff / (n_chunks > 0 ? n_chunks : 1)) return RADAR_ERR_UNSUPPORTED;
    if (2 * vocab_pass_partial_bytes(a->B * kMaxNodes, n_chunks) > kNoAllocScratchBytes) return RADAR_ERR_UNSUPPORTED;     // 16 bytes a record: the documented limit
    if (!a->target_logits || !a->tree_tok || !a->tree_parent || !a->n_nodes || !a->retrieve || !a->n_leaves ||
        !a->accept_len || !a->path_nodes || !a->path_tokens || !a->next_token || !a->best_retrieve_row)
        return RADAR_ERR_INVALID_ARG;

    int cur = -1;
    RADAR_CUDA_CHECK(cudaGetDevice(&cur));
    if (cur != ctx->device || cur < 0 || cur >= kNoAllocMaxDevices) return RADAR_ERR_INVALID_ARG;
    void* scratch = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_noalloc_mutex);
        if (g_noalloc_addr[cur] == nullptr) {
            void* p = nullptr;
            if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || p == nullptr) return RADAR_ERR_CUDA;
            g_noalloc_addr[cur] = p;
        }
        scratch = g_noalloc_addr[cur];
    }

    GreedyParams gp;
    gp.a = *a;
    gp.a.workspace = scratch;
    gp.a.workspace_bytes = kNoAllocScratchBytes;
    VocabPassParams& vp = gp.vp;
    vp.logits = a->target_logits;
    vp.dtype = a->logits_dtype;
    vp.row_stride = a->V;
    vp.seq_stride = (int64_t)kMaxNodes * a->V;
    vp.n_seq = a->B;
    vp.F = kMaxNodes;
    vp.V = a->V;
    vp.n_chunks = n_chunks;
    vp.chunk = chunk;
    vp.seq_rows = a->n_nodes;
    vp.status = ctx->d_status;
    vocab_pass_carve(scratch, a->B * kMaxNodes, n_chunks, &vp);
    RADAR_CUDA_CHECK(vocab_pass_launch(ctx, vp, stream));
    {
        radar_launch_scope scope(ctx, RADAR_K_GREEDY_WALK, stream);
        RADAR_CUDA_CHECK(launch_chained(greedy_walk_kernel, dim3(a->B), dim3(kGreedyThreads), 0, stream, gp));
    }
    RADAR_CUDA_CHECK(cudaGetLastError());
    return RADAR_OK;
}
