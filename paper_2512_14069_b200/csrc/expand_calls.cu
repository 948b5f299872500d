// radar_expand_calls: all draft calls of a step on draft logits that are there already.
//
//   vocab_pass_kernel      one vocabulary pass over the rows of all calls;
//   row_merge_kernel       chunk records -> the row's top-k tokens and log-probabilities (fp64), a block of two warps per row: it
//                          is a chain of dependent steps, so one warp ranks the records beside the other's fp64 normaliser
//                          (against one warp for both, whole steps: B = 4, V = 32000 137.3 -> 135.0 us, bf16 B = 6 104.5 -> 103.2);
//   expand_calls_kernel    one cluster per sequence goes through the calls: candidates, pool, frontier, prediction model.
//
// Call by call, a step is a chain of a dozen launches whose blocks each reload the gate's weights, merge a row's records and
// hand the state on through global memory: 7 to 12 us a call, whatever the size.  Here the passes and merges, which depend on
// nothing the calls decide, run once over all rows, and the calls themselves are a loop whose weights and state stay in
// shared memory, 2 us a call (B = 1, V = 128256, 8 calls: 77 us call by call, 39 together).  What it costs: rows of calls that
// a sequence never makes are read too, so long passes go call by call (calls_logits).  It takes draft logits that exist before
// the first call (recorded ones, or a draft model that does not look at the frontier); where the draft model runs between the
// calls, radar_expand_step is the form.
#include <algorithm>
#include <cstdint>

#include "select.cuh"

namespace radar {
namespace {

constexpr size_t kMergeStageLimit = 40 * 1024;
constexpr int32_t kNanRow = INT32_MIN;               // set in the tokens of a row with a NaN logit

__global__ void __launch_bounds__(64) row_merge_kernel(const VocabPassParams vp, int staged, int32_t* tok, double* logp) {
    chain_wait();
    extern __shared__ __align__(16) unsigned char merge_smem[];
    __shared__ double s_lse;
    __shared__ int32_t s_mark;
    __shared__ float s_v[RADAR_MAX_K];
    __shared__ int s_t[RADAR_MAX_K];
    const int k = vp.k, tid = threadIdx.x;
    const size_t row = blockIdx.x;
    if (tid < 32) {
        const int stride = staged ? (vp.n_chunks * k + 3) & ~3 : 0;
        float* pv_s = reinterpret_cast<float*>(merge_smem + (size_t)kSurvCap * 8);
        merge_row(vp, row, staged != 0, pv_s, reinterpret_cast<int*>(pv_s + stride), reinterpret_cast<unsigned long long*>(merge_smem), [] {},
                  [&](int rank, float v, int t) { s_v[rank] = v; s_t[rank] = t; });
    } else {
        bool nan = false;                            // reported by the call that uses the row: nobody may ever
        for (int c = tid - 32; c < vp.n_chunks; c += 32) nan |= isnan(vp.part_m[row * vp.n_chunks + c]);
        const double lse = row_normaliser(vp, row);
        const bool any = __any_sync(kFull, nan);
        if (tid == 32) { s_lse = lse; s_mark = any ? kNanRow : 0; }
    }
    __syncthreads();
    if (tid < k) {
        tok[row * k + tid] = s_t[tid] | s_mark;
        logp[row * k + tid] = (double)s_v[tid] - s_lse;
    }
}

struct CallsParams {
    radar_expand_args a;                             // the arguments of call 1
    int32_t* topk_tok_next;                          // [t_max-1][B][k][k] of calls 2..
    float* topk_logp_next;
    const int32_t* row_tok;                          // [B][R][k] merged rows
    const double* row_logp;
    int* status;
};

// bounded wait for a phase of a barrier that other blocks of the cluster complete
__device__ __forceinline__ bool cluster_wait(const uint64_t* bar, uint32_t parity) {
    bool ok = false;
    for (uint32_t it = 0; it < (1u << 22) && !(ok = mbar_try_wait_cluster(bar, parity)); ++it) {}
    return ok;
}
__device__ __forceinline__ uint32_t cluster_addr(const void* p, uint32_t rank) {
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_addr(p)), "r"(rank));
    return a;
}
// a word into another block's shared memory, counted by a barrier there: the message needs no release of what came before it
__device__ __forceinline__ void send_f32(uint32_t addr, uint32_t bar, float v) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(addr), "r"(__float_as_uint(v)), "r"(bar) : "memory");
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

// Block 0 of a cluster goes through the calls of its sequence; with the recurrent policy the other blocks hold W_hh (256 KB) in
// their registers: they receive h as soon as the cell has produced it and deliver W_hh h + biases while block 0 finishes
// the call and ranks the next one's candidates.  What bounds a call is block 0's chain of steps, each a few dozen dependent
// instructions and a block barrier.  So weights sit in registers or conflict-free in shared memory, candidates are
// compared as integers, messages between the blocks are counted stores (a release by each sender, 2500 cycles with the
// calls' global stores in front of it, was the longest step), and the stores of a call's results are issued by warps that
// have nothing else to do.  The arithmetic and its order are those of expand_select_gate_kernel.
template <bool kRecurrent>
__global__ void __launch_bounds__(kSelThreads, 1) expand_calls_kernel(const CallsParams P) {
    const radar_expand_args& a = P.a;
    constexpr int H = kHidden, kBlocks = kRecurrent ? kSelCluster : 1, kHelp = kBlocks - 1;
    constexpr int kRows = kRecurrent ? (4 * H + kHelp - 1) / kHelp : 1;          // rows of W_hh per helper block
    constexpr uint32_t kStateBytes = (H + 1) * 4, kProductBytes = 4 * H * 4;     // the two messages: h and a stop flag; W_hh h + biases
    const int b = blockIdx.x / kBlocks, B = a.B, k = a.k, t_max = a.t_max;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    extern __shared__ __align__(16) unsigned char calls_smem[];
    __shared__ float s_pre[4 * H];                     // block 0: W_hh h + biases of the call
    __shared__ __align__(16) float s_h[H + 4];         // helpers: the h they were sent; [H]: not 0 if it is the last message
    __shared__ __align__(8) uint64_t s_bar;            // completes with the message the block expects next
    uint32_t crank = 0;
    if (kRecurrent) asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(crank));

    // The predecessor is row_merge_kernel, whose blocks wait for everything before them: only the merged rows need the wait.
    if (crank != 0) {
        // ---- helper block: rows [r0, r1) of W_hh h + biases, into block 0's s_pre ----
        const int r0 = ((int)crank - 1) * kRows, r1 = min(4 * H, r0 + kRows);
        constexpr int kPer = (kRows + kSelWarps - 1) / kSelWarps;                // rows per warp, four weights of each per lane
        static_assert(!kRecurrent || (kPer <= 8 && kRows >= kSelWarps), "every warp has rows, at most eight");
        float4 w[kPer];
#pragma unroll
        for (int i = 0; i < kPer; ++i) w[i] = *reinterpret_cast<const float4*>(a.w_hh + (size_t)min(r0 + warp + i * kSelWarps, r1 - 1) * H + 4 * lane);
        const int my_row = r0 + warp + (lane >> 2) * kSelWarps;                  // the row whose sum ends up in this lane
        const bool sender = (lane & 3) == 0 && (lane >> 2) < kPer && my_row < r1;
        const float bi = sender ? a.b_ih[my_row] : 0.f, bh = sender ? a.b_hh[my_row] : 0.f;
        if (tid == 0) init_message_barrier(&s_bar, kStateBytes);
        const uint32_t to = cluster_addr(&s_pre[min(my_row, 4 * H - 1)], 0), to_bar = cluster_addr(&s_bar, 0);
        cluster_barrier();                             // every block has started and its barrier word is initialised
        chain_sync();
        chain_trigger();
        for (int t = 2; t < t_max; ++t) {              // W_hh h of call t - 1, for call t's gate
            if (!cluster_wait(&s_bar, (uint32_t)(t & 1))) { set_status(P.status, RADAR_ERR_TIMEOUT); break; }
            const float4 h4 = *reinterpret_cast<const float4*>(s_h + lane * 4);
            if (*(volatile float*)&s_h[H] != 0.f) break;
            if (tid == 0) expect_bytes(&s_bar, kStateBytes);
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
            const float sum = transposed_sum<8>(acc);
            if (sender) send_f32(to, to_bar, sum + bi + bh);
        }
        cluster_barrier();
        return;
    }

    __shared__ unsigned long long s_key[kMaxF * RADAR_MAX_K];         // the next call's surviving candidates: order keys,
    __shared__ float s_score[kMaxF * RADAR_MAX_K];     // scores,
    __shared__ short s_cand[kMaxF * RADAR_MAX_K];      // flat indices (f, j)
    __shared__ short s_rank[kMaxF * RADAR_MAX_K];      // rank of every candidate (k: not among the k best)
    __shared__ float s_head[RADAR_MAX_K];              // best candidate of every parent
    __shared__ float s_x[2][RADAR_MAX_K];              // gate input of a call (t & 1)
    __shared__ float s_fscore[RADAR_MAX_K];            // the frontier: next call's parents
    __shared__ int s_fidx[RADAR_MAX_K];
    __shared__ float s_hn[H], s_hid[2][H], s_c[H], s_b1[H], s_w2[2 * H], s_b2[2];
    __shared__ int s_cont, s_count;
    float* s_w = reinterpret_cast<float*>(calls_smem);                // W_ih [4H][k | 1]; without recurrence w1 [H][k | 1]
    const int ws = k | 1;                                             // odd: a column of rows meets all banks
    // head: a warp's four rows of w1, in registers
    static_assert(kHidden == 4 * kSelWarps, "four rows of the hidden layer per warp");
    float w1r[4][4], w1x[4];
    if (t_max > 1) {
        for (int e = tid; e < (kRecurrent ? 4 * H : H) * k; e += kSelThreads) cp_async4(s_w + e / k * ws + e % k, (kRecurrent ? a.w_ih : a.w1) + e);
        if (kRecurrent) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float* w = a.w1 + (size_t)(warp + i * kSelWarps) * (H + k);
#pragma unroll
                for (int c = 0; c < 4; ++c) w1r[i][c] = w[lane + 32 * c];
                w1x[i] = lane < k ? w[H + lane] : 0.f;
            }
            if (tid < 4 * H) s_pre[tid] = a.b_ih[tid] + a.b_hh[tid];  // call 1: h is zero
        }
        if (tid < H) { s_b1[tid] = a.b1[tid]; s_c[tid] = 0.f; }
        if (tid < 2 * H) s_w2[tid] = a.w2[tid];
        if (tid < 2) s_b2[tid] = a.b2[tid];
    }
    const int forced = a.force_calls != nullptr ? a.force_calls[b] : -1;
    const float root_score = a.parent_score[b];
    const int root_idx = a.parent_pool_idx[b];
    uint32_t to[kHelp > 0 ? kHelp : 1], to_bar[kHelp > 0 ? kHelp : 1];
    uint32_t to_flag = 0;
    if (kRecurrent) {
        if (tid == 0) init_message_barrier(&s_bar, kProductBytes);
#pragma unroll
        for (int r = 0; r < kHelp; ++r) { to[r] = cluster_addr(&s_h[tid & (H - 1)], r + 1); to_bar[r] = cluster_addr(&s_bar, r + 1); }
        if (tid < kHelp) to_flag = cluster_addr(&s_h[H], tid + 1);
        cluster_barrier();
    }
    chain_sync();
    chain_trigger();
    const size_t rows0 = (size_t)b * (1 + (t_max - 1) * k);           // the sequence's first row
    // A call is three steps between block barriers:
    //   1  gate: W_ih x and the activations | the logits of the call before, its decision | candidates of the next call
    //   2  gate: the cell, h to the helpers | results of this call, the next call's candidates that can matter
    //   3  gate: the head's hidden layer    | the next call's frontier | the helpers' product
    // The selection of call t + 1 needs nothing of the gate's decision at call t and the input product of call t + 1 is cheap,
    // so both run ahead of the decision; what they leave in shared memory is dropped if the sequence stops.  The last
    // k * k threads of the block handle the candidates (the first ones work on the gate): candidate e, of parent f.
    const int e = tid - (kSelThreads - k * k), f = e >= 0 ? e / k : 0;
    double lp = 0.0;                                                  // log-probability and token of the next candidate
    int tok = 0, my_tok = 0, my_parent = 0;                           // (my_*: of the candidate whose results are stored next)
    float my_score = 0.f, my_lp = 0.f;
    auto fetch = [&](int t) {
        if (e >= 0 && t <= t_max && (t > 1 || e < k)) {
            const size_t o = (t == 1 ? rows0 : rows0 + 1 + (size_t)(t - 2) * k) * k + e;
            lp = P.row_logp[o];
            tok = P.row_tok[o];
        }
    };
    auto frontier = [&](int rank, float score, int cand, int base, int buf) {
        s_fscore[rank] = score;
        s_fidx[rank] = base + cand;
        s_x[buf][rank] = expf(score);                                 // confidence score in [0,1]
        s_rank[cand] = (short)rank;
    };
    fetch(1);
    if (e >= 0 && e < k) {                                            // call 1: one row, already in order
        my_tok = tok;
        my_lp = (float)lp;
        my_score = (float)((double)root_score + lp);
        my_parent = root_idx;
        frontier(e, my_score, e, 0, 1);
    }
    fetch(2);
    cp_async_wait_all();
    __syncthreads();

    int base = 0, sent = 0, t = 1;
    for (;; ++t) {
        const int n_cand = t == 1 ? k : k * k;
        const bool run_gate = t < t_max;
        // ---- 1 ----
        if (run_gate && kRecurrent && tid < 4 * H) {
            float acc = s_pre[tid];
            const float* w = s_w + tid * ws;
            const float* x = s_x[t & 1];
#pragma unroll 4
            for (int j = 0; j < k; ++j) acc = fmaf(w[j], x[j], acc);
            s_pre[tid] = warp / (H / 32) == 2 ? tanhf(acc) : sigmoidf_(acc);
        }
        if (run_gate && !kRecurrent && tid < H) {
            float acc = s_b1[tid];
            const float* w = s_w + tid * ws;
            const float* x = s_x[t & 1];
            for (int j = 0; j < k; ++j) acc = fmaf(w[j], x[j], acc);
            s_hid[t & 1][tid] = fmaxf(acc, 0.f);
        }
        if (t > 1 && warp == 4 * H / 32) {
            const float* hid = s_hid[(t - 1) & 1];
            float y0 = 0.f, y1 = 0.f;
#pragma unroll
            for (int c = 0; c < H; c += 32) {
                y0 = fmaf(s_w2[c + lane], hid[c + lane], y0);
                y1 = fmaf(s_w2[H + c + lane], hid[c + lane], y1);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                y0 += __shfl_xor_sync(kFull, y0, o);
                y1 += __shfl_xor_sync(kFull, y1, o);
            }
            y0 += s_b2[0];
            y1 += s_b2[1];
            const bool c = forced >= 0 ? t - 1 < forced : y1 > y0;
            if (lane == 0) s_cont = c;
            if (lane < 2) a.gate_logits[((size_t)(t - 2) * B + b) * 2 + lane] = lane == 0 ? y0 : y1;
            if (lane == 0) {
                a.cont[(size_t)(t - 2) * B + b] = c ? 1 : 0;
                a.active[b] = c ? 1 : 0;
            }
        }
        unsigned long long key = 0;
        float next_score = 0.f;
        int next_parent = 0;
        if (run_gate && e >= 0) {
            const double cand = (double)s_fscore[f] + lp;
            key = order_key64(cand);
            next_score = (float)cand;
            next_parent = s_fidx[f];
            if (e == f * k) s_head[f] = next_score;
        }
        if (tid == 0) s_count = 0;
        __syncthreads();
        if (t > 1 && s_cont == 0) { --t; break; }                     // t: the last call the sequence made
        if (base + n_cand > a.pool_capacity) {                        // never write past the pool
            if (tid == 0) { set_status(P.status, RADAR_ERR_INVALID_ARG); a.cont[(size_t)(t - 1) * B + b] = 0; a.active[b] = 0; }
            break;
        }
        // ---- 2 ----
        if (run_gate && kRecurrent && tid < H) {
            const float cn = s_pre[H + tid] * s_c[tid] + s_pre[tid] * s_pre[2 * H + tid];
            const float hn = s_pre[3 * H + tid] * tanhf(cn);
            s_c[tid] = cn;
            s_hn[tid] = hn;
            if (t + 1 < t_max) {
#pragma unroll
                for (int r = 0; r < kHelp; ++r) send_f32(to[r], to_bar[r], hn);
                if (tid < kHelp) send_f32(to_flag, cluster_addr(&s_bar, tid + 1), 0.f);
            }
        }
        if (t + 1 < t_max) sent = t;
        if (e >= 0 && e < n_cand) {                                   // results of this call
            const size_t o = (size_t)b * a.pool_capacity + base + e;
            const int rank = s_rank[e];
            if (my_tok < 0) set_status(P.status, RADAR_ERR_NUMERIC);
            const int tk = my_tok & ~kNanRow;
            a.pool_tok[o] = tk;
            a.pool_parent[o] = my_parent;
            a.pool_score[o] = my_score;
            a.pool_depth[o] = t;
            a.pool_draft_row[o] = rank < k ? 1 + (t - 1) * k + rank : -1;
            const size_t q = t == 1 ? (size_t)b * k + e : ((size_t)(t - 2) * B + b) * k * k + e;
            (t == 1 ? a.topk_tok : P.topk_tok_next)[q] = tk;
            (t == 1 ? a.topk_logp : P.topk_logp_next)[q] = my_lp;
            if (rank < k) {
                const size_t u = ((size_t)(t - 1) * B + b) * k + rank;
                a.frontier_tok[u] = tk;
                a.frontier_score[u] = my_score;
                a.frontier_pool_idx[u] = base + e;
                a.frontier_src_row[u] = t == 1 ? 0 : f;
            }
        }
        base += n_cand;
        if (tid == kSelThreads - 1) a.pool_len[b] = base;
        if (!run_gate) {
            if (tid < 2) a.gate_logits[((size_t)(t - 1) * B + b) * 2 + tid] = 0.f;
            if (tid == 0) { a.cont[(size_t)(t - 1) * B + b] = 0; a.active[b] = 0; }
            break;
        }
        if (warp >= (kSelThreads - k * k) / 32) {
            // the worst of the parents' best candidates is a lower bound of the k-th best: what reaches it (some 2 k) is listed
            const float low = warp_min_value(lane < k ? s_head[lane] : CUDART_INF_F);
            const bool keep = e >= 0 && !(next_score < low);
            const unsigned m = __ballot_sync(kFull, keep);
            int at = 0;
            if (lane == 0) at = atomicAdd(&s_count, __popc(m));
            at = __shfl_sync(kFull, at, 0) + __popc(m & ((1u << lane) - 1u));
            if (keep) {
                s_key[at] = key;
                s_score[at] = next_score;
                s_cand[at] = (short)e;
            }
            if (e >= 0) {
                s_rank[e] = (short)k;                                 // (until it is found among the k best)
                my_tok = tok;
                my_lp = (float)lp;
                my_score = next_score;
                my_parent = next_parent;
                fetch(t + 2);
            }
        }
        __syncthreads();
        // ---- 3 ----
        if (kRecurrent) {
            const float hv[4] = {s_hn[lane], s_hn[lane + 32], s_hn[lane + 64], s_hn[lane + 96]};
            const float xv = lane < k ? s_x[t & 1][lane] : 0.f;
            float acc[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float v = w1r[i][0] * hv[0];
                v = fmaf(w1r[i][1], hv[1], v);
                v = fmaf(w1r[i][2], hv[2], v);
                v = fmaf(w1r[i][3], hv[3], v);
                if (lane < k) v = fmaf(w1x[i], xv, v);
                acc[i] = v;
            }
            const float sum = transposed_sum<4>(acc);
            const int r = warp + (lane >> 3) * kSelWarps;
            if ((lane & 7) == 0) s_hid[t & 1][r] = fmaxf(sum + s_b1[r], 0.f);
        }
        {
            // the k best survivors (score desc, flat index asc): sixteen threads share a rank count
            const int n = s_count, part = tid & 15;
            for (int c0 = 0; c0 + warp * 2 < n; c0 += kSelThreads / 16) {
                const int c = min(c0 + (tid >> 4), n - 1);
                const unsigned long long mine = s_key[c];
                const int idx = s_cand[c];
                int rank = 0;
#pragma unroll 2
                for (int j = part; j < n; j += 16) {
                    const unsigned long long kj = s_key[j];
                    const int ij = s_cand[j];
                    rank += (int)(kj > mine) | ((int)(kj == mine) & (int)(ij < idx));
                }
#pragma unroll
                for (int o = 8; o > 0; o >>= 1) rank += __shfl_xor_sync(kFull, rank, o);
                if (part == 0 && rank < k && c0 + (tid >> 4) < n) frontier(rank, s_score[c], idx, base, (t + 1) & 1);
            }
        }
        if (kRecurrent) {
            if (tid >= kSelThreads - H) {
                const int c = tid - (kSelThreads - H);
                a.c[(size_t)b * H + c] = s_c[c];
                a.h[(size_t)b * H + c] = s_hn[c];
            }
            // one thread waits for the helpers' product of the next call, the barrier publishes it
            if (t + 1 < t_max && tid == kSelThreads - 1) {
                if (!cluster_wait(&s_bar, (uint32_t)((t + 1) & 1))) set_status(P.status, RADAR_ERR_TIMEOUT);
                expect_bytes(&s_bar, kProductBytes);
            }
        }
        __syncthreads();
    }
    for (int u = t + 1 + tid; u <= t_max; u += kSelThreads) a.cont[(size_t)(u - 1) * B + b] = 0;     // calls the sequence does not make
    if (kRecurrent) {
        if (tid < H) {
            // The product of the last h has been waited for, so that nothing is on its way into this block and every helper warp
            // is past its wait (a barrier may not run two phases ahead of a waiter).
            if (sent < t_max - 2) {                                   // helpers that still expect an h
#pragma unroll
                for (int r = 0; r < kHelp; ++r) send_f32(to[r], to_bar[r], 0.f);
                if (tid < kHelp) send_f32(to_flag, cluster_addr(&s_bar, tid + 1), 1.f);
            }
        }
        cluster_barrier();                                            // the helpers have received their last message
    }
}

struct CallsPlan {
    int R, rows, n_chunks, chunk;
    size_t part_bytes, merged_bytes;
};
CallsPlan plan_calls(const radar_ctx* ctx, int B, int V, int k, int t_max) {
    CallsPlan p;
    p.R = 1 + (t_max - 1) * k;
    p.rows = B * p.R;
    p.n_chunks = vocab_pass_plan_chunks(ctx->sm_count, p.rows, V, &p.chunk);
    p.part_bytes = align_up(vocab_pass_partial_bytes(p.rows, p.n_chunks, k), 256);
    p.merged_bytes = align_up((size_t)p.rows * k * sizeof(double), 256) + align_up((size_t)p.rows * k * sizeof(int32_t), 256);
    return p;
}

// The line: calls whose passes are short (B k V logits at most), where each also costs a cluster of blocks when it is made one by
// one, whether a sequence is still active or not.  Together, the rows of all calls are read, one by one those of a call more
// than is made.  Expansion in us, together / one by one, fp32, where every sequence makes 1, 2, 3 and all calls:
//   1.2M logits  V = 128256, B = 1, k = 10  t_max  4: 21 / 21, 23 / 27, 25 / 33, 26 / 39     8: 25 / 35, 27 / 41, 30 / 45, 39 / 73
//   2.4M         V = 32000, B = 8, k = 10   t_max  4: 23 / 23, 25 / 27, 28 / 35, 29 / 39    16: 49 / 66, 53 / 72, 55 / 76, 85 / 150
//   3.7M         V = 128256, B = 3, k = 10  t_max  3: 25 / 19, 27 / 27, 27 / 31              8: 41 / 37, 45 / 42, -, 57 / 82
//   3.9M         V = 128256, B = 8, k = 4   t_max  4: 25 / 23, 28 / 27, 29 / 35, 29 / 39    16: 63 / 68, 66 / 72, 68 / 78, 94 / 154
//   4.9M         V = 128256, B = 4, k = 10  t_max  4: 31 / 21, 33 / 27, 35 / 36, 35 / 41     8: 49 / 27, 51 / 35, 53 / 43, 64 / 89
// Up to the line together is the faster form from two calls on (but for 3 us at 3.7M), and at one call at most 8 us the
// slower one; above it, one by one drops the clusters, a call that is not made costs 2 us, and it takes five made calls out of
// eight for the rows to pay.  From k = 16 on, where a call by itself merges and ranks more than twice the candidates, three do
// (t_max = 8; 4.6M logits, V = 152000, k = 16, B = 2: 50 / 31, 53 / 43, 55 / 55, 68 / 123; k = 32, B = 1: 80 / 47, 85 / 150, 91 / 252,
// 111 / 767), and the line lies a little higher.
inline long long calls_logits(int k) { return k < 16 ? kShortPassLogits : 5LL << 20; }

}  // namespace
}  // namespace radar

using namespace radar;

static bool calls_together(const radar_ctx* ctx, int B, int V, int k, int t_max) {
    return B > 0 && k > 0 && t_max > 0 && k <= RADAR_MAX_K && V >= k && (long long)B * k * V <= calls_logits(k) &&
           B * kSelCluster <= ctx->sm_count && 1 + (long long)(t_max - 1) * k <= 65535;
}

extern "C" size_t radar_expand_calls_workspace_bytes(const radar_ctx* ctx, int B, int V, int k, int t_max) {
    if (!ctx || !calls_together(ctx, B, V, k, t_max)) return 0;
    const CallsPlan p = plan_calls(ctx, B, V, k, t_max);
    return align_up(vocab_pass_workspace_bytes(ctx->sm_count, p.rows, V, k), 256) + p.merged_bytes;
}

extern "C" int radar_expand_calls(radar_ctx* ctx, const radar_expand_calls_args* args, void* stream_) {
    if (!ctx || !args) return RADAR_ERR_INVALID_ARG;
    const radar_expand_args* a = &args->call;
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
    if (a->B <= 0 || a->F != 1 || a->V <= 0 || a->k <= 0 || a->t != 1 || a->t_max < 1) return RADAR_ERR_INVALID_ARG;
    if (a->k > RADAR_MAX_K || a->V < a->k) return RADAR_ERR_UNSUPPORTED;
    if (a->logits_dtype != RADAR_F32 && a->logits_dtype != RADAR_BF16) return RADAR_ERR_UNSUPPORTED;
    if (a->policy != RADAR_POLICY_LSTM_SCORES && a->policy != RADAR_POLICY_MLP_SCORES) return RADAR_ERR_UNSUPPORTED;
    if (!calls_together(ctx, a->B, a->V, a->k, a->t_max)) return RADAR_ERR_UNSUPPORTED;
    if (a->logits_row_stride < a->V) return RADAR_ERR_INVALID_ARG;
    if (!a->logits || !a->parent_score || !a->parent_pool_idx || !a->active || !a->h || !a->c || !a->pool_tok || !a->pool_parent ||
        !a->pool_depth || !a->pool_draft_row || !a->pool_score || !a->pool_len || !a->frontier_tok || !a->frontier_score ||
        !a->frontier_pool_idx || !a->frontier_src_row || !a->topk_tok || !a->topk_logp || !a->gate_logits || !a->cont || !a->workspace)
        return RADAR_ERR_INVALID_ARG;
    const bool gate_runs = a->t_max > 1, recurrent = a->policy == RADAR_POLICY_LSTM_SCORES;
    if (gate_runs && (!args->topk_tok_next || !args->topk_logp_next || !a->w1 || !a->b1 || !a->w2 || !a->b2 ||
                      (reinterpret_cast<uintptr_t>(a->w1) & 15) != 0))
        return RADAR_ERR_INVALID_ARG;
    if (gate_runs && recurrent &&
        (!a->w_ih || !a->w_hh || !a->b_ih || !a->b_hh || ((reinterpret_cast<uintptr_t>(a->w_hh) | reinterpret_cast<uintptr_t>(a->w_ih)) & 15) != 0))
        return RADAR_ERR_INVALID_ARG;
    if (a->pool_capacity < a->k) return RADAR_ERR_INVALID_ARG;
    const CallsPlan plan = plan_calls(ctx, a->B, a->V, a->k, a->t_max);
    if ((reinterpret_cast<uintptr_t>(a->workspace) & 255) != 0 || plan.part_bytes + plan.merged_bytes > a->workspace_bytes) return RADAR_ERR_WORKSPACE;

    VocabPassParams vp;
    vp.logits = a->logits;
    vp.dtype = a->logits_dtype;
    vp.row_stride = a->logits_row_stride;
    vp.seq_stride = a->logits_seq_stride;
    vp.n_seq = a->B;
    vp.F = plan.R;
    vp.V = a->V;
    vp.k = a->k;
    vp.n_chunks = plan.n_chunks;
    vp.chunk = plan.chunk;
    vp.want_lse = 1;
    vp.seq_active = nullptr;
    vp.seq_rows = nullptr;
    vp.status = nullptr;
    vocab_pass_carve(a->workspace, plan.rows, plan.n_chunks, a->k, &vp);
    char* merged = reinterpret_cast<char*>(a->workspace) + plan.part_bytes;
    double* row_logp = reinterpret_cast<double*>(merged);
    int32_t* row_tok = reinterpret_cast<int32_t*>(merged + align_up((size_t)plan.rows * a->k * sizeof(double), 256));
    RADAR_CUDA_CHECK(vocab_pass_launch(ctx, RADAR_K_VOCAB_EXPAND, vp, stream));
    {
        radar_launch_scope scope(ctx, RADAR_K_ROW_MERGE, stream);
        const size_t stage = (size_t)((vp.n_chunks * a->k + 3) & ~3) * 8;
        const int staged = stage <= kMergeStageLimit ? 1 : 0;
        const size_t smem = (size_t)kSurvCap * 8 + (staged ? stage : 0);
        RADAR_CUDA_CHECK(launch_chained(row_merge_kernel, dim3((unsigned)plan.rows), dim3(64), smem, stream, vp, staged, row_tok, row_logp));
    }
    {
        CallsParams cp;
        cp.a = *a;
        cp.topk_tok_next = args->topk_tok_next;
        cp.topk_logp_next = args->topk_logp_next;
        cp.row_tok = row_tok;
        cp.row_logp = row_logp;
        cp.status = ctx->d_status;
        radar_launch_scope scope(ctx, RADAR_K_EXPAND_CALLS, stream);
        const int blocks = recurrent && gate_runs ? kSelCluster : 1;
        const size_t smem = gate_runs ? sizeof(float) * (size_t)((recurrent ? 4 : 1) * kHidden) * (a->k | 1) : 0;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(a->B * blocks));
        cfg.blockDim = dim3(kSelThreads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = stream;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = (unsigned)blocks;
        attr[1].val.clusterDim.y = 1;
        attr[1].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = blocks > 1 ? 2 : 1;
        if (blocks > 1) {
            RADAR_CUDA_CHECK(radar_opt_in_smem(ctx, RADAR_SMEM_EXPAND_CALLS, expand_calls_kernel<true>, smem));
            RADAR_CUDA_CHECK(cudaLaunchKernelEx(&cfg, expand_calls_kernel<true>, cp));
        } else {
            RADAR_CUDA_CHECK(radar_opt_in_smem(ctx, RADAR_SMEM_EXPAND_CALLS_PLAIN, expand_calls_kernel<false>, smem));
            RADAR_CUDA_CHECK(cudaLaunchKernelEx(&cfg, expand_calls_kernel<false>, cp));
        }
    }
    RADAR_CUDA_CHECK(cudaGetLastError());
    return RADAR_OK;
}
