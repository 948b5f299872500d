// radar_expand_calls: all draft calls of a step on draft logits that are there already.
//
//   row_topk_kernel        one pass over the rows of all calls: their top-k tokens and log-probabilities (fp64);
//   expand_calls_kernel    one cluster per sequence goes through the calls: candidates, pool, frontier, prediction model.
//
// Call by call, a step is a chain of two dozen launches whose blocks each reload the gate's weights and hand the state on through
// global memory: 8 us a call, whatever the size.  Here the passes, which depend on nothing the calls decide, run once over all
// rows of a range of calls, and the calls themselves are a loop whose weights and state stay on chip, 2.3 us a call (B = 1,
// V = 128256, 8 calls: 65 us call by call, 32 together).  What it costs: rows of calls that a sequence never makes are read
// too, so with long passes a step is made in several ranges; what one range leaves, the next one starts from.  It takes
// draft logits that exist before the range's first call (recorded ones, or a draft model that does not look at the frontier);
// where the draft model runs between the calls, radar_expand_step is the form.
#include <algorithm>
#include <cstdint>

#include "select.cuh"

namespace radar {
namespace {

struct CallsParams {
    radar_expand_args a;                             // the arguments of call 1
    int32_t* topk_tok_next;                          // [t_max-1][B][k][k] of calls 2..
    float* topk_logp_next;
    int t_first, t_last;                             // the calls that are made
    const int32_t* row_tok;                          // [B][rows of these calls][k] merged rows
    const double* row_logp;
    const float* feat_pre;                           // hidden-state policy: [calls made][B][4H] W_ih f and [..][H] W_1[:, H:] f
    const float* feat_hid;
    int* status;
};

// Rank of candidate c among n (key desc, index asc), by the 16 threads of a half-warp.  For more than 64 of them, where two to a
// warp with ballots (ranks_of) takes longer: five calls of two sequences, V = 32000, k = 32, 70.6 -> 55.0 us, k = 16, eight 35.2 -> 33.0.
// Not inlined: in the calls' loop its instructions cost the others 0.8 us a step.
__device__ __noinline__ int rank_among_many(const unsigned long long* keys, const short* index, int n, int c) {
    const unsigned long long mine = keys[c];
    const int idx = index[c];
    int rank = 0;
#pragma unroll 2
    for (int j = threadIdx.x & 15; j < n; j += 16) {
        const unsigned long long kj = keys[j];
        const int ij = index[j];
        rank += (int)(kj > mine) | ((int)(kj == mine) & (int)(ij < idx));
    }
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) rank += __shfl_xor_sync(kFull, rank, o);
    return rank;
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
    constexpr uint32_t kStateBytes = (H + 1) * 4, kProductBytes = HelperRows::kProductBytes;     // the two messages: h and a stop flag; W_hh h + biases
    const int b = blockIdx.x / kBlocks, B = a.B, k = a.k, t_max = a.t_max;
    const int t_first = P.t_first, t_last = P.t_last, t_gate = min(t_last, t_max - 1);     // (t_gate: the last call whose gate runs)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    extern __shared__ __align__(16) unsigned char calls_smem[];
    __shared__ float s_pre[4 * H];                     // block 0: W_hh h + biases of the call
    __shared__ __align__(16) float s_h[H + 4];         // helpers: the h they were sent; [H]: not 0 if it is the last message
    __shared__ __align__(8) uint64_t s_bar;            // completes with the message the block expects next
    uint32_t crank = 0;
    if (kRecurrent) asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(crank));

    // The predecessor is row_topk_kernel, whose CTAs let this one start behind their own wait: only the rows need the wait.
    if (t_first > 1 && a.active[b] == 0) {             // the sequence has stopped
        chain_sync();
        chain_trigger();
        if (crank == 0 && tid <= t_last - t_first) a.cont[(size_t)(t_first - 1 + tid) * B + b] = 0;
        return;
    }
    if (crank != 0) {
        // ---- helper block: its rows of W_hh h + biases, into block 0's s_pre ----
        const HelperRows R(a, (int)crank);
        if (tid == 0) init_message_barrier(&s_bar, kStateBytes);
        const uint32_t to = cluster_addr(&s_pre[min(R.row, 4 * H - 1)], 0), to_bar = cluster_addr(&s_bar, 0);
        cluster_barrier();                             // every block has started and its barrier word is initialised
        if (t_first > 1 && t_first <= t_gate) {        // of the h that the calls before have left
            const float* hb = a.h + (size_t)b * H + 4 * lane;
            const float sum = R.product(make_float4(hb[0], hb[1], hb[2], hb[3]));
            if (R.sender) send_f32(to, to_bar, sum);
        }
        chain_sync();
        chain_trigger();
        for (int t = t_first + 1; t <= t_gate; ++t) {  // W_hh h of call t - 1, for call t's gate
            if (!cluster_wait(&s_bar, (uint32_t)((t - t_first - 1) & 1))) { set_status(P.status, RADAR_ERR_TIMEOUT); break; }
            const float4 h4 = *reinterpret_cast<const float4*>(s_h + lane * 4);
            if (*(volatile float*)&s_h[H] != 0.f) break;
            if (tid == 0) expect_bytes(&s_bar, kStateBytes);
            const float sum = R.product(h4);
            if (R.sender) send_f32(to, to_bar, sum);
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
    const bool hidden = kRecurrent && a.policy == RADAR_POLICY_LSTM_HIDDEN;
    if (t_max > 1) {
        if (!hidden) copy_rows(s_w, kRecurrent ? a.w_ih : a.w1, kRecurrent ? 4 * H : H, k);
        if (kRecurrent) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float* w = a.w1 + (size_t)(warp + i * kSelWarps) * (H + (hidden ? a.feat_dim : k));
#pragma unroll
                for (int c = 0; c < 4; ++c) w1r[i][c] = w[lane + 32 * c];
                w1x[i] = !hidden && lane < k ? w[H + lane] : 0.f;
            }
        }
        // (nothing is waited for here: the block has to reach the cluster's barrier, and what it copies may land behind the rows)
        if (tid < H) cp_async4(s_b1 + tid, a.b1 + tid);
        if (tid < 2 * H) cp_async4(s_w2 + tid, a.w2 + tid);
        if (tid < 2) cp_async4(s_b2 + tid, a.b2 + tid);
        if (kRecurrent && t_first > 1 && tid < H) cp_async4(s_c + tid, a.c + (size_t)b * H + tid);
    }
    const bool first_bias = kRecurrent && t_max > 1 && t_first == 1 && tid < 4 * H;      // call 1: h is zero
    const float bias_ih = first_bias ? a.b_ih[tid] : 0.f, bias_hh = first_bias ? a.b_hh[tid] : 0.f;
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
    const size_t rows0 = (size_t)b * (t_first == 1 ? 1 + (t_last - 1) * k : (t_last - t_first + 1) * k);     // the sequence's first row
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
        if (e >= 0 && t <= t_last && (t > 1 || e < k)) {
            const size_t o = (t == 1 ? rows0 : rows0 + (t_first == 1 ? 1 + (t - 2) * k : (t - t_first) * k)) * k + e;
            lp = P.row_logp[o];
            tok = P.row_tok[o];
        }
    };
    // hidden-state policy: this thread's share of the input-side products of the gate's next call
    float feat_p = 0.f, feat_h = 0.f;
    const int head_row = warp + (lane >> 3) * kSelWarps;              // the row of the hidden layer whose sum ends up in this lane
    auto fetch_features = [&](int t) {
        if (!hidden || t < t_first || t > t_gate) return;
        const size_t o = (size_t)(t - t_first) * B + b;
        if (tid < 4 * H) feat_p = P.feat_pre[o * 4 * H + tid];
        if ((lane & 7) == 0) feat_h = P.feat_hid[o * H + head_row];
    };
    auto frontier = [&](int rank, float score, int cand, int base, int buf) {
        s_fscore[rank] = score;
        s_fidx[rank] = base + cand;
        s_x[buf][rank] = expf(score);                                 // confidence score in [0,1]
        s_rank[cand] = (short)rank;
    };
    if (t_first == 1) fetch(1);
    if (t_first == 1 && e >= 0 && e < k) {                            // call 1: one row, already in order
        my_tok = tok;
        my_lp = (float)lp;
        my_score = (float)((double)root_score + lp);
        my_parent = root_idx;
        frontier(e, my_score, e, 0, 1);
    }
    if (t_first > 1 && tid < k) {                                     // the frontier that the calls before have left
        const size_t o = ((size_t)(t_first - 2) * B + b) * k + tid;
        s_fscore[tid] = a.frontier_score[o];
        s_fidx[tid] = a.frontier_pool_idx[o];
    }
    fetch(max(t_first, 2));
    if (first_bias) s_pre[tid] = bias_ih + bias_hh;
    if (t_first == 1 && tid < H) s_c[tid] = 0.f;
    if (t_first == 1) fetch_features(1);
    cp_async_wait_all();
    __syncthreads();

    // (calls that go on from others: a first turn, t = t_first - 1, only selects call t_first's frontier; a last one, where
    // the gate of the last call runs, only takes its decision)
    int base = t_first > 1 ? a.pool_len[b] : 0, sent = t_first - 1, t = max(t_first - 1, 1);
    for (;; ++t) {
        const bool made = t >= t_first, more = t < t_last;            // more: call t + 1 may follow
        const int n_cand = !made ? 0 : t == 1 ? k : k * k;
        const bool run_gate = made && t <= t_gate;
        // ---- 1 ----
        if (run_gate && kRecurrent && tid < 4 * H) {
            float acc = s_pre[tid] + feat_p;
            const float* w = s_w + tid * ws;
            const float* x = s_x[t & 1];
#pragma unroll 4
            for (int j = 0; j < (hidden ? 0 : k); ++j) acc = fmaf(w[j], x[j], acc);
            s_pre[tid] = warp / (H / 32) == 2 ? tanhf(acc) : sigmoidf_(acc);
        }
        if (run_gate && !kRecurrent && tid < H) {
            float acc = s_b1[tid];
            const float* w = s_w + tid * ws;
            const float* x = s_x[t & 1];
            for (int j = 0; j < k; ++j) acc = fmaf(w[j], x[j], acc);
            s_hid[t & 1][tid] = fmaxf(acc, 0.f);
        }
        if (t > t_first && warp == 4 * H / 32) {
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
        if (more && e >= 0) {
            const double cand = (double)s_fscore[f] + lp;
            key = order_key64(cand);
            next_score = (float)cand;
            next_parent = s_fidx[f];
            if (e == f * k) s_head[f] = next_score;
        }
        if (tid == 0) s_count = 0;
        __syncthreads();
        if (t > t_first && (s_cont == 0 || t > t_last)) { --t; break; }                     // t: the last call the sequence made
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
            if (t + 1 <= t_gate) {
#pragma unroll
                for (int r = 0; r < kHelp; ++r) send_f32(to[r], to_bar[r], hn);
                if (tid < kHelp) send_f32(to_flag, cluster_addr(&s_bar, tid + 1), 0.f);
            }
        }
        if (made && t + 1 <= t_gate) sent = t;
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
        if (made && tid == kSelThreads - 1) a.pool_len[b] = base;
        if (t == t_max) {
            if (tid < 2) a.gate_logits[((size_t)(t - 1) * B + b) * 2 + tid] = 0.f;
            if (tid == 0) { a.cont[(size_t)(t - 1) * B + b] = 0; a.active[b] = 0; }
            break;
        }
        if (more && warp >= (kSelThreads - k * k) / 32) {
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
        if (kRecurrent && run_gate) {
            const float hv[4] = {s_hn[lane], s_hn[lane + 32], s_hn[lane + 64], s_hn[lane + 96]};
            const float xv = !hidden && lane < k ? s_x[t & 1][lane] : 0.f;
            float acc[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float v = w1r[i][0] * hv[0];
                v = fmaf(w1r[i][1], hv[1], v);
                v = fmaf(w1r[i][2], hv[2], v);
                v = fmaf(w1r[i][3], hv[3], v);
                if (!hidden && lane < k) v = fmaf(w1x[i], xv, v);
                acc[i] = v;
            }
            const float sum = transposed_sum<4>(acc);
            if ((lane & 7) == 0) s_hid[t & 1][head_row] = fmaxf(sum + s_b1[head_row] + feat_h, 0.f);
        }
        fetch_features(t + 1);
        // the k best survivors (score desc, flat index asc): up to 64, a warp to two of them, else a half-warp to each
        const int n = more ? s_count : 0;
        if (n <= 2 * kSelWarps) {
            if (warp < n) {
                const int c1 = min(warp + kSelWarps, n - 1), idx0 = s_cand[warp], idx1 = s_cand[c1];
                const int2 rank = ranks_of(s_key, s_cand, n, s_key[warp], idx0, s_key[c1], idx1);
                if (lane == 0 && rank.x < k) frontier(rank.x, s_score[warp], idx0, base, (t + 1) & 1);
                if (lane == 1 && rank.y < k && warp + kSelWarps < n) frontier(rank.y, s_score[c1], idx1, base, (t + 1) & 1);
            }
        } else {
            for (int c0 = 0; c0 + warp * 2 < n; c0 += kSelThreads / 16) {
                const int c = min(c0 + (tid >> 4), n - 1), rank = rank_among_many(s_key, s_cand, n, c);
                if ((tid & 15) == 0 && rank < k && c0 + (tid >> 4) < n) frontier(rank, s_score[c], s_cand[c], base, (t + 1) & 1);
            }
        }
        if (kRecurrent) {
            if (run_gate && tid >= kSelThreads - H) {
                const int c = tid - (kSelThreads - H);
                a.c[(size_t)b * H + c] = s_c[c];
                a.h[(size_t)b * H + c] = s_hn[c];
            }
            // one thread waits for the helpers' product of the next call, the barrier publishes it
            if (t + 1 <= t_gate && tid == kSelThreads - 1) {
                if (!cluster_wait(&s_bar, (uint32_t)((t_first == 1 ? t - 1 : t + 1 - t_first) & 1))) set_status(P.status, RADAR_ERR_TIMEOUT);
                expect_bytes(&s_bar, kProductBytes);
            }
        }
        __syncthreads();
    }
    for (int u = t + 1 + tid; u <= t_last; u += kSelThreads) a.cont[(size_t)(u - 1) * B + b] = 0;     // calls the sequence does not make
    if (kRecurrent) {
        if (tid < H) {
            // The product of the last h has been waited for, so that nothing is on its way into this block and every helper warp
            // is past its wait (a barrier may not run two phases ahead of a waiter).
            if (sent < t_gate - 1) {                                   // helpers that still expect an h
#pragma unroll
                for (int r = 0; r < kHelp; ++r) send_f32(to[r], to_bar[r], 0.f);
                if (tid < kHelp) send_f32(to_flag, cluster_addr(&s_bar, tid + 1), 1.f);
            }
        }
        cluster_barrier();                                            // the helpers have received their last message
    }
}

// The line of radar_expand_calls, calls of at most 4 Mi logits (5 Mi from k = 16 on): all rows of a step in one range.  Longer
// passes read too much in vain where sequences stop early; radar_expand_range makes such a step in several ranges.
inline long long calls_logits(int k) { return k < 16 ? kShortPassLogits : 5LL << 20; }

}  // namespace
}  // namespace radar

using namespace radar;

// rows of a sequence in calls t_first .. t_last; 0: this form does not take them
static int range_rows(const radar_ctx* ctx, int B, int V, int k, int t_first, int t_last) {
    if (B <= 0 || k <= 0 || k > RADAR_MAX_K || V < k || t_first < 1 || t_last < t_first || (long long)B * kSelCluster > ctx->sm_count) return 0;
    const long long rows = (t_first == 1 ? 1 : k) + (long long)(t_last - t_first) * k;
    return rows <= 65535 ? (int)rows : 0;
}
// the input-side products of the hidden-state policy
static size_t feature_bytes(int B, int calls) { return (size_t)std::max(calls, 0) * B * 5 * kHidden * sizeof(float); }
static bool calls_together(const radar_ctx* ctx, int B, int V, int k, int t_max) {
    return range_rows(ctx, B, V, k, 1, t_max) > 0 && (long long)B * k * V <= calls_logits(k);
}

extern "C" size_t radar_expand_range_workspace_bytes(const radar_ctx* ctx, int B, int V, int k, int t_first, int t_last) {
    const int rows = ctx ? range_rows(ctx, B, V, k, t_first, t_last) : 0;
    return rows ? row_topk_workspace_bytes(B * rows, V, k) + feature_bytes(B, t_last - t_first + 1) : 0;
}

extern "C" size_t radar_expand_calls_workspace_bytes(const radar_ctx* ctx, int B, int V, int k, int t_max) {
    return ctx && calls_together(ctx, B, V, k, t_max) ? row_topk_workspace_bytes(B * range_rows(ctx, B, V, k, 1, t_max), V, k) : 0;
}

extern "C" int radar_expand_calls(radar_ctx* ctx, const radar_expand_calls_args* args, void* stream) {
    if (!ctx || !args) return RADAR_ERR_INVALID_ARG;
    const radar_expand_args& a = args->call;
    if (a.B > 0 && a.F == 1 && a.t == 1 && a.V >= a.k && a.k > 0 && a.k <= RADAR_MAX_K && a.t_max >= 1 && !calls_together(ctx, a.B, a.V, a.k, a.t_max))
        return RADAR_ERR_UNSUPPORTED;
    if (a.policy != RADAR_POLICY_LSTM_SCORES && a.policy != RADAR_POLICY_MLP_SCORES) return RADAR_ERR_UNSUPPORTED;
    const radar_expand_range_args r = {a, args->topk_tok_next, args->topk_logp_next, 1, a.t_max};
    return radar_expand_range(ctx, &r, stream);
}

extern "C" int radar_expand_range(radar_ctx* ctx, const radar_expand_range_args* args, void* stream_) {
    if (!ctx || !args) return RADAR_ERR_INVALID_ARG;
    const radar_expand_args* a = &args->call;
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
    if (a->B <= 0 || a->F != 1 || a->V <= 0 || a->k <= 0 || a->t != 1 || a->t_max < 1) return RADAR_ERR_INVALID_ARG;
    if (args->t_first < 1 || args->t_last < args->t_first || args->t_last > a->t_max) return RADAR_ERR_INVALID_ARG;
    if (a->k > RADAR_MAX_K || a->V < a->k) return RADAR_ERR_UNSUPPORTED;
    if (a->logits_dtype != RADAR_F32 && a->logits_dtype != RADAR_BF16) return RADAR_ERR_UNSUPPORTED;
    if (a->policy != RADAR_POLICY_LSTM_SCORES && a->policy != RADAR_POLICY_MLP_SCORES && a->policy != RADAR_POLICY_LSTM_HIDDEN)
        return RADAR_ERR_INVALID_ARG;
    const int rows = range_rows(ctx, a->B, a->V, a->k, args->t_first, args->t_last);
    if (rows == 0) return RADAR_ERR_UNSUPPORTED;
    if (a->logits_row_stride < a->V) return RADAR_ERR_INVALID_ARG;
    if (!a->logits || !a->parent_score || !a->parent_pool_idx || !a->active || !a->h || !a->c || !a->pool_tok || !a->pool_parent ||
        !a->pool_depth || !a->pool_draft_row || !a->pool_score || !a->pool_len || !a->frontier_tok || !a->frontier_score ||
        !a->frontier_pool_idx || !a->frontier_src_row || !a->topk_tok || !a->topk_logp || !a->gate_logits || !a->cont || !a->workspace)
        return RADAR_ERR_INVALID_ARG;
    const bool gate_runs = a->t_max > 1, recurrent = a->policy != RADAR_POLICY_MLP_SCORES, hidden = a->policy == RADAR_POLICY_LSTM_HIDDEN;
    if (gate_runs && (!args->topk_tok_next || !args->topk_logp_next || !a->w1 || !a->b1 || !a->w2 || !a->b2 ||
                      (reinterpret_cast<uintptr_t>(a->w1) & 15) != 0))
        return RADAR_ERR_INVALID_ARG;
    if (gate_runs && recurrent &&
        (!a->w_ih || !a->w_hh || !a->b_ih || !a->b_hh || ((reinterpret_cast<uintptr_t>(a->w_hh) | reinterpret_cast<uintptr_t>(a->w_ih)) & 15) != 0))
        return RADAR_ERR_INVALID_ARG;
    if (gate_runs && hidden && (!a->features || a->feat_dim < 4 || a->feat_dim > 16384 || (a->feat_dim & 3) != 0 ||
                                (reinterpret_cast<uintptr_t>(a->features) & 15) != 0))
        return RADAR_ERR_INVALID_ARG;
    if (a->pool_capacity < a->k) return RADAR_ERR_INVALID_ARG;
    const int n_gates = std::min(args->t_last, a->t_max - 1) - args->t_first + 1;
    const size_t row_bytes = row_topk_workspace_bytes(a->B * rows, a->V, a->k);
    if ((reinterpret_cast<uintptr_t>(a->workspace) & 255) != 0 || row_bytes + (hidden ? feature_bytes(a->B, n_gates) : 0) > a->workspace_bytes)
        return RADAR_ERR_WORKSPACE;
    float* feat_pre = reinterpret_cast<float*>(static_cast<char*>(a->workspace) + row_bytes);
    if (hidden && n_gates > 0) {                           // of all calls of the range: the weights are read once
        radar_expand_args f = *a;
        f.B = a->B * n_gates;
        f.features = a->features + (size_t)(args->t_first - 1) * a->B * a->feat_dim;
        RADAR_CUDA_CHECK(gate_features_launch(ctx, f, feat_pre, stream));
    }

    const int64_t first_row = args->t_first == 1 ? 0 : 1 + (int64_t)(args->t_first - 2) * a->k;
    RowTopkParams rp;
    rp.logits = static_cast<const char*>(a->logits) + first_row * a->logits_row_stride * (a->logits_dtype == RADAR_F32 ? 4 : 2);
    rp.dtype = a->logits_dtype;
    rp.row_stride = a->logits_row_stride;
    rp.seq_stride = a->logits_seq_stride;
    rp.n_seq = a->B;
    rp.F = rows;
    rp.V = a->V;
    rp.k = a->k;
    rp.seq_active = args->t_first > 1 ? a->active : nullptr;
    row_topk_carve(rp, a->workspace);
    RADAR_CUDA_CHECK(row_topk_launch(ctx, rp, stream));
    {
        CallsParams cp;
        cp.a = *a;
        cp.topk_tok_next = args->topk_tok_next;
        cp.topk_logp_next = args->topk_logp_next;
        cp.t_first = args->t_first;
        cp.t_last = args->t_last;
        cp.row_tok = rp.tok;
        cp.row_logp = rp.logp;
        cp.feat_pre = feat_pre;
        cp.feat_hid = feat_pre + (size_t)a->B * std::max(n_gates, 0) * 4 * kHidden;
        cp.status = ctx->d_status;
        radar_launch_scope scope(ctx, RADAR_K_EXPAND_CALLS, stream);
        const int blocks = recurrent && gate_runs ? kSelCluster : 1;
        const size_t smem = gate_runs && !hidden ? sizeof(float) * (size_t)((recurrent ? 4 : 1) * kHidden) * (a->k | 1) : 0;
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
