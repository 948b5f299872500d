// radar_expand_step: vocabulary pass and row merge (row_topk.cu), then one block per sequence that forms the candidate scores,
// appends them to the pool, selects the k best over all parents and runs the prediction model (LSTM cell + MLP head) on their
// confidence scores.
#include <algorithm>

#include "select.cuh"

namespace radar {
namespace {

struct SelectParams {
    radar_expand_args a;
    const int32_t* row_tok;                          // [B][F][k] merged rows
    const double* row_logp;
    int split;                                       // 1: launched on its own (RADAR_EXPAND_SELECT)
    const float* feat_pre;                           // hidden-state policy: [B][4H] W_ih f and [B][H] W_1[:, H:] f,
    const float* feat_hid;                           // written by gate_features_kernel
    int* status;
};

// Hidden-state policy (Table 3): the input-side products of the prediction model, W_ih f_b (4H rows) and the
// head's columns for the input, W_1[:, H:] f_b (H rows), for every sequence.  One block per output row, one
// warp per 512-element segment of it: every weight is requested at once (the matrix is read at memory speed,
// once), the feature rows come from L1/L2, the segments meet in shared memory.  It needs nothing from the
// vocabulary pass and is launched ahead of it.
constexpr int kFeatSeg = 512;                        // elements of a row per warp: 4 x float4 per lane
__global__ void __launch_bounds__(1024) gate_features_kernel(const radar_expand_args a, float* pre, float* hid) {
    chain_wait();
    const int H = kHidden, lane = threadIdx.x & 31, seg = threadIdx.x >> 5, nseg = blockDim.x >> 5;
    const int r = blockIdx.x;                        // 0 .. 5H-1
    const int d = a.feat_dim;
    __shared__ float s_part[32][8];
    const float* w = r < 4 * H ? a.w_ih + (size_t)r * d : a.w1 + (size_t)(r - 4 * H) * (H + d) + H;
    float4 wv[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int c = seg * kFeatSeg + i * 128 + lane * 4;
        wv[i] = c < d ? __ldg(reinterpret_cast<const float4*>(w + c)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    for (int b0 = 0; b0 < a.B; b0 += 8) {
        float acc[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[j] = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int c = seg * kFeatSeg + i * 128 + lane * 4;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                if (c < d && b0 + j < a.B) {
                    const float4 f = __ldg(reinterpret_cast<const float4*>(a.features + (size_t)(b0 + j) * d + c));
                    acc[j] = fmaf(wv[i].x, f.x, fmaf(wv[i].y, f.y, fmaf(wv[i].z, f.z, fmaf(wv[i].w, f.w, acc[j]))));
                }
            }
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float v = warp_sum(acc[j]);
            if (lane == 0) s_part[seg][j] = v;
        }
        __syncthreads();
        if (threadIdx.x < 8 && b0 + (int)threadIdx.x < a.B) {
            float v = 0.f;
            for (int q = 0; q < nseg; ++q) v += s_part[q][threadIdx.x];
            const int b = b0 + threadIdx.x;
            if (r < 4 * H) pre[(size_t)b * 4 * H + r] = v;
            else hid[(size_t)b * H + (r - 4 * H)] = v;
        }
        __syncthreads();
    }
}

// One block per sequence.  What bounds it is its chain of steps between block barriers; all that does not depend on the call's
// rows (weights, the previous state, W_hh h) is fetched and multiplied before the wait for the merge.  The arithmetic and its order are those of expand_calls_kernel.
//
// Behind its own rows' kernel, the block reads the weights and what the previous call left (active, h, c, pool_len, the frontier)
// before it waits: that kernel's CTAs let it start behind their own wait.  Launched on its own (split), its predecessor is the
// block of the call before, or anything: it waits first.
template <bool kHelpers>
__global__ void __launch_bounds__(kSelThreads, 1) expand_select_gate_kernel(const SelectParams P) {
    if (P.split) chain_sync();
    chain_trigger();
    const radar_expand_args& a = P.a;
    constexpr int H = kHidden, kBlocks = kHelpers ? kSelCluster : 1;
    const int b = blockIdx.x / kBlocks, F = a.F, k = a.k;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool run_gate = a.t < a.t_max, lstm = run_gate && a.policy != RADAR_POLICY_MLP_SCORES;
    const bool hidden = a.policy == RADAR_POLICY_LSTM_HIDDEN;
    extern __shared__ __align__(16) float s_w[];       // W_ih [4H][k | 1], or w1 [H][k | 1] of the MLP policy
    __shared__ float s_pre[4 * H];                     // W_hh h + biases
    __shared__ __align__(8) uint64_t s_bar;            // completes when the helpers have delivered it
    uint32_t crank = 0;
    if (kHelpers) asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(crank));
    const bool live = a.t == 1 || a.active[b] != 0;    // call 1 always runs: it (re)starts every sequence
    const float* hb = a.h + (size_t)b * H;

    if (kHelpers && crank != 0) {
        // ---- helper block (calls from the second on): its rows of W_hh h + biases, into block 0's s_pre ----
        const HelperRows R(a, (int)crank);
        const float4 h4 = make_float4(hb[4 * lane], hb[4 * lane + 1], hb[4 * lane + 2], hb[4 * lane + 3]);
        const float sum = R.product(h4);
        cluster_barrier();                             // block 0 has started and its barrier word is initialised
        if (live && R.sender) send_f32(cluster_addr(&s_pre[R.row], 0), cluster_addr(&s_bar, 0), sum);
        chain_sync();
        return;
    }

    __shared__ unsigned long long s_key[kMaxF * RADAR_MAX_K];         // candidates that can matter: order keys,
    __shared__ float s_score[kMaxF * RADAR_MAX_K];     // scores,
    __shared__ short s_cand[kMaxF * RADAR_MAX_K];      // flat indices (f, j)
    __shared__ short s_rank[kMaxF * RADAR_MAX_K];      // rank of every candidate (k: not among the k best)
    __shared__ float s_head[kMaxF];                    // of every parent, the candidate the bound is taken from
    __shared__ float s_x[RADAR_MAX_K];                 // gate input
    __shared__ float s_hn[H], s_hid[H], s_c[H], s_b1[H], s_w2[2 * H], s_b2[2];
    __shared__ int s_count;
    const int ws = k | 1;                              // odd: a column of rows meets all banks
    const int w1_stride = H + (hidden ? a.feat_dim : k);
    float w1r[4][4], w1x[4];                           // a warp's four rows of the head's hidden layer
    static_assert(H == 4 * kSelWarps, "four rows of the hidden layer per warp");
    if (run_gate) {
        if (!hidden) copy_rows(s_w, lstm ? a.w_ih : a.w1, lstm ? 4 * H : H, k);
        if (lstm) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float* w = a.w1 + (size_t)(warp + i * kSelWarps) * w1_stride;
#pragma unroll
                for (int c = 0; c < 4; ++c) w1r[i][c] = w[lane + 32 * c];
                w1x[i] = !hidden && lane < k ? w[H + lane] : 0.f;
            }
        }
        // (nothing is waited for here)
        if (tid < H) cp_async4(s_b1 + tid, a.b1 + tid);
        if (tid < 2 * H) cp_async4(s_w2 + tid, a.w2 + tid);
        if (tid < 2) cp_async4(s_b2 + tid, a.b2 + tid);
        if (tid < H && lstm) {
            if (a.t > 1) cp_async4(s_c + tid, a.c + (size_t)b * H + tid);
            else s_c[tid] = 0.f;
        }
    }
    if (kHelpers) {
        if (tid == 0) init_message_barrier(&s_bar, HelperRows::kProductBytes);
        cluster_barrier();
    }
    if (!live) {
        cp_async_wait_all();                           // nothing of this block is in flight when it leaves
        chain_sync();
        if (tid == 0) a.cont[b] = 0;
        return;
    }
    if (lstm && a.t == 1) {                            // h is zero
        if (tid < 4 * H) s_pre[tid] = a.b_ih[tid] + a.b_hh[tid];
    } else if (lstm && !kHelpers) {
        const float4 h4 = make_float4(hb[4 * lane], hb[4 * lane + 1], hb[4 * lane + 2], hb[4 * lane + 3]);
#pragma unroll
        for (int r0 = warp * 16; r0 < warp * 16 + 16; r0 += 8) {
            float4 w[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) w[i] = __ldg(reinterpret_cast<const float4*>(a.w_hh + (size_t)(r0 + i) * H) + lane);
            float acc[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                acc[i] = w[i].x * h4.x;
                acc[i] = fmaf(w[i].y, h4.y, acc[i]);
                acc[i] = fmaf(w[i].z, h4.z, acc[i]);
                acc[i] = fmaf(w[i].w, h4.w, acc[i]);
            }
            const float sum = transposed_sum<8>(acc);
            const int r = r0 + (lane >> 2);
            if ((lane & 3) == 0) s_pre[r] = sum + a.b_ih[r] + a.b_hh[r];
        }
    }
    const int n_cand = F * k, e = tid, f = e / k;      // candidate e, of parent f
    const bool mine = e < n_cand;
    const float parent_score = mine ? a.parent_score[(size_t)b * F + f] : 0.f;
    const int parent = mine ? a.parent_pool_idx[(size_t)b * F + f] : 0;
    const int base = a.t > 1 ? a.pool_len[b] : 0;
    const int forced = a.force_calls != nullptr ? a.force_calls[b] : -1;
    const float feat_h = hidden && lstm && tid < H ? P.feat_hid[(size_t)b * H + tid] : 0.f;
    const float feat_p = hidden && lstm && tid < 4 * H ? P.feat_pre[(size_t)b * 4 * H + tid] : 0.f;
    if (tid == 0) s_count = 0;
    cp_async_wait_all();
    chain_sync();
    if (base + n_cand > a.pool_capacity) {             // never write past the pool
        if (mine) {
            const size_t q = (size_t)b * n_cand + e;
            const int tk = P.row_tok[q];
            if (tk < 0) set_status(P.status, RADAR_ERR_NUMERIC);
            a.topk_tok[q] = tk & ~kNanRow;
            a.topk_logp[q] = (float)P.row_logp[q];
        }
        __syncthreads();
        if (tid == 0) {
            if (kHelpers) cluster_wait(&s_bar, 0);     // what the helpers send has landed
            set_status(P.status, RADAR_ERR_INVALID_ARG);
            a.cont[b] = 0;
            a.active[b] = 0;
        }
        return;
    }

    // ---- 1. candidates ----
    static_assert(kMaxF * RADAR_MAX_K <= kSelThreads, "one candidate per thread");
    int tok = 0;
    float lp32 = 0.f, score = 0.f;
    unsigned long long key = 0;
    const int depth = (k + F - 1) / F - 1;             // with that many of every (sorted) row, the rows have k candidates
    if (mine) {
        const double lp = P.row_logp[(size_t)b * n_cand + e];
        tok = P.row_tok[(size_t)b * n_cand + e];
        const double cand = (double)parent_score + lp;
        lp32 = (float)lp;
        score = (float)cand;
        key = order_key64(cand);
        s_rank[e] = (short)k;
        if (e - f * k == depth) s_head[f] = score;
    }
    if (kHelpers && tid == kSelThreads - 1 && !cluster_wait(&s_bar, 0)) set_status(P.status, RADAR_ERR_TIMEOUT);
    __syncthreads();
    {
        // the worst of the rows' candidates at that depth is a lower bound of the k-th best: what reaches it is listed
        const float low = warp_min_value(lane < F ? s_head[lane] : CUDART_INF_F);
        const bool keep = mine && !(score < low);
        const unsigned m = __ballot_sync(kFull, keep);
        if (m != 0) {
            int at = 0;
            if (lane == 0) at = atomicAdd(&s_count, __popc(m));
            at = __shfl_sync(kFull, at, 0) + __popc(m & ((1u << lane) - 1u));
            if (keep) {
                s_key[at] = key;
                s_score[at] = score;
                s_cand[at] = (short)e;
            }
        }
    }
    __syncthreads();

    // ---- 2. the k best (score desc, flat index asc): a warp to two candidates ----
    for (int c = warp, n = s_count; c < n; c += 2 * kSelWarps) {
        const int c1 = min(c + kSelWarps, n - 1), idx0 = s_cand[c], idx1 = s_cand[c1];
        const int2 rank = ranks_of(s_key, s_cand, n, s_key[c], idx0, s_key[c1], idx1);
        if (lane == 0 && rank.x < k) { s_rank[idx0] = (short)rank.x; s_x[rank.x] = expf(s_score[c]); }       // confidence score in [0,1]
        if (lane == 1 && rank.y < k && c + kSelWarps < n) { s_rank[idx1] = (short)rank.y; s_x[rank.y] = expf(s_score[c1]); }
    }
    __syncthreads();

    // ---- 3. the gate's input, and the call's results ----
    if (lstm && tid < 4 * H) {
        float acc = s_pre[tid];
        if (hidden) {
            acc += feat_p;
        } else {
            const float* w = s_w + tid * ws;
#pragma unroll 4
            for (int j = 0; j < k; ++j) acc = fmaf(w[j], s_x[j], acc);
        }
        s_pre[tid] = warp / (H / 32) == 2 ? tanhf(acc) : sigmoidf_(acc);
    }
    if (run_gate && !lstm && tid < H) {
        float acc = s_b1[tid];
        const float* w = s_w + tid * ws;
        for (int j = 0; j < k; ++j) acc = fmaf(w[j], s_x[j], acc);
        s_hid[tid] = fmaxf(acc, 0.f);
    }
    auto store_results = [&] {
        if (mine) {
            if (tok < 0) set_status(P.status, RADAR_ERR_NUMERIC);
            const int tk = tok & ~kNanRow, rank = s_rank[e];
            const size_t o = (size_t)b * a.pool_capacity + base + e, q = (size_t)b * n_cand + e;
            a.pool_tok[o] = tk;
            a.pool_parent[o] = parent;
            a.pool_score[o] = score;
            a.pool_depth[o] = a.t;
            a.pool_draft_row[o] = rank < k ? 1 + (a.t - 1) * k + rank : -1;
            a.topk_tok[q] = tk;
            a.topk_logp[q] = lp32;
            if (rank < k) {
                const size_t u = (size_t)b * k + rank;
                a.frontier_tok[u] = tk;
                a.frontier_score[u] = score;
                a.frontier_pool_idx[u] = base + e;
                a.frontier_src_row[u] = f;
            }
        }
        if (tid == kSelThreads - 1) a.pool_len[b] = base + n_cand;
    };
    if (!run_gate) {
        store_results();
        if (tid < 2) a.gate_logits[(size_t)b * 2 + tid] = 0.f;
        if (tid == 0) { a.cont[b] = 0; a.active[b] = 0; }
        return;
    }
    __syncthreads();
    if (lstm) {
        if (tid < H) {
            const float cn = s_pre[H + tid] * s_c[tid] + s_pre[tid] * s_pre[2 * H + tid];
            const float hn = s_pre[3 * H + tid] * tanhf(cn);
            s_hn[tid] = hn;
            a.c[(size_t)b * H + tid] = cn;
            a.h[(size_t)b * H + tid] = hn;
        }
        __syncthreads();
        const float hv[4] = {s_hn[lane], s_hn[lane + 32], s_hn[lane + 64], s_hn[lane + 96]};
        const float xv = !hidden && lane < k ? s_x[lane] : 0.f;
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
        const int r = warp + (lane >> 3) * kSelWarps;
        if ((lane & 7) == 0) s_hid[r] = hidden ? sum + s_b1[r] : fmaxf(sum + s_b1[r], 0.f);
        __syncthreads();
        if (hidden) {                                  // the features' share of the hidden layer
            if (tid < H) s_hid[tid] = fmaxf(s_hid[tid] + feat_h, 0.f);
            __syncthreads();
        }
    }
    if (warp == 0) {                                   // both logits in one warp: nothing else has to wait for them
        float y0 = 0.f, y1 = 0.f;
#pragma unroll
        for (int c = 0; c < H; c += 32) {
            y0 = fmaf(s_w2[c + lane], s_hid[c + lane], y0);
            y1 = fmaf(s_w2[H + c + lane], s_hid[c + lane], y1);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            y0 += __shfl_xor_sync(kFull, y0, o);
            y1 += __shfl_xor_sync(kFull, y1, o);
        }
        y0 += s_b2[0];
        y1 += s_b2[1];
        const bool cont = forced >= 0 ? a.t < forced : y1 > y0;
        if (lane < 2) a.gate_logits[(size_t)b * 2 + lane] = lane == 0 ? y0 : y1;
        if (lane == 0) { a.cont[b] = cont ? 1 : 0; a.active[b] = cont ? 1 : 0; }
    }
    store_results();
}

}  // namespace

cudaError_t gate_features_launch(radar_ctx* ctx, const radar_expand_args& a, float* pre, cudaStream_t stream) {
    radar_launch_scope scope(ctx, RADAR_K_GATE_FEATURES, stream);
    const int nseg = (a.feat_dim + kFeatSeg - 1) / kFeatSeg;
    return launch_chained(gate_features_kernel, dim3(5 * kHidden), dim3(nseg * 32), 0, stream, a, pre, pre + (size_t)a.B * 4 * kHidden);
}
}  // namespace radar

using namespace radar;

extern "C" size_t radar_expand_workspace_bytes(const radar_ctx* ctx, int B, int F, int V, int k) {
    if (!ctx || B <= 0 || F <= 0 || V <= 0 || k <= 0) return 0;
    return row_topk_workspace_bytes(B * F, V, k) + (size_t)B * 5 * kHidden * sizeof(float);
}

extern "C" int radar_expand_step(radar_ctx* ctx, const radar_expand_args* a, void* stream_) {
    if (!ctx || !a) return RADAR_ERR_INVALID_ARG;
    cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
    if (a->B <= 0 || a->F <= 0 || a->V <= 0 || a->k <= 0 || a->t < 1 || a->t > a->t_max) return RADAR_ERR_INVALID_ARG;
    if (a->k > RADAR_MAX_K || a->F > kMaxF || a->V < a->k) return RADAR_ERR_UNSUPPORTED;
    if (a->logits_dtype != RADAR_F32 && a->logits_dtype != RADAR_BF16) return RADAR_ERR_UNSUPPORTED;
    if (a->logits_row_stride < a->V) return RADAR_ERR_INVALID_ARG;
    if (a->phase != RADAR_EXPAND_ALL && a->phase != RADAR_EXPAND_VOCAB && a->phase != RADAR_EXPAND_SELECT) return RADAR_ERR_INVALID_ARG;
    if (!a->logits || !a->parent_score || !a->parent_pool_idx || (!a->active && a->phase != RADAR_EXPAND_VOCAB) || !a->h || !a->c || !a->pool_tok ||
        !a->pool_parent || !a->pool_depth || !a->pool_draft_row || !a->pool_score || !a->pool_len ||
        !a->frontier_tok || !a->frontier_score || !a->frontier_pool_idx || !a->frontier_src_row || !a->topk_tok ||
        !a->topk_logp || !a->gate_logits || !a->cont || !a->workspace)
        return RADAR_ERR_INVALID_ARG;
    if (a->policy != RADAR_POLICY_LSTM_SCORES && a->policy != RADAR_POLICY_MLP_SCORES && a->policy != RADAR_POLICY_LSTM_HIDDEN)
        return RADAR_ERR_INVALID_ARG;
    const bool gate_runs = a->t < a->t_max;
    if (gate_runs && (!a->w1 || !a->b1 || !a->w2 || !a->b2 || (reinterpret_cast<uintptr_t>(a->w1) & 15) != 0))
        return RADAR_ERR_INVALID_ARG;
    if (gate_runs && a->policy != RADAR_POLICY_MLP_SCORES &&
        (!a->w_ih || !a->w_hh || !a->b_ih || !a->b_hh ||
         ((reinterpret_cast<uintptr_t>(a->w_hh) | reinterpret_cast<uintptr_t>(a->w_ih)) & 15) != 0))
        return RADAR_ERR_INVALID_ARG;
    if (gate_runs && a->policy == RADAR_POLICY_LSTM_HIDDEN &&
        (!a->features || a->feat_dim < 4 || a->feat_dim > 16384 || (a->feat_dim & 3) != 0 ||
         (reinterpret_cast<uintptr_t>(a->features) & 15) != 0))
        return RADAR_ERR_INVALID_ARG;
    if (a->pool_capacity < a->F * a->k) return RADAR_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(a->workspace) & 255) != 0) return RADAR_ERR_WORKSPACE;

    RowTopkParams rp;
    rp.logits = a->logits;
    rp.dtype = a->logits_dtype;
    rp.row_stride = a->logits_row_stride;
    rp.seq_stride = a->logits_seq_stride;
    rp.n_seq = a->B;
    rp.F = a->F;
    rp.V = a->V;
    rp.k = a->k;
    rp.seq_active = a->t > 1 ? a->active : nullptr;          // RADAR_EXPAND_VOCAB: the caller's (possibly older) mask, or NULL
    const size_t row_bytes = row_topk_workspace_bytes(a->B * a->F, a->V, a->k);
    if (row_bytes + (size_t)a->B * 5 * kHidden * sizeof(float) > a->workspace_bytes) return RADAR_ERR_WORKSPACE;
    float* feat_pre = reinterpret_cast<float*>(reinterpret_cast<char*>(a->workspace) + row_bytes);
    if (gate_runs && a->policy == RADAR_POLICY_LSTM_HIDDEN && a->phase != RADAR_EXPAND_SELECT) {
        RADAR_CUDA_CHECK(gate_features_launch(ctx, *a, feat_pre, stream));
    }

    row_topk_carve(rp, a->workspace);
    if (a->phase != RADAR_EXPAND_SELECT) RADAR_CUDA_CHECK(row_topk_launch(ctx, rp, stream));
    if (a->phase == RADAR_EXPAND_VOCAB) return RADAR_OK;
    SelectParams sp;
    sp.a = *a;
    sp.split = a->phase == RADAR_EXPAND_SELECT ? 1 : 0;
    sp.row_tok = rp.tok;
    sp.row_logp = rp.logp;
    sp.feat_pre = feat_pre;
    sp.feat_hid = feat_pre + (size_t)a->B * 4 * kHidden;
    sp.status = ctx->d_status;
    const bool recurrent = gate_runs && a->policy != RADAR_POLICY_MLP_SCORES;
    const size_t weights = gate_runs && a->policy != RADAR_POLICY_LSTM_HIDDEN ? sizeof(float) * (size_t)((recurrent ? 4 : 1) * kHidden) * (a->k | 1) : 0;
    // Blocks per sequence.  With a recurrent policy, three more blocks per sequence hold W_hh in their registers, loaded while
    // the predecessors still run, and deliver W_hh h + biases into block 0.  That pays while the draft calls are a chain of short,
    // latency-bound kernels; with longer passes they only take SMs from the pass that runs beside this kernel.
    const bool short_pass = (long long)a->B * a->k * a->V <= kShortPassLogits;
    const int cluster = recurrent && a->t > 1 && short_pass && a->B * kSelCluster * 2 <= ctx->sm_count ? kSelCluster : 1;
    radar_launch_scope scope(ctx, RADAR_K_SELECT_GATE, stream);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(a->B * cluster));
    cfg.blockDim = dim3(kSelThreads);
    cfg.dynamicSmemBytes = weights;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    if (cluster > 1) {
        RADAR_CUDA_CHECK(radar_opt_in_smem(ctx, RADAR_SMEM_SELECT_GATE_CLUSTER, expand_select_gate_kernel<true>, weights));
        RADAR_CUDA_CHECK(cudaLaunchKernelEx(&cfg, expand_select_gate_kernel<true>, sp));
    } else {
        RADAR_CUDA_CHECK(radar_opt_in_smem(ctx, RADAR_SMEM_SELECT_GATE, expand_select_gate_kernel<false>, weights));
        RADAR_CUDA_CHECK(cudaLaunchKernelEx(&cfg, expand_select_gate_kernel<false>, sp));
    }
    RADAR_CUDA_CHECK(cudaGetLastError());
    return RADAR_OK;
}
