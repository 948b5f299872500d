// One REINFORCE step of the prediction model (Sec. 4.2, Eq. 3-10; data points {S, D} of Sec. 4.3).
//
// Three kernels:
//   train_rollout_kernel   one block per one, two or four data points: rolls the LSTM + MLP out over the states with
//                          sampled actions, draws the acceptance length from d_T, forms the returns, and runs
//                          backpropagation through time.  What the parameter gradients need - the deltas of
//                          every layer and the activations they multiply - goes to a record per (data point,
//                          decision) in the workspace.
//   train_outer_kernel     the parameter gradients: sums over all records of delta (x) activation, one output
//                          tile and one slice of the records per block, each slice in a fixed order into its own
//                          partial buffer (no atomics: the result does not depend on scheduling).
//   train_adam_kernel      adds the slices up (fixed order), batch loss (fixed-order sum) and the Adam update.
// The network is the one expand.cu runs at inference; the forward arithmetic is fp32 like there.
#include "common.cuh"

namespace radar {
namespace {

constexpr int H = kHidden;            // 128
constexpr int kTrainThreads = 4 * H;  // one thread per LSTM gate row
constexpr int kMaxSteps = 16;
constexpr int kGroups = kTrainThreads / 32;   // row groups of the rollout's transposed products
constexpr int kXPad = 32;             // room for the k scores behind h in the head's input
constexpr int kSlices = 8;            // the records are summed in this many slices, one block each per output tile

// record of one decision (floats)
constexpr int R_DPRE = 0;                       // [4H] delta of the LSTM pre-activations
constexpr int R_DPRE1 = R_DPRE + 4 * H;         // [H]  delta of the head's hidden pre-activations
constexpr int R_DY = R_DPRE1 + H;               // [2]  delta of the logits (+2 padding)
constexpr int R_HPREV = R_DY + 4;               // [H]  h before the step
constexpr int R_CAT = R_HPREV + H;              // [H + kXPad]  h after the step, then the k scores
constexpr int R_HID = R_CAT + H + kXPad;        // [H]  relu output
constexpr int R_GATES = R_HID + H;              // [4H] i, f, g, o after their non-linearities
constexpr int R_C = R_GATES + 4 * H;            // [H]  c after the step
constexpr int R_CPREV = R_C + H;                // [H]
constexpr int R_STRIDE = R_CPREV + H;

struct Theta {
    float *w_ih, *w_hh, *b_ih, *b_hh, *w1, *b1, *w2, *b2;
};
__host__ __device__ inline Theta carve_theta(float* t, int k) {
    Theta o;
    o.w_ih = t;
    o.w_hh = o.w_ih + (size_t)4 * H * k;
    o.b_ih = o.w_hh + (size_t)4 * H * H;
    o.b_hh = o.b_ih + 4 * H;
    o.w1 = o.b_hh + 4 * H;
    o.b1 = o.w1 + (size_t)H * (H + k);
    o.w2 = o.b1 + H;
    o.b2 = o.w2 + 2 * H;
    return o;
}
__host__ __device__ inline size_t param_count(int k) { return (size_t)4 * H * k + 4 * H * H + 8 * H + (size_t)H * (H + k) + H + 2 * H + 2; }

struct TrainParams {
    radar_train_args a;
    float* rec;          // [n][t_max - 1][R_STRIDE]
    int* ndec;           // [n] decisions taken
    float* point_loss;   // [n]
    float* part;         // [kSlices][parameters] partial gradient sums
};

__device__ __forceinline__ float sigmoidf(float v) { return 1.f / (1.f + __expf(-v)); }
__device__ __forceinline__ void copy4(float* smem, const float* gmem) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(gmem) : "memory");
}
__device__ __forceinline__ void copy16(float* smem, const float* gmem) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(gmem) : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int kLeft>
__device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(kLeft) : "memory"); }
__device__ __forceinline__ float softplusf(float v) { return v > 0.f ? v + log1pf(expf(-v)) : log1pf(expf(v)); }

// A block takes kP data points side by side.  What bounds it is the way of the weights from L2 into the SM (256 KB of W_hh
// and 70 KB of W_1 for every decision, forwards and backwards, 64 B a clock) and the latency of that way: the points of
// a block share every weight that is loaded, and a thread has eight or more loads of a product in flight.  With one point
// a block, a row at a time and five shuffles a row, n = 148 took 134 us and n = 1024 332; now 65 and 139.
// W_1, W_ih, the states and the uniform numbers are in shared memory before the first decision, so that W_hh is all that is
// read again for every one (and not for the first: its h is zero).  Whole step, us, before / after: 256 points that
// make one call 31.2 / 27.0, 64 points of two calls on average 76.9 / 68.5, 1024 of them 211 / 205.
template <int kP>
__global__ void __launch_bounds__(kTrainThreads, 1) train_rollout_kernel(const TrainParams P) {
    chain_wait();
    const radar_train_args& a = P.a;
    const int j0 = blockIdx.x * kP, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int k = a.k, t_max = a.t_max, n = a.n;
    const Theta W = carve_theta(a.theta, k);
    __shared__ __align__(16) float sh[kP][H], sc[kP][H], sx[kP][kXPad], sg[kP][4 * H], shid[kP][H], sd1[kP][H], sdp[kP][4 * H], sdh[kP][H], sdc[kP][H];
    extern __shared__ __align__(16) float train_smem[];
    float (*spart)[kGroups][H] = reinterpret_cast<float (*)[kGroups][H]>(train_smem);      // [kP]
    float* s_w1 = train_smem + kP * kGroups * H;         // [H][H + k]
    float* s_wih = s_w1 + H * (H + k);                   // [4H][k]
    float* s_state = s_wih + 4 * H * k;                  // [kP][t_max - 1][k] log states
    __shared__ float sy[kP][2], spi1[kP][kMaxSteps], sG[kP][kMaxSteps], s_u[kP][kMaxSteps];
    __shared__ double s_dist[kP][kMaxSteps + 1];
    __shared__ int sact[kP][kMaxSteps], sT[kP], sndec[kP], s_going[kP];
    // What every decision needs, once: the head's and the input's weights, all states, the uniform numbers.  (Fetched where they are
    // used, each is a wait of a microsecond in the chain of every decision.)
    for (int e = tid; e < 4 * H * k / 4; e += kTrainThreads) copy16(s_wih + 4 * e, W.w_ih + 4 * e);
    for (int e = tid; e < kP * (t_max - 1) * k; e += kTrainThreads) {
        const int p = e / ((t_max - 1) * k), r = e % ((t_max - 1) * k);
        if (j0 + p < n) copy4(s_state + e, a.log_states + ((size_t)(r / k) * n + j0 + p) * k + r % k);
    }
    for (int e = tid; e < kP * (t_max - 1); e += kTrainThreads) {
        const int p = e / (t_max - 1), r = e % (t_max - 1);
        if (j0 + p < n) copy4(&s_u[p][r], a.u_action + (size_t)(j0 + p) * t_max + r);
    }
    copies_commit();
    for (int e = tid; e < H * (H + k) / 4; e += kTrainThreads) copy16(s_w1 + 4 * e, W.w1 + 4 * e);
    copies_commit();
    for (int e = tid; e < kP * H; e += kTrainThreads) { (&sh[0][0])[e] = 0.f; (&sc[0][0])[e] = 0.f; }
    if (tid < kP) { s_going[tid] = j0 + tid < n; sT[tid] = t_max; sndec[tid] = 0; }
    copies_wait<1>();                                    // all but the head's weights
    __syncthreads();
    auto record = [&](int p, int s) { return P.rec + ((size_t)(j0 + p) * (t_max - 1) + s) * R_STRIDE; };

    // ---- rollout ----
    for (int t = 1; t < t_max; ++t) {
        bool going[kP], any = false;                          // the same in every thread
#pragma unroll
        for (int p = 0; p < kP; ++p) { going[p] = s_going[p] != 0; any |= going[p]; }
        if (!any) break;
        for (int e = tid; e < kP * kXPad; e += kTrainThreads) {
            const int p = e / kXPad, c = e % kXPad;
            sx[p][c] = c < k && going[p] ? __expf(s_state[(p * (t_max - 1) + t - 1) * k + c]) : 0.f;
        }
        for (int e = tid; e < kP * H; e += kTrainThreads) {
            const int p = e / H, c = e % H;
            if (going[p]) {
                float* rec = record(p, t - 1);
                rec[R_HPREV + c] = sh[p][c];
                rec[R_CPREV + c] = sc[p][c];
            }
        }
        __syncthreads();
        // LSTM pre-activations: warp w owns rows 32 w .. 32 w + 31 in two batches of 16, the lanes share each row's dot
        // product; even lanes end up with a row of the first batch, odd lanes with one of the second
        float mine[kP];
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const int r0 = warp * 32 + half * 16;
            const float* wx = s_wih + r0 * k + lane;
            if (t == 1) {                                     // the state before the first call is zero
#pragma unroll
                for (int p = 0; p < kP; ++p) {
                    const float x = sx[p][lane];
                    float v[16];
#pragma unroll
                    for (int i = 0; i < 16; ++i) v[i] = lane < k ? wx[i * k] * x : 0.f;
                    const float sum = transposed_sum<16>(v);
                    if ((lane & 1) == half) mine[p] = sum;
                }
                continue;
            }
            float4 w[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) w[i] = *reinterpret_cast<const float4*>(W.w_hh + (size_t)(r0 + i) * H + 4 * lane);
            float wr[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) wr[i] = lane < k ? wx[i * k] : 0.f;
#pragma unroll
            for (int p = 0; p < kP; ++p) {
                const float4 h4 = *reinterpret_cast<const float4*>(&sh[p][4 * lane]);
                const float x = sx[p][lane];
                float v[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) v[i] = fmaf(wr[i], x, w[i].x * h4.x + w[i].y * h4.y + w[i].z * h4.z + w[i].w * h4.w);
                const float sum = transposed_sum<16>(v);
                if ((lane & 1) == half) mine[p] = sum;
            }
        }
        {
            const int row = warp * 32 + (lane & 1) * 16 + (lane >> 1);
            const float b = W.b_ih[row] + W.b_hh[row];
#pragma unroll
            for (int p = 0; p < kP; ++p) {
                const float pre = mine[p] + b;
                const float g = (row >= 2 * H && row < 3 * H) ? tanhf(pre) : sigmoidf(pre);
                sg[p][row] = g;
                if (going[p]) record(p, t - 1)[R_GATES + row] = g;
            }
        }
        __syncthreads();
        for (int e = tid; e < kP * (H + kXPad); e += kTrainThreads) {
            const int p = e / (H + kXPad), c = e % (H + kXPad);
            if (!going[p]) continue;
            float* rec = record(p, t - 1);
            if (c < H) {
                const float cn = sg[p][H + c] * sc[p][c] + sg[p][c] * sg[p][2 * H + c];
                const float hn = sg[p][3 * H + c] * tanhf(cn);
                sc[p][c] = cn;
                sh[p][c] = hn;
                rec[R_C + c] = cn;
                rec[R_CAT + c] = hn;
            } else {
                rec[R_CAT + c] = sx[p][c - H];
            }
        }
        if (t == 1) copies_wait<0>();
        __syncthreads();
        // head: warp w owns hidden rows 8 w .. 8 w + 7
        {
            float w[8][4], wx[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float* wr = s_w1 + (warp * 8 + i) * (H + k);
#pragma unroll
                for (int c = 0; c < 4; ++c) w[i][c] = wr[lane + 32 * c];
                wx[i] = lane < k ? wr[H + lane] : 0.f;
            }
            const int row = warp * 8 + (lane >> 2);
            const float b1 = W.b1[row];
#pragma unroll
            for (int p = 0; p < kP; ++p) {
                float v[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    v[i] = wx[i] * sx[p][lane];
#pragma unroll
                    for (int c = 0; c < 4; ++c) v[i] = fmaf(w[i][c], sh[p][lane + 32 * c], v[i]);
                }
                const float hv = fmaxf(transposed_sum<8>(v) + b1, 0.f);
                if ((lane & 3) == 0) {
                    shid[p][row] = hv;
                    if (going[p]) record(p, t - 1)[R_HID + row] = hv;
                }
            }
        }
        __syncthreads();
        if (warp < 2 * kP) {
            const int p = warp >> 1, o = warp & 1;
            float v = 0.f;
            for (int c = lane; c < H; c += 32) v += W.w2[o * H + c] * shid[p][c];
            v = warp_sum(v);
            if (lane == 0) sy[p][o] = v + W.b2[o];
        }
        __syncthreads();
        if (tid < kP && going[tid]) {
            const int p = tid;
            const float d = sy[p][1] - sy[p][0];
            const float pi1 = 1.f / (1.f + expf(-d));
            const int act = s_u[p][t - 1] < pi1 ? 1 : 0;
            spi1[p][t - 1] = pi1;
            sact[p][t - 1] = act;
            sG[p][t - 1] = act ? -softplusf(-d) : -softplusf(d);       // log pi(a_t) for now
            sndec[p] = t;
            if (!act) { sT[p] = t; s_going[p] = 0; }
        }
        __syncthreads();
    }
    __syncthreads();
    if (warp < kP && j0 + warp < n && lane <= t_max) s_dist[warp][lane] = a.dists[((size_t)(sT[warp] - 1) * n + j0 + warp) * (t_max + 1) + lane];
    __syncthreads();

    // ---- acceptance length, reward, returns, loss (one thread per point, fp64) ----
    if (tid < kP && j0 + tid < n) {
        const int p = tid, j = j0 + p, T = sT[p], ndec = sndec[p];
        const double* drow = s_dist[p];
        double total = 0.0;
        for (int i = 0; i <= t_max; ++i) total += drow[i];
        const double target = (double)a.u_length[j] * total;
        double run = 0.0;
        int len = -1, last_pos = -1;
        for (int i = 0; i <= t_max; ++i) {
            run += drow[i];
            if (drow[i] > 0.0) last_pos = i;
            if (run > target) { len = i; break; }
        }
        if (len < 0) len = last_pos;
        const double t_pred = (double)a.T_p * (T < t_max ? T + 1 : T);
        const double reward_T = (double)len / ((double)a.T_o + (double)a.T_d * T + t_pred);
        // G_t = r_t + gamma G_{t+1}, backwards from the last call
        double g = reward_T, loss = 0.0;
        for (int t = T; t >= 1; --t) {
            if (t < T) g = -(double)a.alpha + (double)a.gamma * g;
            if (t <= ndec) {
                loss -= g * (double)sG[p][t - 1];
                sG[p][t - 1] = (float)g;
            }
        }
        P.point_loss[j] = (float)loss;
        P.ndec[j] = ndec;
        a.calls[j] = T;
        a.l_acc[j] = len;
        for (int t = 1; t <= t_max; ++t) a.actions[(size_t)j * t_max + (t - 1)] = t <= ndec ? (uint8_t)sact[p][t - 1] : (uint8_t)255;
    }
    for (int e = tid; e < kP * H; e += kTrainThreads) { (&sdh[0][0])[e] = 0.f; (&sdc[0][0])[e] = 0.f; }
    __syncthreads();
    int steps = 0;
#pragma unroll
    for (int p = 0; p < kP; ++p) steps = max(steps, sndec[p]);

    // ---- backpropagation through time (a point joins at its own last decision) ----
    const int q = tid >> 7, col = tid & (H - 1);
    static_assert(kP * H <= kTrainThreads, "one unit of one point to a thread");
    for (int s = steps - 1; s >= 0; --s) {
        // what the cell's derivative takes from the record, on its way while the head's is worked out
        const int up = tid / H, uc = tid % H;
        const bool mine = up < kP && s < sndec[up < kP ? up : 0];
        float gi = 0.f, gf = 0.f, gg = 0.f, go = 0.f, cell = 0.f, cell_before = 0.f;
        if (mine) {
            const float* rec = record(up, s);
            gi = rec[R_GATES + uc]; gf = rec[R_GATES + H + uc]; gg = rec[R_GATES + 2 * H + uc]; go = rec[R_GATES + 3 * H + uc];
            cell = rec[R_C + uc]; cell_before = rec[R_CPREV + uc];
        }
        for (int e = tid; e < kP * H; e += kTrainThreads) {
            const int p = e / H, c = e % H;
            float v = 0.f;
            if (s < sndec[p]) {
                float* rec = record(p, s);
                const float G = sG[p][s], pi1 = spi1[p][s];
                const int act = sact[p][s];
                const float dy0 = -G * ((act == 0 ? 1.f : 0.f) - (1.f - pi1));
                const float dy1 = -G * ((act == 1 ? 1.f : 0.f) - pi1);
                if (c == 0) { rec[R_DY] = dy0; rec[R_DY + 1] = dy1; }
                v = rec[R_HID + c] > 0.f ? W.w2[c] * dy0 + W.w2[H + c] * dy1 : 0.f;
                rec[R_DPRE1 + c] = v;
            }
            sd1[p][c] = v;
        }
        __syncthreads();
        {   // dh = W1[:, :H]^T dpre1 + dh from the next step: thread (q, col) sums 32 rows
            float acc[kP];
#pragma unroll
            for (int p = 0; p < kP; ++p) acc[p] = 0.f;
#pragma unroll 16
            for (int r = q * 32; r < q * 32 + 32; ++r) {
                const float w = s_w1[r * (H + k) + col];
#pragma unroll
                for (int p = 0; p < kP; ++p) acc[p] += w * sd1[p][r];
            }
#pragma unroll
            for (int p = 0; p < kP; ++p) spart[p][q][col] = acc[p];
        }
        __syncthreads();
        if (up < kP) {
            const int p = up, c = uc;
            float di = 0.f, df = 0.f, dg = 0.f, dob = 0.f;
            if (mine) {
                float* rec = record(p, s);
                const float dh = spart[p][0][c] + spart[p][1][c] + spart[p][2][c] + spart[p][3][c] + sdh[p][c];
                const float tc = tanhf(cell);
                const float dc = dh * go * (1.f - tc * tc) + sdc[p][c];
                di = dc * gg * gi * (1.f - gi); df = dc * cell_before * gf * (1.f - gf);
                dg = dc * gi * (1.f - gg * gg); dob = dh * tc * go * (1.f - go);
                rec[R_DPRE + c] = di; rec[R_DPRE + H + c] = df; rec[R_DPRE + 2 * H + c] = dg; rec[R_DPRE + 3 * H + c] = dob;
                sdc[p][c] = dc * gf;
            }
            sdp[p][c] = di; sdp[p][H + c] = df; sdp[p][2 * H + c] = dg; sdp[p][3 * H + c] = dob;
        }
        if (s == 0) break;                                    // the state before the first call is a constant
        __syncthreads();
        {   // dh for the step before: W_hh^T dpre; thread (warp, lane) sums 32 rows of four columns
            float4 acc[kP];
#pragma unroll
            for (int p = 0; p < kP; ++p) acc[p] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 16
            for (int i = 0; i < 32; ++i) {
                const int r = warp * 32 + i;
                const float4 w = *reinterpret_cast<const float4*>(W.w_hh + (size_t)r * H + 4 * lane);
#pragma unroll
                for (int p = 0; p < kP; ++p) {
                    const float d = sdp[p][r];
                    acc[p].x += w.x * d; acc[p].y += w.y * d; acc[p].z += w.z * d; acc[p].w += w.w * d;
                }
            }
#pragma unroll
            for (int p = 0; p < kP; ++p) *reinterpret_cast<float4*>(&spart[p][warp][4 * lane]) = acc[p];
        }
        __syncthreads();
        for (int e = tid; e < kP * H; e += kTrainThreads) {
            const int p = e / H, c = e % H;
            float v = 0.f;
#pragma unroll
            for (int g = 0; g < kGroups; ++g) v += spart[p][g][c];
            sdh[p][c] = v;                                    // (zero for a point that has not joined: its sdp was)
        }
        __syncthreads();
    }
}

// out[m][c] = sum over valid records of A[rec][m] * B[rec][c], c < N; column N of B is ones, and its sums are the biases'
struct OuterJob {
    int a_off, M, b_off, N;     // offsets into a record
    int first;                  // first decision whose record counts (1: B is zero before the first call)
    long long out_off;          // [M][N] in grad
    long long bias_off[2];      // [M] each, or -1
};
constexpr int kJobs = 4;
constexpr int kTile = 64, kBatchRecs = 32;
struct OuterParams {
    OuterJob job[kJobs];
    int first[kJobs + 1];       // first output tile of each job (and their number)
    const float* rec;
    const int* ndec;
    float* part;                // [kSlices][count]
    long long count;
    int n, steps;               // records per data point = t_max - 1
};

// Block (tile, slice): a 64 x 64 tile of one output, four by four to a thread, summed over the records of the slice's data points.
// Only decisions that were taken have a record, on average two of a point's t_max - 1: the block lists them first, 256 points at a
// time, and goes through the list in batches of 32 (in the order of the points, so the sum does not depend on
// scheduling).  Visiting every possible record cost 60 us at 256 points and 205 at 1024; the list 23 and 57.  What bounds it is the
// issue of instructions: with four products a thread, nine instructions for them, 32 x 32 tiles and the biases as
// tiles of their own, 256 points of one / two calls took 12.8 / 21.0 us, now 10.7 / 13.5; 1024 points 31.3 / 50.5, now 19.8 / 29.2.
__global__ void __launch_bounds__(256) train_outer_kernel(const OuterParams P) {
    chain_wait();
    int job = 0;
    while ((int)blockIdx.x >= P.first[job + 1]) ++job;
    const OuterJob J = P.job[job];
    const int tile = blockIdx.x - P.first[job], columns = J.bias_off[0] >= 0 ? J.N + 1 : J.N, tiles_x = (columns + kTile - 1) / kTile;
    const int m0 = tile / tiles_x * kTile, c0 = tile % tiles_x * kTile;
    __shared__ __align__(16) float As[kBatchRecs][kTile], Bs[kBatchRecs][kTile];
    __shared__ int s_rec[256 * (kMaxSteps - 1)], s_sum[8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, tx = tid & 15, ty = tid >> 4;
    float acc[4][4] = {};
    const int p_end = (int)((long long)P.n * (blockIdx.y + 1) / kSlices);
    for (int p0 = (int)((long long)P.n * blockIdx.y / kSlices); p0 < p_end; p0 += 256) {
        // list of the records of points p0 .. p0 + 255
        const int pt = p0 + tid;
        const int mine = pt < p_end ? max(P.ndec[pt] - J.first, 0) : 0;
        int incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += v;
        }
        __syncthreads();                                        // the previous list has been read
        if (lane == 31) s_sum[warp] = incl;
        __syncthreads();
        int at = incl - mine, total = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            if (w < warp) at += s_sum[w];
            total += s_sum[w];
        }
        for (int s = 0; s < mine; ++s) s_rec[at + s] = pt * P.steps + J.first + s;
        __syncthreads();
        for (int r0 = 0; r0 < total; r0 += kBatchRecs) {
            // 32 records x 64 columns of each operand; past the list zero, past the edges whatever the record holds there
            // (those sums are not kept)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int e = ty + 16 * i;
                float4 av = make_float4(0.f, 0.f, 0.f, 0.f), bv = av;
                if (r0 + e < total) {
                    const float* rec = P.rec + (size_t)s_rec[r0 + e] * R_STRIDE + 4 * tx;
                    av = *reinterpret_cast<const float4*>(rec + J.a_off + m0);
                    bv = *reinterpret_cast<const float4*>(rec + J.b_off + c0);
                    const int one = J.N - c0 - 4 * tx;
                    if (one == 0) bv.x = 1.f;
                    if (one == 1) bv.y = 1.f;
                    if (one == 2) bv.z = 1.f;
                    if (one == 3) bv.w = 1.f;
                }
                *reinterpret_cast<float4*>(&As[e][4 * tx]) = av;
                *reinterpret_cast<float4*>(&Bs[e][4 * tx]) = bv;
            }
            __syncthreads();
            const int live = min(kBatchRecs, total - r0);
#pragma unroll 4
            for (int e = 0; e < live; ++e) {
                const float4 av = *reinterpret_cast<const float4*>(&As[e][4 * ty]), bv = *reinterpret_cast<const float4*>(&Bs[e][4 * tx]);
                const float x[4] = {av.x, av.y, av.z, av.w}, y[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[i][j] += x[i] * y[j];
            }
            __syncthreads();
        }
    }
    float* out = P.part + (long long)blockIdx.y * P.count;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int m = m0 + 4 * ty + i;
        if (m >= J.M) break;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int c = c0 + 4 * tx + j;
            if (c < J.N) out[J.out_off + (long long)m * J.N + c] = acc[i][j];
            if (c == J.N) {
                if (J.bias_off[0] >= 0) out[J.bias_off[0] + m] = acc[i][j];
                if (J.bias_off[1] >= 0) out[J.bias_off[1] + m] = acc[i][j];
            }
        }
    }
}

__global__ void __launch_bounds__(256) train_adam_kernel(const TrainParams P, size_t count) {
    chain_wait();
    const radar_train_args& a = P.a;
    if (blockIdx.x == gridDim.x - 1) {
        // the last block: batch loss, a fixed-order sum
        __shared__ double part[256];
        double s = 0.0;
        for (int j = threadIdx.x; j < a.n; j += 256) s += (double)P.point_loss[j];
        part[threadIdx.x] = s;
        __syncthreads();
        for (int o = 128; o > 0; o >>= 1) {
            if (threadIdx.x < o) part[threadIdx.x] += part[threadIdx.x + o];
            __syncthreads();
        }
        if (threadIdx.x == 0) a.loss[0] = (float)(part[0] / a.n);
        return;
    }
    const float c1 = 1.f - powf(a.beta1, (float)max(a.step, 1)), c2 = 1.f - powf(a.beta2, (float)max(a.step, 1));
    const float scale = 1.f / (float)a.n;
    const size_t i = (size_t)blockIdx.x * 256 + threadIdx.x;            // one parameter a thread: every load in flight at once
    if (i >= count) return;
    const bool update = a.step >= 1;
    float part_sum[kSlices];
#pragma unroll
    for (int sl = 0; sl < kSlices; ++sl) part_sum[sl] = P.part[(size_t)sl * count + i];
    const float m0 = update ? a.adam_m[i] : 0.f, v0 = update ? a.adam_v[i] : 0.f, theta = update ? a.theta[i] : 0.f;
    float g = 0.f;
#pragma unroll
    for (int sl = 0; sl < kSlices; ++sl) g += part_sum[sl];
    g *= scale;
    a.grad[i] = g;
    if (!update) return;
    const float m = a.beta1 * m0 + (1.f - a.beta1) * g;
    const float v = a.beta2 * v0 + (1.f - a.beta2) * g * g;
    a.adam_m[i] = m;
    a.adam_v[i] = v;
    a.theta[i] = theta - a.lr * (m / c1) / (sqrtf(v / c2) + a.eps);
}

}  // namespace
}  // namespace radar

using namespace radar;

extern "C" size_t radar_policy_param_count(int k) { return k >= 1 && k <= RADAR_MAX_K ? param_count(k) : 0; }

extern "C" size_t radar_train_workspace_bytes(const radar_ctx*, int n, int k, int t_max) {
    if (n < 1 || k < 1 || t_max < 2) return 0;
    return align_up((size_t)n * (t_max - 1) * R_STRIDE * sizeof(float), 256) + align_up((size_t)n * sizeof(int), 256) +
           align_up((size_t)n * sizeof(float), 256) + align_up((size_t)kSlices * param_count(k) * sizeof(float), 256);
}

extern "C" int radar_policy_train_step(radar_ctx* ctx, const radar_train_args* a, void* stream_) {
    if (!ctx || !a) return RADAR_ERR_INVALID_ARG;
    if (a->n < 1 || a->k < 1 || a->k > RADAR_MAX_K || a->t_max < 2 || a->t_max > kMaxSteps) return RADAR_ERR_INVALID_ARG;
    if (!a->log_states || !a->dists || !a->u_action || !a->u_length || !a->theta || !a->grad || !a->loss || !a->calls ||
        !a->l_acc || !a->actions || !a->workspace)
        return RADAR_ERR_INVALID_ARG;
    if (a->step < 0 || (a->step >= 1 && (!a->adam_m || !a->adam_v))) return RADAR_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(a->theta) & 15) || (reinterpret_cast<uintptr_t>(a->workspace) & 15)) return RADAR_ERR_INVALID_ARG;
    if (a->workspace_bytes < radar_train_workspace_bytes(ctx, a->n, a->k, a->t_max)) return RADAR_ERR_WORKSPACE;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    TrainParams P;
    P.a = *a;
    unsigned char* w = static_cast<unsigned char*>(a->workspace);
    P.rec = reinterpret_cast<float*>(w);
    w += align_up((size_t)a->n * (a->t_max - 1) * R_STRIDE * sizeof(float), 256);
    P.ndec = reinterpret_cast<int*>(w);
    w += align_up((size_t)a->n * sizeof(int), 256);
    P.point_loss = reinterpret_cast<float*>(w);
    w += align_up((size_t)a->n * sizeof(float), 256);
    P.part = reinterpret_cast<float*>(w);
    const int k = a->k;
    {
        radar_launch_scope scope(ctx, RADAR_K_TRAIN_ROLLOUT, stream);
        const unsigned n = (unsigned)a->n, sms = (unsigned)ctx->sm_count;
        // Points per block: one wave of blocks, four points at most.  Whole step in us with 1 / 2 / 4 points a block, where the
        // trajectories are 2, 3.1 and 6.8 calls long on average (a gate that has been trained makes 5 to 7):
        //   n = 200   91 / 95 / 117    105 / 99 / 123    165 / 115 / 139
        //   n = 290   106 / 99 / 121   132 / 114 / 137   184 / 135 / 160
        //   n = 310   97 / 99 / 121    137 / 126 / 139   188 / 183 / 160
        //   n = 420   122 / 117 / 131  158 / 149 / 144   255 / 220 / 180
        //   n = 592   146 / 137 / 140  200 / 192 / 159   351 / 258 / 214
        //   n = 1024  220 / 207 / 212  308 / 281 / 275   552 / 450 / 370
        // A block lasts as long as its longest trajectory, so with short, mixed ones two points would do a little longer.
        const int kp = n <= sms ? 1 : n <= 2 * sms ? 2 : 4;
        const size_t smem = ((size_t)kp * kGroups * H + (size_t)H * (H + k) + (size_t)4 * H * k + (size_t)kp * (a->t_max - 1) * k) * sizeof(float);
        auto launch = [&](int slot, auto kernel) {
            const cudaError_t e = radar_opt_in_smem(ctx, RADAR_SMEM_TRAIN_ROLLOUT + slot, kernel, smem);
            return e != cudaSuccess ? e : launch_chained(kernel, dim3((n + kp - 1) / kp), dim3(kTrainThreads), smem, stream, P);
        };
        if (kp == 1) RADAR_CUDA_CHECK(launch(0, train_rollout_kernel<1>));
        else if (kp == 2) RADAR_CUDA_CHECK(launch(1, train_rollout_kernel<2>));
        else RADAR_CUDA_CHECK(launch(2, train_rollout_kernel<4>));
    }
    {
        // offsets of the tensors inside theta / grad
        const long long o_w_ih = 0, o_w_hh = o_w_ih + 4LL * H * k, o_b_ih = o_w_hh + 4LL * H * H, o_b_hh = o_b_ih + 4 * H;
        const long long o_w1 = o_b_hh + 4 * H, o_b1 = o_w1 + (long long)H * (H + k), o_w2 = o_b1 + H, o_b2 = o_w2 + 2 * H;
        OuterParams O = {};
        O.rec = P.rec; O.ndec = P.ndec; O.part = P.part; O.count = (long long)param_count(k); O.n = a->n; O.steps = a->t_max - 1;
        O.job[0] = {R_DPRE, 4 * H, R_CAT + H, k, 0, o_w_ih, {o_b_ih, o_b_hh}};        // w_ih and both LSTM biases: dpre (x) [x; 1]
        O.job[1] = {R_DPRE, 4 * H, R_HPREV, H, 1, o_w_hh, {-1, -1}};                  // w_hh: dpre (x) h before the step
        O.job[2] = {R_DPRE1, H, R_CAT, H + k, 0, o_w1, {o_b1, -1}};                   // w1 and b1: dpre1 (x) [h; x; 1]
        O.job[3] = {R_DY, 2, R_HID, H, 0, o_w2, {o_b2, -1}};                          // w2 and b2: dy (x) [relu output; 1]
        O.first[0] = 0;
        for (int x = 0; x < kJobs; ++x) {
            const OuterJob& J = O.job[x];
            const int columns = J.bias_off[0] >= 0 ? J.N + 1 : J.N;
            O.first[x + 1] = O.first[x] + (J.M + kTile - 1) / kTile * ((columns + kTile - 1) / kTile);
        }
        radar_launch_scope scope(ctx, RADAR_K_TRAIN_OUTER, stream);
        RADAR_CUDA_CHECK(launch_chained(train_outer_kernel, dim3((unsigned)O.first[kJobs], kSlices), dim3(256), 0, stream, O));
    }
    {
        const size_t count = param_count(k);
        radar_launch_scope scope(ctx, RADAR_K_TRAIN_ADAM, stream);
        RADAR_CUDA_CHECK(launch_chained(train_adam_kernel, dim3((unsigned)((count + 255) / 256 + 1)), dim3(256), 0, stream, P, count));
    }
    return RADAR_OK;
}
