// Tree-masked GQA attention for bf16 on the 5th-generation tensor cores (tcgen05 + tensor memory),
// with K/V tiles staged by TMA.
//
// Work decomposition.  All G query heads of one KV head, for all tree rows, form R = n_nodes * G
// query rows (row r = node * G + head-in-group), cut into row blocks of whole nodes, up to 128 rows
// (the MMA M dimension), and these into pairs.  A unit is (sequence, KV head, row-block pair); it has to visit the
// sequence's prefix in tiles of 128 keys plus one tile holding the tree's own 64 keys.  The tiles of
// all units, weighted by their cost, are laid end to end and cut into equal ranges, one per CTA, so
// every CTA gets about the same amount of time whatever the mix of prefix lengths and tree sizes;
// the grid is one CTA per SM.  A CTA therefore works through a few segments (unit, tile range).  A
// unit that falls into one CTA is normalised and written to O directly; the pieces of a unit that
// was cut are written as fp32 partials (m, l, O) and merged by tree_attn_tc_combine_kernel.  When
// there are several pairs per KV head, CTAs alternate between them so that they stream the same K/V
// at the same time and all but the first read hit L2.
//
// Inside the CTA (16 warps; the registers are shared out by warpgroup):
//   warp 12    TMA producer: works out the CTA's segments for itself and, through a ring in shared memory, for the others;
//              per segment the Q rows, then K and V tiles into two rings (128-byte swizzle), in the order the MMA warp
//              consumes them.
//   warp 13    MMA issuer: S = Q K^T into one of two tensor-memory score buffers, and O (+)= P V with P read back from
//              tensor memory (bf16, overlaying S) and V consumed N-major straight from the row-major tile.
//   warps 0-3 / 4-7  softmax groups 0 / 1, one thread per query row: the row's scores from tensor memory into registers,
//              running max with lazy rescaling of the O accumulator, exp2, P back to tensor memory.
//              Unit with two live row blocks: group s owns row block s and sees every tile, so each
//              K/V tile is loaded once for 256 query rows.  Unit with one live row block: the
//              groups take alternate tiles with separate (m, l, O) and are merged at the end.
//              Either way one group's softmax overlaps the other's MMAs.
//   warps 8-11 epilogue: a finished accumulator to O or to the partials, while the others are in the next segment.
//   warps 14, 15 only fill up the producer's warpgroup.
// What is rare (ends of segments, tiles that are not full) shares its code with what is not, or is written as loops: with every
// wait, schedule and mask unrolled in line the kernel had up to 145 KB of code (112 now), a segment's end missed the instruction
// cache all along, and 8.5 thousand cycles lay between a segment's last product and the next one's first.
// Every mbarrier wait is bounded; a wait that runs out sets RADAR_ERR_TIMEOUT on the device status
// word, the CTA drains, frees its tensor memory and returns.
#include <cuda.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "common.cuh"
#include "tc05.cuh"

namespace radar {
namespace {

using namespace tc05;

constexpr int kTcThreads = 512;
constexpr int kEpilogueWarp = 8, kProducerWarp = 12, kMmaWarp = 13;
// Registers a thread: 128 at launch, then shared out by warpgroup (two of softmax; what they take the other two give).
constexpr int kSoftmaxRegs = 176, kEpilogueRegs = 88, kIssueRegs = 72;
static_assert(2 * kSoftmaxRegs + kEpilogueRegs + kIssueRegs <= 512, "a block shares out the registers it was launched with");
constexpr int kStaticSmem = 3072;    // barriers and exchange arrays: with the tiles exactly the 227 KB a block may have
constexpr int kTileKeys = 128;       // keys per prefix tile
constexpr int kFirstKeys = 64;       // keys of a tile whose products start before the rest of its probabilities is there
constexpr int kTreeKeys = 64;        // keys of the tree tile (RADAR_MAX_NODES)
constexpr int kPairRows = 256;       // query rows of a row-block pair (and the stride of partial records)
constexpr long long kLatencyWork = 9 << 15;   // sequences x query heads x keys x head dimension: tree_attn_tc_supported
constexpr float kRescaleThreshold = 8.f;   // in log2 units: P stays below 2^8

// Written by every CTA of the attention kernel, read by the combine kernel: the pieces are worked out by the producer warp
// behind its last load, where nothing waits for it, and not by every warp of the combine (two 64-bit divisions a piece).
constexpr int kMaxPerClass = 160;    // CTAs of a class at most (plan_grid)
struct __align__(16) CutUnit {
    int valid;           // 1: this CTA's last segment starts a unit that continues in the following CTAs
    int b, g, layer;     // the unit
    int slot;            // partial slot of that first piece in this CTA (0 or 1)
    int rows;            // live query rows of the unit
    int n_pieces;        // CTAs of the class from this one on whose range begins before the unit's end
    uint32_t live[kMaxPerClass / 32];    // bit j: piece j's range holds the start of a tile of the unit
};

// ... and what its table of pieces follows from.
struct Cut {
    CutUnit unit;
    long long u0, tot;   // start of the unit, size of the class's space (all layers)
    int nt, w;           // tiles of the unit and their cost
};

struct TcParams {
    radar_attn_args a;
    int G, nodes_per_rb; // a row block holds whole nodes: nodes_per_rb = 128 / G (rounded down) of them
    int rb_rows;         // ... so rb_rows = nodes_per_rb * G of its 128 rows can be live (all of them if G divides 128)
    uint32_t g_magic;    // ceil(2^16 / G): row / G == row * g_magic >> 16 for row < 128 and G <= 128
    int n_blk;           // row blocks of a class's units: 2 (they share each K/V tile) or 1
    int pair_rows;       // query rows of a class's units: n_blk * rb_rows
    int n_layers;        // layers run by this launch (the same tree, masks and prefix lengths for all)
    long long o_ls, lse_ls;   // elements between consecutive layers of O and of lse
    int n_cls;           // classes = units per KV head
    int ncc;             // CTAs per class; grid = n_cls * ncc
    int cost_one, cost_two, unit_cost;   // tile_costs(n_cls)
    float scale_log2;
    float scale_log2_lo; // two parts of P: what scale_log2 is below the scale itself (positive)
    long long cache_rows;
    float2* part_ml;     // [grid][2][256]     (m in natural-log units, with two parts of P in log2 units; l)
    float* part_o;       // [grid][2][256][D]
    CutUnit* cut;        // [grid]
    int* status;
};

__device__ __forceinline__ float max3(float a, float b, float c) {
    float y;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
    return y;
}
// one 32-byte store: a whole sector per lane (the epilogue's lanes write to different rows, so every store
// instruction is split into one transaction per lane; with 16-byte stores each of them filled half a sector)
__device__ __forceinline__ void st_global_32b(void* p, const uint32_t (&w)[8]) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]),
                 "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
                 : "memory");
}
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// the same and the other steps of a probability, kept in the order in which they are written
__device__ __forceinline__ float ex2_in_order(float x) {
    float y;
    asm volatile("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float2 fma2_in_order(float2 a, float2 b, float2 c) {
    float2 d;
    asm volatile("{\n\t.reg .b64 a, b, c, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tmov.b64 c, {%6, %7};\n\t"
                 "fma.rn.f32x2 d, a, b, c;\n\tmov.b64 {%0, %1}, d;\n\t}"
                 : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}
__device__ __forceinline__ float2 add2_in_order(float2 a, float2 b) {
    float2 d;
    asm volatile("{\n\t.reg .b64 a, b, d;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tadd.rn.f32x2 d, a, b;\n\tmov.b64 {%0, %1}, d;\n\t}"
                 : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ uint32_t bf16x2_in_order(float lo, float hi) {
    uint32_t d;
    asm volatile("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}
template <int N> __device__ __forceinline__ void regs_inc() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N)); }
template <int N> __device__ __forceinline__ void regs_dec() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N)); }
// m ln 2 + ln l, m in log2 units
__device__ __forceinline__ float lse_of(float m, float l) {
    constexpr float kHi = 0.693147182f, kLo = (float)(0.6931471805599453 - (double)kHi);
    return fmaf(m, kHi, fmaf(m, kLo, logf(l)));
}

// ---- the tile space of one class (unit index pp within a KV head) ---------------------------------
// Positions are in cost units: a tile of a unit with two live row blocks (four MMAs) weighs cost_two, a tile of
// a unit with one live row block cost_one, and every unit books cost_unit in front of its first tile for what it
// costs beside its tiles (pipeline fill, epilogue), so that a CTA whose range holds several unit starts gets fewer
// tiles; equal position ranges are then about equal amounts of time.  A tile belongs to the CTA whose range
// contains the tile's start position.  The weights are measured, not derived (us a launch with its combine, against 3 : 5 without
// the unit term): several classes per KV head, 3 : 5 + 15: 32 / 8 heads, B = 1, 2048 tokens 18.7 -> 17.1; 64 / 8 heads, B = 8, 2000
// to 8192 tokens, trees of two calls 114 -> 111; one class, 2 : 4 + 12: 32 / 8 heads, B = 32, 4096 to 32768 tokens 780 -> 772.
// It is the unit term that counts; 2 : 4 + 12 everywhere gives 17.3, 103 to 108 and 764, other sets lie within 2 %.
struct TileCosts { int one, two, unit; };
inline TileCosts tile_costs(int n_cls) { return n_cls == 1 ? TileCosts{2, 4, 12} : TileCosts{3, 5, 15}; }

struct SeqInfo {
    int M, Pb, nt;       // tree rows, prefix length, tiles of a unit (prefix tiles + the tree tile)
    int rows;            // live query rows of this class's unit (0: it does not exist for this sequence)
    int w;               // cost of one tile
    long long kv0;
};

template <bool PAGED>
__device__ __forceinline__ SeqInfo seq_info(const TcParams& P, int b, int pp) {
    const radar_attn_args& a = P.a;
    SeqInfo s;
    s.M = min(max(a.n_nodes[b], 0), kMaxNodes);
    s.Pb = a.prefix_len[b];
    s.kv0 = PAGED ? 0 : a.kv_start[b];          // paged: the host has checked max_pages * page_size >= max_prefix_len
    const bool ok = s.Pb >= 0 && s.Pb <= a.max_prefix_len && s.kv0 >= 0 && s.kv0 + s.Pb <= P.cache_rows;
    s.rows = ok ? min(max(s.M * P.G - pp * P.pair_rows, 0), P.pair_rows) : 0;
    s.nt = (max(s.Pb, 0) + kTileKeys - 1) / kTileKeys + 1;
    s.w = s.rows > P.rb_rows ? P.cost_two : P.cost_one;
    return s;
}
template <bool PAGED>
__device__ __forceinline__ long long seq_cost(const TcParams& P, int b, int pp) {
    const SeqInfo s = seq_info<PAGED>(P, b, pp);
    return s.rows > 0 ? (long long)P.a.Hkv * (s.nt * s.w + P.unit_cost) : 0;
}
// number of tiles of a unit (start position U, nt tiles of cost w) that start before position x
__device__ __forceinline__ int tiles_before(long long x, long long U, int nt, int w, int unit_cost) {
    const long long d = x - U - unit_cost;           // clamped first, so that the division is a 32-bit one
    if (d <= 0) return 0;
    if (d >= (long long)nt * w) return nt;
    return ((int)d + w - 1) / w;
}

// One CTA's walk over its range [.., hi) of the class's space: segments (sequence b, KV head g, tiles [t0, t1)).
template <bool PAGED>
struct Cursor {
    int b, g, t0, t1;
    int layer;           // layers follow one another in the space, each with the same sequence of units
    long long U, hi;     // start position of the current unit, end of the CTA's range
    int unit_cost;
    SeqInfo s;
    __device__ __forceinline__ bool valid() const { return t1 > t0; }
    __device__ __forceinline__ void clip() { t1 = tiles_before(hi, U, s.nt, s.w, unit_cost); }
    __device__ __forceinline__ void next_unit(const TcParams& P, int pp) {
        U += (long long)s.nt * s.w + unit_cost;
        t0 = 0;
        if (++g == P.a.Hkv) {
            g = 0;
            do {
                if (++b >= P.a.B) {                               // the next layer starts over at the first sequence
                    if (++layer >= P.n_layers) { t1 = 0; return; }
                    b = 0;
                }
                s = seq_info<PAGED>(P, b, pp);
            } while (s.rows == 0);
        }
        clip();
    }
    __device__ __forceinline__ void next(const TcParams& P, int pp) {
        if (t1 < s.nt) { t0 = t1; return; }                  // the range ended inside this unit
        next_unit(P, pp);
    }
    __device__ __forceinline__ bool complete() const { return t0 == 0 && t1 == s.nt; }
    __device__ __forceinline__ bool two_rb(const TcParams& P) const { return s.rows > P.rb_rows; }
};

// The first segment of CTA ci of a class, by a whole warp: the unit that contains the start of its range, from the unit's first
// tile that starts at or after it.  tot_all: size of the class's space (all layers).
template <bool PAGED>
__device__ __forceinline__ Cursor<PAGED> first_segment(const TcParams& P, int pp, int ci, long long& tot_all) {
    const radar_attn_args& a = P.a;
    const int lane = threadIdx.x & 31;
    long long tot = 0;
#pragma unroll 1
    for (int b0 = 0; b0 < a.B; b0 += 32) {
        const int b = b0 + lane;
        if (pp == 0 && ci == 0 && b < a.B) {
            const int Pb = a.prefix_len[b];
            const long long kv0 = PAGED ? 0 : a.kv_start[b];
            if (Pb < 0 || Pb > a.max_prefix_len || kv0 < 0 || kv0 + Pb > P.cache_rows) set_status(P.status, RADAR_ERR_INVALID_ARG);
        }
        tot += warp_sum(b < a.B ? seq_cost<PAGED>(P, b, pp) : 0ll);
    }
    // the space of all layers: layer l occupies [l * tot, (l + 1) * tot)
    tot_all = tot * P.n_layers;
    const long long lo_all = tot_all * ci / P.ncc;
    Cursor<PAGED> cur;
    cur.hi = tot_all * (ci + 1) / P.ncc;
    cur.unit_cost = P.unit_cost;
    cur.layer = tot > 0 ? (int)(lo_all / tot) : 0;
    cur.t0 = cur.t1 = 0;
    cur.b = -1;
    cur.g = 0;
    cur.U = 0;
    const long long lo = lo_all - (long long)cur.layer * tot;
    long long cum = 0;
#pragma unroll 1
    for (int b0 = 0; b0 < a.B && cur.b < 0; b0 += 32) {
        const int b = b0 + lane;
        const long long sz = b < a.B ? seq_cost<PAGED>(P, b, pp) : 0;
        long long incl = sz;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long v = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += v;
        }
        const unsigned hit = __ballot_sync(kFull, cum + incl > lo);
        if (hit) {
            const int src = __ffs(hit) - 1;
            const long long before = cum + __shfl_sync(kFull, incl - sz, src);
            cur.b = b0 + src;
            cur.s = seq_info<PAGED>(P, cur.b, pp);
            const long long unit = (long long)cur.s.nt * cur.s.w + P.unit_cost;
            cur.g = (int)((lo - before) / unit);
            cur.U = before + cur.g * unit + (long long)cur.layer * tot;
        }
        cum += __shfl_sync(kFull, incl, 31);
    }
    if (cur.b >= 0 && cur.layer < P.n_layers) {
        cur.t0 = tiles_before(lo_all, cur.U, cur.s.nt, cur.s.w, P.unit_cost);
        if (cur.t0 >= cur.s.nt) cur.next_unit(P, pp);       // every tile of that unit starts before the range
        else cur.clip();
    }
    return cur;
}

// What a CTA leaves to the combine, by a whole warp that agrees on `cut`.
__device__ __forceinline__ void write_cut_unit(const TcParams& P, int ci, const Cut& cut) {
    const int lane = threadIdx.x & 31;
    CutUnit* out = P.cut + blockIdx.x;
    int n_pieces = 0;
    if (cut.unit.valid) {
        const long long u0 = cut.u0, tot = cut.tot;
        const int nt = cut.nt, w = cut.w;
        const long long u1 = u0 + (long long)nt * w + P.unit_cost;
#pragma unroll 1
        for (int k = 0; k < kMaxPerClass / 32; ++k) {
            const int c = ci + k * 32 + lane;
            const long long lo = tot * c / P.ncc, hi = tot * (c + 1) / P.ncc;
            const bool piece = c < P.ncc && lo < u1;
            const bool live = piece && tiles_before(hi, u0, nt, w, P.unit_cost) > tiles_before(lo, u0, nt, w, P.unit_cost);
            const uint32_t pieces = __ballot_sync(kFull, piece), bits = __ballot_sync(kFull, live);
            n_pieces += __popc(pieces);
            if (lane == 0) out->live[k] = bits;
            if (pieces != 0xffffffffu) break;
        }
    }
    if (lane == 0) {
        const CutUnit& u = cut.unit;
        out->valid = u.valid; out->b = u.b; out->g = u.g; out->layer = u.layer;
        out->slot = u.slot; out->rows = u.rows; out->n_pieces = n_pieces;
    }
}

// What the other warps know of a segment.
constexpr int kSegRing = 4;
struct __align__(16) Segment {
    int n;                               // tiles; 0: there is no further segment
    int t0, nt, Pb, M, rows;             // first tile, tiles of the unit, prefix length, tree rows, live query rows
    int b, g, layer;
    int pad[3];
};

template <int D, bool TWO>
struct Smem {
    static constexpr int kHalves = D / 64;
    static constexpr int kQBlock = 128 * D * 2;
    static constexpr int kQBytes = (TWO ? 2 : 1) * kQBlock;
    static constexpr int kTileBytes = kTileKeys * D * 2;
    static constexpr int kRingK = 3;
    static constexpr int kRingV = TWO ? 2 : 3;
    static constexpr int kTotal = kQBytes + (kRingK + kRingV) * kTileBytes;
    static constexpr int kDynamic = kTotal;                 // starts on a 1024-byte boundary behind the static block
};

// TWO: the launch may contain units with two live row blocks; decides the shared-memory layout
// PAGED: the prefix cache is read through a block table (a separate instantiation, so that the contiguous
// layout's code is not touched by it)
template <int D, bool TWO, bool PAGED>
__global__ void __launch_bounds__(kTcThreads, 1)
tree_attn_tc_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmKc,
                    const __grid_constant__ CUtensorMap tmVc, const __grid_constant__ CUtensorMap tmKt,
                    const __grid_constant__ CUtensorMap tmVt, const TcParams P) {
    chain_trigger();                     // every warp waits for the predecessor where its role begins; the barrier,
                                         // tensor-memory and descriptor set-up needs nothing from global memory
    using SM = Smem<D, TWO>;
    constexpr int H = SM::kHalves;
    constexpr int RK = SM::kRingK, RV = SM::kRingV;
    const radar_attn_args& a = P.a;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int pp = blockIdx.x % P.n_cls;                    // class
    const int ci = blockIdx.x / P.n_cls;
    const int G = P.G;

    // Static block first (padded to a multiple of 1024 bytes and aligned to it), the tiles behind it: the
    // swizzled tiles need a 1024-byte boundary and there is no room left for alignment slack.
    struct __align__(1024) Static {
        uint64_t bar_qfull, bar_qempty, bar_kfull[3], bar_kempty[3], bar_vfull[3], bar_vempty[3];
        uint64_t bar_sfull[2], bar_odone[2], bar_ofree[2], bar_mlfull, bar_mlempty;
        uint64_t bar_idle;               // every product issued has run
        uint32_t q_last, k_next, v_next, spare[3];   // the producer's: phase parity of the last Q, slot and parity of the next K and V
        uint64_t bar_pfirst[2];          // the probabilities of the tile's first kFirstKeys keys are there
        uint64_t bar_pready[2];          // ... all of them
        uint64_t bar_segfull[kSegRing], bar_segempty[kSegRing];
        Segment seg[kSegRing];
        Cut cut;                         // (paged: the producer's)
        float2 ml[2][128];               // per group: (m in log2 units, l) of the rows at the end of a segment
        uint32_t tmem_base;
        int abort;
        unsigned char pad[kStaticSmem - ((30 + 2 * kSegRing) * 8 + kSegRing * (int)sizeof(Segment) + (int)sizeof(Cut) + 2 * 128 * 8 + 8)];
    };
    static_assert(sizeof(Static) == kStaticSmem, "static shared-memory block");
    __shared__ Static st;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* sQ = smem_raw;
    unsigned char* sK = sQ + SM::kQBytes;
    unsigned char* sV = sK + RK * SM::kTileBytes;

    // ---- set-up ----
    if (warp == 0) {
        if (lane == 0) {
            st.abort = 0;
            mbar_init(&st.bar_qfull, 1);
            mbar_init(&st.bar_qempty, 1);
            for (int i = 0; i < 3; ++i) {
                mbar_init(&st.bar_kfull[i], 1); mbar_init(&st.bar_kempty[i], 1);
                mbar_init(&st.bar_vfull[i], 1); mbar_init(&st.bar_vempty[i], 1);
            }
            for (int i = 0; i < 2; ++i) {
                mbar_init(&st.bar_sfull[i], 1); mbar_init(&st.bar_pfirst[i], 4); mbar_init(&st.bar_pready[i], 4);
                mbar_init(&st.bar_odone[i], 1); mbar_init(&st.bar_ofree[i], 4);
            }
            for (int i = 0; i < kSegRing; ++i) { mbar_init(&st.bar_segfull[i], 1); mbar_init(&st.bar_segempty[i], kProducerWarp + 1); }
            mbar_init(&st.bar_idle, 1);
            st.q_last = 1;
            mbar_init(&st.bar_mlfull, 8);
            mbar_init(&st.bar_mlempty, 4);
            fence_barrier_init();
        }
    } else if (warp == kMmaWarp) {
        tmem_alloc(&st.tmem_base, 512);
        tmem_relinquish();
        if (lane == 0) {
            tma_prefetch_desc(&tmQ); tma_prefetch_desc(&tmKc); tma_prefetch_desc(&tmVc);
            tma_prefetch_desc(&tmKt); tma_prefetch_desc(&tmVt);
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    // All of tensor memory is this CTA's, so its addresses are constants (the producer checks): S/P buffers in columns 0 and
    // 128, O accumulators in 256 and 384.  An address that the compiler does not know to be the same in every lane costs the
    // issuing warp a handful of instructions for every product.
    constexpr uint32_t tmem = 0;
    bool ok = true;                         // no wait of this thread has run out
    // Each role starts with chain_sync(): the bounds of the waits behind it are for this kernel's own work.  (A warp that went
    // straight to its first wait would spend them on whatever is left of the predecessor.)
    // the producer's next segment; false behind the last one
    auto take_segment = [&](uint32_t seg, Segment& s) {
        ok = mbar_wait_while(ok, &st.bar_segfull[seg % kSegRing], (seg / kSegRing) & 1);
        ok = __all_sync(kFull, ok);
        s = st.seg[seg % kSegRing];
        __syncwarp();
        if (lane == 0) mbar_arrive(&st.bar_segempty[seg % kSegRing]);
        return ok && s.n > 0;
    };

    if (warp < kEpilogueWarp) {
        regs_inc<kSoftmaxRegs>();
        chain_sync();
        // =================================== softmax groups ===================================
        // One thread per query row, which holds the tile's 128 scores in registers: tensor memory is read once and no two
        // threads have to agree on a maximum.  (Two threads a row, 64 scores each read twice for want of registers, was the
        // form before: 32 layers, 8 sequences of 6000 to 8192 tokens, 64 / 8 heads 4118 -> 3930 us; one layer of it within a
        // step 307 -> 295; 32 layers of one sequence of 2048 tokens, 32 / 8 heads 105 -> 101.)
        const int grp = warp >> 2;
        const int row = (warp & 3) * 32 + lane;                 // row of the block == tensor-memory lane
        const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t tS = tmem + grp * 128 + lane_addr;
        const uint32_t tO = tmem + 256 + grp * 128 + lane_addr;
        const int rb_node = (int)(((uint32_t)row * P.g_magic) >> 16);        // row / G
        uint32_t sc = 0;                         // S tiles this group has waited for
        Segment s;
        for (uint32_t seg = 0; take_segment(seg, s); ++seg) {
            const bool two = TWO && s.rows > P.rb_rows;
            const int blk = two ? grp : 0;                       // row block within the unit
            const int node = (pp * P.n_blk + blk) * P.nodes_per_rb + rb_node;
            const int rows_here = min(s.rows - blk * P.rb_rows, P.rb_rows);  // live rows of this row block
            // A warp none of whose 32 rows is live does no arithmetic (the products of its rows are never read):
            // it only keeps the barriers going.
            const bool warp_live = row - lane < rows_here;
            // the row's ancestor word is needed by the tree tile only (the unit's last): it is loaded here and first
            // touched there, so that the segment does not start with a wait for global memory
            uint32_t mask_lo, mask_hi;
            asm volatile("ld.global.v2.u32 {%0, %1}, [%2];" : "=r"(mask_lo), "=r"(mask_hi) : "l"(a.mask + (int64_t)s.b * kMaxNodes + min(node, kMaxNodes - 1)));
            const int n_my = two ? s.n : (s.n - grp + 1) >> 1;
            float m_run = -CUDART_INF_F, l_run = 0.f;

#pragma unroll 1
            for (int j = 0; j < n_my; ++j) {
                const int t = s.t0 + (two ? j : 2 * j + grp);
                ok = mbar_wait_while(ok, &st.bar_sfull[grp], sc & 1);
                ok = __all_sync(kFull, ok);                      // warp-uniform: guards .aligned ops
                ++sc;
                tc_fence_after_sync();
                if (ok && warp_live) {
                    uint32_t sv[4][32];
                    const int valid = s.Pb - t * kTileKeys;
                    if (t == s.nt - 1 || valid < kTileKeys) {
                        // Keys that the row may not attend to (and, of the tree tile, which has 64, the columns that are stale)
                        // become -inf in tensor memory, 32 at a time: one tile of a unit or two need it, and an unrolled path
                        // for them would be fetched into the instruction cache anew each time.
#pragma unroll 1
                        for (int c = 0; c < 4; ++c) {
                            uint32_t al;
                            if (t == s.nt - 1) {
                                const int live = s.M - c * 32;
                                al = row < rows_here && c < 2 && live > 0 ? (c == 0 ? mask_lo : mask_hi) & (live >= 32 ? 0xffffffffu : (1u << live) - 1u) : 0u;
                            } else {
                                const int lim = valid - c * 32;
                                al = lim >= 32 ? 0xffffffffu : (lim <= 0 ? 0u : ((1u << lim) - 1u));
                            }
                            tmem_ld32(tS + c * 32, sv[0]);
                            tmem_wait_ld();
#pragma unroll
                            for (int e = 0; e < 32; ++e)
                                if (!((al >> e) & 1u)) sv[0][e] = 0xff800000u;     // -inf
                            tmem_st32(tS + c * 32, sv[0]);
                        }
                        tmem_wait_st();
                    }
#pragma unroll
                    for (int c = 0; c < 4; ++c) tmem_ld32(tS + c * 32, sv[c]);
                    tmem_wait_ld();
                    float mxa[4];
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        mxa[c] = __uint_as_float(sv[c][0]);
#pragma unroll
                        for (int e = 1; e < 31; e += 2)                     // three-input maxima: half the instructions
                            mxa[c] = max3(mxa[c], __uint_as_float(sv[c][e]), __uint_as_float(sv[c][e + 1]));
                        mxa[c] = fmaxf(mxa[c], __uint_as_float(sv[c][31]));
                    }
                    const float mx = fmaxf(max3(mxa[0], mxa[1], mxa[2]), mxa[3]);
                    // ---- running max (log2 units), lazy rescale of the accumulator when some row of the warp moved its max ----
                    const float m_tile = mx * P.scale_log2;
                    float factor = 1.f;
                    if (j == 0) {
                        m_run = m_tile;
                    } else if (m_tile > m_run + kRescaleThreshold) {
                        factor = ex2(m_run - m_tile);           // m_run may be -inf: factor 0 clears O and l
                        m_run = m_tile;
                    }
                    const float m_use = m_run == -CUDART_INF_F ? 0.f : m_run;
                    if (j > 0 && __any_sync(kFull, factor != 1.f)) {
#pragma unroll 1
                        for (int c = 0; c < D; c += 16) {
                            uint32_t o[16];
                            tmem_ld16(tO + c, o);
                            tmem_wait_ld();
#pragma unroll
                            for (int e = 0; e < 16; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * factor);
                            tmem_st16(tO + c, o);
                        }
                    }
                    // ---- P = exp2(s * scale - m), row sum, bf16 pairs back to tensor memory ----
                    // (the scaling and the row sum work on pairs: one packed fp32x2 instruction per two values)
                    // The warp issues in order and an exponential takes its unit 8 cycles: what else there is to do stands between
                    // two of them.
                    float2 ls[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
                    const float2 sc2 = make_float2(P.scale_log2, P.scale_log2), nm2 = make_float2(-m_use, -m_use);
                    uint32_t pk[16];
                    auto scale = [&](const int p) {
                        uint32_t &x = sv[p >> 4][2 * (p & 15)], &y = sv[p >> 4][2 * (p & 15) + 1];
                        const float2 s2 = make_float2(__uint_as_float(x), __uint_as_float(y));
                        const float2 t2 = fma2_in_order(s2, sc2, nm2);
                        x = __float_as_uint(t2.x);
                        y = __float_as_uint(t2.y);
                    };
                    auto finish = [&](const int p) {
                        const float p0 = __uint_as_float(sv[p >> 4][2 * (p & 15)]), p1 = __uint_as_float(sv[p >> 4][2 * (p & 15) + 1]);
                        ls[p & 1] = add2_in_order(ls[p & 1], make_float2(p0, p1));
                        pk[p & 15] = bf16x2_in_order(p0, p1);
                        if ((p & 15) == 15) tmem_st16(tS + (p >> 4) * 16, pk);
                    };
                    // pairs that the scaling is ahead, that the rest is behind, and that the first stores are given to land in
                    constexpr int kAhead = 2, kLag = 4, kLanding = 4;
#pragma unroll
                    for (int p = 0; p < kAhead; ++p) scale(p);
#pragma unroll
                    for (int p = 0; p < 64 + kLag; ++p) {
                        if (p < 64) sv[p >> 4][2 * (p & 15)] = __float_as_uint(ex2_in_order(__uint_as_float(sv[p >> 4][2 * (p & 15)])));
                        if (p + kAhead < 64) scale(p + kAhead);
                        if (p < 64) sv[p >> 4][2 * (p & 15) + 1] = __float_as_uint(ex2_in_order(__uint_as_float(sv[p >> 4][2 * (p & 15) + 1])));
                        if (p >= kLag) finish(p - kLag);
                        if (p == kFirstKeys / 2 - 1 + kLag + kLanding) {
                            tmem_wait_st();
                            tc_fence_before_sync();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(&st.bar_pfirst[grp]);
                        }
                    }
                    l_run = l_run * factor + ((ls[0].x + ls[0].y) + (ls[1].x + ls[1].y));
                    tmem_wait_st();
                }
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) {
                    if (!(ok && warp_live)) mbar_arrive(&st.bar_pfirst[grp]);
                    mbar_arrive(&st.bar_pready[grp]);
                }
            }

            // the rows' (m, l) go to the epilogue, which has taken those of the segment before
            ok = mbar_wait_while(ok, &st.bar_mlempty, (seg & 1) ^ 1);
            st.ml[grp][row] = make_float2(m_run, l_run);
            __syncwarp();
            if (lane == 0) mbar_arrive(&st.bar_mlfull);
        }
    } else if (warp < kProducerWarp) {
        regs_dec<kEpilogueRegs>();
        chain_sync();
        // =================================== epilogue ===================================
        // One thread per tensor-memory lane takes the finished accumulators to O (or to the partials) while the softmax
        // groups and the tensor cores are already in the next segment; each accumulator is handed back as soon as it is read.
        const int row = (warp - kEpilogueWarp) * 32 + lane;
        const uint32_t tO = tmem + 256 + ((uint32_t)((warp - kEpilogueWarp) * 32) << 16);
        const int rb_node = (int)(((uint32_t)row * P.g_magic) >> 16);        // row / G
        uint32_t oc[2] = {0, 0};             // accumulators waited for
        Segment s;
        for (uint32_t seg = 0; take_segment(seg, s); ++seg) {
            const bool two = TWO && s.rows > P.rb_rows;
            const bool final_rows = s.n == s.nt;                 // the whole unit
            const int slot = seg == 0 ? 0 : 1;                   // a CTA has at most a cut first and a cut last segment
            ok = mbar_wait_lazy(ok, &st.bar_mlfull, seg & 1);
            const float2 ml0 = st.ml[0][row], ml1 = st.ml[1][row];
            __syncwarp();
            if (lane == 0) mbar_arrive(&st.bar_mlempty);
#pragma unroll 1
            for (int blk = 0; blk < 2; ++blk) {
                // two live row blocks: accumulator blk is row block blk; one: both belong to it, merged in the first trip
                if (blk == 1 && !two) {
                    if (lane == 0) mbar_arrive(&st.bar_ofree[1]);
                    break;
                }
                ok = mbar_wait_while(ok, &st.bar_odone[blk], oc[blk] & 1);
                ++oc[blk];
                const bool merge = !two && s.n > 1;
                if (merge) {
                    ok = mbar_wait_while(ok, &st.bar_odone[1], oc[1] & 1);
                    ++oc[1];
                }
                ok = __all_sync(kFull, ok);
                tc_fence_after_sync();
                const int rows_here = min(s.rows - blk * P.rb_rows, P.rb_rows);  // live rows of this row block
                const bool row_live = row < rows_here;
                if (ok && row - lane < rows_here) {
                    float m_out = blk == 0 ? ml0.x : ml1.x, l_out = blk == 0 ? ml0.y : ml1.y, w0 = 1.f, w1 = 0.f;
                    if (merge) {
                        m_out = fmaxf(ml0.x, ml1.x);
                        const float ms = m_out == -CUDART_INF_F ? 0.f : m_out;
                        w0 = ex2(ml0.x - ms);                        // exp2(-inf) = 0
                        w1 = ex2(ml1.x - ms);
                        l_out = ml0.y * w0 + ml1.y * w1;
                    }
                    const float m_safe = m_out == -CUDART_INF_F ? 0.f : m_out;
                    const float inv = final_rows ? 1.f / l_out : 1.f;
                    const int node = (pp * P.n_blk + blk) * P.nodes_per_rb + rb_node;
                    const int hq = s.g * G + row - rb_node * G;
                    const int64_t out_row = ((int64_t)s.b * kMaxNodes + node) * a.Hq + hq;
                    const int64_t rec = ((int64_t)blockIdx.x * 2 + slot) * kPairRows + blk * 128 + row;
                    __nv_bfloat16* dst_o = reinterpret_cast<__nv_bfloat16*>(a.O) + s.layer * P.o_ls + out_row * D;
                    float* dst_p = P.part_o + rec * D;                  // 128-byte aligned (workspace carve)
                    const bool wide = (reinterpret_cast<uintptr_t>(dst_o) & 31) == 0;
#pragma unroll 1
                    for (int col = 0; col < D; col += 16) {
                        uint32_t o[16], o2[16];
                        tmem_ld16(tO + blk * 128 + col, o);
                        if (merge) tmem_ld16(tO + 128 + col, o2);
                        tmem_wait_ld();
                        float v[16];
#pragma unroll
                        for (int e = 0; e < 16; ++e) v[e] = __uint_as_float(o[e]) * w0;
                        if (merge) {
#pragma unroll
                            for (int e = 0; e < 16; ++e) v[e] = fmaf(__uint_as_float(o2[e]), w1, v[e]);
                        }
                        if (row_live) {
                            uint32_t w[8];
                            if (final_rows) {
#pragma unroll
                                for (int e = 0; e < 8; ++e) {
                                    const __nv_bfloat162 t2 = __floats2bfloat162_rn(v[2 * e] * inv, v[2 * e + 1] * inv);
                                    w[e] = *reinterpret_cast<const uint32_t*>(&t2);
                                }
                                if (wide) {
                                    st_global_32b(dst_o + col, w);
                                } else {
                                    *reinterpret_cast<uint4*>(dst_o + col) = make_uint4(w[0], w[1], w[2], w[3]);
                                    *reinterpret_cast<uint4*>(dst_o + col + 8) = make_uint4(w[4], w[5], w[6], w[7]);
                                }
                            } else {
#pragma unroll
                                for (int q = 0; q < 2; ++q) {
#pragma unroll
                                    for (int e = 0; e < 8; ++e) w[e] = __float_as_uint(v[q * 8 + e]);
                                    st_global_32b(dst_p + col + q * 8, w);
                                }
                            }
                        }
                    }
                    if (row_live) {
                        const float m_nat = m_safe * 0.6931471805599453f;
                        if (final_rows) {
                            if (a.lse != nullptr) a.lse[s.layer * P.lse_ls + ((int64_t)s.b * a.Hq + hq) * kMaxNodes + node] = m_nat + logf(l_out);
                        } else {
                            P.part_ml[rec] = make_float2(m_out == -CUDART_INF_F ? m_out : m_nat, l_out);
                        }
                    }
                }
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(&st.bar_ofree[blk]);
            }
        }
    } else {
        regs_dec<kIssueRegs>();
        chain_sync();                            // every global access of the CTA comes behind one
        if (warp == kProducerWarp) {
            // =================================== TMA producer ===================================
            // One lane does everything for the contiguous cache.  With a paged cache the whole warp walks the same
            // loop and lane p looks up and fetches page p of a tile (up to eight boxes per tile), the leading lane
            // still doing the waits, the byte counts, Q and the tree tile.
            const bool lead = lane == 0;
            const bool usable = (smem_u32(smem_raw) & 1023u) == 0 && st.tmem_base == 0;     // (else the tiles would not sit on their swizzle boundary)
            if (!usable && lead) set_status(P.status, RADAR_ERR_CUDA);
            long long tot_all;
            Cursor<PAGED> cur = first_segment<PAGED>(P, pp, ci, tot_all);
            if (!usable) cur.t0 = cur.t1 = 0;
            // Needed behind the last load only, and a dozen registers.  With a paged cache, whose producer would spill for them
            // (132 bytes, in its loop over the tiles), in shared memory: B = 1, 32 / 8 heads, 2048 tokens in pages of 16 21.9 ->
            // 20.2 us, of 256 19.4 -> 17.7; B = 8, 64 / 8 heads, 8192 tokens, pages of 16 198.3 -> 192.8.  Without one, where
            // nothing is spilled, in registers (8 layers of B = 8, 64 / 8 heads 1073, in shared memory 1081).
            Cut own;
            Cut& cut = PAGED ? st.cut : own;
            cut.unit.valid = 0;
            cut.tot = tot_all;
            uint32_t k_slot = 0, k_par = 1, v_slot = 0, v_par = 1;   // ring slot to fill next and the phase that frees it
            const int n_cache_pages = PAGED ? (int)P.cache_rows / a.page_size : 0;            // (cache_rows: below 2^31)
            const int box_shift = PAGED ? __ffs(min(a.page_size, kTileKeys)) - 1 : 0, tiles_per_page = PAGED ? max(a.page_size / kTileKeys, 1) : 1;
            auto first_page = [&](int t) { return tiles_per_page > 1 ? t / tiles_per_page : t << (7 - box_shift); };     // of tile t
            // asks for the lines of the block table that tiles [t0, t1) of a sequence are looked up in
            auto fetch_pages = [&](int b, int t0, int t1) {
                const int last = min(first_page(t1), a.max_pages - 1);
                for (int i = first_page(t0) + lane * 32; i <= last; i += 32 * 32)
                    asm volatile("prefetch.global.L1 [%0];" ::"l"(a.block_table + (long long)b * a.max_pages + i));
            };
            for (uint32_t seg = 0;; ++seg) {
                const bool on = cur.valid();
                const int b = cur.b, g = cur.g, n = cur.t1 - cur.t0, t0 = cur.t0, layer = cur.layer, nt = cur.s.nt, Pb = cur.s.Pb;
                const long long kv0 = cur.s.kv0;
                const bool two = TWO && cur.two_rb(P);
                if (lead) {
                    ok = mbar_wait_while(ok, &st.bar_segempty[seg % kSegRing], ((seg / kSegRing) & 1) ^ 1);
                    Segment s;                       // (behind a wait that ran out the others are sent home)
                    s.n = on && ok ? n : 0; s.t0 = t0; s.nt = nt; s.Pb = Pb; s.M = cur.s.M; s.rows = cur.s.rows; s.b = b; s.g = g; s.layer = layer;
                    st.seg[seg % kSegRing] = s;
                    mbar_arrive(&st.bar_segfull[seg % kSegRing]);
                }
                if (!on) break;
                if (t0 == 0 && n < nt) {                             // necessarily the last segment of this CTA
                    cut.unit.valid = 1; cut.unit.b = b; cut.unit.g = g; cut.unit.slot = seg == 0 ? 0 : 1; cut.unit.layer = layer; cut.unit.rows = cur.s.rows;
                    cut.nt = nt; cut.w = cur.s.w; cut.u0 = cur.U;
                }
                cur.next(P, pp);
                if (!PAGED && !lead) continue;
                // Order: the first K tile(s), Q (behind them, for its slot is free only after the last S of the segment before; the
                // CTA's first segment finds it free), then V(i), K(i + la), the order in which the MMA warp consumes them.
                const int la = two ? 1 : 2;
#pragma unroll 1
                for (int j = -2 * la; j < 2 * n; ++j) {              // even: V(j / 2), odd: K(j / 2 + la)
                    const bool is_k = (j & 1) != 0;
                    const int i = (j >> 1) + (is_k ? la : 0);
                    if (i >= 0 && i < n) {
                        const int t = t0 + i;
                        const bool tree = t == nt - 1, boxes = PAGED && !tree;
                        // paged cache: one box per page (or per tile when a page holds whole tiles); only pages
                        // that hold live keys are fetched, what stays stale in the slot is masked / never read.
                        // The pages are looked up while the slot is not free yet.
                        int n_ld = 0, per = 0, page_row = 0;
                        if (boxes) {
                            per = min(a.page_size, kTileKeys);
                            n_ld = (min(kTileKeys, Pb - t * kTileKeys) + per - 1) >> box_shift;
                            if (lane < n_ld) {
                                const int index = first_page(t) + lane;
                                int page = __ldg(a.block_table + (long long)b * a.max_pages + index);
                                if (page < 0 || page >= n_cache_pages) { set_status(P.status, RADAR_ERR_INVALID_ARG); page = 0; }
                                page_row = page * a.page_size + (tiles_per_page > 1 ? (t - index * tiles_per_page) * kTileKeys : 0);   // (below cache_rows)
                            }
                        }
                        const uint32_t slot = is_k ? k_slot : v_slot;
                        uint64_t* full = is_k ? &st.bar_kfull[slot] : &st.bar_vfull[slot];
                        unsigned char* dst = (is_k ? sK : sV) + slot * SM::kTileBytes;
                        if (lead) ok = mbar_wait_while(ok, is_k ? &st.bar_kempty[slot] : &st.bar_vempty[slot], is_k ? k_par : v_par);
                        if (PAGED) ok = __shfl_sync(kFull, ok, 0);
                        if (!ok) break;                              // (the ring's position stays that of the last load)
                        if (is_k) { if (++k_slot == RK) { k_slot = 0; k_par ^= 1; } }
                        else if (++v_slot == RV) { v_slot = 0; v_par ^= 1; }
                        if (!boxes) {
                            if (lead) {
                                const int keys = tree ? kTreeKeys : kTileKeys;
                                const CUtensorMap* tm = tree ? (is_k ? &tmKt : &tmVt) : (is_k ? &tmKc : &tmVc);
                                const int row = tree ? b * kMaxNodes : (int)(kv0 + (long long)t * kTileKeys);
                                mbar_arrive_expect_tx(full, keys * D * 2);
                                for (int h = 0; h < H; ++h) tma_load_4d(dst + h * (keys * 128), tm, full, h * 64, g, row, layer);
                            }
                        } else {
                            if (lead) mbar_arrive_expect_tx(full, n_ld * per * D * 2);
                            __syncwarp();
                            if (lane < n_ld)
                                for (int h = 0; h < H; ++h)
                                    tma_load_4d(dst + h * (kTileKeys * 128) + lane * per * 128, is_k ? &tmKc : &tmVc, full, h * 64, g, page_row, layer);
                        }
                    }
                    if (j == (seg == 0 ? -2 * la : -1) && lead) {
                        ok = mbar_wait_while(ok, &st.bar_qempty, (seg & 1) ^ 1);
                        const int blocks = two ? 2 : 1, node0 = b * kMaxNodes + pp * P.n_blk * P.nodes_per_rb;
                        if (ok) {
                            st.q_last = seg & 1;
                            mbar_arrive_expect_tx(&st.bar_qfull, blocks * P.rb_rows * D * 2);   // rows past rb_rows stay stale: never read back
                            for (int q = 0; q < blocks; ++q)
                                for (int h = 0; h < H; ++h)
                                    tma_load_4d(sQ + q * SM::kQBlock + h * (128 * 128), &tmQ, &st.bar_qfull, h * 64, g * G, node0 + q * P.nodes_per_rb, layer);
                        }
                        // ... so the next segment's Q waits for it in L2
                        if (cur.valid()) {
                            const int next0 = cur.b * kMaxNodes + pp * P.n_blk * P.nodes_per_rb;
                            for (int q = 0; q < (TWO && cur.two_rb(P) ? 2 : 1); ++q)
                                for (int h = 0; h < H; ++h) tma_prefetch_4d(&tmQ, h * 64, cur.g * G, next0 + q * P.nodes_per_rb, cur.layer);
                        }
                    }
                    if (PAGED && j == 0 && cur.valid()) fetch_pages(cur.b, cur.t0, cur.t1);
                }
            }
            __syncwarp();
            write_cut_unit(P, ci, cut);
            if (lead) { st.k_next = k_slot | k_par << 8; st.v_next = v_slot | v_par << 8; }
            __syncwarp();
        } else if (warp == kMmaWarp) {
            // =================================== MMA issuer ===================================
            // The warp runs converged: every lane waits on the barriers and executes the same straight-line issue
            // sequences with warp-uniform descriptor words, and the elected lane issues the instructions and the
            // commits (predicated, no branch around them).  Whatever this warp executes between two MMAs costs
            // tensor-pipe time, so no control flow depends on a wait's outcome: after a wait that ran out the
            // predicate is off and the loops run dry.
            constexpr uint32_t idesc_s128 = idesc_bf16_f32(128, kTileKeys, false, false);
            constexpr uint32_t idesc_s64 = idesc_bf16_f32(128, kTreeKeys, false, false);
            constexpr uint32_t idesc_pv = idesc_bf16_f32(128, D, false, true);
            // high word of every shared-memory descriptor (stride between 8-row groups 1024 B, version, swizzle)
            constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);
            const uint32_t q_lo = ((smem_u32(sQ) & 0x3ffff) >> 4) | (1u << 16);
            const uint32_t k_lo = ((smem_u32(sK) & 0x3ffff) >> 4) | (1u << 16);
            const uint32_t v_lo = (smem_u32(sV) & 0x3ffff) >> 4;
            const uint32_t elected = elect_one();
            uint32_t k_next = 0, k_par = 0, v_next = 0, v_par = 0;   // ring slot to take next and its phase parity
            uint32_t p_par[2] = {0, 0};              // phase parity of the next P tile per group
            // The segment's shape comes from memory; passing it through a broadcast from lane 0 tells the
            // compiler that it is the same in every lane, so that the loops below and the descriptor arithmetic in
            // them stay on the uniform datapath (this warp's own instruction stream is what bounds the issue rate).
            auto uni = [](int v) { return __shfl_sync(kFull, v, 0); };
            Segment s;
            for (uint32_t seg = 0; take_segment(seg, s); ++seg) {
                const int seg_t0 = uni(s.t0), n = uni(s.n), M = uni(s.M), Pb = uni(s.Pb), last = uni(s.nt) - 1;
                const bool two = TWO && uni(s.rows) > P.rb_rows;
                ok = mbar_wait_while(ok, &st.bar_qfull, seg & 1);
                uint32_t k_slot = 0, v_slot = 0;      // ring slots of the K and V tiles in use
                bool acc[2] = {false, false};         // accumulator holds a product of this segment
                auto take_v = [&]() {
                    v_slot = v_next;
                    ok = mbar_wait_while(ok, &st.bar_vfull[v_slot], v_par);
                    if (++v_next == RV) { v_next = 0; v_par ^= 1; }
                };
                auto take_k = [&]() {
                    k_slot = k_next;
                    ok = mbar_wait_while(ok, &st.bar_kfull[k_slot], k_par);
                    if (++k_next == RK) { k_next = 0; k_par ^= 1; }
                };
                // the accumulator's first product of the segment: the epilogue of the previous one has read it
                auto take_o = [&](const int q) {
                    if (!acc[q]) ok = mbar_wait_while(ok, &st.bar_ofree[q], (seg & 1) ^ 1);
                };

                // ---- O[q] (+)= P[q] V for tile i (q is a literal at every call site) ----
                auto pv = [&](const int q, const int i, const bool fresh_v, const bool release_v) {
                    const bool tree = seg_t0 + i == last;
                    const int nk = tree ? kTreeKeys : kTileKeys;
                    const int valid = tree ? M : min(kTileKeys, Pb - (seg_t0 + i) * kTileKeys);
                    const int ksteps = (valid + 15) >> 4;
                    if (fresh_v) {
                        take_v();
                        if (valid < ksteps * 16) {
                            // rows past the last live key meet P = 0; they must not hold NaN/Inf bit patterns
                            unsigned char* vtile = sV + v_slot * SM::kTileBytes;
                            const int nrows = ksteps * 16 - valid;
#pragma unroll 1
                            for (int e = lane; e < nrows * 8 * H; e += 32) {
                                const int h = e / (nrows * 8), rem = e % (nrows * 8);
                                const int r = valid + rem / 8, c = rem % 8;
                                *reinterpret_cast<uint4*>(vtile + h * (nk * 128) + r * 128 + c * 16) = make_uint4(0, 0, 0, 0);
                            }
                            fence_proxy_async_smem();
                            __syncwarp();
                        }
                    }
                    take_o(q);
                    ok = mbar_wait_while(ok, &st.bar_pready[q], p_par[q]);
                    p_par[q] ^= 1;
                    tc_fence_after_sync();
                    const uint32_t go = ok ? elected : 0u;
                    // V is consumed N-major: 16 keys are 2048 B; 64-column blocks are nk * 128 B apart
                    const uint32_t b_lo = (v_lo + v_slot * (SM::kTileBytes >> 4)) | ((uint32_t)(nk * 128 >> 4) << 16);
                    mma_ts_x4(go, ksteps, tmem + 256 + q * 128, tmem + q * 128, b_lo, kDescHi, idesc_pv, acc[q]);
                    mma_ts_x4(go, ksteps - 4, tmem + 256 + q * 128, tmem + q * 128 + 32, b_lo + 4 * 128, kDescHi, idesc_pv, true);
                    acc[q] = true;
                    if (release_v) mma_commit_if(go, &st.bar_vempty[v_slot]);
                    if (two ? i == n - 1 : i + 2 >= n) mma_commit_if(go, &st.bar_odone[q]);
                };
                // ---- S[q] = Q K^T for tile si.  Nothing in tensor memory changes hands here: K arrives through the
                // async proxy, and the buffer was last read by this thread's own P V, which runs first. ----
                auto qk = [&](const int q, const int si, const bool fresh_k, const bool release_k) {
                    if (fresh_k) take_k();
                    const uint32_t go = ok ? elected : 0u;
                    const bool tree = seg_t0 + si == last;
                    const uint32_t a0 = q_lo + (two ? q : 0) * (SM::kQBlock >> 4);
                    const uint32_t b0 = k_lo + k_slot * (SM::kTileBytes >> 4);
                    const uint32_t idesc = tree ? idesc_s64 : idesc_s128;
                    mma_ss_x4(go, tmem + q * 128, a0, b0, kDescHi, idesc, false);
                    if (D == 128)                     // second 64-column block of Q and K
                        mma_ss_x4(go, tmem + q * 128, a0 + (128 * 128 >> 4), b0 + ((uint32_t)((tree ? kTreeKeys : kTileKeys) * 128) >> 4),
                                  kDescHi, idesc, true);
                    if (release_k) mma_commit_if(go, &st.bar_kempty[k_slot]);
                    mma_commit_if(go, &st.bar_sfull[q]);
                    // the last S of the segment: Q may be overwritten once it has run
                    if (si == n - 1 && release_k) mma_commit_if(go, &st.bar_qempty);
                };
                // Schedule.  Two live row blocks: group s owns row block s; per tile PV0(i) S0(i+1) PV1(i) S1(i+1),
                // both groups sharing K(i+1) and V(i).  One live row block: the groups take alternate tiles,
                // PV(i) S(i+2) for group i & 1.  S of the first tile(s) comes from the iterations with i < 0.
                // Steady state (all tiles involved are full prefix tiles): the same steps with nothing to decide,
                // so that the issuing warp executes as few instructions per MMA as possible.  The waits for K and V, which are
                // there most of the time, stand where the warp would wait for P.
                auto full = [&](const int q, const uint32_t a0, const bool fresh, const bool release) {
                    static_assert(kFirstKeys == 64 && kTileKeys == 128, "four steps before and behind the second wait");
                    const uint32_t o_col = tmem + 256 + q * 128, p_col = tmem + q * 128;
                    if (fresh) take_v();
                    take_o(q);
                    const uint32_t b_lo = (v_lo + v_slot * (SM::kTileBytes >> 4)) | ((uint32_t)(kTileKeys * 128 >> 4) << 16);
                    ok = mbar_wait_while(ok, &st.bar_pfirst[q], p_par[q]);
                    tc_fence_after_sync();
                    mma_ts_x4(ok ? elected : 0u, o_col, p_col, b_lo, kDescHi, idesc_pv, acc[q]);
                    if (fresh) take_k();
                    const uint32_t b0 = k_lo + k_slot * (SM::kTileBytes >> 4);
                    ok = mbar_wait_while(ok, &st.bar_pready[q], p_par[q]);
                    p_par[q] ^= 1;
                    acc[q] = true;
                    tc_fence_after_sync();
                    const uint32_t go = ok ? elected : 0u;
                    mma_ts_x4(go, o_col, p_col + 32, b_lo + 4 * 128, kDescHi, idesc_pv, true);
                    if (release) mma_commit_if(go, &st.bar_vempty[v_slot]);
                    mma_ss_x4(go, p_col, a0, b0, kDescHi, idesc_s128, false);
                    if (D == 128) mma_ss_x4(go, p_col, a0 + (128 * 128 >> 4), b0 + (kTileKeys * 128 >> 4), kDescHi, idesc_s128, true);
                    mma_commit_if(go, &st.bar_sfull[q]);
                    if (release) mma_commit_if(go, &st.bar_kempty[k_slot]);
                };
                const uint32_t a_q0 = q_lo, a_q1 = q_lo + (SM::kQBlock >> 4);
                const int n_full = min(n, Pb / kTileKeys - seg_t0);   // tiles [0, n_full) of the segment are full prefix tiles
                if (two) {
#pragma unroll 1
                    for (int i = -1; i < n; ++i) {
                        if (i >= 0 && i + 2 < n_full) {           // tiles i and i+1 full, and S(i+1) is not the segment's last
                            full(0, a_q0, true, false);
                            full(1, a_q1, false, true);
                        } else {
                            if (i >= 0) pv(0, i, true, false);
                            if (i + 1 < n) qk(0, i + 1, true, false);
                            if (i >= 0) pv(1, i, false, true);
                            if (i + 1 < n) qk(1, i + 1, false, true);
                        }
                    }
                } else {
#pragma unroll 1
                    for (int i = -2; i < n; i += 2) {
                        if (i >= 0 && i + 4 < n_full) {           // tiles i to i+3 full, S(i+3) not the last
                            full(0, a_q0, true, true);
                            full(1, a_q0, true, true);
                        } else {
                            if (i >= 0) pv(0, i, true, true);
                            if (i + 2 < n) qk(0, i + 2, true, true);
                            if (i >= 0 && i + 1 < n) pv(1, i + 1, true, true);
                            if (i + 3 < n) qk(1, i + 3, true, true);
                        }
                    }
                }
            }
            // no product may read shared memory or write tensor memory that the CTA has given back
            mma_commit_if(elected, &st.bar_idle);
            ok &= mbar_drain(&st.bar_idle, 0);
            __syncwarp();
        }
    }

    // ---- teardown ----
    if (!ok) st.abort = 1;
    tc_fence_before_sync();
    __syncthreads();
    if (warp == kMmaWarp) {
        if (lane == 0 && st.abort) {
            // No load may land in shared memory that the CTA has left.  (Without an abort the roles have waited for every
            // one; seven more waits at the end of every producer cost launches up to 1.2 %: 16 / 1 heads, B = 8, 8192 tokens
            // 51.9 -> 52.4 us.)
            const uint32_t k = st.k_next, v = st.v_next;
            mbar_drain(&st.bar_qfull, st.q_last);
            for (int i = 0; i < RK; ++i) mbar_drain(&st.bar_kfull[i], last_armed_parity(i, k & 255, k >> 8));
            for (int i = 0; i < RV; ++i) mbar_drain(&st.bar_vfull[i], last_armed_parity(i, v & 255, v >> 8));
            set_status(P.status, RADAR_ERR_TIMEOUT);
        }
        __syncwarp();
        tmem_dealloc(st.tmem_base, 512);
    }
}

// The form for head ratios that do not divide 128, which came from the FMA kernel, whose probabilities are fp32, and keep its
// precision: P goes to the tensor cores as the sum of two bf16 numbers (its value to 2^-18) in place of one (2^-9), and the
// scores' scale is applied in two parts (error against fp64, 2-norm, of 24 / 8 heads, 2048 tokens: FMA 1.6545e-3, one bf16
// 2.1607e-3, two 1.6545e-3, all of it the rounding of O to bf16).  That doubles the instructions between two exponentials,
// which one thread a row issues one after the other and two a row side by side: 16 softmax warps here, which also do the
// epilogue, TMA producer and MMA issuer (this form / the one above with two parts: 24 / 8 heads, B = 6, 300 to 4500 tokens
// 33.8 / 37.3 us, paged 39.1 / 43.6; 16 layers, B = 2, 1000 to 2000 tokens 105 / 131).
constexpr int kFineThreads = 576;
constexpr int kFineProducerWarp = 16, kFineMmaWarp = 17;
template <int D, bool TWO, bool PAGED>
__global__ void __launch_bounds__(kFineThreads, 1)      // 18 warps are allocated as 20: 96 registers per thread
tree_attn_tc_fine_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmKc,
                    const __grid_constant__ CUtensorMap tmVc, const __grid_constant__ CUtensorMap tmKt,
                    const __grid_constant__ CUtensorMap tmVt, const TcParams P) {
    chain_trigger();                     // warp 0 waits for the predecessor below; the barrier, tensor-memory and
                                         // descriptor set-up of the other warps needs nothing from global memory
    using SM = Smem<D, TWO>;
    constexpr int H = SM::kHalves;
    constexpr int RK = SM::kRingK, RV = SM::kRingV;
    const radar_attn_args& a = P.a;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int pp = blockIdx.x % P.n_cls;                    // class
    const int ci = blockIdx.x / P.n_cls;
    const int G = P.G;

    // Static block first (padded to a multiple of 1024 bytes and aligned to it), the tiles behind it: the
    // swizzled tiles need a 1024-byte boundary and there is no room left for alignment slack.
    struct __align__(1024) Static {
        uint64_t bar_qfull, bar_qempty, bar_kfull[3], bar_kempty[3], bar_vfull[3], bar_vempty[3];
        uint64_t bar_sfull[2], bar_pfirst[2], bar_pready[2], bar_odone[2], bar_ofree[2];
        uint64_t bar_idle;       // every product issued has run
        uint32_t armed[4];       // K and V loads of the producer, phase parity of its last Q
        long long range[4];      // this CTA's range [lo, hi), size of the class's space (all layers), start of its first unit
        int start[3];            // sequence, KV head and layer of the unit that contains lo
        int start_pad;
        uint32_t tmem_base;
        int abort;
        float xm[128];           // group 1's running max at the end of a segment (one live row block)
        float mx[2][2][128];     // per group and column half: row maxima of a tile; row sums at the end of a segment
        unsigned char pad[kStaticSmem - (25 * 8 + 4 * 4 + 4 * 8 + 4 * 4 + 4 + 4 + 128 * 4 + 2 * 2 * 128 * 4)];
    };
    static_assert(sizeof(Static) == kStaticSmem, "static shared-memory block");
    __shared__ Static st;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = smem_raw;
    unsigned char* sQ = smem;
    unsigned char* sK = smem + SM::kQBytes;
    unsigned char* sV = sK + RK * SM::kTileBytes;
    uint64_t& bar_qfull = st.bar_qfull;
    uint64_t& bar_qempty = st.bar_qempty;
    uint64_t (&bar_kfull)[3] = st.bar_kfull;
    uint64_t (&bar_kempty)[3] = st.bar_kempty;
    uint64_t (&bar_vfull)[3] = st.bar_vfull;
    uint64_t (&bar_vempty)[3] = st.bar_vempty;
    uint64_t (&bar_sfull)[2] = st.bar_sfull;
    uint64_t (&bar_pfirst)[2] = st.bar_pfirst;       // the first chunk of every thread's P is there
    uint64_t (&bar_pready)[2] = st.bar_pready;       // ... all of it
    uint64_t (&bar_odone)[2] = st.bar_odone;
    uint64_t (&bar_ofree)[2] = st.bar_ofree;
    uint32_t& s_tmem_base = st.tmem_base;
    int& s_abort = st.abort;
    float (&s_xm)[128] = st.xm;
    float (&s_mx)[2][2][128] = st.mx;
    float (&s_xl)[2][2][128] = st.mx;        // same storage: the two uses never overlap in time
    long long (&s_range)[4] = st.range;
    int (&s_start)[3] = st.start;
    const bool smem_aligned = (smem_u32(smem_raw) & 1023u) == 0;

    // ---- set-up: warp 0 finds this CTA's range while the barriers and tensor memory are prepared ----
    // (The steps of first_segment, which has to give the same ranges.  That function called here: 24 / 8 heads, B = 1, 2048 tokens
    // 19.2 -> 19.5 us, 28 / 4 heads, B = 1, 1000 tokens 16.8 -> 17.0, others within 2 % either way.)
    if (warp == 0) {
        chain_sync();                    // every global access of the CTA comes after the block barrier below
        long long tot = 0;
        for (int b0 = 0; b0 < a.B; b0 += 32) {
            const int b = b0 + lane;
            long long sz = b < a.B ? seq_cost<PAGED>(P, b, pp) : 0;
            if (pp == 0 && ci == 0 && b < a.B) {
                const int Pb = a.prefix_len[b];
                const long long kv0 = PAGED ? 0 : a.kv_start[b];
                if (Pb < 0 || Pb > a.max_prefix_len || kv0 < 0 || kv0 + Pb > P.cache_rows) set_status(P.status, RADAR_ERR_INVALID_ARG);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sz += __shfl_xor_sync(kFull, sz, o);
            tot += sz;
        }
        // the space of all layers: layer l occupies [l * tot, (l + 1) * tot)
        const long long tot_all = tot * P.n_layers;
        const long long lo_all = tot_all * ci / P.ncc, hi = tot_all * (ci + 1) / P.ncc;
        const int layer0 = tot > 0 ? (int)(lo_all / tot) : 0;
        const long long lo = lo_all - (long long)layer0 * tot;
        long long cum = 0, fU = 0;
        int fb = -1, fg = 0;
        for (int b0 = 0; b0 < a.B && fb < 0; b0 += 32) {
            const int b = b0 + lane;
            const long long sz = b < a.B ? seq_cost<PAGED>(P, b, pp) : 0;
            long long incl = sz;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const long long v = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += v;
            }
            const unsigned hit = __ballot_sync(kFull, cum + incl > lo);
            if (hit) {
                const int src = __ffs(hit) - 1;
                const long long before = cum + __shfl_sync(kFull, incl - sz, src);
                fb = b0 + src;
                const SeqInfo si = seq_info<PAGED>(P, fb, pp);
                const long long unit = (long long)si.nt * si.w + P.unit_cost;
                fg = (int)((lo - before) / unit);
                fU = before + fg * unit;
            }
            cum += __shfl_sync(kFull, incl, 31);
        }
        if (lane == 0) {
            s_range[0] = lo_all; s_range[1] = hi; s_range[2] = tot_all; s_range[3] = fU + (long long)layer0 * tot;
            s_start[0] = layer0 < P.n_layers ? fb : -1; s_start[1] = fg; s_start[2] = layer0;
        }
    } else if (warp == 1) {
        if (lane == 0) {
            s_abort = 0;
            mbar_init(&bar_qfull, 1);
            mbar_init(&bar_qempty, 1);
            mbar_init(&st.bar_idle, 1);
            st.armed[2] = 1;
            for (int i = 0; i < 3; ++i) {
                mbar_init(&bar_kfull[i], 1); mbar_init(&bar_kempty[i], 1);
                mbar_init(&bar_vfull[i], 1); mbar_init(&bar_vempty[i], 1);
            }
            for (int i = 0; i < 2; ++i) {
                mbar_init(&bar_sfull[i], 1); mbar_init(&bar_pfirst[i], 8); mbar_init(&bar_pready[i], 8);
                mbar_init(&bar_odone[i], 1); mbar_init(&bar_ofree[i], 8);
            }
            fence_barrier_init();
        }
    } else if (warp == kFineProducerWarp) {
        tmem_alloc(&s_tmem_base, 512);
        tmem_relinquish();
        if (lane == 0) {
            tma_prefetch_desc(&tmQ); tma_prefetch_desc(&tmKc); tma_prefetch_desc(&tmVc);
            tma_prefetch_desc(&tmKt); tma_prefetch_desc(&tmVt);
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = s_tmem_base;      // columns: S/P buffers at 0 and 128, O accumulators at 256 and 384
    volatile int* ab = &s_abort;

    // first segment: the unit that contains the range's start, from its first tile starting at or after it
    Cursor<PAGED> cur;
    cur.b = s_start[0]; cur.g = s_start[1]; cur.layer = s_start[2];
    cur.hi = s_range[1];
    cur.unit_cost = P.unit_cost;
    cur.U = s_range[3];
    cur.t0 = cur.t1 = 0;
    if (cur.b >= 0) {
        cur.s = seq_info<PAGED>(P, cur.b, pp);
        cur.t0 = tiles_before(s_range[0], cur.U, cur.s.nt, cur.s.w, P.unit_cost);
        if (cur.t0 >= cur.s.nt) cur.next_unit(P, pp);       // every tile of that unit starts before the range
        else cur.clip();
    }
    if (!cur.valid() || !smem_aligned) {                    // nothing for this CTA (uniform)
        if (tid == 0) {
            P.cut[blockIdx.x].valid = 0;
            if (!smem_aligned) set_status(P.status, RADAR_ERR_CUDA);   // the tiles would not sit on their swizzle boundary
        }
        tc_fence_before_sync();
        __syncthreads();
        if (warp == kFineProducerWarp) tmem_dealloc(tmem, 512);
        return;
    }

    if (warp == kFineProducerWarp) {
        // =================================== TMA producer ===================================
        // One lane does everything for the contiguous cache.  With a paged cache the whole warp walks the same
        // loop and lane p looks up and fetches page p of a tile (up to eight boxes per tile), the leading lane
        // still doing the waits, the byte counts, Q and the tree tile.
        Cut cut;
        cut.unit.valid = 0;
        cut.nt = cut.w = 0;
        cut.u0 = 0;
        if (PAGED || lane == 0) {
            const bool lead = lane == 0;
            uint32_t kc = 0, vc = 0;
            bool ok = true;
            for (uint32_t seg = 0; cur.valid(); cur.next(P, pp), ++seg) {
                const int b = cur.b, g = cur.g, n = cur.t1 - cur.t0;
                const bool two = TWO && cur.two_rb(P);
                if (cur.t0 == 0 && cur.t1 < cur.s.nt) {          // necessarily the last segment of this CTA
                    cut.unit.valid = 1; cut.unit.b = b; cut.unit.g = g; cut.unit.slot = seg == 0 ? 0 : 1;
                    cut.unit.layer = cur.layer; cut.unit.rows = cur.s.rows;
                    cut.nt = cur.s.nt; cut.w = cur.s.w; cut.u0 = cur.U;
                }
                if (lead) ok = ok && mbar_wait(&bar_qempty, (seg & 1) ^ 1, ab);
                if (lead && ok) {
                    st.armed[2] = seg & 1;
                    mbar_arrive_expect_tx(&bar_qfull, (two ? 2 : 1) * P.rb_rows * D * 2);   // rows past rb_rows stay stale: never read back
                    for (int q = 0; q < (two ? 2 : 1); ++q)
                        for (int h = 0; h < H; ++h)
                            tma_load_4d(sQ + q * SM::kQBlock + h * (128 * 128), &tmQ, &bar_qfull, h * 64, g * G,
                                        b * kMaxNodes + (pp * P.n_blk + q) * P.nodes_per_rb, cur.layer);
                }
                auto load_tile = [&](int t, bool is_k) {
                    uint32_t& cnt = is_k ? kc : vc;
                    const int ring = is_k ? RK : RV;
                    const int slot = cnt % ring;
                    const uint32_t use = cnt / ring;
                    uint64_t* full = is_k ? &bar_kfull[slot] : &bar_vfull[slot];
                    uint64_t* empty = is_k ? &bar_kempty[slot] : &bar_vempty[slot];
                    unsigned char* dst = (is_k ? sK : sV) + slot * SM::kTileBytes;
                    if (lead && (!ok || !mbar_wait(empty, (use & 1) ^ 1, ab))) ok = false;
                    if (PAGED) ok = __shfl_sync(kFull, ok, 0);
                    if (!ok) return;
                    ++cnt;                           // loads armed
                    if (t == cur.s.nt - 1) {
                        if (lead) {
                            mbar_arrive_expect_tx(full, kTreeKeys * D * 2);
                            for (int h = 0; h < H; ++h)
                                tma_load_4d(dst + h * (kTreeKeys * 128), is_k ? &tmKt : &tmVt, full, h * 64, g, b * kMaxNodes, cur.layer);
                        }
                    } else if (!PAGED) {
                        mbar_arrive_expect_tx(full, kTileKeys * D * 2);
                        const int row = (int)(cur.s.kv0 + (long long)t * kTileKeys);
                        for (int h = 0; h < H; ++h)
                            tma_load_4d(dst + h * (kTileKeys * 128), is_k ? &tmKc : &tmVc, full, h * 64, g, row, cur.layer);
                    } else {
                        // paged cache: one box per page (or per tile when a page holds whole tiles); only pages
                        // that hold live keys are fetched, what stays stale in the slot is masked / never read
                        const int ps = a.page_size, per = min(ps, kTileKeys);
                        const int key0 = t * kTileKeys;
                        const int n_ld = (min(kTileKeys, cur.s.Pb - key0) + per - 1) / per;
                        const long long n_cache_pages = P.cache_rows / ps;
                        if (lead) mbar_arrive_expect_tx(full, n_ld * per * D * 2);
                        __syncwarp();
                        if (const int p = lane; p < n_ld) {
                            const int key = key0 + p * per;
                            long long page = __ldg(a.block_table + (long long)b * a.max_pages + key / ps);
                            if (page < 0 || page >= n_cache_pages) { set_status(P.status, RADAR_ERR_INVALID_ARG); page = 0; }
                            const int row = (int)(page * ps + key % ps);
                            for (int h = 0; h < H; ++h)
                                tma_load_4d(dst + h * (kTileKeys * 128) + p * per * 128, is_k ? &tmKc : &tmVc, full, h * 64, g, row, cur.layer);
                        }
                    }
                };
                // same order as the MMA warp consumes: the first K tile(s), then V(i), K(i + lookahead)
                const int la = two ? 1 : 2;
                for (int i = 0; i < la && i < n; ++i) load_tile(cur.t0 + i, true);
                for (int i = 0; i < n; ++i) {
                    load_tile(cur.t0 + i, false);
                    if (i + la < n) load_tile(cur.t0 + i + la, true);
                }
            }
            if (lead) { st.armed[0] = kc; st.armed[1] = vc; }
        }
        __syncwarp();
        if (!PAGED) {                    // lane 0 alone has gone through the segments
            cut.unit.valid = __shfl_sync(kFull, cut.unit.valid, 0);
            cut.nt = __shfl_sync(kFull, cut.nt, 0); cut.w = __shfl_sync(kFull, cut.w, 0); cut.u0 = __shfl_sync(kFull, cut.u0, 0);
        }
        cut.tot = s_range[2];
        write_cut_unit(P, ci, cut);
        __syncwarp();
    } else if (warp == kFineMmaWarp) {
        // =================================== MMA issuer ===================================
        // The warp runs converged: every lane waits on the barriers and executes the same straight-line issue
        // sequences with warp-uniform descriptor words, and the elected lane issues the instructions and the
        // commits (predicated, no branch around them).  Whatever this warp executes between two MMAs costs
        // tensor-pipe time, so no control flow depends on a wait's outcome: after a wait that ran out the
        // predicate is off and the loops run dry.
        constexpr uint32_t idesc_s128 = idesc_bf16_f32(128, kTileKeys, false, false);
        constexpr uint32_t idesc_s64 = idesc_bf16_f32(128, kTreeKeys, false, false);
        constexpr uint32_t idesc_pv = idesc_bf16_f32(128, D, false, true);
        // high word of every shared-memory descriptor (stride between 8-row groups 1024 B, version, swizzle)
        constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);
        const uint32_t q_lo = ((smem_u32(sQ) & 0x3ffff) >> 4) | (1u << 16);
        const uint32_t k_lo = ((smem_u32(sK) & 0x3ffff) >> 4) | (1u << 16);
        const uint32_t v_lo = (smem_u32(sV) & 0x3ffff) >> 4;
        const uint32_t elected = elect_one();
        uint32_t k_next = 0, k_par = 0, v_next = 0, v_par = 0;   // ring slot to take next and its phase parity
        uint32_t p_par[2] = {0, 0};              // phase parity of the next P tile per group
        bool ok = true;
        // The segment's shape comes from global memory; passing it through a broadcast from lane 0 tells the
        // compiler that it is the same in every lane, so that the loops below and the descriptor arithmetic in
        // them stay on the uniform datapath (this warp's own instruction stream is what bounds the issue rate).
        auto uni = [](int v) { return __shfl_sync(kFull, v, 0); };
        for (uint32_t seg = 0; uni(cur.valid()); cur.next(P, pp), ++seg) {
            const int seg_t0 = uni(cur.t0);
            const int n = uni(cur.t1) - seg_t0;
            const bool two = TWO && uni(cur.two_rb(P));
            const int M = uni(cur.s.M), Pb = uni(cur.s.Pb), nt_unit = uni(cur.s.nt);
            ok = ok && mbar_wait(&bar_qfull, seg & 1, ab);
            uint32_t k_slot = 0, v_slot = 0;      // ring slots of the K and V tiles in use
            bool acc[2] = {false, false};         // accumulator holds a product of this segment

            // ---- O[q] (+)= P[q] V for tile i (q is a literal at every call site) ----
            auto pv = [&](const int q, const int i, const bool fresh_v, const bool release_v) {
                const bool tree = seg_t0 + i == nt_unit - 1;
                const int nk = tree ? kTreeKeys : kTileKeys;
                const int valid = tree ? M : min(kTileKeys, Pb - (seg_t0 + i) * kTileKeys);
                const int ksteps = (valid + 15) >> 4;
                ok = ok && mbar_wait(&bar_pfirst[q], p_par[q], ab);
                ok = ok && mbar_wait(&bar_pready[q], p_par[q], ab);
                p_par[q] ^= 1;
                if (fresh_v) {
                    v_slot = v_next;
                    ok = ok && mbar_wait(&bar_vfull[v_slot], v_par, ab);
                    if (++v_next == RV) { v_next = 0; v_par ^= 1; }
                    if (valid < ksteps * 16) {
                        // rows past the last live key meet P = 0; they must not hold NaN/Inf bit patterns
                        unsigned char* vtile = sV + v_slot * SM::kTileBytes;
                        const int nrows = ksteps * 16 - valid;
                        for (int e = lane; e < nrows * 8 * H; e += 32) {
                            const int h = e / (nrows * 8), rem = e % (nrows * 8);
                            const int r = valid + rem / 8, c = rem % 8;
                            *reinterpret_cast<uint4*>(vtile + h * (nk * 128) + r * 128 + c * 16) = make_uint4(0, 0, 0, 0);
                        }
                        fence_proxy_async_smem();
                        __syncwarp();
                    }
                    if (i == 0) {                 // the previous segment's epilogue has read both accumulators
                        ok = ok && mbar_wait(&bar_ofree[0], (seg & 1) ^ 1, ab);
                        ok = ok && mbar_wait(&bar_ofree[1], (seg & 1) ^ 1, ab);
                    }
                }
                tc_fence_after_sync();
                const uint32_t go = ok ? elected : 0u;
                // V is consumed N-major: 16 keys are 2048 B; 64-column blocks are nk * 128 B apart
                const uint32_t b_lo = (v_lo + v_slot * (SM::kTileBytes >> 4)) | ((uint32_t)(nk * 128 >> 4) << 16);
                // P of the first half of the tile's keys sits at column 0 of the group's buffer, of the second half
                // at column 64 (each softmax thread writes inside its own column range)
                const int hs = tree ? 2 : 4;
                const uint32_t n1 = (uint32_t)min(ksteps, hs), n2 = (uint32_t)ksteps - n1;
                mma_ts_two_x4(go, n1, tmem + 256 + q * 128, tmem + q * 128, b_lo, kDescHi, idesc_pv, acc[q]);
                mma_ts_two_x4(go, n2, tmem + 256 + q * 128, tmem + q * 128 + 64, b_lo + hs * 128, kDescHi, idesc_pv, true);
                acc[q] = true;
                if (release_v) mma_commit_if(go, &bar_vempty[v_slot]);
                if (two ? i == n - 1 : i + 2 >= n) mma_commit_if(go, &bar_odone[q]);
            };
            // ---- S[q] = Q K^T for tile si.  Nothing in tensor memory changes hands here: K arrives through the
            // async proxy, and the buffer was last read by this thread's own P V, which runs first. ----
            auto qk = [&](const int q, const int si, const bool fresh_k, const bool release_k) {
                if (fresh_k) {
                    k_slot = k_next;
                    ok = ok && mbar_wait(&bar_kfull[k_slot], k_par, ab);
                    if (++k_next == RK) { k_next = 0; k_par ^= 1; }
                }
                const uint32_t go = ok ? elected : 0u;
                const bool tree = seg_t0 + si == nt_unit - 1;
                const uint32_t a0 = q_lo + (two ? q : 0) * (SM::kQBlock >> 4);
                const uint32_t b0 = k_lo + k_slot * (SM::kTileBytes >> 4);
                const uint32_t idesc = tree ? idesc_s64 : idesc_s128;
                mma_ss_x4(go, tmem + q * 128, a0, b0, kDescHi, idesc, false);
                if (D == 128)                     // second 64-column block of Q and K
                    mma_ss_x4(go, tmem + q * 128, a0 + (128 * 128 >> 4), b0 + ((uint32_t)((tree ? kTreeKeys : kTileKeys) * 128) >> 4),
                              kDescHi, idesc, true);
                if (release_k) mma_commit_if(go, &bar_kempty[k_slot]);
                mma_commit_if(go, &bar_sfull[q]);
                // the last S of the segment: Q may be overwritten once it has run
                if (si == n - 1 && release_k) mma_commit_if(go, &bar_qempty);
            };
            // Schedule.  Two live row blocks: group s owns row block s; per tile PV0(i) S0(i+1) PV1(i) S1(i+1),
            // both groups sharing K(i+1) and V(i).  One live row block: the groups take alternate tiles,
            // PV(i) S(i+2) for group i & 1.  S of the first tile(s) comes from the iterations with i < 0.
            // Steady state (both tiles involved are full prefix tiles): the same steps with nothing to decide,
            // so that the issuing warp executes as few instructions per MMA as possible.
            const uint32_t a_q0 = q_lo, a_q1 = q_lo + (SM::kQBlock >> 4);
            auto wait_all = [&](uint64_t* bar, uint32_t parity) { ok = mbar_wait(bar, parity, ab) && ok; };
            auto pv_full = [&](const int q, const bool fresh_v, const bool release_v) {
                wait_all(&bar_pfirst[q], p_par[q]);
                if (fresh_v) {
                    v_slot = v_next;
                    wait_all(&bar_vfull[v_slot], v_par);
                    if (++v_next == RV) { v_next = 0; v_par ^= 1; }
                }
                tc_fence_after_sync();
                const uint32_t b_lo = (v_lo + v_slot * (SM::kTileBytes >> 4)) | ((uint32_t)(kTileKeys * 128 >> 4) << 16);
                mma_ts_two_x2x2_full(ok ? elected : 0u, tmem + 256 + q * 128, tmem + q * 128, b_lo, kDescHi, idesc_pv, acc[q]);
                wait_all(&bar_pready[q], p_par[q]);
                p_par[q] ^= 1;
                tc_fence_after_sync();
                const uint32_t go = ok ? elected : 0u;
                mma_ts_two_x2x2_full(go, tmem + 256 + q * 128, tmem + q * 128 + 32, b_lo + 2 * 128, kDescHi, idesc_pv, true);
                acc[q] = true;
                if (release_v) mma_commit_if(go, &bar_vempty[v_slot]);
            };
            auto qk_full = [&](const int q, const uint32_t a0, const bool fresh_k, const bool release_k) {
                if (fresh_k) {
                    k_slot = k_next;
                    wait_all(&bar_kfull[k_slot], k_par);
                    if (++k_next == RK) { k_next = 0; k_par ^= 1; }
                }
                const uint32_t go = ok ? elected : 0u;
                const uint32_t b0 = k_lo + k_slot * (SM::kTileBytes >> 4);
                mma_ss_x4(go, tmem + q * 128, a0, b0, kDescHi, idesc_s128, false);
                if (D == 128) mma_ss_x4(go, tmem + q * 128, a0 + (128 * 128 >> 4), b0 + (kTileKeys * 128 >> 4), kDescHi, idesc_s128, true);
                if (release_k) mma_commit_if(go, &bar_kempty[k_slot]);
                mma_commit_if(go, &bar_sfull[q]);
            };
            const int n_full = min(n, Pb / kTileKeys - seg_t0);   // tiles [0, n_full) of the segment are full prefix tiles
            if (two) {
                for (int i = -1; i < n; ++i) {
                    if (i >= 0 && i + 2 < n_full) {           // tiles i and i+1 full, and S(i+1) is not the segment's last
                        pv_full(0, true, false);
                        qk_full(0, a_q0, true, false);
                        pv_full(1, false, true);
                        qk_full(1, a_q1, false, true);
                    } else {
                        if (i >= 0) pv(0, i, true, false);
                        if (i + 1 < n) qk(0, i + 1, true, false);
                        if (i >= 0) pv(1, i, false, true);
                        if (i + 1 < n) qk(1, i + 1, false, true);
                    }
                }
            } else {
                for (int i = -2; i < n; ++i) {
                    const bool fast = i >= 0 && i + 3 < n_full;   // tiles i and i+2 full, S(i+2) not the last
                    if (i & 1) {
                        if (fast) { pv_full(1, true, true); qk_full(1, a_q0, true, true); }
                        else {
                            if (i >= 0) pv(1, i, true, true);
                            if (i + 2 < n) qk(1, i + 2, true, true);
                        }
                    } else {
                        if (fast) { pv_full(0, true, true); qk_full(0, a_q0, true, true); }
                        else {
                            if (i >= 0) pv(0, i, true, true);
                            if (i + 2 < n) qk(0, i + 2, true, true);
                        }
                    }
                }
            }
        }
        // no product may read shared memory or write tensor memory that the CTA has given back
        mma_commit_if(elected, &st.bar_idle);
        if (!mbar_drain(&st.bar_idle, 0)) s_abort = 1;
        __syncwarp();
    } else {
        // =================================== softmax groups ===================================
        // Two threads per query row: warp w of a group's eight serves tensor-memory lanes 32 (w & 3) .. + 31
        // and the column half (w >> 2) & 1, so a row's 128 scores are exponentiated by two threads at once
        // and the chain S -> softmax -> P V of a group is about half as long.
        // That chain is what a tile costs, so the products of a thread's first 32 columns start while the second 32 are
        // exponentiated, and only the two warps that share rows wait for each other's maxima.
        const int grp = warp >> 3;
        const int half = (warp >> 2) & 1;
        const int pair_bar = 1 + grp * 4 + (warp & 3);          // barriers 1 .. 8: the two warps that share 32 rows
        const int row = (warp & 3) * 32 + lane;                 // row of the block == tensor-memory lane
        const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t tS = tmem + grp * 128 + lane_addr;
        const uint32_t tO = tmem + 256 + grp * 128 + lane_addr;
        const uint32_t tO_other = tmem + 256 + (grp ^ 1) * 128 + lane_addr;
        constexpr int DH = D / 2;                               // accumulator columns per thread
        uint32_t sc = 0, oc = 0;                 // S tiles and accumulators this group has waited for
        bool ok = true;
        for (uint32_t seg = 0; cur.valid(); cur.next(P, pp), ++seg) {
            const int b = cur.b, g = cur.g, n = cur.t1 - cur.t0;
            const bool two = TWO && cur.two_rb(P);
            const int M = cur.s.M, Pb = cur.s.Pb, nt_unit = cur.s.nt;
            const int blk = two ? grp : 0;                       // row block within the unit
            const int rb_node = (int)(((uint32_t)row * P.g_magic) >> 16);        // row / G
            const int node = (pp * P.n_blk + blk) * P.nodes_per_rb + rb_node;
            const int rows_here = min(cur.s.rows - blk * P.rb_rows, P.rb_rows);  // live rows of this row block
            const bool row_live = row < rows_here;
            // A warp none of whose 32 rows is live does no arithmetic (the products of its rows are never read):
            // it only keeps the barriers going.
            const bool warp_live = row - lane < rows_here;
            const unsigned long long live_bits = M >= 64 ? ~0ull : ((1ull << M) - 1ull);
            // the row's ancestor word is needed by the tree tile only (the unit's last): it is loaded here and first
            // touched there, so that the segment does not start with a wait for global memory
            const unsigned long long mask_word = a.mask[(int64_t)b * kMaxNodes + min(node, kMaxNodes - 1)];
            const int n_my = two ? n : (n - grp + 1) >> 1;
            float m_run = -CUDART_INF_F, l_run = 0.f;            // l_run: this thread's columns only

            for (int j = 0; j < n_my; ++j) {
                const int i = two ? j : 2 * j + grp;             // local tile index
                const int t = cur.t0 + i;
                ok = __all_sync(kFull, ok && mbar_wait(&bar_sfull[grp], sc & 1, ab));    // warp-uniform: guards .aligned ops
                ++sc;
                tc_fence_after_sync();
                // This thread's chunks of 32 score columns: a prefix tile has four (two per thread), the tree tile
                // two (one per thread).  Half h of a row works in columns 64 h .. 64 h + 63 of the buffer only: its
                // scores sit there (the tree tile's second chunk is read from columns 32 .. 63 but belongs to
                // half 1 alone) and its P goes to columns 64 h + 32 cc, 16 of each part, so the halves
                // never touch each other's columns and a thread overwrites only scores it has already taken into registers.
                const bool tree = t == nt_unit - 1;
                const int nch = tree ? 1 : 2;
                const int c0 = tree ? half : 2 * half;
                const int valid = tree ? kTreeKeys : min(kTileKeys, Pb - t * kTileKeys);
                const bool partial = tree || valid < kTileKeys;
                auto allowed_bits = [&](int c) -> uint32_t {        // keys of chunk c this row may attend to
                    if (tree) return row_live ? (uint32_t)((mask_word & live_bits) >> (c * 32)) : 0u;
                    const int lim = valid - c * 32;
                    return lim >= 32 ? 0xffffffffu : (lim <= 0 ? 0u : ((1u << lim) - 1u));
                };
                float mx = -CUDART_INF_F;
                if (ok && warp_live) {
#pragma unroll 1
                    for (int cc = 0; cc < nch; ++cc) {
                        uint32_t sv[32];
                        tmem_ld32(tS + (c0 + cc) * 32, sv);
                        tmem_wait_ld();
                        if (partial) {
                            const uint32_t al = allowed_bits(c0 + cc);
#pragma unroll
                            for (int e = 0; e < 32; ++e)
                                if (!((al >> e) & 1u)) sv[e] = 0xff800000u;     // -inf
                        }
                        float mxa[4] = {-CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F};
#pragma unroll
                        for (int e = 0; e < 32; e += 2)                     // three-input maxima: half the instructions
                            mxa[(e >> 1) & 3] = max3(mxa[(e >> 1) & 3], __uint_as_float(sv[e]), __uint_as_float(sv[e + 1]));
                        mx = fmaxf(mx, fmaxf(fmaxf(mxa[0], mxa[1]), fmaxf(mxa[2], mxa[3])));
                    }
                }
                // the two halves of a row exchange their maxima
                s_mx[grp][half][row] = mx;
                asm volatile("bar.sync %0, 64;" ::"r"(pair_bar) : "memory");
                if (ok && warp_live) {
                    mx = fmaxf(mx, s_mx[grp][half ^ 1][row]);
                    // ---- running max (log2 units), lazy rescale decision: the same in both halves of a row ----
                    const float m_tile = mx * P.scale_log2;
                    float factor = 1.f;
                    if (j == 0) {
                        m_run = m_tile;
                    } else if (m_tile > m_run + kRescaleThreshold) {
                        factor = ex2(m_run - m_tile);           // m_run may be -inf: factor 0 clears O and l
                        m_run = m_tile;
                    }
                    const float m_use = m_run == -CUDART_INF_F ? 0.f : m_run;
                    // ---- rescale this thread's half of the accumulator when some row of the warp moved its max
                    // (the products of the first chunk start before the second is there) ----
                    if (j > 0 && __any_sync(kFull, factor != 1.f)) {
#pragma unroll 1
                        for (int c = 0; c < DH / 32; ++c) {
                            uint32_t o[32];
                            tmem_ld32(tO + half * DH + c * 32, o);
                            tmem_wait_ld();
#pragma unroll
                            for (int e = 0; e < 32; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * factor);
                            tmem_st32(tO + half * DH + c * 32, o);
                        }
                    }
                    // ---- P = exp2(s * scale - m), row sum, bf16 pairs back to tensor memory ----
                    // (the scaling and the row sum work on pairs: one packed fp32x2 instruction per two values)
                    float2 ls[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
                    const float2 sc2 = make_float2(P.scale_log2, P.scale_log2), nm2 = make_float2(-m_use, -m_use);
#pragma unroll 1
                    for (int cc = 0; cc < nch; ++cc) {
                        uint32_t sv[32];
                        tmem_ld32(tS + (c0 + cc) * 32, sv);
                        tmem_wait_ld();
                        if (partial) {
                            const uint32_t al = allowed_bits(c0 + cc);
#pragma unroll
                            for (int e = 0; e < 32; ++e)
                                if (!((al >> e) & 1u)) sv[e] = 0xff800000u;
                        }
                        uint32_t pk[16], pl[16];
#pragma unroll
                        for (int e = 0; e < 16; ++e) {
                            const float2 s2 = make_float2(__uint_as_float(sv[2 * e]), __uint_as_float(sv[2 * e + 1]));
                            float2 t = __ffma2_rn(s2, sc2, nm2);
                            t = __ffma2_rn(s2, make_float2(P.scale_log2_lo, P.scale_log2_lo), t);
                            const float p0 = ex2(t.x), p1 = ex2(t.y);
                            ls[e & 1] = __fadd2_rn(ls[e & 1], make_float2(p0, p1));
                            const __nv_bfloat162 v = __floats2bfloat162_rn(p0, p1);
                            pk[e] = *reinterpret_cast<const uint32_t*>(&v);
                            const __nv_bfloat162 r = __floats2bfloat162_rn(p0 - __uint_as_float(pk[e] << 16), p1 - __uint_as_float(pk[e] & 0xffff0000u));
                            pl[e] = *reinterpret_cast<const uint32_t*>(&r);
                        }
                        tmem_st16(tS + half * 64 + cc * 32, pk);
                        tmem_st16(tS + half * 64 + cc * 32 + 16, pl);
                        if (cc == 0) {
                            tmem_wait_st();
                            tc_fence_before_sync();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(&bar_pfirst[grp]);
                        }
                    }
                    l_run = l_run * factor + ((ls[0].x + ls[0].y) + (ls[1].x + ls[1].y));
                    tmem_wait_st();
                }
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) {
                    if (!(ok && warp_live)) mbar_arrive(&bar_pfirst[grp]);
                    mbar_arrive(&bar_pready[grp]);
                }
            }

            // ---- epilogue of the segment ----
            if (n_my > 0) {
                ok = __all_sync(kFull, ok && mbar_wait(&bar_odone[grp], oc & 1, ab));
                ++oc;
            }
            tc_fence_after_sync();
            const bool final_rows = cur.complete();
            const int slot = seg == 0 ? 0 : 1;                   // a CTA has at most a cut first and a cut last segment
            const int64_t rec = ((int64_t)blockIdx.x * 2 + slot) * kPairRows + blk * 128 + row;
            // the row sum is the two halves' sums; with one live row block group 1 also hands its (m, l) to group 0
            s_xl[grp][half][row] = l_run;
            if (grp == 1 && half == 0) s_xm[row] = n_my > 0 ? m_run : -CUDART_INF_F;
            asm volatile("bar.sync 9, 512;" ::: "memory");
            float l_out = s_xl[grp][0][row] + s_xl[grp][1][row];
            float m_out = m_run, w0 = 1.f, w1 = 0.f;
            bool writer = true, merge_any = false;
            if (!two) {
                // group 0 merges group 1's accumulator, which sits in the same tensor-memory lanes
                writer = grp == 0;
                if (writer) {
                    const float m1 = s_xm[row], l1 = s_xl[1][0][row] + s_xl[1][1][row];
                    const bool merge = m1 != -CUDART_INF_F;
                    m_out = fmaxf(m_run, m1);
                    const float ms = m_out == -CUDART_INF_F ? 0.f : m_out;
                    w0 = ex2(m_run - ms);                        // exp2(-inf) = 0
                    w1 = ex2(m1 - ms);
                    l_out = l_out * w0 + l1 * w1;
                    merge_any = __any_sync(kFull, merge);        // rows that do not merge carry w1 = 0
                }
            }
            if (writer && ok && warp_live) {
                const float m_safe = m_out == -CUDART_INF_F ? 0.f : m_out;
                const float inv = final_rows ? 1.f / l_out : 1.f;
                const int hq = g * G + row - (int)(((uint32_t)row * P.g_magic) >> 16) * G;
                const int64_t out_row = ((int64_t)b * kMaxNodes + node) * a.Hq + hq;
#pragma unroll 1
                for (int c = 0; c < DH / 32; ++c) {
                    const int col = half * DH + c * 32;          // first accumulator column of this chunk
                    uint32_t o[32];
                    tmem_ld32(tO + col, o);
                    tmem_wait_ld();
                    float v[32];
#pragma unroll
                    for (int e = 0; e < 32; ++e) v[e] = __uint_as_float(o[e]) * w0;
                    if (merge_any) {
                        tmem_ld32(tO_other + col, o);
                        tmem_wait_ld();
#pragma unroll
                        for (int e = 0; e < 32; ++e) v[e] = fmaf(__uint_as_float(o[e]), w1, v[e]);
                    }
                    if (row_live) {
                        if (final_rows) {
                            __nv_bfloat16* dst = reinterpret_cast<__nv_bfloat16*>(a.O) + cur.layer * P.o_ls + out_row * D + col;
                            const bool wide = (reinterpret_cast<uintptr_t>(dst) & 31) == 0;
#pragma unroll
                            for (int q = 0; q < 2; ++q) {
                                uint32_t w[8];
#pragma unroll
                                for (int e = 0; e < 8; ++e) {
                                    const __nv_bfloat162 t2 = __floats2bfloat162_rn(v[q * 16 + 2 * e] * inv, v[q * 16 + 2 * e + 1] * inv);
                                    w[e] = *reinterpret_cast<const uint32_t*>(&t2);
                                }
                                if (wide) {
                                    st_global_32b(dst + q * 16, w);
                                } else {
                                    *reinterpret_cast<uint4*>(dst + q * 16) = make_uint4(w[0], w[1], w[2], w[3]);
                                    *reinterpret_cast<uint4*>(dst + q * 16 + 8) = make_uint4(w[4], w[5], w[6], w[7]);
                                }
                            }
                        } else {
                            float* dst = P.part_o + rec * D + col;          // 128-byte aligned (workspace carve)
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                uint32_t w[8];
#pragma unroll
                                for (int e = 0; e < 8; ++e) w[e] = __float_as_uint(v[q * 8 + e]);
                                st_global_32b(dst + q * 8, w);
                            }
                        }
                    }
                }
                if (row_live && half == 0) {
                    if (final_rows) {
                        if (a.lse != nullptr) a.lse[cur.layer * P.lse_ls + ((int64_t)b * a.Hq + hq) * kMaxNodes + node] = lse_of(m_safe, l_out);
                    } else {
                        P.part_ml[rec] = make_float2(m_out, l_out);
                    }
                }
            }
            asm volatile("bar.sync 10, 512;" ::: "memory");       // the exchanged (m, l) and group 1's accumulator have been read
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_ofree[grp]);
        }
    }

    // ---- teardown ----
    tc_fence_before_sync();
    __syncthreads();
    if (warp == kFineProducerWarp) {
        if (s_abort) {
            // no load may land in shared memory that the CTA has left
            if (lane == 0) {
                int dummy = 0;
                const uint32_t nk = st.armed[0], nv = st.armed[1];
                mbar_wait(&bar_qfull, st.armed[2], &dummy, 1u << 12);
                for (int i = 0; i < RK; ++i) {
                    mbar_wait(&bar_kfull[i], last_armed_parity(i, nk % RK, (nk / RK & 1) ^ 1), &dummy, 1u << 12);
                    if (i < RV) mbar_wait(&bar_vfull[i], last_armed_parity(i, nv % RV, (nv / RV & 1) ^ 1), &dummy, 1u << 12);
                }
                set_status(P.status, RADAR_ERR_TIMEOUT);
            }
            __syncwarp();
        }
        tmem_dealloc(tmem, 512);
    }
}

// Merges the pieces of the units that were cut across CTAs.  Blocks (c, *): CTA c of the attention kernel holds the first
// piece of a cut unit (or the blocks exit); the following CTAs of the same class hold the rest, each as its first
// segment.  A warp merges one query row, every piece of it in flight together: the work is a chain of three trips to L2,
// and many warps hide it better than many rows a warp do (148 cut units of 256 rows: 17.1 us event-timed with one row a
// warp, 18.4 with two, 20.6 with four; 72 cut units of 128 rows: 10.0, 10.8, 14.7).
template <int D, bool FINE>
__global__ void __launch_bounds__(256) tree_attn_tc_combine_kernel(const TcParams P) {
    chain_wait();
    auto weight = [](float d) { return FINE ? ex2(d) : __expf(d); };      // of two pieces' maxima that differ by d
    const radar_attn_args& a = P.a;
    const CutUnit& cu = P.cut[blockIdx.x];
    const int valid = cu.valid, b = cu.b, g = cu.g, layer = cu.layer, slot = cu.slot, rows = cu.rows, n_pieces = cu.n_pieces;
    const uint32_t live0 = cu.live[0];
    if (!valid) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int r = blockIdx.y * 8 + warp;
    if (r >= rows) return;                                   // rows of a unit are live from 0 up
    constexpr int E = D / 32;                                // output elements per lane
    // the row's record in piece j's partials (row blocks start 128 records apart, whatever part of them is live)
    const int blk = r < P.rb_rows ? 0 : 1, in_blk = r - blk * P.rb_rows;
    auto rec_of = [&](int j) {
        const int64_t cta = (int64_t)blockIdx.x + (int64_t)j * P.n_cls;
        return (cta * 2 + (j == 0 ? slot : 0)) * kPairRows + blk * 128 + in_blk;
    };
    auto store_row = [&](const float (&o)[E], float mx, float den) {
        const float inv = 1.f / den;
        const int rb_node = (int)(((uint32_t)in_blk * P.g_magic) >> 16);
        const int node = ((blockIdx.x % P.n_cls) * P.n_blk + blk) * P.nodes_per_rb + rb_node, hq = g * P.G + in_blk - rb_node * P.G;
        __nv_bfloat16* dst = reinterpret_cast<__nv_bfloat16*>(a.O) + layer * P.o_ls + (((int64_t)b * kMaxNodes + node) * a.Hq + hq) * D + lane * E;
        __nv_bfloat162 w[E / 2];
#pragma unroll
        for (int q = 0; q < E; q += 2) w[q / 2] = __floats2bfloat162_rn(o[q] * inv, o[q + 1] * inv);
        if (E == 4) *reinterpret_cast<uint2*>(dst) = *reinterpret_cast<const uint2*>(w);
        else *reinterpret_cast<uint32_t*>(dst) = *reinterpret_cast<const uint32_t*>(w);
        if (a.lse != nullptr && lane == 0) a.lse[layer * P.lse_ls + ((int64_t)b * a.Hq + hq) * kMaxNodes + node] = FINE ? lse_of(mx, den) : mx + logf(den);
    };
    auto load_row = [&](const float* src, float (&v)[E]) {
        if (E == 4) {
            const float4 t = *reinterpret_cast<const float4*>(src);
            v[0] = t.x; v[1] = t.y; v[E - 2] = t.z; v[E - 1] = t.w;
        } else {
            const float2 t = *reinterpret_cast<const float2*>(src);
            v[0] = t.x; v[1] = t.y;
        }
    };

    if (n_pieces <= 4) {
        // ---- the usual case: a unit spread over a few CTAs.  (A CTA whose range holds no tile start has no piece.) ----
        float2 ml[4];
        float v[4][E], o[E];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const bool on = ((live0 >> j) & 1u) && j < n_pieces;
            const int64_t rec = rec_of(on ? j : 0);
            ml[j] = P.part_ml[rec];
            load_row(P.part_o + rec * D + lane * E, v[j]);
            if (!on) ml[j] = make_float2(-CUDART_INF_F, 0.f);
        }
        const float mx = fmaxf(fmaxf(ml[0].x, ml[1].x), fmaxf(ml[2].x, ml[3].x));
        float den = 0.f;
#pragma unroll
        for (int q = 0; q < E; ++q) o[q] = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (ml[j].x == -CUDART_INF_F) continue;
            const float w = weight(ml[j].x - mx);
            den = fmaf(ml[j].y, w, den);
#pragma unroll
            for (int q = 0; q < E; ++q) o[q] = fmaf(v[j][q], w, o[q]);
        }
        store_row(o, mx, den);
        return;
    }

    // ---- a unit spread over many CTAs (few units, long prefixes): lane j holds piece j's (m, l) ----
    float den = 0.f, mx = -CUDART_INF_F, o[E];
#pragma unroll
    for (int q = 0; q < E; ++q) o[q] = 0.f;
    for (int j0 = 0; j0 < n_pieces; j0 += 32) {
        const int jl = j0 + lane;
        const uint32_t live = cu.live[j0 >> 5];
        float2 ml = make_float2(-CUDART_INF_F, 0.f);
        if (jl < n_pieces && ((live >> lane) & 1u)) ml = P.part_ml[rec_of(jl)];
        const float mnew = fmaxf(mx, warp_max(ml.x));
        if (mnew == -CUDART_INF_F) continue;
        const float rescale = weight(mx - mnew);             // 0 on the first live batch
        den *= rescale;
#pragma unroll
        for (int q = 0; q < E; ++q) o[q] *= rescale;
        mx = mnew;
        const float wl = ml.x == -CUDART_INF_F ? 0.f : weight(ml.x - mx);
        den += warp_sum(ml.y * wl);
        const int nb = min(32, n_pieces - j0);
        for (int u0 = 0; u0 < nb; u0 += 4) {
            float v[4][E], w[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                w[u] = u0 + u < nb ? __shfl_sync(kFull, wl, u0 + u) : 0.f;
                if (w[u] != 0.f) {
                    load_row(P.part_o + rec_of(j0 + u0 + u) * D + lane * E, v[u]);
                } else {
#pragma unroll
                    for (int q = 0; q < E; ++q) v[u][q] = 0.f;
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int q = 0; q < E; ++q) o[q] = fmaf(v[u][q], w[u], o[q]);
        }
    }
    store_row(o, mx, den);
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = []() -> EncodeTiledFn {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess) return nullptr;
        return q == cudaDriverEntryPointSuccess ? reinterpret_cast<EncodeTiledFn>(p) : nullptr;
    }();
    return fn;
}

// [layers][rows][heads][d] bf16 tensor (layer_stride elements between layers), box = (64 elements, box_heads,
// box_rows, one layer), 128-byte swizzle, zero fill
bool make_map(CUtensorMap* tm, const void* base, int d, int heads, long long rows, int box_heads, int box_rows, int layers,
              long long layer_stride) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) return false;
    if (layers <= 1) { layers = 1; layer_stride = rows * heads * d; }
    cuuint64_t dims[4] = {(cuuint64_t)d, (cuuint64_t)heads, (cuuint64_t)rows, (cuuint64_t)layers};
    cuuint64_t strides[3] = {(cuuint64_t)d * 2, (cuuint64_t)d * 2 * heads, (cuuint64_t)layer_stride * 2};
    cuuint32_t box[4] = {64, (cuuint32_t)box_heads, (cuuint32_t)box_rows, 1};
    cuuint32_t es[4] = {1, 1, 1, 1};
    return enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Grid shape.  A class is one row-block pair (256 query rows: both row blocks share every K/V tile in
// shared memory) or, when such fused units would leave most SMs without work, one row block (128 rows).
// CTAs per class: the grid is one CTA per SM, but at least two tiles per CTA when every sequence has the longest prefix (four
// instead of two, us: 32 / 8 heads, 1000 tokens 16.0 / 14.6; 4 / 4 heads, d = 64, 500 tokens 13.6 / 11.5; 16 / 16 heads, 1000 tokens
// 14.5 / 13.6; but 32 / 8 heads, 2048 tokens 16.5 / 17.1).  Both decisions look at the tiles of the whole launch, all its
// layers: 32 layers of one sequence with 2048 tokens (32 / 8 heads, d = 128) run as 148 CTAs of fused units, where one layer
// alone would be split into half units on 128 CTAs.
void plan_grid(const radar_ctx* ctx, int B, int Hq, int Hkv, int max_prefix_len, int layers, int* n_blk, int* n_cls, int* ncc,
               bool* whole) {
    const int G = Hq / Hkv;
    const int blocks = (kMaxNodes + 128 / G - 1) / (128 / G);         // row blocks of a full tree
    const long long unit_tiles = (long long)layers * B * Hkv * ((max_prefix_len + kTileKeys - 1) / kTileKeys + 1);
    int nb = 2;
    if (blocks > 1 && unit_tiles * ((blocks + 1) / 2) < 4LL * ctx->sm_count) nb = 1;
    const int cls = (blocks + nb - 1) / nb;
    long long per = std::min(ctx->sm_count / cls, kMaxPerClass);
    const long long cap = (unit_tiles + 1) / 2;
    if (per > cap) per = cap;
    if (per < 1) per = 1;
    // All units of one sequence are alike, so where they are no more than the CTAs of a class a grid can be chosen in
    // which every CTA has one piece of one unit and pays for one segment (fill and epilogue, what tile_costs books per
    // unit) and not for two.  Not where that leaves so many CTAs unused that the pieces get longer than what it saves.
    // (Attention + combine, d = 128: 40 / 40 heads, 2048 tokens 22.9 -> 19.6 us; 16 / 16 heads, 1000 tokens 14.8 -> 13.6.)
    const long long units = (long long)layers * Hkv, tiles = unit_tiles / (B * units);
    *whole = false;
    if (B == 1 && units <= per) {
        const TileCosts tc = tile_costs(cls);
        const int w = nb > 1 && blocks > 1 ? tc.two : tc.one;
        const long long pieces = std::max(1ll, std::min(tiles / 2, per / units));
        *whole = (tiles + pieces - 1) / pieces * w <= units * (tiles * w + tc.unit) / per + 2 * tc.unit / 3;
        if (*whole) per = units * pieces;
    }
    *n_blk = nb;
    *n_cls = cls;
    *ncc = (int)per;
}

}  // namespace

bool tree_attn_tc_supported(const radar_attn_args* a) {
    if (a->dtype != RADAR_BF16 || (a->d != 64 && a->d != 128)) return false;
    const int G = a->Hq / a->Hkv;
    if (G < 1 || G > kTcMaxRatio) return false;
    // Ratios that do not divide 128 leave the last 128 % G rows of a row block idle (2 of 128 at G = 3 and 7) and take two
    // products a tile for their probabilities, and are still far ahead of the FMA kernel (one layer, 61 tree rows, d = 128, us
    // FMA / this kernel: 24 / 8 heads, B = 1, 2048 tokens 119 / 21; B = 4, 300 tokens 101 / 23; 28 / 4 heads, B = 2, 4096 tokens
    // 444 / 31), but for launches that are all latency, where the FMA kernel's one wave of small blocks is done before this
    // one's pipeline has filled.  Where the two cross is a matter of the work (61 rows, FMA / this one; in units of the line
    // below): 24 / 8 heads of d = 64, B = 1, 64 tokens (0.7) 10.5 / 12.3, 128 (1.0) 10.6 / 11.8, 192 (1.3) 13.6 / 13.1; 28 / 4 heads,
    // 128 (1.2) 13.5 / 12.0; 3 heads, 256 (0.2) 8.4 / 13.0; d = 128: 3 / 1 heads, B = 4, 128 (1.0) 10.0 / 13.1, 28 / 4 heads, 0 (0.8)
    // 13.3 / 15.6, 64 (1.6) 13.9 / 13.3.  Several layers are one launch here and one each there.
    if ((128 % G) != 0 && a->n_layers <= 1 && (long long)a->B * a->Hq * (a->max_prefix_len + kMaxNodes) * a->d <= kLatencyWork) return false;
    if (a->cache_rows < 0 || a->cache_rows >= (1ll << 31) || (long long)a->B * kMaxNodes >= (1ll << 31)) return false;
    const uintptr_t al = reinterpret_cast<uintptr_t>(a->Q) | reinterpret_cast<uintptr_t>(a->Kc) |
                         reinterpret_cast<uintptr_t>(a->Vc) | reinterpret_cast<uintptr_t>(a->Kt) |
                         reinterpret_cast<uintptr_t>(a->Vt) | reinterpret_cast<uintptr_t>(a->O);
    return (al & 15) == 0 && encode_fn() != nullptr;
}

// partial records (two per CTA) and the cut-unit table of a grid
static size_t partial_bytes(size_t grid, int d) {
    const size_t rec = grid * 2 * kPairRows;
    return align_up(rec * sizeof(float2), 256) + align_up(rec * d * sizeof(float), 256) + align_up(grid * sizeof(CutUnit), 256);
}

size_t tree_attn_tc_workspace_bytes(const radar_ctx* ctx, int B, int Hq, int Hkv, int d, int max_prefix_len) {
    // the grid of any number of layers: it grows with them up to one CTA per SM
    int n_blk, n_cls, ncc;
    bool whole;
    plan_grid(ctx, B, Hq, Hkv, max_prefix_len, 1, &n_blk, &n_cls, &ncc, &whole);
    return partial_bytes((size_t)std::max(n_cls * ncc, ctx->sm_count), d);
}

template <int D, bool TWO, bool PAGED, bool FINE>
static int launch_tc(radar_ctx* ctx, TcParams& P, cudaStream_t stream) {
    const radar_attn_args& a = P.a;
    CUtensorMap tmQ, tmKc, tmVc, tmKt, tmVt;
    const long long tree_rows = (long long)a.B * kMaxNodes;
    const bool have_prefix = a.Kc != nullptr && a.Vc != nullptr && a.cache_rows > 0;
    const int cache_box = a.block_table != nullptr && a.page_size < kTileKeys ? a.page_size : kTileKeys;   // rows per TMA box
    const int L = P.n_layers;
    if (!make_map(&tmQ, a.Q, D, a.Hq, tree_rows, P.G, P.nodes_per_rb, L, a.q_layer_stride) ||
        !make_map(&tmKt, a.Kt, D, a.Hkv, tree_rows, 1, kTreeKeys, L, a.tree_kv_layer_stride) ||
        !make_map(&tmVt, a.Vt, D, a.Hkv, tree_rows, 1, kTreeKeys, L, a.tree_kv_layer_stride) ||
        !make_map(&tmKc, have_prefix ? a.Kc : a.Kt, D, a.Hkv, have_prefix ? a.cache_rows : tree_rows, 1, cache_box, L,
                  have_prefix ? a.cache_layer_stride : a.tree_kv_layer_stride) ||
        !make_map(&tmVc, have_prefix ? a.Vc : a.Vt, D, a.Hkv, have_prefix ? a.cache_rows : tree_rows, 1, cache_box, L,
                  have_prefix ? a.cache_layer_stride : a.tree_kv_layer_stride))
        return RADAR_ERR_CUDA;
    auto* const kernel = FINE ? tree_attn_tc_fine_kernel<D, TWO, PAGED> : tree_attn_tc_kernel<D, TWO, PAGED>;
    RADAR_CUDA_CHECK(radar_opt_in_smem(ctx, RADAR_SMEM_ATTN_TC + 8 * FINE + 4 * (D == 128) + 2 * TWO + PAGED, kernel, (size_t)Smem<D, TWO>::kDynamic));
    {
        radar_launch_scope scope(ctx, RADAR_K_ATTN, stream);
        RADAR_CUDA_CHECK(launch_chained(kernel, dim3((unsigned)(P.n_cls * P.ncc)), dim3(FINE ? kFineThreads : kTcThreads),
                                        (size_t)Smem<D, TWO>::kDynamic, stream, tmQ, tmKc, tmVc, tmKt, tmVt, P));
    }
    RADAR_CUDA_CHECK(cudaGetLastError());
    {
        radar_launch_scope scope(ctx, RADAR_K_ATTN_COMBINE, stream);
        RADAR_CUDA_CHECK(launch_chained(tree_attn_tc_combine_kernel<D, FINE>, dim3((unsigned)(P.n_cls * P.ncc), kPairRows / 8), dim3(256), 0, stream, P));
    }
    RADAR_CUDA_CHECK(cudaGetLastError());
    return RADAR_OK;
}

int tree_attn_tc_launch(radar_ctx* ctx, const radar_attn_args* a, cudaStream_t stream) {
    TcParams P;
    P.a = *a;
    P.G = a->Hq / a->Hkv;
    P.g_magic = (65536u + P.G - 1) / P.G;
    P.nodes_per_rb = 128 / P.G;
    P.rb_rows = P.nodes_per_rb * P.G;
    const float scale = a->scale > 0.f ? a->scale : 1.f / sqrtf((float)a->d);
    const bool fine = 128 % P.G != 0;
    P.scale_log2 = scale * 1.4426950408889634f;
    P.scale_log2_lo = 0.f;
    if (fine) {                          // the second part positive: a score of -inf (a masked one) stays -inf
        const double exact = (a->scale > 0.f ? (double)a->scale : 1.0 / std::sqrt((double)a->d)) * 1.4426950408889634;
        if ((double)P.scale_log2 >= exact) P.scale_log2 = std::nextafterf(P.scale_log2, 0.f);
        P.scale_log2_lo = (float)(exact - (double)P.scale_log2);
    }
    P.cache_rows = a->cache_rows;
    P.status = ctx->d_status;
    P.n_layers = a->n_layers > 1 ? a->n_layers : 1;
    P.o_ls = P.n_layers > 1 ? a->o_layer_stride : 0;
    P.lse_ls = P.n_layers > 1 ? a->lse_layer_stride : 0;
    bool whole;
    plan_grid(ctx, a->B, a->Hq, a->Hkv, a->max_prefix_len, P.n_layers, &P.n_blk, &P.n_cls, &P.ncc, &whole);
    P.pair_rows = P.n_blk * P.rb_rows;
    const TileCosts tc = tile_costs(P.n_cls);
    P.cost_one = tc.one; P.cost_two = tc.two; P.unit_cost = whole ? 0 : tc.unit;
    if (partial_bytes((size_t)P.n_cls * P.ncc, a->d) > a->workspace_bytes)
        return RADAR_ERR_WORKSPACE;
    const size_t rec = (size_t)P.n_cls * P.ncc * 2 * kPairRows;
    P.part_ml = reinterpret_cast<float2*>(a->workspace);
    P.part_o = reinterpret_cast<float*>(reinterpret_cast<char*>(a->workspace) + align_up(rec * sizeof(float2), 256));
    P.cut = reinterpret_cast<CutUnit*>(reinterpret_cast<char*>(P.part_o) + align_up(rec * a->d * sizeof(float), 256));
    const bool two = P.n_blk > 1 && P.nodes_per_rb < kMaxNodes;       // some unit can have two live row blocks
    auto launch = [&](auto d, auto fine_c) {
        constexpr int D = decltype(d)::value;
        constexpr bool F = decltype(fine_c)::value;
        if (a->block_table != nullptr) return two ? launch_tc<D, true, true, F>(ctx, P, stream) : launch_tc<D, false, true, F>(ctx, P, stream);
        return two ? launch_tc<D, true, false, F>(ctx, P, stream) : launch_tc<D, false, false, F>(ctx, P, stream);
    };
    using d64 = std::integral_constant<int, 64>;
    using d128 = std::integral_constant<int, 128>;
    if (a->d == 128) return fine ? launch(d128{}, std::true_type{}) : launch(d128{}, std::false_type{});
    return fine ? launch(d64{}, std::true_type{}) : launch(d64{}, std::false_type{});
}

}  // namespace radar
