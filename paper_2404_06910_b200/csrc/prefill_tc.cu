// Fork-join prefill attention on the Blackwell tensor cores (bf16, head_dim 64 and 128).
// Section 3.2: a row attends to its prompt's preamble and, causally, to its own path.
//
// Work unit ("item"): one or two consecutive query tiles of one segment, for one head; with grouped query heads a tile's 128
// rows are 128 / G rows of the segment for each of G = 2, 4 or 8 heads that share a KV head, so that K and V are loaded once for
// all of them and a tile's rows lie closer to the diagonal.  Its keys are
// the preamble's rows (all visible) followed by the segment's own rows up to the diagonal, as one sequence cut into tiles
// of 64 (the preamble is padded to a multiple of 16 in front of the own rows, so one tile may hold both); key tiles that the
// fork-join mask excludes are never loaded or multiplied.  Short paths behind a preamble are cut into tiles without regard to where one
// ends and the next begins (the rule and its figures: across_pays()): a tile's own keys then start with its first path, and
// every row has a first own key too.  Per query tile and key tile:
//   S = Q K^T     tcgen05.mma, A and B from TMA-staged 128B-swizzled shared memory, fp32 in tensor memory
//   P = softmax   4 warps, one thread per query row, the row's 64 scores in registers: maximum, then exp2 with a lazily
//                 updated reference maximum; P is rounded to bf16 and written over S
//   O += P V      tcgen05.mma with A = P from tensor memory, B = V from shared memory (MN-major)
//
// One persistent block per SM with two "lanes": each lane owns a query tile at a time, with its own softmax
// warpgroup, issuing warp, two S / P buffers and O accumulator (256 tensor-memory columns).  The two tiles of an
// item go to different lanes and share every K and V stage, so a path's keys are loaded once per tile pair; the tiles of
// consecutive items swap lanes (tile B has more keys than tile A), and nothing but the shared stages couples the lanes.
// All of the SM's shared memory is one pool: query slots (the next tile's Q is loaded while the current ones are worked
// on) and four stages each of K and V.
// What sets the pace: 1 024 clk of the exponential unit per key tile of both lanes, 1 280 clk of shared-memory reads by
// their MMAs, a softmax warp's own instruction stream, and for short paths HBM.
// Roles: warps 0-7 softmax (a warpgroup per lane), 8-11 epilogue (O / l -> bf16 -> global), 12 / 13 / 14 K / V / Q loads, 15
// key positions (ALiBi), 16 / 17 MMA issuer of lane 0 / 1, 18 / 19 pass landed K / V tiles on to the lanes (19 cleans ragged V
// tiles).
// A K or V stage may be of use to one lane only, and a waiter that left out fills of a two-phase barrier could mistake an
// older fill for the one it waits for.  So loads arrive on a barrier that one warp waits on fill by fill, which passes the
// stage on to the lanes that use it, on barriers of their own; query slots have a barrier per lane to begin with.
// A lane's issuing warp issues O += P V of tile g and then S = Q K^T of tile g+2 into the same columns without a wait between
// the two: tensor-core operations of one thread execute in order, so S(g+2) overwrites P(g) only after it has been read.
// The warp runs as a whole and only the tcgen05 instructions are predicated on one elected thread: descriptors then live in
// uniform registers and an MMA takes 20 clk to issue (46 to 94 from the branch of one thread, longer than it runs).
// Every mbarrier wait is bounded: on expiry the block records a timeout in the workspace status word, unwinds, frees its
// tensor memory and exits.
// sp_superpose_prefill_rope rotates Q into `out` first and runs the same kernel on it.
// Measured (32 heads of 128, us; before: two blocks per SM, a tile each, K and V loaded per tile): 2 prompts x 400 documents of
// 128-512 rows 3208 -> 2580, 64 prompts x 17 paths behind a prefix of some 390 rows 3224 -> 2724, ALiBi 1366 -> 954; head_dim 64
// (before: fp32 arithmetic) 9387 -> 172.  These launches run at the board's power limit (1.3 to 1.55 GHz): leaving out all
// exponentials gains 2 %, so time follows the energy of the loads and products rather than any one pipe.
#include <climits>

#include "common.cuh"
#include "prefill_plan.cuh"
#include "tc_ptx.cuh"
#include "tensor_map.cuh"

namespace sp {

using namespace ptx;

constexpr int kBM = 128;              // query rows per tile
constexpr int kBN = kPairKeys;        // keys per tile
constexpr int kTmemCols = 512;        // lane l: S / P buffers at 256 l and 256 l + 64, O at 256 l + 128
constexpr int kLaneCols = 256, kOCol = 128;
constexpr int kTcThreads = 640;
constexpr float kLog2eT = 1.4426950408889634f;
constexpr float kLn2T = 0.6931471805599453f;
constexpr float kRescaleThreshold = 8.f;   // log2 units: rescale O only when the max grows by > 2^8

enum { WARP_EPI = 8, WARP_K = 12, WARP_V, WARP_Q, WARP_POS, WARP_MMA, WARP_PASS = WARP_MMA + 2 };

// SPLIT_P: P is carried as the sum of two bf16 numbers (16 bits of mantissa) and the second product runs twice.  Set for
// head_dim 64, which is then as precise as fp32 arithmetic, and for query rows only: relative to the maximum over a first
// key tile, P in one bf16 number is 2.27e-3 of the norm from 64-bit results there (8 prompts x 100 documents), as two it is
// 1.66e-3, the rounding of the output.  Cost: 8 prompts x 100 documents, two heads to a KV head, 326 -> 341 us; four, 197 -> 217.
template <int D, bool ALIBI, bool SPLIT> struct TcConfig {
    static constexpr bool SPLIT_P = SPLIT, EXACT = D == 64;
    static constexpr int HALVES = D / 64;                       // 64-column halves of a row (one 128-byte swizzle atom each)
    static constexpr int Q_BYTES = kBM * D * 2, KV_BYTES = kBN * D * 2;
    static constexpr int NQ = D == 64 ? 4 : 3;                  // query slots
    static constexpr int NKV = 4;                               // K and V stages, each (a power of two)
    static constexpr int X_OFF = NQ * Q_BYTES + 2 * NKV * KV_BYTES;
    static constexpr int PK_OFF = X_OFF + 2 * kBM * 4;          // behind the row sums [lane][row]
    static constexpr int BAR_OFF = PK_OFF + (ALIBI ? NKV * kBN * 4 : 0);   // behind the key positions [V stage][key] (ALiBi)
    // barriers; [lane][n] where a barrier is a lane's own (S_FULL, O_DONE, P: [lane][buffer])
    static constexpr int BAR_Q_FULL = 0, BAR_Q_EMPTY = BAR_Q_FULL + 2 * NQ, BAR_K_FULL = BAR_Q_EMPTY + NQ,
                         BAR_K_READY = BAR_K_FULL + NKV, BAR_V_FULL = BAR_K_READY + 2 * NKV, BAR_V_READY = BAR_V_FULL + NKV,
                         BAR_POS = BAR_V_READY + 2 * NKV, BAR_S_FULL = BAR_POS + 2 * NKV, BAR_O_DONE = BAR_S_FULL + 4,
                         BAR_DRAIN = BAR_O_DONE + 4, BAR_K_EMPTY = BAR_DRAIN + 2, BAR_V_EMPTY = BAR_K_EMPTY + NKV, BAR_P = BAR_V_EMPTY + NKV,
                         BAR_L_READY = BAR_P + 4, BAR_X_FREE = BAR_L_READY + 2, BAR_O_FREE = BAR_X_FREE + 2,
                         BAR_COUNT = BAR_O_FREE + 2;
    static constexpr int SMEM = BAR_OFF + BAR_COUNT * 8 + 16;
    // No other block with operands in shared memory fits on the SM: less than 1 KB of it is left besides the 1 KB that each block
    // has reserved (and 4 096 registers).
    static constexpr bool ALONE = SMEM + 3 * 1024 > 228 * 1024;
    // Registers per thread: at launch (what __launch_bounds__ makes of 65 536), and after the split.  The softmax warps take
    // what the others give back, which has to add up; only they grow.
    static constexpr int R_LAUNCH = 96, R_SOFT = 128, R_EPI = 96, R_LOAD = 56, R_MMA = 64;
    static_assert(2 * R_SOFT + R_EPI + R_LOAD + R_MMA <= kTcThreads / 128 * R_LAUNCH, "registers of a block");
    static_assert(R_EPI == R_LAUNCH, "a function called from the epilogue may use what the kernel was launched with");
    static_assert(R_SOFT >= R_LAUNCH && R_LOAD <= R_LAUNCH && R_MMA <= R_LAUNCH, "direction of setmaxnreg");
};
static_assert(TcConfig<128, false, false>::SMEM <= 232448 && TcConfig<128, true, false>::SMEM <= 232448, "one block's shared memory");

static_assert(TcConfig<128, false, true>::ALONE && TcConfig<128, true, true>::ALONE && !TcConfig<64, true, true>::ALONE, "who shares an SM");

// The instruction stream of the softmax warps is what paces a lane: three-input maxima and two-lane fp32 forms.
__device__ __forceinline__ float fmax3(float a, float b, float c)
{
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ float ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// n ones from bit 0 up, for any n (negative: none, above 32: all)
__device__ __forceinline__ uint32_t low_bits(int n)
{
    uint32_t m;
    asm("bmsk.clamp.b32 %0, 0, %1;" : "=r"(m) : "r"(max(n, 0)));
    return m;
}

// Which rows make up a tile.
enum TileRows {
    SEGMENT_ROWS,                     // of one segment and head
    HEAD_ROWS,                        // of one segment and several heads of a KV head
    ACROSS_ROWS                       // of consecutive paths of a prompt and one head
};

struct TcParams {
    CUtensorMap maps[3][3];           // [K, V, Q][box: a whole tile of a head's rows, 32 rows x 64 columns, 16 rows x 64 columns]
    const TcHeader *hdr;
    const TcPair *pairs;
    uint32_t *status;
    __nv_bfloat16 *out;
    float *lse;
    const __nv_bfloat16 *q, *k, *v;
    int n_heads, n_kv_heads;
    int log_rows, n_units, units_per_kv;   // rows of a head in a tile (log2); units of G heads in all and per KV head
    int64_t total_tokens;
    float scale_log2e;
    int wide_stores;                  // out is 32-byte aligned
    const float *pos, *slopes;        // ALiBi variant: token positions [T], head slopes [H]
    const int32_t *path_start;        // ACROSS_ROWS
    int n_paths;
    int stall_producer;               // test hook: the producers issue no load, so every wait runs out
};

// Every role walks the block's items in the same grid-stride order; heads vary fastest, so blocks running side by
// side read neighbouring head slices of the same token rows.
// Keys are numbered u = 0 .. : the preamble at [0, pre_len), own rows at [p16, ...), p16 = pre_len rounded up to 16.
template <bool ACROSS> struct Walk {
    const TcPair *pairs;
    uint32_t pair, n_pairs, item_no;
    int h, n_units, dp, dh;           // h: unit of G heads
    TcPair t;
    int first_path, lo_b;             // ACROSS: tile A's first path (-1: one segment), key number where tile B's first one starts
    __device__ __forceinline__ explicit Walk(const TcParams &p)
    {
        pairs = p.pairs; n_pairs = p.hdr->n_tiles; n_units = p.n_units; item_no = 0xffffffffu;
        dp = gridDim.x / n_units; dh = gridDim.x - dp * n_units;
        pair = blockIdx.x / n_units; h = blockIdx.x - pair * n_units;
        // one step back: next() comes before every item, the first one included, so that its code exists once per role
        h -= dh; pair -= dp;
        if (h < 0) { h += n_units; --pair; }
    }
    __device__ __forceinline__ bool next()
    {
        ++item_no; pair += dp; h += dh;
        if (h >= n_units) { h -= n_units; ++pair; }
        if (pair >= n_pairs) return false;
        const int4 *src = reinterpret_cast<const int4 *>(pairs + pair);
        const int4 a = src[0], b = src[1];
        t.own_base = a.x; t.q_u = a.y; t.pre_row = a.z; t.pre_len = a.w;
        t.p16 = b.x; t.rows_ab = b.y; t.steps_a = b.z; t.steps = b.w;
        if (ACROSS) {
            first_path = b.x; lo_b = b.z;
            t.p16 = (t.pre_len + 15) & ~15;
            t.steps_a = (t.q_u + rows_a() + kBN - 1) / kBN;
        }
        return true;
    }
    __device__ __forceinline__ int rows_a() const { return t.rows_ab & 0xffff; }
    __device__ __forceinline__ int rows_b() const { return t.rows_ab >> 16; }
    __device__ __forceinline__ int n_q() const { return rows_b() ? 2 : 1; }
    __device__ __forceinline__ int end() const { return t.q_u + rows_a() + rows_b(); }                  // keys of the item
    __device__ __forceinline__ int lane_a() const { return item_no & 1; }                               // tile A's lane
    // ACROSS: tile B has no use for key tiles behind the preamble and in front of its first path (there are more behind them)
    __device__ __forceinline__ int gap_at() const { return (t.pre_len + kBN - 1) / kBN; }
    __device__ __forceinline__ int gap() const { return ACROSS ? max(lo_b / kBN - gap_at(), 0) : 0; }
    __device__ __forceinline__ bool in_gap(int j) const { return ACROSS && (uint32_t)(j - gap_at()) < (uint32_t)gap(); }
    __device__ __forceinline__ bool used_by(int lane, int j) const { return lane == lane_a() ? j < t.steps_a : rows_b() > 0 && !in_gap(j); }
    __device__ __forceinline__ bool one_lane(int j) const { return rows_b() == 0 || j >= t.steps_a || in_gap(j); }
};

// What a lane does in an item: tile A goes to lane item_no & 1, tile B (if any) to the other one.
struct LaneTile {
    int b, q_u, rows, end, steps;     // b: it is tile B; q_u: key number of its first row; no steps: the lane has none
    int gap_at, gap;                  // ACROSS: its steps without [gap_at, gap_at + gap)
    LaneTile() = default;
    template <bool ACROSS> __device__ __forceinline__ LaneTile(const Walk<ACROSS> &w, int lane)
    {
        b = (w.item_no & 1) ^ lane;
        rows = b ? w.rows_b() : w.rows_a();
        q_u = w.t.q_u + (b ? w.rows_a() : 0);
        end = q_u + rows;
        steps = b ? (rows ? w.t.steps : 0) : w.t.steps_a;
        gap_at = w.gap_at();
        gap = b ? w.gap() : 0;
    }
};

template <int N> struct Ring {        // stage and parity of a ring of N barriers
    uint32_t i = 0, ph = 0;
    __device__ __forceinline__ void skip(uint32_t n)      // n <= N, or N a power of two
    {
        i += n;
        if ((N & (N - 1)) == 0) { ph ^= i / N & 1; i &= N - 1; }
        else if (i >= N) { i -= N; ph ^= 1; }
    }
    __device__ __forceinline__ void next() { skip(1); }
};

// ---- rows with values that are not finite ------------------------------------------------
// Keys that a row does not see have a P of exactly zero, but 0 x Inf and 0 x NaN reach O.  Where such keys share tiles with those it does
// see, the row's values that are not finite are computed again, in fp32 over exactly the keys it sees, by the row's warp: a lane takes
// every 32nd key's score, then D / 32 columns of the sums.  Not where nothing hidden can be the cause: a value of the preamble or of the row's
// own keys belongs there.  A row of 740 keys takes its warp 36 us; a look at the rows alone doubles a launch's time.
// A lane's columns of a row: D / 64 words of two bf16 numbers each.
template <int D> struct Words {
    uint32_t w[D / 64];
    __device__ __forceinline__ void load(const void *row)
    {
        if constexpr (D == 128) { const uint2 x = static_cast<const uint2 *>(row)[threadIdx.x & 31]; w[0] = x.x; w[1] = x.y; }
        else w[0] = static_cast<const uint32_t *>(row)[threadIdx.x & 31];
    }
    __device__ __forceinline__ void store(void *row) const
    {
        if constexpr (D == 128) static_cast<uint2 *>(row)[threadIdx.x & 31] = make_uint2(w[0], w[1]);
        else static_cast<uint32_t *>(row)[threadIdx.x & 31] = w[0];
    }
};
// Ones in the halves of a word that are not finite, or NaN.
__device__ __forceinline__ uint32_t not_finite(uint32_t x)
{
    return ((x & 0x7f80u) == 0x7f80u ? 0xffffu : 0u) | ((x & 0x7f800000u) == 0x7f800000u ? 0xffff0000u : 0u);
}
__device__ __forceinline__ uint32_t is_nan(uint32_t x) { return ((x & 0x7fffu) > 0x7f80u ? 0xffffu : 0u) | ((x & 0x7fff0000u) > 0x7f800000u ? 0xffff0000u : 0u); }
template <int D> __device__ __forceinline__ const __nv_bfloat16 *value_row(const TcParams &p, int64_t row, int kv_head) { return p.v + (row * p.n_kv_heads + kv_head) * D; }

// The first and the last of the segment's keys [u0, u1) whose values are not all finite.
template <int D>
__device__ __forceinline__ void bad_values(const TcParams &p, const TcPair &t, int kv_head, int u0, int u1, int &first, int &last)
{
    constexpr int PIECES = D / 8;                        // of 16 bytes in a row
    const int lane = threadIdx.x & 31;
    first = INT_MAX; last = -1;
#pragma unroll 8
    for (int u = u0 + lane / PIECES; u < u1; u += 32 / PIECES) {
        const uint4 v = reinterpret_cast<const uint4 *>(value_row<D>(p, t.own_base + u, kv_head))[lane % PIECES];
        if (not_finite(v.x) | not_finite(v.y) | not_finite(v.z) | not_finite(v.w)) { first = min(first, u); last = u; }
    }
    first = __reduce_min_sync(0xffffffffu, first);
    last = __reduce_max_sync(0xffffffffu, last);
}

// The row with key number `last`, whose own keys start at number `from`; y: its columns of this lane.
template <int D, bool ALIBI>
__device__ __forceinline__ void exact_row(const TcParams &p, const TcPair &t, int head, int kv_head, int from, int last, Words<D> &y)
{
    const int lane = threadIdx.x & 31, n = t.pre_len + last - from + 1;
    const int64_t own = t.own_base + last;
    Words<D> v;
    v.load(value_row<D>(p, own, kv_head));
    bool cause = false;                                  // a NaN of the row's own value is its own
#pragma unroll
    for (int i = 0; i < D / 64; ++i) cause |= (not_finite(y.w[i]) & ~is_nan(v.w[i])) != 0u;
    if (!__any_sync(0xffffffffu, cause)) return;
    const uint4 *q = reinterpret_cast<const uint4 *>(p.q + (own * p.n_heads + head) * D);
    const float pq = ALIBI ? p.pos[own] : 0.f, slope = ALIBI ? p.slopes[head] * kLog2eT : 0.f;
    auto packed_row = [&](int i) { return (int64_t)i + (i < t.pre_len ? t.pre_row : t.own_base + from - t.pre_len); };
    float m = -INFINITY, l = 0.f, acc[D / 32];
#pragma unroll
    for (int e = 0; e < D / 32; ++e) acc[e] = 0.f;
#pragma unroll 1
    for (int i0 = 0; i0 < n; i0 += 32) {
        const int64_t row = packed_row(min(i0 + lane, n - 1));
        const uint4 *k = reinterpret_cast<const uint4 *>(p.k + (row * p.n_kv_heads + kv_head) * D);
        float s = 0.f;
#pragma unroll 4
        for (int c = 0; c < D / 8; ++c) {
            const uint4 x = q[c], z = k[c];
            s = fmaf(bf16_lo(x.x), bf16_lo(z.x), s); s = fmaf(bf16_hi(x.x), bf16_hi(z.x), s);
            s = fmaf(bf16_lo(x.y), bf16_lo(z.y), s); s = fmaf(bf16_hi(x.y), bf16_hi(z.y), s);
            s = fmaf(bf16_lo(x.z), bf16_lo(z.z), s); s = fmaf(bf16_hi(x.z), bf16_hi(z.z), s);
            s = fmaf(bf16_lo(x.w), bf16_lo(z.w), s); s = fmaf(bf16_hi(x.w), bf16_hi(z.w), s);
        }
        s *= p.scale_log2e;
        if (ALIBI) s -= slope * fabsf(pq - p.pos[row]);
        if (i0 + lane >= n) s = -INFINITY;
        const float m_new = fmaxf(m, warp_max(s)), ref = m_new == -INFINITY ? 0.f : m_new, a = ex2(m - ref), w = ex2(s - ref);
        m = m_new;
        l = fmaf(l, a, warp_sum(w));
#pragma unroll
        for (int e = 0; e < D / 32; ++e) acc[e] *= a;
        const int here = min(32, n - i0);
#pragma unroll 8
        for (int j = 0; j < here; ++j) {
            const float wj = __shfl_sync(0xffffffffu, w, j);
            v.load(value_row<D>(p, packed_row(i0 + j), kv_head));
#pragma unroll
            for (int i = 0; i < D / 64; ++i) {
                acc[2 * i] = fmaf(wj, bf16_lo(v.w[i]), acc[2 * i]);
                acc[2 * i + 1] = fmaf(wj, bf16_hi(v.w[i]), acc[2 * i + 1]);
            }
        }
    }
    const float inv = 1.f / l;
#pragma unroll
    for (int i = 0; i < D / 64; ++i) {                   // the finite ones are right as they are
        const uint32_t again = not_finite(y.w[i]);
        y.w[i] = (y.w[i] & ~again) | (pack_bf16x2(acc[2 * i] * inv, acc[2 * i + 1] * inv) & again);
    }
}

// The same for tiles of one segment, head_dim 64, before a row is stored (the output may take Q's place): the rows of the warp that
// are not finite; o: the bf16 pairs of this thread's.  Rows in front of one whose values are not finite share tiles with it.  Called, not
// inlined, because it is rare and the loop it is called from is sensitive to registers (inlined, ALiBi, 16 prompts x 20 documents: 344 -> 357
// us); the epilogue's warps keep the registers that the kernel was launched with, so any called function has enough.
template <bool ALIBI, TileRows ROWS>
__device__ __noinline__ void exact_rows64(const TcParams &p, uint32_t pair, int unit, int b, int quad, uint32_t *o)
{
    const TcPair t = p.pairs[pair];
    const int lane = threadIdx.x & 31, log_rows = ROWS == HEAD_ROWS ? p.log_rows : 7, row = quad * 32 + lane, hr = row & ((1 << log_rows) - 1);
    const int rows_a = t.rows_ab & 0xffff, rows_b = t.rows_ab >> 16, q_u = t.q_u + (b ? rows_a : 0), n_rows = b ? rows_b : rows_a;
    const int kv_head = unit / p.units_per_kv, head = (unit << (7 - log_rows)) + (row >> log_rows);
    uint32_t bad = 0u;
    for (int i = 0; i < 32; ++i) bad |= not_finite(o[i]);
    uint32_t rows = __ballot_sync(0xffffffffu, bad && hr < n_rows);
    int bad_first, bad_last;
    bad_values<64>(p, t, kv_head, q_u, min((q_u + n_rows + 15) & ~15, t.q_u + rows_a + rows_b), bad_first, bad_last);
#pragma unroll 1
    for (; rows; rows &= rows - 1) {
        const int r = __ffs(rows) - 1, last = q_u + __shfl_sync(0xffffffffu, hr, r);
        if (bad_last <= last) continue;
        Words<64> y;                                     // row r from its thread to a lane each, and back
#pragma unroll 1
        for (int i = 0; i < 32; ++i) {
            const uint32_t x = __shfl_sync(0xffffffffu, o[i], r);
            if (lane == i) y.w[0] = x;
        }
        exact_row<64, ALIBI>(p, t, __shfl_sync(0xffffffffu, head, r), kv_head, t.p16, last, y);
#pragma unroll 1
        for (int i = 0; i < 32; ++i) {
            const uint32_t x = __shfl_sync(0xffffffffu, y.w[0], i);
            if (lane == r) o[i] = x;
        }
    }
}

// Tiles across paths: the rows that other paths' values may have reached, once more, by the warp that has stored them: behind the last item,
// when no other warp waits for this one, and from the stored output.
template <int D, bool ALIBI> __device__ __forceinline__ void exact_rows_across(const TcParams &p, int quad)
{
#pragma unroll 1
    for (Walk<true> w(p); w.next();) {
        // rows of one segment meet only their own later rows, head_dim 128: as in a launch without tiles across paths
        if (D == 128 && w.first_path < 0) continue;
#pragma unroll 1
        for (int b = 0; b < w.n_q(); ++b) {
            const LaneTile t(w, w.lane_a() ^ b);
            const int kv_head = w.h / p.units_per_kv, row0 = w.t.own_base + t.q_u + quad * 32, n = min(32, t.rows - quad * 32);
            auto out_row = [&](int r) { return p.out + ((int64_t)(row0 + r) * p.n_heads + w.h) * D; };
            uint32_t rows = 0u;                  // a bit per row with values that are not finite
#pragma unroll 4
            for (int r = 0; r < n; ++r) {
                Words<D> y;
                y.load(out_row(r));
#pragma unroll
                for (int i = 0; i < D / 64; ++i) rows |= not_finite(y.w[i]) ? 1u << r : 0u;
            }
            rows = __reduce_or_sync(0xffffffffu, rows);
            int bad_first = INT_MAX, bad_last = -1;
            if (rows) bad_values<D>(p, w.t, kv_head, w.t.p16, min((t.end + 15) & ~15, w.end()), bad_first, bad_last);
#pragma unroll 1
            for (; rows; rows &= rows - 1) {
                const int r = __ffs(rows) - 1, last = t.q_u + quad * 32 + r;
                int start = w.t.own_base + w.t.p16;               // of the row's own path
                if (w.first_path >= 0)
                    for (int i = w.first_path + 1; i < p.n_paths && p.path_start[i] > start && p.path_start[i] <= row0 + r; ++i) start = p.path_start[i];
                const int from = start - w.t.own_base;
                if (bad_first >= from && bad_last <= last) continue;
                Words<D> y;
                y.load(out_row(r));
                exact_row<D, ALIBI>(p, w.t, w.h, kv_head, from, last, y);
                y.store(out_row(r));
            }
        }
    }
}

// Inlined it made head_dim 64 slower (16 prompts x 17 paths behind 390 rows 459 -> 473 us), called head_dim 128 (497 -> 507).
template <bool ALIBI> __device__ __noinline__ void exact_rows_across64(const TcParams &p, int quad) { exact_rows_across<64, ALIBI>(p, quad); }

template <int N> __device__ __forceinline__ void reg_alloc() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N)); }
template <int N> __device__ __forceinline__ void reg_dealloc() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N)); }

// ALIBI: scores get -slope_h * |pos_q - pos_k| before the softmax (Section 3.2.2: real-valued positions are no obstacle
// for ALiBi).
// ROWS: what makes up a tile.  Tiles of several heads are a kernel of their own because their index arithmetic cost a launch of single heads
// 1.5 % (630 against 621 us, measured on 32 query rows of 800 paths, which go to prefill_qonly.cu now).
template <int D, bool ALIBI, TileRows ROWS, bool SPLIT>
__global__ void __launch_bounds__(kTcThreads, 1) prefill_tc_kernel(const __grid_constant__ TcParams p)
{
    constexpr bool ACROSS = ROWS == ACROSS_ROWS;
    using C = TcConfig<D, ALIBI, SPLIT>;
    using Walk = Walk<ACROSS>;
    const int log_rows = ROWS == HEAD_ROWS ? p.log_rows : 7;
    extern __shared__ __align__(1024) unsigned char smem[];
    unsigned char *sQ = smem, *sK = smem + C::NQ * C::Q_BYTES, *sV = sK + C::NKV * C::KV_BYTES;
    float *x_l = reinterpret_cast<float *>(smem + C::X_OFF);                            // [lane][row] row sums
    float *s_pos = reinterpret_cast<float *>(smem + C::PK_OFF);                         // [V stage][key] positions (ALiBi)
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + C::BAR_OFF);
    uint32_t *tmem_base_s = reinterpret_cast<uint32_t *>(bars + C::BAR_COUNT);

    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    if (threadIdx.x < C::BAR_COUNT) {
        const int i = threadIdx.x;
        int count = 1;
        if (i >= C::BAR_K_EMPTY && i < C::BAR_P) count = 2;      // both lanes
        if (i >= C::BAR_P) count = 4;                            // four warps
        mbar_init(&bars[i], count);
        fence_mbar_init();
    } else if (threadIdx.x >= 96 && threadIdx.x < 105) {
        prefetch_tmap(&p.maps[0][0] + (threadIdx.x - 96));
    }
    auto take_tmem = [&]() {
        if (warp == WARP_MMA) { tmem_alloc(tmem_base_s, kTmemCols); tmem_relinquish(); }
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        pdl_trigger();
    };
    // pdl_wait(): the tile list and everything before it in the stream.  Where another kernel's block fits beside this one, tensor
    // memory is taken behind the wait and before the next kernel is let in: a block that held it while it waits, or one of a
    // dependent's that took it first, could keep its neighbour waiting for columns that are freed only after that neighbour has
    // ended.  Costs 0.2 us of a launch.
    if (C::ALONE) { take_tmem(); pdl_wait(); } else { pdl_wait(); take_tmem(); }
    const uint32_t tb = *tmem_base_s;
    bool ok = (smem_u32(smem) & 1023u) == 0;      // the swizzle atoms need it; reported like an expired wait

    // Each warpgroup's branch starts with its own setmaxnreg and the branches do not meet again before the end: the
    // compiler allots registers by region, and a region reached with two different limits could use more than one of them has.
    if (warp >= WARP_K && warp < WARP_MMA) {
        reg_dealloc<C::R_LOAD>();
        if (warp != WARP_POS) {
            // ---------------------------------------------------------------- K, V and Q tiles (TMA), one code for the three
            // A tile lands as [half][64 (Q: 128) rows][128 bytes], swizzled.  A whole tile of one segment is one box; otherwise
            // 32- and 16-row boxes per half, so that a key tile may hold the end of the preamble and the start of the own rows
            // and ragged ends pull in at most 15 rows nobody needs.
            if (!p.stall_producer) {
                const uint32_t lead = elect_one();
                const bool is_q = warp == WARP_Q;
                const int kind = warp - WARP_K, slots = is_q ? C::NQ : C::NKV, tile_rows = is_q ? kBM : kBN;
                uint64_t *full = &bars[is_q ? C::BAR_Q_FULL : (kind ? C::BAR_V_FULL : C::BAR_K_FULL)];
                uint64_t *empty = &bars[is_q ? C::BAR_Q_EMPTY : (kind ? C::BAR_V_EMPTY : C::BAR_K_EMPTY)];
                unsigned char *base = is_q ? sQ : (kind ? sV : sK);
                const CUtensorMap *maps = p.maps[kind];
                uint64_t pol;                         // query tiles are read once: leave L2 to the K / V rows
                if (is_q) pol = l2_policy_evict_first(); else pol = l2_policy_evict_normal();
                const int log_g = 7 - log_rows, heads = is_q ? 1 << log_g : 1;       // heads in a tile of this kind
                int slot = 0;
                uint32_t ph = 1, n = 0, last = 0, fills = 0;      // per slot: barrier of its last fill; per barrier: parity of the next one
#pragma unroll 1
                for (Walk w(p); ok && w.next();) {
                    const int head = (is_q ? w.h << log_g : w.h / p.units_per_kv) * C::HALVES, units = is_q ? w.n_q() : w.t.steps;
#pragma unroll 1
                    for (int j = 0; j < units; ++j) {
                        if (!(ok = mbar_wait_warp(empty + slot, ph))) break;
                        // rows [u0, u1) of the segment's key numbering; a query tile is part of its own rows
                        const int u0 = is_q ? w.t.q_u + (j ? w.rows_a() : 0) : j * kBN;
                        const int have = is_q ? (j ? w.rows_b() : w.rows_a()) : min(kBN, w.end() - u0);
                        const int u1 = u0 + ((have + 15) & ~15), split = is_q ? u0 : min(max(w.t.p16, u0), u1);
                        const int to = is_q ? (w.lane_a() ^ j) * C::NQ + slot : slot;
                        uint64_t *bar = full + to;
                        last = (last & ~(0xffu << (8 * slot))) | (uint32_t)to << (8 * slot);
                        fills ^= 1u << to;
                        unsigned char *dst = base + slot * (tile_rows * D * 2);
                        if (lead) mbar_expect_tx(bar, (uint32_t)((u1 - u0) * heads) * (D * 2));
                        __syncwarp();
#pragma unroll 1
                        for (int hq = 0; hq < heads; ++hq) {
                            unsigned char *to_rows = dst + (hq << log_rows) * 128;
#pragma unroll 1
                            for (int u = u0; u < u1;) {
                                const bool pre = u < split;                         // preamble part, then own part
                                const int left = (pre ? split : u1) - u, row = u + (pre ? w.t.pre_row : w.t.own_base);
                                const int box = left == tile_rows ? 0 : (left >= 32 ? 1 : 2);
#pragma unroll 1
                                for (int hh = 0; hh < (box ? C::HALVES : 1); ++hh)
                                    tma_load_3d_hint(lead, to_rows + hh * (tile_rows * 128) + (u - u0) * 128, maps + box, 0, row,
                                                     head + hq * C::HALVES + hh, bar, pol);
                                u += box == 0 ? tile_rows : (box == 1 ? 32 : 16);
                            }
                        }
                        if (lead && !is_q && w.one_lane(j)) mbar_arrive(empty + slot);      // for the lane that has no use for it
                        ++n;
                        if (++slot == slots) { slot = 0; ph ^= 1; }
                    }
                }
                // a wait ran out: the copies in flight must land before the block may exit (bounded)
                if (!ok)
                    for (int i = 0; i < slots && i < (int)n; ++i) {
                        const uint32_t to = last >> (8 * i) & 0xff;
                        mbar_wait_warp(full + to, (fills >> to & 1) ^ 1);
                    }
            }
        } else if (ALIBI) {
            // ---------------------------------------------------------------- key positions, one set per V stage
            Ring<C::NKV> v;
#pragma unroll 1
            for (Walk w(p); ok && w.next();) {
                const int end = w.end();
#pragma unroll 1
                for (int j = 0; j < w.t.steps; ++j, v.next()) {
                    float x[kBN / 32];
#pragma unroll
                    for (int i = 0; i < kBN / 32; ++i) {
                        const int u = j * kBN + i * 32 + lane;
                        x[i] = u < w.t.pre_len || (u >= w.t.p16 && u < end) ? p.pos[u + (u < w.t.pre_len ? w.t.pre_row : w.t.own_base)] : 0.f;
                    }
                    if (!(ok = mbar_wait_warp(&bars[C::BAR_V_EMPTY + v.i], v.ph ^ 1))) break;
#pragma unroll
                    for (int i = 0; i < kBN / 32; ++i) s_pos[v.i * kBN + i * 32 + lane] = x[i];
                    __syncwarp();
                    if (lane < 2 && w.used_by(lane, j)) mbar_arrive(&bars[C::BAR_POS + lane * C::NKV + v.i]);
                }
            }
        }
        __syncwarp();
    } else if (warp >= WARP_MMA) {
        reg_dealloc<C::R_MMA>();
        if (warp < WARP_PASS) {
            // ---------------------------------------------------------------- MMA issuer of one lane
            const int ln = warp - WARP_MMA;
            const uint32_t lead = elect_one();
            // Descriptor words are loop-invariant up to a small address offset.  High word: stride-dimension offset
            // 1024 B (8-row groups), descriptor version 1, 128B swizzle; V: leading-dimension offset = one half.
            const uint64_t d_hi = (uint64_t)((1024u >> 4) | (1u << 14) | (2u << 29)) << 32;
            const uint32_t q_lo = ((smem_u32(sQ) & 0x3ffffu) >> 4) | (1u << 16);
            const uint32_t k_lo = ((smem_u32(sK) & 0x3ffffu) >> 4) | (1u << 16);
            const uint32_t v_lo = ((smem_u32(sV) & 0x3ffffu) >> 4) | (((uint32_t)(kBN * 128) >> 4) << 16);
            const uint32_t id_o = idesc_bf16(kBM, D, 0, 1), s_col = tb + ln * kLaneCols, o_col = s_col + kOCol;
            uint64_t *own2 = bars + ln, *own_buf = bars + 2 * ln, *own_kv = bars + ln * C::NKV, *own_q = bars + ln * C::NQ;
            Ring<C::NKV> k;                                 // K and V stages advance together
            Ring<C::NQ> q;
            uint32_t kv_ph = 0, q_ph = 0;                   // parity of the lane's own barriers, a bit per slot (V: 8 bits up)
            uint32_t g_s = 0, g_o = 0, tiles = 0, skip = 0; // S and O += P V issued so far
            // The (at most two) steps whose O += P V is still to be issued, oldest in the low half: 16-key steps, V stage (<< 3),
            // first of its tile (<< 8), parity of its tile number (<< 10), not the lane's first tile (<< 11)
            uint32_t pending = 0;
            Walk w(p);
            LaneTile t = {};
            int j = 0, q_slot = 0;
            bool more = true;
#pragma unroll 1
            while (true) {
#pragma unroll 1
                while (j >= t.steps && more) {              // the lane's next tile
                    more = w.next();
                    if (!more) break;
                    t = LaneTile(w, ln);
                    j = 0;
                    q_slot = q.i + t.b;
                    if (q_slot >= C::NQ) q_slot -= C::NQ;
                    q.skip(w.n_q());
                    k.skip(skip);                           // the item before: key tiles this lane had no use for
                    skip = w.t.steps - t.steps;
                    if (t.steps) ++tiles;
                }
                // What the next S needs is looked at before the wait for P, so that in the steady state (two steps pending) a turn
                // is: wait for P(g), issue O += P V (g), issue S (g+2).
                uint64_t *k_bar = own_kv + C::BAR_K_READY + k.i, *q_bar = own_q + C::BAR_Q_FULL + q_slot;
                auto look = [&]() { return more && __all_sync(0xffffffffu, mbar_test(k_bar, kv_ph >> k.i & 1) && (j > 0 || mbar_test(q_bar, q_ph >> q_slot & 1))); };
                const int n_mma = (min(kBN, t.end - j * kBN) + 15) & ~15;
                const uint64_t qd = d_hi | uniform(q_lo + q_slot * (C::Q_BYTES >> 4)), kd = d_hi | uniform(k_lo + k.i * (C::KV_BYTES >> 4));
                const uint32_t id_s = uniform(idesc_bf16(kBM, 0, 0, 0) | ((uint32_t)(n_mma >> 3) << 17)), d_s = uniform(s_col + (g_s & 1) * kBN);
                bool ready = look();
                if (g_s - g_o == 2 || (g_s != g_o && !ready)) {
                    const uint32_t vs = pending >> 3 & 3, buf = g_o & 1;
                    const uint32_t n = uniform(pending & 7), fresh = uniform(pending & 256u), a = uniform(s_col + buf * kBN);
                    const uint64_t vd = d_hi | uniform(v_lo + vs * (C::KV_BYTES >> 4));
                    if (!(ok = mbar_wait_warp(own_kv + C::BAR_V_READY + vs, kv_ph >> (8 + vs) & 1))) break;
                    kv_ph ^= 256u << vs;
                    // the first O = P V of a tile overwrites O: the lane's previous tile must have been read out
                    if ((pending & (256u | 2048u)) == (256u | 2048u) && !(ok = mbar_wait_warp(own2 + C::BAR_O_FREE, pending >> 10 & 1))) break;
                    if (!(ok = mbar_wait_warp(own_buf + C::BAR_P + buf, g_o >> 1 & 1))) break;
                    tc_fence_after();
#pragma unroll
                    for (int kk = 0; kk < kBN / 16; ++kk)           // contraction over keys
                        if (kk < n) {
                            const uint32_t at = a + (C::SPLIT_P ? (kk >> 1) * 32 + (kk & 1) * 8 : kk * 8);
                            umma_ts(lead, o_col, at, vd + kk * (2048 >> 4), id_o, kk > 0 || !fresh ? 1u : 0u);
                            if (C::SPLIT_P) umma_ts(lead, o_col, at + 16, vd + kk * (2048 >> 4), id_o, 1u);
                        }
                    if (lead) {
                        umma_commit(own_buf + C::BAR_O_DONE + buf);
                        umma_commit(bars + C::BAR_V_EMPTY + vs);
                    }
                    __syncwarp();
                    pending >>= 16;
                    ++g_o;
                    if (!ready) ready = look();
                }
                if (!more) {
                    if (g_s == g_o) break;
                    continue;
                }
                if (!ready) {
                    // With a step pending there is no waiting for K or Q: they may lie behind tiles of the other lane that need
                    // the V stages still held here.
                    if (g_s != g_o) continue;
                    if (!(ok = mbar_wait_warp(k_bar, kv_ph >> k.i & 1))) break;
                    if (j == 0 && !(ok = mbar_wait_warp(q_bar, q_ph >> q_slot & 1))) break;
                }
                tc_fence_after();
#pragma unroll
                for (int kk = 0; kk < D / 16; ++kk)                 // contraction over head_dim
                    umma_ss(lead, d_s, qd + (kk >> 2) * ((kBM * 128) >> 4) + (kk & 3) * 2, kd + (kk >> 2) * ((kBN * 128) >> 4) + (kk & 3) * 2,
                            id_s, kk > 0 ? 1u : 0u);
                const bool last = j == t.steps - 1;
                if (lead) {
                    umma_commit(own_buf + C::BAR_S_FULL + (g_s & 1));
                    umma_commit(bars + C::BAR_K_EMPTY + k.i);
                    if (last) umma_commit(bars + C::BAR_Q_EMPTY + q_slot);
                }
                __syncwarp();
                kv_ph ^= 1u << k.i;
                if (j == 0) q_ph ^= 1u << q_slot;
                const uint32_t info = (uint32_t)(n_mma >> 4) | k.i << 3 | (j == 0 ? 256u : 0u) | (tiles & 1) << 10 | (tiles > 1 ? 2048u : 0u);
                pending |= info << (16 * (g_s - g_o));
                ++j; ++g_s;
                k.next();
                if (ACROSS && j == t.gap_at) { j += t.gap; k.skip(t.gap); }
            }
            if (!ok) {
                // a wait ran out: every MMA of this lane must finish (bounded) before its tensor memory is freed
                if (lead) umma_commit(own2 + C::BAR_DRAIN);
                __syncwarp();
                mbar_wait_warp(own2 + C::BAR_DRAIN, 0);
            }
        } else {
            // ---------------------------------------------------------------- passes tiles on to the lanes, cleans V
            // O += P V contracts over whole 16-key steps.  The V rows of keys that do not exist (behind a preamble whose length
            // is not a multiple of 16, behind the last key) hold whatever follows in the packed tensor, another path's rows;
            // their P is exactly zero, but 0 x Inf or 0 x NaN would still reach O.  They are zeroed before the stage is passed
            // on, so a path's output depends on nothing outside its own keys (Section 3.2: paths do not see each other).
            const bool is_v = warp != WARP_PASS;
            uint64_t *full = &bars[is_v ? C::BAR_V_FULL : C::BAR_K_FULL], *ready = &bars[is_v ? C::BAR_V_READY : C::BAR_K_READY];
            Ring<C::NKV> k;
#pragma unroll 1
            for (Walk w(p); ok && w.next();) {
#pragma unroll 1
                for (int j = 0; j < w.t.steps; ++j, k.next()) {
                    if (!(ok = mbar_wait_warp(full + k.i, k.ph))) break;
                    if (is_v) {
                        const int u0 = j * kBN, e0 = min(kBN, w.end() - u0);
                        const int g0 = min(max(w.t.pre_len - u0, 0), kBN), n_gap = min(max(w.t.p16 - u0, 0), kBN) - g0;
                        const int n = n_gap + (-e0 & 15);
                        if (n > 0) {
                            // lane & 7: 16-byte piece of a row (the swizzle permutes pieces inside a row), then half, then row
                            unsigned char *vs = sV + k.i * C::KV_BYTES + (lane >> 3 & (C::HALVES - 1)) * (kBN * 128) + (lane & 7) * 16;
#pragma unroll 1
                            for (int i = lane / (8 * C::HALVES); i < n; i += 4 / C::HALVES)
                                *reinterpret_cast<uint4 *>(vs + (i < n_gap ? g0 + i : e0 + i - n_gap) * 128) = make_uint4(0u, 0u, 0u, 0u);
                            fence_proxy_async();         // generic-proxy stores -> visible to the MMA's reads
                        }
                        __syncwarp();
                    }
                    if (lane < 2 && w.used_by(lane, j)) mbar_arrive(ready + lane * C::NKV + k.i);
                }
            }
        }
        __syncwarp();
    } else if (warp < WARP_EPI) {
        // -------------------------------------------------------------------- softmax, one thread per query row
        reg_alloc<C::R_SOFT>();
        const int ln = warp >> 2, quad = warp & 3, row = quad * 32 + lane;
        const int rows_per_head = 1 << log_rows, hr = row & (rows_per_head - 1);            // row of the tile, for head row >> log_rows
        const int hr0 = quad * 32 & (rows_per_head - 1), hr1 = hr0 + min(32, rows_per_head);  // ... of the warp
        const uint32_t s_base = tb + ln * kLaneCols + ((uint32_t)(quad * 32) << 16);
        const float sc = p.scale_log2e;
        uint64_t *own2 = bars + ln, *own_buf = bars + 2 * ln;
        uint32_t g = 0, tiles = 0, pos_ph = 0;
        Ring<C::NKV> v;
#pragma unroll 1
        for (Walk w(p); ok && w.next();) {
            const LaneTile t(w, ln);
            const bool live_w = hr0 < t.rows;            // rows past the tile's last one take part in barriers only
            const int head = (w.h << (7 - log_rows)) + (row >> log_rows);
            float m_ref = -INFINITY, l = 0.f;            // reference maximum (log2 units) and row sum
            float pq = 0.f, neg_slope = 0.f;
            if (ALIBI && t.steps) {
                pq = hr < t.rows ? p.pos[w.t.own_base + t.q_u + hr] : 0.f;
                neg_slope = -p.slopes[head] * (kLog2eT / sc);     // in units of the unscaled score: one scaling serves both
            }
            // counted from the key tile's first key: the first one this row may not see, the padding behind the preamble
            int lim = min(t.q_u + hr + 1, t.end), g0 = w.t.pre_len, g1 = w.t.p16;
            int see = live_w ? min(t.q_u + hr1, t.end) : 0;      // keys some row of the warp may see
            // ACROSS: path starts from tile A's on, a lane each; looked at where the first own keys come (g0 < kBN), by when they are here
            const int row_w = w.t.own_base + t.q_u + hr0, start_a = w.t.own_base + w.t.p16;
            int see_from = 0, start = INT_MAX;
            if (ACROSS && t.steps && w.first_path >= 0 && w.first_path + lane < p.n_paths) start = p.path_start[w.first_path + lane];
            bool look = ACROSS && w.first_path >= 0;
#pragma unroll 1
            for (int j = 0; j < t.steps; ++j, ++g, lim -= kBN, g0 -= kBN, g1 -= kBN, see -= kBN) {
                if (ACROSS && look && g0 < kBN) {
                    // the path of the warp's first row, and a bit for each of its rows that is the first of another one
                    look = false;
                    int before = start_a;
                    uint32_t firsts = 0;
                    for (int base = w.first_path + lane;; ) {
                        // a row of another prompt's path is none of the item's: those lie in front of its first row or behind its last
                        const uint32_t at = (uint32_t)(start - row_w);
                        before = max(before, start <= row_w ? start : INT_MIN);
                        if (at - 1u < 31u) firsts |= 1u << at;
                        if (!__shfl_sync(0xffffffffu, start >= start_a && start < row_w + 32, 31)) break;
                        base += 32;
                        start = base < p.n_paths ? p.path_start[base] : INT_MAX;
                    }
                    before = __reduce_max_sync(0xffffffffu, before);
                    firsts = __reduce_or_sync(0xffffffffu, firsts) & low_bits(lane + 1);
                    const int passed = j * kBN + w.t.own_base;
                    g1 = (firsts ? row_w + 31 - __clz(firsts) : before) - passed;
                    see_from = before - w.t.own_base;
                }
                const uint32_t buf = g & 1, s_addr = s_base + buf * kBN;
                if (!(ok = mbar_wait_warp(own_buf + C::BAR_S_FULL + buf, g >> 1 & 1))) break;
                if (ALIBI && !(ok = mbar_wait_warp(&bars[C::BAR_POS + ln * C::NKV + v.i], pos_ph >> v.i & 1))) break;
                tc_fence_after();
                if (see > 0 && !(ACROSS && g0 <= 0 && see_from - j * kBN >= kBN)) {
                    uint32_t r[2][32];
                    tmem_ld32(s_addr, r[0]);
                    tmem_ld32(s_addr + 32, r[1]);
                    tmem_ld_wait();
                    float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        if (c == 1 && see <= 32) break;
                        // keys this row may not see (causal diagonal, ragged end) or that do not exist -> -inf
                        const uint32_t vis = low_bits(lim - c * 32) & (low_bits(g0 - c * 32) | ~low_bits(g1 - c * 32));
                        if (ALIBI) {              // score - slope * |distance|; key positions are broadcast reads
                            const uint64_t pq2 = pack_f32x2(-pq, -pq), ns2 = pack_f32x2(neg_slope, neg_slope);
#pragma unroll
                            for (int i = 0; i < 32; i += 4) {
                                const ulonglong2 kp = *reinterpret_cast<const ulonglong2 *>(s_pos + v.i * kBN + c * 32 + i);
#pragma unroll
                                for (int e = 0; e < 4; e += 2) {
                                    const uint64_t d = add_f32x2(e ? kp.y : kp.x, pq2) & 0x7fffffff7fffffffull;
                                    float x0, x1;
                                    unpack_f32x2(fma_f32x2(d, ns2, pack_f32x2(__uint_as_float(r[c][i + e]), __uint_as_float(r[c][i + e + 1]))), x0, x1);
                                    r[c][i + e] = __float_as_uint(x0); r[c][i + e + 1] = __float_as_uint(x1);
                                }
                            }
                        }
                        if (__any_sync(0xffffffffu, vis != 0xffffffffu)) {
#pragma unroll
                            for (int i = 0; i < 32; ++i) r[c][i] = vis & (1u << i) ? r[c][i] : 0xff800000u;
                        }
#pragma unroll
                        for (int i = 0; i < 32; i += 2) mx[(i >> 1) & 3] = fmax3(mx[(i >> 1) & 3], __uint_as_float(r[c][i]), __uint_as_float(r[c][i + 1]));
                    }
                    const float m_tile = fmaxf(fmax3(mx[0], mx[1], mx[2]), mx[3]) * sc;
                    const bool grow = j > 0 && m_tile > m_ref + kRescaleThreshold;
                    if (__any_sync(0xffffffffu, grow)) {      // rare: bring O and l to the new reference
                        // needs the lane's previous O += P V complete
                        if (!(ok = mbar_wait_warp(own_buf + C::BAR_O_DONE + (buf ^ 1), (g - 1) >> 1 & 1))) break;
                        tc_fence_after();
                        const float alpha = grow ? ex2(m_ref - m_tile) : 1.f;
                        l *= alpha;
#pragma unroll 1
                        for (int cc = 0; cc < D / 16; ++cc) {
                            uint32_t o[16];
                            tmem_ld16(s_base + kOCol + cc * 16, o);
                            tmem_ld_wait();
#pragma unroll
                            for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
                            tmem_st16(s_base + kOCol + cc * 16, o);
                        }
                    }
                    if (j == 0 || grow) m_ref = m_tile;
                    // P = exp2(score - reference) as bf16
                    const uint64_t sc2 = pack_f32x2(sc, sc), nm2 = pack_f32x2(-m_ref, -m_ref);
                    uint64_t sum[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        uint32_t hi[16], lo[C::SPLIT_P ? 16 : 1];
                        if (c == 0 || see > 32) {
#pragma unroll
                            for (int i = 0; i < 32; i += 2) {        // hidden scores are -inf: exp2 gives exactly 0 for them
                                float x0, x1;
                                unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(r[c][i]), __uint_as_float(r[c][i + 1])), sc2, nm2), x0, x1);
                                const float p0 = ex2(x0), p1 = ex2(x1);
                                sum[(i >> 1) & 3] = add_f32x2(sum[(i >> 1) & 3], pack_f32x2(p0, p1));
                                if (C::SPLIT_P) split_bf16(p0, p1, hi[i >> 1], lo[C::SPLIT_P ? i >> 1 : 0]);
                                else hi[i >> 1] = pack_bf16x2(p0, p1);
                            }
                        } else {                                     // no row of this warp sees these keys
#pragma unroll
                            for (int i = 0; i < 16; ++i) { hi[i] = 0u; if (C::SPLIT_P) lo[C::SPLIT_P ? i : 0] = 0u; }
                        }
                        tmem_st16(s_addr + c * (C::SPLIT_P ? 32 : 16), hi);
                        if constexpr (C::SPLIT_P) tmem_st16(s_addr + c * 32 + 16, lo);
                    }
                    float a0, a1;
                    unpack_f32x2(add_f32x2(add_f32x2(sum[0], sum[1]), add_f32x2(sum[2], sum[3])), a0, a1);
                    l += a0 + a1;
                } else if (live_w) {
                    const uint32_t z[32] = {0u};
                    tmem_st32(s_addr, z);
                    if (C::SPLIT_P) tmem_st32(s_addr + 32, z);
                }
                tmem_st_wait();                           // P is in tensor memory: release it to the issuer
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(own_buf + C::BAR_P + buf);
                if (ALIBI) { pos_ph ^= 1u << v.i; v.next(); }
                if (ACROSS && j + 1 == t.gap_at) {
                    j += t.gap; lim -= t.gap * kBN; g0 -= t.gap * kBN; g1 -= t.gap * kBN; see -= t.gap * kBN;
                    if (ALIBI) v.skip(t.gap);
                }
            }
            if (!ok) break;
            if (ALIBI) v.skip(w.t.steps - t.steps);
            if (!t.steps) continue;
            // hand the tile's row sums to the epilogue warps, which must have read the previous ones
            if (tiles > 0 && !(ok = mbar_wait_warp(own2 + C::BAR_X_FREE, (tiles - 1) & 1))) break;
            x_l[ln * kBM + row] = l;
            __syncwarp();
            if (lane == 0) mbar_arrive(own2 + C::BAR_L_READY);
            ++tiles;
            if (p.lse && hr < t.rows) p.lse[(int64_t)head * p.total_tokens + w.t.own_base + t.q_u + hr] = (m_ref + log2f(l)) * kLn2T;
        }
    } else {
        // -------------------------------------------------------------------- epilogue
        // O / l -> bf16 -> global, off the softmax warps' path.  A thread owns a row and writes it in full 32-byte sectors;
        // the accumulator is handed back before the last 64 columns are stored.
        reg_dealloc<C::R_EPI>();
        const int quad = warp - WARP_EPI, row = quad * 32 + lane;
        const int hr = row & ((1 << log_rows) - 1), hr0 = quad * 32 & ((1 << log_rows) - 1);
        uint32_t ph = 0, g[2] = {0, 0};                  // tiles so far, mod 2, a bit per lane; key tiles so far
        bool not_all_finite = false;                     // ACROSS: some value that this thread has stored is not finite
#pragma unroll 1
        for (Walk w(p); ok && w.next();) {
#pragma unroll 1
            for (int b = 0; b < w.n_q(); ++b) {
                const int ln = w.lane_a() ^ b;
                const LaneTile t(w, ln);
                if (!(ok = mbar_wait_warp(&bars[C::BAR_L_READY + ln], ph >> ln & 1))) break;
                const float inv = __fdividef(1.f, x_l[ln * kBM + row]);
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars[C::BAR_X_FREE + ln]);
                const uint32_t g_last = (ln ? g[1] : g[0]) + t.steps - t.gap - 1;
                if (ln) g[1] = g_last + 1; else g[0] = g_last + 1;
                if (!(ok = mbar_wait_warp(&bars[C::BAR_O_DONE + 2 * ln + (g_last & 1)], g_last >> 1 & 1))) break;      // last O += P V
                ph ^= 1u << ln;
                tc_fence_after();
                const uint32_t o_addr = tb + ln * kLaneCols + kOCol + ((uint32_t)(quad * 32) << 16);
                const uint64_t inv2 = pack_f32x2(inv, inv);
                unsigned char *dst = reinterpret_cast<unsigned char *>(p.out) +
                                     ((int64_t)(w.t.own_base + t.q_u + hr) * p.n_heads + (w.h << (7 - log_rows)) + (row >> log_rows)) * (D * 2);
                uint32_t nan = 0u;
#pragma unroll 1
                for (int cc = 0; cc < C::HALVES; ++cc) {       // 64 columns
                    uint32_t o[32];
                    if (hr0 < t.rows) {
                        uint32_t r0[32], r1[32];
                        tmem_ld32(o_addr + cc * 64, r0);
                        tmem_ld32(o_addr + cc * 64 + 32, r1);
                        tmem_ld_wait();
#pragma unroll
                        for (int i = 0; i < 32; ++i) {
                            const uint32_t *r = i < 16 ? r0 : r1;
                            float x0, x1;
                            unpack_f32x2(mul_f32x2(pack_f32x2(__uint_as_float(r[2 * (i & 15)]), __uint_as_float(r[2 * (i & 15) + 1])), inv2), x0, x1);
                            o[i] = pack_bf16x2(x0, x1);
                        }
                    }
                    if (cc == C::HALVES - 1) {                 // O is in registers: the accumulator may be overwritten
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&bars[C::BAR_O_FREE + ln]);
                    }
                    if (ACROSS) {
#pragma unroll
                        for (int i = 0; i < 32; ++i) asm("fma.rn.bf16x2 %0, %1, %2, %0;" : "+r"(nan) : "r"(o[i]), "r"(0u));
                    }
                    if constexpr (C::EXACT && !ACROSS) {
                        uint32_t nan = 0u;
#pragma unroll
                        for (int i = 0; i < 32; ++i) asm("fma.rn.bf16x2 %0, %1, %2, %0;" : "+r"(nan) : "r"(o[i]), "r"(0u));
                        if (__any_sync(0xffffffffu, hr < t.rows && (nan & 0x7fff7fffu))) {
                            uint32_t copy[32];
#pragma unroll
                            for (int i = 0; i < 32; ++i) copy[i] = o[i];
                            exact_rows64<ALIBI, ROWS>(p, w.pair, w.h, b, quad, copy);
#pragma unroll
                            for (int i = 0; i < 32; ++i) o[i] = copy[i];
                        }
                    }
                    if (hr < t.rows) {
                        if (p.wide_stores) {
#pragma unroll
                            for (int i = 0; i < 4; ++i) st_global_32b(dst + cc * 128 + i * 32, *reinterpret_cast<const uint32_t (*)[8]>(&o[i * 8]));
                        } else {
#pragma unroll
                            for (int i = 0; i < 8; ++i)
                                __stcs(reinterpret_cast<uint4 *>(dst + cc * 128) + i, make_uint4(o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]));
                        }
                    }
                }
                not_all_finite |= hr < t.rows && (nan & 0x7fff7fffu);
            }
        }
        if (ACROSS && ok && __any_sync(0xffffffffu, not_all_finite)) {
            if constexpr (D == 128) exact_rows_across<D, ALIBI>(p, quad);
            else exact_rows_across64<ALIBI>(p, quad);
        }
    }

    if (!ok && lane == 0) atomicExch(p.status, (uint32_t)STATUS_TIMEOUT);
    tc_fence_before();
    __syncthreads();
    if (warp == WARP_MMA) tmem_dealloc(tb, kTmemCols);
}

// ---- rotation of Q for sp_superpose_prefill_rope -----------------------------------------
// Rotates the rows of every item from q into out, where the attention kernel then reads its query tiles: an item's tile
// is in shared memory long before its epilogue overwrites those rows (one head's columns of one tile's rows belong to one
// item), so no other buffer is needed and q stays as it is.  One read and one write of Q at HBM speed.  The rotation inside
// the attention kernel that this replaced (on the softmax warps, from a per-token table) cost 1.2 ms of a 2.9 ms launch at
// 236 000 tokens x 32 heads; this pass costs 0.6.  Rows that belong to no segment are left alone.
constexpr int kRopeRows = 4;          // rows per block iteration: 256 angles, one per thread
struct RopeRows {
    const __nv_bfloat16 *q;
    __nv_bfloat16 *out;
    const float *pos;
    const TcHeader *hdr;
    const TcPair *pairs;
    int n_heads, half_split;
    uint32_t item_groups;             // of kRopeRows rows, in an item at most
    double inv_freq[64];
};
__global__ void __launch_bounds__(256, 8) rope_rows_kernel(const __grid_constant__ RopeRows a)
{
    __shared__ float2 cs[kRopeRows][64];
    pdl_wait();
    pdl_trigger();
    const uint32_t n_groups = a.hdr->n_tiles * a.item_groups;
    for (uint32_t g = blockIdx.x; g < n_groups; g += gridDim.x) {
        const TcPair t = a.pairs[g / a.item_groups];
        const int r0 = (int)(g % a.item_groups) * kRopeRows, n = min(kRopeRows, (t.rows_ab & 0xffff) + (t.rows_ab >> 16) - r0);
        if (n <= 0) continue;
        const int64_t row = t.own_base + t.q_u + r0;
        __syncthreads();
        const int r = threadIdx.x >> 6, m = threadIdx.x & 63;
        if (r < n) {
            double sn, cn;
            sincos((double)a.pos[row + r] * a.inv_freq[m], &sn, &cn);
            cs[r][m] = make_float2((float)cn, (float)sn);
        }
        __syncthreads();
        // 16 elements of a head per thread: a piece of each half (half-split) or two neighbouring pieces
        for (int i = threadIdx.x; i < n * a.n_heads * 8; i += 256) {
            const int rr = i / (a.n_heads * 8), j = i & 7;
            const int64_t at = (row + rr) * a.n_heads * 128 + (int64_t)(i - rr * a.n_heads * 8 >> 3) * 128 + (a.half_split ? j * 8 : j * 16);
            float x[8], y[8];
            Vec<__nv_bfloat16>::load(a.q + at, x);
            Vec<__nv_bfloat16>::load(a.q + at + (a.half_split ? 64 : 8), y);
            if (a.half_split) {
#pragma unroll
                for (int e = 0; e < 8; ++e) rope_rotate(x[e], y[e], cs[rr][j * 8 + e].x, cs[rr][j * 8 + e].y, x[e], y[e]);
            } else {
#pragma unroll
                for (int e = 0; e < 8; e += 2) {
                    const float2 wx = cs[rr][j * 8 + e / 2], wy = cs[rr][j * 8 + 4 + e / 2];
                    rope_rotate(x[e], x[e + 1], wx.x, wx.y, x[e], x[e + 1]);
                    rope_rotate(y[e], y[e + 1], wy.x, wy.y, y[e], y[e + 1]);
                }
            }
            uint4 *dst = reinterpret_cast<uint4 *>(a.out + at);
            dst[0] = make_uint4(pack_bf16x2(x[0], x[1]), pack_bf16x2(x[2], x[3]), pack_bf16x2(x[4], x[5]), pack_bf16x2(x[6], x[7]));
            dst[a.half_split ? 8 : 1] = make_uint4(pack_bf16x2(y[0], y[1]), pack_bf16x2(y[2], y[3]), pack_bf16x2(y[4], y[5]), pack_bf16x2(y[6], y[7]));
        }
    }
}

// ---- host side ---------------------------------------------------------------------------
// Failure-detection test hook (host-injected, no GPU fault): while set, the producers load no
// tile, every bounded wait expires, the blocks unwind and the call reports SP_ERR_TIMEOUT
// through the workspace status word.  Set only through sp_test_stall_producer(), a symbol for
// the test suite that the public header does not declare.
bool g_stall_producer = false;

size_t prefill_tc_workspace_bytes(int n_prompts, int n_paths, int max_pre_len, int max_path_len, int)
{
    if (n_prompts < 0 || n_paths < 0 || max_pre_len < 0 || max_path_len < 0) return 256;
    // the head counts are not known yet: items of 2 x 16 rows, those of eight heads in a tile
    return 256 + round_up((size_t)plan_max_tiles(n_prompts, n_paths, max_pre_len, max_path_len, 32) * sizeof(TcPair), 256);
}

template <int D, bool ALIBI, TileRows ROWS, bool SPLIT> static int launch_kernel(const TcParams &p, int grid, cudaStream_t st)
{
    using C = TcConfig<D, ALIBI, SPLIT>;
    SP_CUDA(cudaFuncSetAttribute(prefill_tc_kernel<D, ALIBI, ROWS, SPLIT>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM));
    return launch(prefill_tc_kernel<D, ALIBI, ROWS, SPLIT>, grid, kTcThreads, C::SMEM, st, 1, p);
}

// Tiles over the rows of consecutive paths (one head to a tile): full ones, and the preamble's keys loaded and multiplied once per pair of
// tiles instead of once per path, but every tile also meets the keys of all of its paths.  Both ways are counted from the host
// mirror: key tiles of all query tiles, in the share that the busiest block gets.  A key tile takes up to a tenth longer across (two
// lanes that agree less about which keys they need), and with less than three items to a block one block's items are a chain too
// long.  us segment by segment / across, 32 heads of 128, 20 documents to a prompt, about 120 000 rows (key tiles across in
// proportion): documents of 8-24 rows behind 64 1495 / 716 (0.37), behind 400 3359 / 1191 (0.28); 32-64 behind 64 758 / 691 (0.85),
// behind 16 645 / 652 (0.99); 60-180 behind 400 1625 / 1375 (0.84), behind 64 715 / 749 (0.97); 64-256 behind 400 1497 / 1436
// (0.89); 128-512 behind 64 901 / 970 (1.05); ALiBi 60-180 behind 400 2118 / 1855; head_dim 64 1439 / 1231.  One prompt of 20
// documents of 32-64 rows behind 128 (0.74, one item to a block): 19.6 / 22.8.
static bool across_pays(const sp_layout *lay, int n_units)
{
    const sp_layout_host *m = lay->host_mirror;
    if (!m) return false;
    int64_t alone = 0, across = 0, items_alone = 0, items_across = 0;      // key tiles of all query tiles; pairs of them
    for (int b = 0; b < lay->n_prompts; ++b) {
        const int i0 = m->prompt_path_off[b], i1 = m->prompt_path_off[b + 1], p16 = (m->pre_len[b] + 15) & ~15;
        if (i0 == i1) continue;
        if (m->pre_len[b] == 0) return false;            // every row has to see the first key tile
        int run = 0;
        for (int i = i0; i < i1; ++i) {
            const int n = m->doc_len[i] + m->qry_len[i], h = even_height(n, kBM);
            if (n == 0 || m->path_start[i] != m->path_start[i0] + run) return false;
            run += n;
            for (int r = h; r < n + h; r += h) alone += (p16 + std::min(r, n) + kBN - 1) / kBN;
            items_alone += (n + 2 * h - 1) / (2 * h);
        }
        const int h = even_height(run, kBM), gap_at = (m->pre_len[b] + kBN - 1) / kBN;
        for (int r = 0, i = i0, start = 0, start_a = 0; r < run; r += h) {
            for (int n; start + (n = m->doc_len[i] + m->qry_len[i]) <= r; ++i) start += n;
            const bool is_b = r / h & 1;
            if (!is_b) { start_a = start; ++items_across; }
            const int end = p16 + std::min(r + h, run) - start_a;
            across += (end + kBN - 1) / kBN - (is_b ? std::max((p16 + start - start_a) / kBN - gap_at, 0) : 0);
        }
    }
    if (items_across * n_units < 3 * (int64_t)num_sms()) return false;
    // what the busiest block gets, at the mean number of key tiles
    const auto busiest = [&](int64_t steps, int64_t items) { return (double)((items * n_units + num_sms() - 1) / num_sms()) * steps / items; };
    return busiest(across, items_across) < 0.9 * busiest(alone, items_alone);
}

static int launch_tc(const void *q, const void *k, const void *v, const sp_layout *lay, const float *pos,
                     const float *slopes, const RopeRows *rope, int n_heads, int n_kv_heads, int head_dim,
                     float scale, int rows, void *out, float *lse, void *ws, cudaStream_t st)
{
    TcParams p;
    const int halves = head_dim / 64;
    const int64_t q_cols = (int64_t)n_heads * head_dim, kv_cols = (int64_t)n_kv_heads * head_dim;
    const struct { const void *base; int64_t cols; } src[3] = {{k, kv_cols}, {v, kv_cols}, {q, q_cols}};
    for (int i = 0; i < 3; ++i)
        for (int b = 0; b < 3; ++b)
            if (int rc = encode_rows_map(&p.maps[i][b], src[i].base, lay->total_tokens, src[i].cols,
                                         b == 0 ? (i == 2 ? kBM : kBN) : (b == 1 ? 32 : 16), b == 0 ? halves : 1)) return rc;

    TcHeader *hdr = static_cast<TcHeader *>(ws);
    TcPair *pairs = reinterpret_cast<TcPair *>(static_cast<char *>(ws) + 256);
    PlanArgs pa;
    pa.ppo = lay->prompt_path_off; pa.pre_start = lay->pre_start; pa.pre_len = lay->pre_len;
    pa.path_start = lay->path_start; pa.doc_len = lay->doc_len; pa.qry_len = lay->qry_len;
    // Heads that share a tile: the largest of 8, 4, 2, 1 that divides the group; 16-row boxes rule out more.  Less of a tile is
    // empty (segments of a few hundred rows, queries of 8 to 48) and its rows lie closer to the diagonal.  us with one head a
    // tile / this, 32 heads over 8: 2 prompts x 400 documents of 128-512 rows 2376 / 1972, 64 x 20 of 100-200 rows 1399 / 1054, 32
    // query rows only of 8 x 100 552 / 190, head_dim 64 163 / 127.
    const int group = n_heads / n_kv_heads, log_g = group % 8 == 0 ? 3 : (group % 4 == 0 ? 2 : (group % 2 == 0 ? 1 : 0));
    pa.n_prompts = lay->n_prompts; pa.n_paths = lay->n_paths; pa.rows_mode = rows; pa.tile_rows = kBM >> log_g;
    pa.max_pre_len = lay->max_pre_len; pa.max_path_len = lay->max_path_len; pa.total_tokens = lay->total_tokens;
    pa.max_tiles = plan_max_tiles(lay->n_prompts, lay->n_paths, lay->max_pre_len, lay->max_path_len, 2 * pa.tile_rows);
    // the sort takes a microsecond: worth it from a dozen items per block
    pa.sort_from = 12 * num_sms() / (n_heads >> log_g);
    // (not where the output takes Q's place, as it does with the rotation folded in: a row that has to be computed again would not find it)
    const uintptr_t q_at = reinterpret_cast<uintptr_t>(q), out_at = reinterpret_cast<uintptr_t>(out), q_bytes = (uintptr_t)lay->total_tokens * q_cols * 2;
    const bool over_q = rope || (out_at < q_at + q_bytes && q_at < out_at + q_bytes);
    const bool across = log_g == 0 && rows == SP_ROWS_ALL && !over_q && across_pays(lay, n_heads);
    pa.hdr = hdr; pa.list = pairs;
    if (int rc = launch(across ? prefill_plan_kernel<true, true> : prefill_plan_kernel<true>, 1, 1024, 0, st, 1, pa)) return rc;
    if (pa.max_tiles == 0) return SP_OK;              // no segment can have a row
    if (rope) {
        RopeRows r = *rope;
        r.hdr = hdr; r.pairs = pairs; r.item_groups = 2 * pa.tile_rows / kRopeRows;
        const int64_t groups = pa.max_tiles * r.item_groups;
        if (int rc = launch(rope_rows_kernel, (unsigned)std::min<int64_t>(groups, (int64_t)num_sms() * 16), 256, 0, st, 1, r)) return rc;
    }

    p.hdr = hdr; p.pairs = pairs; p.status = &hdr->status;
    p.out = static_cast<__nv_bfloat16 *>(out); p.lse = lse;
    p.q = static_cast<const __nv_bfloat16 *>(q); p.k = static_cast<const __nv_bfloat16 *>(k); p.v = static_cast<const __nv_bfloat16 *>(v);
    p.n_kv_heads = n_kv_heads;
    p.n_heads = n_heads; p.log_rows = 7 - log_g; p.n_units = n_heads >> log_g; p.units_per_kv = group >> log_g;
    p.total_tokens = lay->total_tokens; p.scale_log2e = scale * kLog2eT;
    p.wide_stores = (reinterpret_cast<uintptr_t>(out) & 31u) == 0;
    p.pos = pos; p.slopes = slopes;
    p.path_start = lay->path_start; p.n_paths = lay->n_paths;
    p.stall_producer = g_stall_producer ? 1 : 0;      // test hook, see sp_test_stall_producer below

    const int64_t items = pa.max_tiles * p.n_units;
    const int grid = (int)std::min<int64_t>(items, num_sms());
    using Launch = int (*)(const TcParams &, int, cudaStream_t);
    const auto run = [&](Launch segment, Launch heads, Launch paths) { return (across ? paths : (log_g ? heads : segment))(p, grid, st); };
    if (head_dim == 64)
        return pos ? run(launch_kernel<64, true, SEGMENT_ROWS, true>, launch_kernel<64, true, HEAD_ROWS, true>, launch_kernel<64, true, ACROSS_ROWS, true>)
                   : run(launch_kernel<64, false, SEGMENT_ROWS, true>, launch_kernel<64, false, HEAD_ROWS, true>, launch_kernel<64, false, ACROSS_ROWS, true>);
    if (rows == SP_ROWS_QUERY_ONLY)               // P as two bf16 numbers, see TcConfig
        return pos ? run(launch_kernel<128, true, SEGMENT_ROWS, true>, launch_kernel<128, true, HEAD_ROWS, true>, nullptr)
                   : run(launch_kernel<128, false, SEGMENT_ROWS, true>, launch_kernel<128, false, HEAD_ROWS, true>, nullptr);
    return pos ? run(launch_kernel<128, true, SEGMENT_ROWS, false>, launch_kernel<128, true, HEAD_ROWS, false>, launch_kernel<128, true, ACROSS_ROWS, false>)
               : run(launch_kernel<128, false, SEGMENT_ROWS, false>, launch_kernel<128, false, HEAD_ROWS, false>, launch_kernel<128, false, ACROSS_ROWS, false>);
}

int launch_prefill_tc(const void *q, const void *k, const void *v, const sp_layout *lay, const float *pos,
                      const float *slopes, int n_heads, int n_kv_heads, int head_dim, float scale, int rows, void *out,
                      float *lse, void *ws, cudaStream_t st)
{
    return launch_tc(q, k, v, lay, pos, slopes, nullptr, n_heads, n_kv_heads, head_dim, scale, rows, out, lse, ws, st);
}

// sp_superpose_prefill_rope.  The size has 512 bytes per token behind the tile list that nothing uses any more (a table of angles
// was there): the entry point has refused less since its first version, and what it refuses is part of the interface.
size_t prefill_tc_rope_workspace_bytes(int n_prompts, int n_paths, int max_pre_len, int max_path_len, int64_t total_tokens)
{
    return prefill_tc_workspace_bytes(n_prompts, n_paths, max_pre_len, max_path_len, 0) +
           round_up((size_t)std::max<int64_t>(total_tokens, 0) * 64 * sizeof(float2), 256);
}

int launch_prefill_tc_rope(const void *q, const void *k, const void *v, const sp_layout *lay, const float *pos, double base,
                           int pairing, int n_heads, int n_kv_heads, float scale, void *out, float *lse, void *ws,
                           cudaStream_t st)
{
    RopeRows r;
    r.q = static_cast<const __nv_bfloat16 *>(q); r.out = static_cast<__nv_bfloat16 *>(out); r.pos = pos;
    r.n_heads = n_heads; r.half_split = pairing == SP_ROPE_HALF_SPLIT;
    rope_inv_freq(base, 128, r.inv_freq);
    return launch_tc(out, k, v, lay, nullptr, nullptr, &r, n_heads, n_kv_heads, 128, scale, SP_ROWS_ALL, out, lse, ws, st);
}

}  // namespace sp

extern "C" void sp_test_stall_producer(int on) { sp::g_stall_producer = on != 0; }
