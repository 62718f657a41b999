// Query rows only: the N query copies of a prompt attend to cached preamble and document
// keys and, causally, to their own rows (Section 3.3, path caching: at serving time only the
// query segments are new).  bf16, head_dim 128.
//
// With 8 to 48 query rows per path the work is a stream over the cached K / V with ~25 flop per byte.  A tensor-core tile has 128
// rows, so here the keys take that side and the queries the other, which may be as narrow as they are:
//   S^T [128 keys x queries] = K Q^T       tcgen05.mma, K and Q from TMA-staged shared memory
//   P^T                                    a thread per key: maximum over the keys of every query, exponentials, to shared memory
//   O^T [128 columns x queries] += V^T P^T tcgen05.mma, V as it lies (MN-major), P^T from shared memory
// Per 128 keys and 32 queries that takes 320 + 320 to 400 clk of the tensor core's shared-memory port, where their 64 KB take some 2 700
// clk of an SM's share of HBM: K and V stages are all that has to be kept in flight.
// Work item: the query rows of one path (at most NQ) and a head, heads fastest, one persistent block per SM.  Items alternate
// between two softmax warpgroups ("lanes") with S^T, P^T and O^T of their own; loads and products run in item order.
// P is (SPLIT) the sum of two bf16 numbers, side by side as columns of one product, or, without a bias, one number relative to the running
// maximum and two for an item's first 32 keys (the rule, and what both cost: prefill.cu).
// Measured (32 heads, 8 x 100 documents of 64-256 rows behind 48): 470 us = 0.95 of the copy bandwidth, 610 with warp-level products
// (mma.sync, two warps to a scheduler, the chain product - softmax - product exposed); 48 rows 553 us = 0.93.
// Behind long preambles (384 rows: 724 us, 456 at the copy bandwidth) it is bound by what L2 gives the SMs, 10 TB/s: every
// path fetches the preamble anew.  Three query slots at least: with two, the loads of K wait behind Q (documents of 32-64 rows 112 -> 128 us).
// Two numbers in a register pair (f32x2) made 48 rows 677 -> 547 us; a look at the scores instead of the maximum where the reference may
// stay (SPLIT) gained 1 % behind 1 200 rows and lost 2 % behind 48: not kept.
// Roles: warps 0-7 softmax and output, 8 S^T, 9 O^T, 10 loads of K and Q, 11 of V.
// Every mbarrier wait is bounded: on expiry the block records a timeout in the workspace status word, unwinds and exits.
#include "common.cuh"
#include "prefill_plan.cuh"
#include "tc_ptx.cuh"
#include "tensor_map.cuh"

namespace sp {

using namespace ptx;

extern bool g_stall_producer;                 // test hook, see prefill_tc.cu

constexpr int kQKeys = 128;                   // keys per tile
constexpr int kQThreads = 384;                // 12 warps, three to a partition: 168 registers a thread
constexpr int kQKvBytes = kQKeys * 256;
constexpr float kLog2eQ = 1.4426950408889634f;
constexpr float kLn2Q = 0.6931471805599453f;

template <int NQ, bool SPLIT> struct QoConfig {
    static constexpr int PC = SPLIT ? 2 * NQ : NQ;             // columns of P^T and O^T
    static constexpr int NK = 2, NV = NQ == 32 ? 3 : 2, NS = NQ == 32 && !SPLIT ? 5 : 3;      // stages of K, V and Q
    static constexpr int Q_BYTES = NQ * 256, P_BYTES = kQKeys * PC * 2;
    static constexpr int V_OFF = NK * kQKvBytes, Q_OFF = V_OFF + NV * kQKvBytes, P_OFF = Q_OFF + NS * Q_BYTES;
    static constexpr int L_OFF = P_OFF + 2 * P_BYTES, L_BYTES = SPLIT ? 0 : 32 * 64;      // not SPLIT: [lane], low parts of 32 keys
    static constexpr int X_OFF = L_OFF + 2 * L_BYTES;          // [lane][2][warp][NQ] floats: what the warps of a lane exchange
    static constexpr int R_OFF = X_OFF + 2 * 2 * 4 * NQ * 4;   // [softmax warp][NQ]: one number per query, for all threads of the warp
    static constexpr int A_OFF = R_OFF + 8 * NQ * 4;           // [lane][NQ]: positions of the queries (ALiBi)
    static constexpr int BAR_OFF = A_OFF + 2 * NQ * 4;
    static constexpr int BAR_K_FULL = 0, BAR_K_EMPTY = BAR_K_FULL + NK, BAR_V_FULL = BAR_K_EMPTY + NK, BAR_V_EMPTY = BAR_V_FULL + NV,
                         BAR_Q_FULL = BAR_V_EMPTY + NV, BAR_Q_EMPTY = BAR_Q_FULL + NS,
                         BAR_S_FULL = BAR_Q_EMPTY + NS, BAR_O_DONE = BAR_S_FULL + 4, BAR_DRAIN = BAR_O_DONE + 2,
                         BAR_S_FREE = BAR_DRAIN + 2, BAR_P = BAR_S_FREE + 4, BAR_COUNT = BAR_P + 2;
    static constexpr int SMEM = BAR_OFF + BAR_COUNT * 8 + 16;
    // tensor memory of a lane: two S^T of NQ columns, O^T
    static constexpr int S_COLS = NQ == 32 ? 32 : 64, O_COL = 2 * S_COLS, LANE_COLS = O_COL + PC, TMEM = 2 * LANE_COLS <= 256 ? 256 : 512;
    static_assert(SMEM <= 232448, "one block's shared memory");
    static_assert(P_OFF % 1024 == 0 && Q_BYTES % 1024 == 0, "swizzle atoms");
};

__device__ __forceinline__ float ex2q(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// 6 clk a maximum over the warp; the exchange of halves by shuffles takes twice that (246 against 513 clk for 32 columns).
__device__ __forceinline__ float warp_max_redux(float x)
{
    float y;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(y) : "f"(x));
    return y;
}
// Barrier of the 128 threads of a lane; true when x holds in all of them.
__device__ __forceinline__ bool lane_barrier_and(int id, bool x)
{
    uint32_t y;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\tbarrier.cta.red.and.aligned.pred q, %2, 128, p;\n\tselp.b32 %0, 1, 0, q;\n\t}"
                 : "=r"(y) : "r"((uint32_t)x), "r"(id) : "memory");
    return y != 0;
}
// n ones from bit 0 up, for any n
__device__ __forceinline__ uint32_t ones(int n) { return n >= 32 ? 0xffffffffu : (1u << max(n, 0)) - 1u; }

// Sums N columns over the warp: lane i gets column i mod N.
template <int N> __device__ __forceinline__ float column_sums(float (&v)[N])
{
    const int lane = threadIdx.x & 31;
    if (N == 16) {
#pragma unroll
        for (int i = 0; i < N; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], 16);
    }
#pragma unroll
    for (int o = N / 2; o > 0; o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < o; ++i) {
            const float keep = up ? v[i + o] : v[i], give = up ? v[i] : v[i + o];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
    return v[0];
}

struct QoParams {
    CUtensorMap kv[2][4];             // [K, V][box: a whole tile, 64, 32, 16 rows x 64 columns]
    CUtensorMap q;                    // NQ rows x 64 columns
    const TcHeader *hdr;
    const TcTile *tiles;
    uint32_t *status;
    __nv_bfloat16 *out;
    float *lse;
    int n_heads, kv_group;
    int64_t total_tokens;
    float scale_log2e;
    const float *pos, *slopes;        // ALiBi variant: token positions [T], head slopes [H]
    int stall_producer;
};

// Every role walks the block's items (query rows of a path, head) in the same order.  Keys are numbered u: the preamble at
// [0, pre_len), own rows from p16, pre_len rounded up to 16.
struct QoWalk {
    const TcTile *tiles;
    uint32_t tile, n_tiles, item_no;
    int h, n_heads, dt, dh;
    int q_row, n_rows, own_base, pre_row, pre_len, p16, q_u;      // packed row of own key u: own_base + u; q_u: key number of query row 0
    __device__ __forceinline__ explicit QoWalk(const QoParams &p)
    {
        tiles = p.tiles; n_tiles = p.hdr->n_tiles; n_heads = p.n_heads; item_no = 0xffffffffu;
        dt = gridDim.x / n_heads; dh = gridDim.x - dt * n_heads;
        tile = blockIdx.x / n_heads; h = blockIdx.x - tile * n_heads;
        h -= dh; tile -= dt;                                      // one step back: next() comes before every item
        if (h < 0) { h += n_heads; --tile; }
    }
    __device__ __forceinline__ bool next()
    {
        ++item_no; tile += dt; h += dh;
        if (h >= n_heads) { h -= n_heads; ++tile; }
        if (tile >= n_tiles) return false;
        const int4 *src = reinterpret_cast<const int4 *>(tiles + tile);
        const int4 a = src[0], b = src[1];
        q_row = a.x; n_rows = a.y; pre_row = b.x; pre_len = b.y;
        p16 = (pre_len + 15) & ~15;
        own_base = a.w - p16;
        q_u = p16 + a.z;
        return true;
    }
    __device__ __forceinline__ int end() const { return q_u + n_rows; }
    __device__ __forceinline__ int steps() const { return (end() + kQKeys - 1) / kQKeys; }
    // Key tile of step j.  ALIBI: from the last one, whose keys are the nearest, to the first: the reference is then found in the first
    // step instead of growing (and O with it) in each.
    template <bool ALIBI> __device__ __forceinline__ int tile_of(int j) const { return ALIBI ? steps() - 1 - j : j; }
};

template <int N> struct QoRing {
    uint32_t i = 0, ph = 0;
    __device__ __forceinline__ void next() { if (++i == N) { i = 0; ph ^= 1; } }
};

// ALIBI: scores get -slope_h * |pos_q - pos_k| before the softmax (Section 3.2.2).
template <int NQ, bool SPLIT, bool ALIBI>
__global__ void __launch_bounds__(kQThreads, 1) prefill_qonly_kernel(const __grid_constant__ QoParams p)
{
    using C = QoConfig<NQ, SPLIT>;
    extern __shared__ __align__(1024) unsigned char smem[];
    unsigned char *sK = smem, *sV = smem + C::V_OFF, *sQ = smem + C::Q_OFF, *sP = smem + C::P_OFF;
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + C::BAR_OFF);
    uint32_t *tmem_base_s = reinterpret_cast<uint32_t *>(bars + C::BAR_COUNT);

    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    if (threadIdx.x < C::BAR_COUNT) {
        mbar_init(&bars[threadIdx.x], threadIdx.x >= C::BAR_S_FREE ? 4 : 1);        // four warps
        fence_mbar_init();
    } else if (threadIdx.x >= 64 && threadIdx.x < 73) {
        prefetch_tmap(threadIdx.x == 72 ? &p.q : &p.kv[0][0] + (threadIdx.x - 64));
    }
    // Tensor memory is taken behind the wait and before the next kernel is let in, as in prefill_tc.cu: no block may hold it while it
    // waits for a neighbour that needs it.
    pdl_wait();
    if (warp == 8) { tmem_alloc(tmem_base_s, C::TMEM); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_trigger();
    const uint32_t tb = *tmem_base_s;
    bool ok = (smem_u32(smem) & 1023u) == 0;      // the swizzle atoms need it; reported like an expired wait

    if (warp < 8) {
        // -------------------------------------------------------------------- softmax and output, one thread per key / column
        const int ln = warp >> 2, quad = warp & 3, key = quad * 32 + lane;
        constexpr int NL = (NQ + 31) / 32;                 // queries lane, lane + 32 are this lane's when it comes to a number per query
        const uint32_t t_lane = tb + ln * C::LANE_COLS + ((uint32_t)(quad * 32) << 16);
        float *x_ln = reinterpret_cast<float *>(smem + C::X_OFF) + ln * 2 * 4 * NQ;
        float *r_w = reinterpret_cast<float *>(smem + C::R_OFF) + warp * NQ;
        float *a_ln = reinterpret_cast<float *>(smem + C::A_OFF) + ln * NQ;
        unsigned char *p_row = sP + ln * C::P_BYTES + key * 64;
        const float sc = p.scale_log2e;
        uint32_t g = 0, xb = 0;                            // tiles and exchanges so far
        // A warp whose wait ran out goes on, waiting for nothing more, to the next exchange, where all four agree to stop: none is left
        // behind at a barrier.
        bool alive = true;
        // each warp's NQ numbers (query lane + 32 i in mine[i]) -> reduced over the four warps, the same in all of them
        auto exchange = [&](float (&mine)[NL], bool is_max) {
            float *x = x_ln + (xb++ & 1) * 4 * NQ;
#pragma unroll
            for (int i = 0; i < NL; ++i) if (lane + 32 * i < NQ) x[quad * NQ + lane + 32 * i] = mine[i];
            alive = lane_barrier_and(1 + ln, ok);
#pragma unroll
            for (int i = 0; i < NL; ++i)
                if (lane + 32 * i < NQ) {
                    const float *y = x + lane + 32 * i;
                    mine[i] = is_max ? fmaxf(fmaxf(y[0], y[NQ]), fmaxf(y[2 * NQ], y[3 * NQ])) : (y[0] + y[NQ]) + (y[2 * NQ] + y[3 * NQ]);
                }
        };
        // a number per query for every thread of the warp to read
        auto publish = [&](const float (&v)[NL]) {
            __syncwarp();
#pragma unroll
            for (int i = 0; i < NL; ++i) if (lane + 32 * i < NQ) r_w[lane + 32 * i] = v[i];
            __syncwarp();
        };
        // ALIBI: position of this thread's key in step j, and what an item needs besides: loaded ahead of their use
        auto key_pos = [&](const QoWalk &w, int j) {
            const int u = w.tile_of<ALIBI>(j) * kQKeys + key;
            return u < w.pre_len || (u >= w.p16 && u < w.end()) ? p.pos[u + (u < w.pre_len ? w.pre_row : w.own_base)] : 0.f;
        };
        QoWalk w(p);
        bool more = w.next() && (ln == 0 || w.next());     // a lane takes every other item
        float pk_ahead = 0.f, pq_ahead = 0.f, slope_ahead = 0.f;
        auto load_ahead = [&]() {
            if (!ALIBI || !more) return;
            pk_ahead = key_pos(w, 0);
            if (key < w.n_rows) pq_ahead = p.pos[w.q_row + key];
            slope_ahead = p.slopes[w.h];
        };
        load_ahead();
#pragma unroll 1
        while (more && alive) {
            const int end = w.end(), steps = w.steps();
            float ref[NL];                                 // log2 units; queries that do not exist: +inf, so that their P is zero
#pragma unroll
            for (int i = 0; i < NL; ++i) ref[i] = lane + 32 * i < w.n_rows ? -INFINITY : INFINITY;
            uint64_t l[NQ / 2];                            // this thread's keys' share of the sums, two queries each
#pragma unroll
            for (int c = 0; c < NQ / 2; ++c) l[c] = 0ull;
            float neg_slope = 0.f;
            if (ALIBI) {
                neg_slope = -slope_ahead * (kLog2eQ / sc);            // in units of the unscaled score
                if (key < NQ) a_ln[key] = key < w.n_rows ? pq_ahead : 0.f;
                alive = lane_barrier_and(1 + ln, ok);
            }
#pragma unroll 1
            for (int j = 0; j < steps && alive; ++j, ++g) {
                const int u_w = w.tile_of<ALIBI>(j) * kQKeys + quad * 32, u = u_w + lane;
                const bool exists = u < w.pre_len || (u >= w.p16 && u < end);
                const bool live_w = u_w < end;             // some key of the warp exists
                const float pk = pk_ahead;
                if (ALIBI && j + 1 < steps) pk_ahead = key_pos(w, j + 1);
                const uint32_t buf = g & 1;
                ok = ok && mbar_wait_warp(&bars[C::BAR_S_FULL + 2 * ln + buf], g >> 1 & 1);
                tc_fence_after();
                uint32_t s[NQ];
                tmem_ld32(t_lane + buf * C::S_COLS, reinterpret_cast<uint32_t (&)[32]>(s));
                if (NQ == 48) tmem_ld16(t_lane + buf * C::S_COLS + 32, reinterpret_cast<uint32_t (&)[16]>(s[NQ - 16]));
                tmem_ld_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars[C::BAR_S_FREE + 2 * ln + buf]);
                if (live_w) {
                    if (ALIBI) {
#pragma unroll
                        for (int c = 0; c < NQ; c += 4) {
                            const float4 pq = *reinterpret_cast<const float4 *>(a_ln + c);
                            const float d[4] = {pq.x, pq.y, pq.z, pq.w};
#pragma unroll
                            for (int e = 0; e < 4; ++e) s[c + e] = __float_as_uint(fmaf(fabsf(d[e] - pk), neg_slope, __uint_as_float(s[c + e])));
                        }
                    }
                    // query c sees key u when u <= q_u + c: hidden from the first u - q_u queries
                    const int hidden = exists ? u - w.q_u : NQ;
                    if (__any_sync(0xffffffffu, hidden > 0)) {
#pragma unroll
                        for (int b = 0; b < NQ; b += 32) {
                            const uint32_t m = ones(hidden - b);
#pragma unroll
                            for (int c = b; c < b + 32 && c < NQ; ++c) s[c] = m >> (c - b) & 1 ? 0xff800000u : s[c];
                        }
                    }
                }
                float top[NL];
#pragma unroll
                for (int i = 0; i < NL; ++i) top[i] = -INFINITY;
                if (live_w) {
#pragma unroll
                    for (int c = 0; c < NQ; ++c) {
                        const float m = warp_max_redux(__uint_as_float(s[c]));
                        top[c / 32] = lane == c % 32 ? m : top[c / 32];
                    }
                }
                exchange(top, true);
                if (!alive) break;
                // new reference: the running maximum; SPLIT (where P's rounding does not matter): only when it is 2^8 above the old one
                float alpha[NL], minus[NL];
                bool grown = false;
#pragma unroll
                for (int i = 0; i < NL; ++i) {
                    const float t = top[i] * sc;
                    const float now = !SPLIT || j == 0 || t > ref[i] + 8.f ? fmaxf(ref[i], t) : ref[i];
                    alpha[i] = now == ref[i] ? 1.f : ex2q(ref[i] - now);
                    grown |= lane + 32 * i < NQ && now != ref[i];
                    ref[i] = now;
                    minus[i] = now == -INFINITY ? 0.f : -now;
                }
                grown = j > 0 && __any_sync(0xffffffffu, grown);
                if (grown) {
                    publish(alpha);
#pragma unroll
                    for (int c = 0; c < NQ; c += 2) l[c / 2] = mul_f32x2(l[c / 2], *reinterpret_cast<const uint64_t *>(r_w + c));
                    // O^T so far to the new reference: every product into it must be complete
                    ok = ok && mbar_wait_warp(&bars[C::BAR_O_DONE + ln], (g - 1) & 1);
                    tc_fence_after();
#pragma unroll
                    for (int b = 0; b < C::PC; b += 16) {
                        uint32_t o[16];
                        tmem_ld16(t_lane + C::O_COL + b, o);
                        tmem_ld_wait();
#pragma unroll
                        for (int c = 0; c < 16; c += 4) {
                            const float4 a = *reinterpret_cast<const float4 *>(r_w + (b + c) % NQ);
                            o[c] = __float_as_uint(__uint_as_float(o[c]) * a.x);
                            o[c + 1] = __float_as_uint(__uint_as_float(o[c + 1]) * a.y);
                            o[c + 2] = __float_as_uint(__uint_as_float(o[c + 2]) * a.z);
                            o[c + 3] = __float_as_uint(__uint_as_float(o[c + 3]) * a.w);
                        }
                        tmem_st16(t_lane + C::O_COL + b, o);
                    }
                    tmem_st_wait();
                }
                if (live_w) {
                    publish(minus);
                    uint32_t pp[C::PC / 2];
                    const uint64_t sc2 = pack_f32x2(sc, sc);
#pragma unroll
                    for (int c = 0; c < NQ; c += 2) {
                        const uint64_t m = *reinterpret_cast<const uint64_t *>(r_w + c);
                        float x0, x1;
                        unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(s[c]), __uint_as_float(s[c + 1])), sc2, m), x0, x1);
                        x0 = ex2q(x0); x1 = ex2q(x1);
                        l[c / 2] = add_f32x2(l[c / 2], pack_f32x2(x0, x1));
                        s[c] = __float_as_uint(x0); s[c + 1] = __float_as_uint(x1);
                    }
                    if (SPLIT) {
#pragma unroll
                        for (int c = 0; c < NQ; c += 2) split_bf16(__uint_as_float(s[c]), __uint_as_float(s[c + 1]), pp[c / 2], pp[SPLIT ? (NQ + c) / 2 : 0]);
                    } else if (j == 0 && quad == 0) {          // the item's first 32 keys: two numbers
#pragma unroll
                        for (int k = 0; k < NQ / 8; ++k) {
                            uint32_t lo[4];
#pragma unroll
                            for (int i = 0; i < 4; ++i) split_bf16(__uint_as_float(s[8 * k + 2 * i]), __uint_as_float(s[8 * k + 2 * i + 1]), pp[4 * k + i], lo[i]);
                            *reinterpret_cast<uint4 *>(smem + C::L_OFF + ln * C::L_BYTES + lane * 64 + ((k ^ (lane >> 1 & 3)) << 4)) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                        }
                    } else {
#pragma unroll
                        for (int c = 0; c < NQ; c += 2) pp[c / 2] = pack_bf16x2(__uint_as_float(s[c]), __uint_as_float(s[c + 1]));
                    }
                    // the product before this one has read the old P^T
                    if (j > 0) ok = ok && mbar_wait_warp(&bars[C::BAR_O_DONE + ln], (g - 1) & 1);
                    // [32 queries][key][64 bytes], 64-byte swizzle
#pragma unroll
                    for (int k = 0; k < C::PC / 8; ++k)
                        *reinterpret_cast<uint4 *>(p_row + (k >> 2) * (kQKeys * 64) + (((k & 3) ^ (key >> 1 & 3)) << 4)) =
                            make_uint4(pp[4 * k], pp[4 * k + 1], pp[4 * k + 2], pp[4 * k + 3]);
                    fence_proxy_async();
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars[C::BAR_P + ln]);
            }
            if (!alive) break;
            const int q_row = w.q_row, n_rows = w.n_rows, h = w.h;
            if (ALIBI) { more = w.next() && w.next(); load_ahead(); }
            // sums over the lane's threads
            float sum[NL], part[32];
#pragma unroll
            for (int c = 0; c < 16; ++c) unpack_f32x2(l[c], part[2 * c], part[2 * c + 1]);
            sum[0] = column_sums(part);
            if constexpr (NQ == 48) {
                float rest[16];
#pragma unroll
                for (int c = 0; c < 8; ++c) unpack_f32x2(l[16 + c], rest[2 * c], rest[2 * c + 1]);
                sum[1] = column_sums(rest);
            }
            exchange(sum, false);
            if (!alive) break;
#pragma unroll
            for (int i = 0; i < NL; ++i) {
                const int c = lane + 32 * i;
                if (p.lse && quad == 0 && c < n_rows)
                    p.lse[(int64_t)h * p.total_tokens + q_row + c] = sum[i] == 0.f ? -INFINITY : (ref[i] + log2f(sum[i])) * kLn2Q;
                sum[i] = sum[i] == 0.f ? 0.f : 1.f / sum[i];
            }
            publish(sum);
            ok = ok && mbar_wait_warp(&bars[C::BAR_O_DONE + ln], (g - 1) & 1);
            tc_fence_after();
            // O^T: this thread holds one column of all queries' outputs; neighbours swap, so that each writes 4 bytes of every other row
            const int odd = lane & 1;
            unsigned char *dst = reinterpret_cast<unsigned char *>(p.out) + ((int64_t)(q_row + odd) * p.n_heads + h) * 256 + (quad * 32 + lane - odd) * 2;
#pragma unroll
            for (int b = 0; b < NQ; b += 16) {
                if (b >= n_rows) break;
                uint32_t o[16], o2[16];
                tmem_ld16(t_lane + C::O_COL + b, o);
                if (SPLIT) tmem_ld16(t_lane + C::O_COL + NQ + b, o2);
                tmem_ld_wait();
#pragma unroll
                for (int c = 0; c < 16; c += 2) {
                    const float2 inv = *reinterpret_cast<const float2 *>(r_w + b + c);
                    float v0 = __uint_as_float(o[c]), v1 = __uint_as_float(o[c + 1]);
                    if (SPLIT) { v0 += __uint_as_float(o2[c]); v1 += __uint_as_float(o2[c + 1]); }
                    v0 *= inv.x; v1 *= inv.y;
                    const float other = __shfl_xor_sync(0xffffffffu, odd ? v0 : v1, 1);
                    if (b + c + odd < n_rows)
                        *reinterpret_cast<uint32_t *>(dst + (int64_t)(b + c) * p.n_heads * 256) = odd ? pack_bf16x2(other, v1) : pack_bf16x2(v0, other);
                }
            }
            if (!ALIBI) more = w.next() && w.next();       // here two items' numbers do not fit in the registers (48 rows: 547 -> 617 us)
        }
    } else if (warp == 8 || warp == 9) {
        // -------------------------------------------------------------------- MMA issuers: S^T and O^T, tiles in item order
        const uint32_t lead = elect_one();
        const bool is_o = warp == 9;
        // High word: stride-dimension offset (8 rows of an atom), descriptor version 1, swizzle: 128 bytes, P^T 64
        const uint64_t d_hi = (uint64_t)((1024u >> 4) | (1u << 14) | (2u << 29)) << 32, p_hi = (uint64_t)((512u >> 4) | (1u << 14) | (4u << 29)) << 32;
        const uint32_t k_lo = ((smem_u32(sK) & 0x3ffffu) >> 4) | (1u << 16), q_lo = ((smem_u32(sQ) & 0x3ffffu) >> 4) | (1u << 16);
        const uint32_t v_lo = ((smem_u32(sV) & 0x3ffffu) >> 4) | ((uint32_t)(kQKeys * 128) >> 4 << 16);     // leading dimension: next half
        const uint32_t p_lo = ((smem_u32(sP) & 0x3ffffu) >> 4) | ((uint32_t)(kQKeys * 64) >> 4 << 16);      // ... next 32 queries
        const uint32_t l_lo = ((smem_u32(smem + C::L_OFF) & 0x3ffffu) >> 4) | (1u << 16);
        uint32_t g[2] = {0, 0};                            // tiles of each lane so far
        QoRing<C::NK> k;
        QoRing<C::NV> v;
        QoRing<C::NS> q;
#pragma unroll 1
        for (QoWalk w(p); ok && w.next();) {
            const int ln = w.item_no & 1, steps = w.steps(), end = w.end();
            const uint32_t t_lane = tb + ln * C::LANE_COLS;
            uint32_t gl = ln ? g[1] : g[0];
#pragma unroll 1
            for (int j = 0; j < steps; ++j, ++gl) {
                if (!is_o) {
                    if (!(ok = mbar_wait_warp(&bars[C::BAR_K_FULL + k.i], k.ph))) break;
                    if (j == 0 && !(ok = mbar_wait_warp(&bars[C::BAR_Q_FULL + q.i], q.ph))) break;
                    const uint32_t buf = gl & 1;
                    if (gl > 1 && !(ok = mbar_wait_warp(&bars[C::BAR_S_FREE + 2 * ln + buf], ((gl >> 1) - 1) & 1))) break;
                    tc_fence_after();
                    const uint64_t kd = d_hi | uniform(k_lo + k.i * (kQKvBytes >> 4)), qd = d_hi | uniform(q_lo + q.i * (C::Q_BYTES >> 4));
                    const uint32_t d = uniform(t_lane + buf * C::S_COLS);
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk)         // contraction over head_dim
                        umma_ss(lead, d, kd + (kk >> 2) * ((kQKeys * 128) >> 4) + (kk & 3) * 2, qd + (kk >> 2) * ((NQ * 128) >> 4) + (kk & 3) * 2,
                                idesc_bf16(128, NQ, 0, 0), kk > 0 ? 1u : 0u);
                    if (lead) {
                        umma_commit(&bars[C::BAR_S_FULL + 2 * ln + buf]);
                        umma_commit(&bars[C::BAR_K_EMPTY + k.i]);
                        if (j == steps - 1) umma_commit(&bars[C::BAR_Q_EMPTY + q.i]);
                    }
                    __syncwarp();
                    k.next();
                } else {
                    if (!(ok = mbar_wait_warp(&bars[C::BAR_V_FULL + v.i], v.ph))) break;
                    // V rows of keys that do not exist hold whatever follows in the packed tensor, another path's rows; their P is exactly
                    // zero, but 0 x Inf or 0 x NaN would still reach O (Section 3.2: paths do not see each other).  Zeroed.
                    const int u0 = w.tile_of<ALIBI>(j) * kQKeys, e0 = min(kQKeys, end - u0);
                    const int g0 = min(max(w.pre_len - u0, 0), kQKeys), n_gap = min(max(w.p16 - u0, 0), kQKeys) - g0, n_zero = n_gap + (-e0 & 15);
                    if (n_zero > 0) {
                        // lane & 7: 16-byte piece of a row (the swizzle permutes pieces inside a row), then half, then row
                        unsigned char *vs = sV + v.i * kQKvBytes + (lane >> 3 & 1) * (kQKeys * 128) + (lane & 7) * 16;
#pragma unroll 1
                        for (int i = lane >> 4; i < n_zero; i += 2) *reinterpret_cast<uint4 *>(vs + (i < n_gap ? g0 + i : e0 + i - n_gap) * 128) = make_uint4(0u, 0u, 0u, 0u);
                        fence_proxy_async();               // generic-proxy stores -> visible to the MMA's reads
                        __syncwarp();
                    }
                    if (!(ok = mbar_wait_warp(&bars[C::BAR_P + ln], gl & 1))) break;
                    tc_fence_after();
                    const uint64_t vd = d_hi | uniform(v_lo + v.i * (kQKvBytes >> 4)), pd = p_hi | uniform(p_lo + ln * (C::P_BYTES >> 4));
                    const uint32_t d = uniform(t_lane + C::O_COL), n = uniform((uint32_t)(e0 + 15) >> 4), fresh = uniform((uint32_t)(j == 0));
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk)         // contraction over keys
                        if (kk < n) umma_ss(lead, d, vd + kk * (2048 >> 4), pd + kk * (1024 >> 4), idesc_bf16(128, C::PC, 1, 1), kk > 0 || !fresh ? 1u : 0u);
                    if (!SPLIT && fresh) {
                        const uint64_t ld = p_hi | uniform(l_lo + ln * (C::L_BYTES >> 4));
#pragma unroll
                        for (int kk = 0; kk < 2; ++kk)
                            if (kk < n) umma_ss(lead, d, vd + kk * (2048 >> 4), ld + kk * (1024 >> 4), idesc_bf16(128, NQ, 1, 1), 1u);
                    }
                    if (lead) {
                        umma_commit(&bars[C::BAR_O_DONE + ln]);
                        umma_commit(&bars[C::BAR_V_EMPTY + v.i]);
                    }
                    __syncwarp();
                    v.next();
                }
            }
            if (ln) g[1] = gl; else g[0] = gl;
            q.next();
        }
        if (!ok) {
            // a wait ran out: every product must finish (bounded) before the tensor memory is freed
            if (lead) umma_commit(&bars[C::BAR_DRAIN + is_o]);
            __syncwarp();
            mbar_wait_warp(&bars[C::BAR_DRAIN + is_o], 0);
        }
    } else {
        // -------------------------------------------------------------------- loads: K and Q, V
        // A tile lands as [half][row][128 bytes], swizzled: one box where it is whole and of one segment, else boxes of 64, 32 and 16
        // rows of a half; ragged ends pull in at most 15 rows nobody needs.
        if (!p.stall_producer) {
            const uint32_t lead = elect_one();
            const bool is_v = warp == 11;
            const int n_slots = is_v ? C::NV : C::NK;
            uint64_t *full = &bars[is_v ? C::BAR_V_FULL : C::BAR_K_FULL], *empty = &bars[is_v ? C::BAR_V_EMPTY : C::BAR_K_EMPTY];
            const CUtensorMap *maps = p.kv[is_v];
            const uint64_t keep = l2_policy_evict_normal(), once = l2_policy_evict_first();
            int slot = 0;
            uint32_t ph = 1, fills = 0, q_fills = 0;
            QoRing<C::NS> q;
#pragma unroll 1
            for (QoWalk w(p); ok && w.next();) {
                const int head = w.h / p.kv_group * 2, steps = w.steps(), end = w.end();
                if (!is_v) {
                    if (!(ok = mbar_wait_warp(&bars[C::BAR_Q_EMPTY + q.i], q.ph ^ 1))) break;
                    uint64_t *bar = &bars[C::BAR_Q_FULL + q.i];
                    if (lead) mbar_expect_tx(bar, C::Q_BYTES);
                    __syncwarp();
#pragma unroll
                    for (int hh = 0; hh < 2; ++hh) tma_load_3d_hint(lead, sQ + q.i * C::Q_BYTES + hh * (NQ * 128), &p.q, 0, w.q_row, w.h * 2 + hh, bar, once);
                    q.next();
                    ++q_fills;
                }
#pragma unroll 1
                for (int j = 0; j < steps; ++j) {
                    if (!(ok = mbar_wait_warp(empty + slot, ph))) break;
                    const int u0 = w.tile_of<ALIBI>(j) * kQKeys, u1 = u0 + ((min(kQKeys, end - u0) + 15) & ~15), split = min(max(w.p16, u0), u1);
                    uint64_t *bar = full + slot;
                    unsigned char *dst = (is_v ? sV : sK) + slot * kQKvBytes;
                    if (lead) mbar_expect_tx(bar, (uint32_t)(u1 - u0) * 256);
                    __syncwarp();
#pragma unroll 1
                    for (int u = u0; u < u1;) {
                        const bool pre = u < split;                         // preamble part, then own part
                        const int left = (pre ? split : u1) - u, row = u + (pre ? w.pre_row : w.own_base);
                        const int box = left == kQKeys ? 0 : (left >= 64 ? 1 : (left >= 32 ? 2 : 3));
#pragma unroll 1
                        for (int hh = 0; hh < (box ? 2 : 1); ++hh)
                            tma_load_3d_hint(lead, dst + hh * (kQKeys * 128) + (u - u0) * 128, maps + box, 0, row, head + hh, bar, keep);
                        u += kQKeys >> box;
                    }
                    ++fills;
                    if (++slot == n_slots) { slot = 0; ph ^= 1; }
                }
            }
            // a wait ran out: the copies in flight must land before the block may exit (bounded)
            if (!ok) {
                for (uint32_t f = fills - min(fills, (uint32_t)n_slots); f < fills; ++f) mbar_wait_warp(full + f % n_slots, f / n_slots & 1);
                for (uint32_t f = q_fills - min(q_fills, (uint32_t)C::NS); f < q_fills; ++f) mbar_wait_warp(&bars[C::BAR_Q_FULL + f % C::NS], f / C::NS & 1);
            }
        }
    }

    __syncwarp();
    if (!ok && lane == 0) atomicExch(p.status, (uint32_t)STATUS_TIMEOUT);
    tc_fence_before();
    __syncthreads();
    if (warp == 8) tmem_dealloc(tb, C::TMEM);
}

size_t prefill_qonly_workspace_bytes(int n_prompts, int n_paths, int max_pre_len, int max_path_len)
{
    if (n_prompts < 0 || n_paths < 0 || max_pre_len < 0 || max_path_len < 0) return 256;
    return 256 + round_up((size_t)plan_max_tiles(0, n_paths, 0, max_path_len, 32) * sizeof(TcTile), 256);
}

template <int NQ, bool SPLIT> static int launch_qonly(QoParams &p, const void *q, int grid, cudaStream_t st)
{
    using C = QoConfig<NQ, SPLIT>;
    if (int rc = encode_rows_map(&p.q, q, p.total_tokens, (int64_t)p.n_heads * 128, NQ, 1)) return rc;
    auto kern = prefill_qonly_kernel<NQ, SPLIT, false>;
    if constexpr (SPLIT)
        if (p.pos) kern = prefill_qonly_kernel<NQ, SPLIT, true>;
    SP_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM));
    return launch(kern, grid, kQThreads, C::SMEM, st, 1, p);
}

// longest: query rows of a path at most; split: P as the sum of two bf16 numbers (always with more than 32 rows and with ALiBi)
int launch_prefill_qonly(const void *q, const void *k, const void *v, const sp_layout *lay, const float *pos,
                         const float *slopes, int n_heads, int n_kv_heads, float scale, int longest, bool split, void *out,
                         float *lse, void *ws, cudaStream_t st)
{
    TcHeader *hdr = static_cast<TcHeader *>(ws);
    TcTile *tiles = reinterpret_cast<TcTile *>(static_cast<char *>(ws) + 256);
    const int nq = longest > 32 ? 48 : 32;
    PlanArgs pa = {};
    pa.ppo = lay->prompt_path_off; pa.pre_start = lay->pre_start; pa.pre_len = lay->pre_len;
    pa.path_start = lay->path_start; pa.doc_len = lay->doc_len; pa.qry_len = lay->qry_len;
    pa.n_prompts = lay->n_prompts; pa.n_paths = lay->n_paths; pa.rows_mode = SP_ROWS_QUERY_ONLY; pa.tile_rows = nq;
    pa.max_pre_len = lay->max_pre_len; pa.max_path_len = lay->max_path_len; pa.total_tokens = lay->total_tokens;
    pa.max_tiles = plan_max_tiles(lay->n_prompts, lay->n_paths, lay->max_pre_len, lay->max_path_len, nq);
    pa.hdr = hdr; pa.list = tiles;
    if (int rc = launch(prefill_plan_kernel<false>, 1, 1024, 0, st, 1, pa)) return rc;

    const int64_t items = plan_max_tiles(0, lay->n_paths, 0, lay->max_path_len, nq) * n_heads;
    if (items == 0) return SP_OK;
    QoParams p;
    const void *kv[2] = {k, v};
    for (int i = 0; i < 2; ++i)
        for (int b = 0; b < 4; ++b)
            if (int rc = encode_rows_map(&p.kv[i][b], kv[i], lay->total_tokens, (int64_t)n_kv_heads * 128, kQKeys >> b, b ? 1 : 2)) return rc;
    p.hdr = hdr; p.tiles = tiles; p.status = &hdr->status;
    p.out = static_cast<__nv_bfloat16 *>(out); p.lse = lse;
    p.n_heads = n_heads; p.kv_group = n_heads / n_kv_heads;
    p.total_tokens = lay->total_tokens; p.scale_log2e = scale * kLog2eQ;
    p.pos = pos; p.slopes = slopes;
    p.stall_producer = g_stall_producer ? 1 : 0;
    const int grid = (int)std::min<int64_t>(items, num_sms());
    if (nq == 48) return launch_qonly<48, true>(p, q, grid, st);
    return split ? launch_qonly<32, true>(p, q, grid, st) : launch_qonly<32, false>(p, q, grid, st);
}

}  // namespace sp
