// Fork-join prefill attention, fp32 SIMT variant (Section 3.2: a row attends to its
// prompt's preamble and, causally, to its own path).
//
// Used for fp32 storage (the tight tolerance rules out reduced-precision products).  A block owns 16 query rows of one
// segment and one head and walks their keys (the preamble's rows, then the segment's own up to its last row) in tiles
// staged in shared memory; masked tiles are never visited.  Half a warp shares two query rows: a thread holds their scores
// against every 16th key of the tile, reduces maxima and sums over the half warp (online softmax, exact exp2f), and then
// owns 2 x D / 16 outputs.  One tile of the small problems this path serves is a handful of dependent memory
// latencies; the warp-per-row loop before it took one per key (176 tokens x 4 heads x 64: 43 us, now 5.6).
#include "common.cuh"

namespace sp {

constexpr int kSimtThreads = 128;
constexpr int kSimtRows = 16;        // query rows per block
constexpr int64_t kSimtMaxBlocks = 1 << 17;      // in a launch, per head
constexpr float kLog2eP = 1.4426950408889634f;
constexpr float kLn2P = 0.6931471805599453f;

struct PrefillSimtArgs {
    const float *q, *k, *v;
    float *out, *lse;
    const int32_t *ppo, *pre_start, *pre_len, *path_start, *doc_len, *qry_len;
    uint32_t *status;            // workspace status word
    int n_prompts, n_paths, n_heads, n_kv_heads, rows_mode;
    int max_pre_len, max_path_len;               // the host's bounds on the lengths
    int n_pre_blocks, tile0;                     // blocks of the preambles (those of the paths follow), first row tile of the launch
    int64_t total_tokens;
    float scale_log2e;
    const float *pos, *slopes;   // ALiBi: token positions [T] and head slopes [H]; NULL = no bias
};

// Sequence seq (prompt preambles first, then paths): its key ranges [pre_lo, pre_lo + pre_n), fully visible, and [own_lo,
// own_lo + own_n), causal, and the first row to compute.  False where the device arrays contradict the host scalars (negative or
// oversized length, rows outside [0, T)), as in the plan of the tensor-core kernels: such a segment is skipped and reported.
struct SimtSegment { int pre_lo, pre_n, own_lo, own_n, first_row; };
__device__ __forceinline__ bool simt_segment(const PrefillSimtArgs &a, int seq, SimtSegment &g)
{
    int dl = 0, ql, most;
    if (seq < a.n_prompts) {
        g.pre_lo = 0; g.pre_n = 0;
        g.own_lo = a.pre_start[seq]; ql = a.pre_len[seq]; most = a.max_pre_len;
    } else {
        const int i = seq - a.n_prompts;
        int lo = 0, hi = a.n_prompts - 1;           // prompt owning path i
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (a.ppo[mid] <= i) lo = mid; else hi = mid - 1;
        }
        g.pre_lo = a.pre_start[lo]; g.pre_n = a.pre_len[lo];
        g.own_lo = a.path_start[i]; dl = a.doc_len[i]; ql = a.qry_len[i]; most = a.max_path_len;
    }
    g.own_n = dl + ql;
    g.first_row = a.rows_mode == SP_ROWS_QUERY_ONLY ? (seq < a.n_prompts ? ql : dl) : 0;
    // all below 2^31 once none is negative: sums of two fit 32 bits
    const uint32_t T = (uint32_t)a.total_tokens;
    return (g.pre_lo | g.pre_n | g.own_lo | dl | ql) >= 0 && (uint32_t)dl + ql <= (uint32_t)most && (uint32_t)g.own_lo + g.own_n <= T &&
           (uint32_t)g.pre_lo + g.pre_n <= T && g.pre_n <= a.max_pre_len;
}

// The status word, written by one block that computes nothing; a function of its own, so that the other blocks, whose time goes
// by the code they have to fetch, do not carry it.
static __device__ __noinline__ void simt_report(const PrefillSimtArgs &a)
{
    bool bad = false;
    for (int s = threadIdx.x; s < a.n_prompts + a.n_paths; s += kSimtThreads) { SimtSegment g; bad |= !simt_segment(a, s, g); }
    bad = __syncthreads_or(bad);
    if (threadIdx.x == 0) *a.status = bad ? STATUS_BAD_LAYOUT : STATUS_OK;
}

// grid: x = row tiles of the preambles, row tiles of the paths, and one block more that reports on the layout; y = head.
// head_dim 64: registers for four blocks per SM, as shared memory would let five in (32 query-row tiles of 4 prompts: 44.2 us with
// five, whose SMs then have unequal shares, 41.6 with four; head_dim 128 is 4 % slower with this bound).
template <int D>
__global__ void __launch_bounds__(kSimtThreads, D == 64 ? 4 : 5)
prefill_simt_kernel(const __grid_constant__ PrefillSimtArgs a)
{
    constexpr int BN = 4096 / D;             // keys per tile: 32 KB of K and V
    constexpr int KPT = BN / 16;             // keys per thread
    constexpr int CPT = D / 64;              // float4 output columns per thread and row
    constexpr int KS = D + 4;                // padded K row: 16 lanes reading 16 rows hit different banks
    __shared__ __align__(16) float sq[kSimtRows][D], sk[BN][KS], sv[BN][D], sp_[kSimtRows][BN];
    __shared__ float s_pos[BN];

    pdl_wait();
    pdl_trigger();
    const int h = blockIdx.y, hk = h / (a.n_heads / a.n_kv_heads);
    const bool pre = (int)blockIdx.x < a.n_pre_blocks;
    const int x = pre ? blockIdx.x : blockIdx.x - a.n_pre_blocks, n = pre ? a.n_prompts : a.n_paths;
    if (blockIdx.x == gridDim.x - 1) {
        if (h == 0) simt_report(a);
        return;
    }
    const int tile = x / n, seq = x - tile * n + (pre ? 0 : a.n_prompts);
    SimtSegment g;
    if (!simt_segment(a, seq, g)) return;
    const int pre_lo = g.pre_lo, pre_n = g.pre_n, own_lo = g.own_lo, own_n = g.own_n, first_row = g.first_row;
    const int r0 = first_row + (a.tile0 + tile) * kSimtRows;    // first row of the tile, counted in the segment
    const int n_rows = min(kSimtRows, own_n - r0);
    if (n_rows <= 0) return;
    const int n_keys = pre_n + r0 + n_rows;

    for (int i = threadIdx.x; i < kSimtRows * (D / 4); i += kSimtThreads) {
        const int r = i / (D / 4), c = i % (D / 4);
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r < n_rows) x = *reinterpret_cast<const float4 *>(a.q + ((int64_t)(own_lo + r0 + r) * a.n_heads + h) * D + c * 4);
        *reinterpret_cast<float4 *>(&sq[r][c * 4]) = make_float4(x.x * a.scale_log2e, x.y * a.scale_log2e, x.z * a.scale_log2e, x.w * a.scale_log2e);
    }

    const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15, row = 2 * ty;
    float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f}, pq[2] = {0.f, 0.f};
    float4 o[2][CPT];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
#pragma unroll
        for (int c = 0; c < CPT; ++c) o[r][c] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (a.pos && row + r < n_rows) pq[r] = a.pos[own_lo + r0 + row + r];
    }
    const float slope_l2 = a.pos ? a.slopes[h] * kLog2eP : 0.f;

    for (int base = 0; base < n_keys; base += BN) {
        __syncthreads();
        for (int i = threadIdx.x; i < BN * (D / 4); i += kSimtThreads) {
            const int key = i / (D / 4), c = i % (D / 4), j = base + key;
            float4 kx = make_float4(0.f, 0.f, 0.f, 0.f), vx = kx;
            if (j < n_keys) {
                const int64_t at = ((int64_t)(j < pre_n ? pre_lo + j : own_lo + j - pre_n) * a.n_kv_heads + hk) * D + c * 4;
                kx = *reinterpret_cast<const float4 *>(a.k + at);
                vx = *reinterpret_cast<const float4 *>(a.v + at);
            }
            *reinterpret_cast<float4 *>(&sk[key][c * 4]) = kx;
            *reinterpret_cast<float4 *>(&sv[key][c * 4]) = vx;
        }
        if (a.pos && threadIdx.x < BN) {
            const int j = base + (int)threadIdx.x;
            s_pos[threadIdx.x] = j < n_keys ? a.pos[j < pre_n ? pre_lo + j : own_lo + j - pre_n] : 0.f;
        }
        __syncthreads();

        float s[2][KPT];
#pragma unroll
        for (int i = 0; i < KPT; ++i) s[0][i] = s[1][i] = 0.f;
#pragma unroll 4
        for (int d = 0; d < D; d += 4) {
            const float4 q0 = *reinterpret_cast<const float4 *>(&sq[row][d]), q1 = *reinterpret_cast<const float4 *>(&sq[row + 1][d]);
#pragma unroll
            for (int i = 0; i < KPT; ++i) {
                const float4 kx = *reinterpret_cast<const float4 *>(&sk[tx + 16 * i][d]);
                s[0][i] = fmaf(q0.x, kx.x, fmaf(q0.y, kx.y, fmaf(q0.z, kx.z, fmaf(q0.w, kx.w, s[0][i]))));
                s[1][i] = fmaf(q1.x, kx.x, fmaf(q1.y, kx.y, fmaf(q1.z, kx.z, fmaf(q1.w, kx.w, s[1][i]))));
            }
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int lim = pre_n + r0 + row + r + 1 - base;         // keys of the tile this row may see
            float mx = -INFINITY;
#pragma unroll
            for (int i = 0; i < KPT; ++i) {
                if (a.pos) s[r][i] -= slope_l2 * fabsf(pq[r] - s_pos[tx + 16 * i]);     // ALiBi: linear distance penalty
                if (tx + 16 * i >= lim) s[r][i] = -INFINITY;
                mx = fmaxf(mx, s[r][i]);
            }
#pragma unroll
            for (int d = 8; d > 0; d >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, d));
            if (mx > m[r]) {                                          // the same in the whole half warp
                const float rs = exp2f(m[r] - mx);
                l[r] *= rs;
#pragma unroll
                for (int c = 0; c < CPT; ++c) { o[r][c].x *= rs; o[r][c].y *= rs; o[r][c].z *= rs; o[r][c].w *= rs; }
                m[r] = mx;
            }
#pragma unroll
            for (int i = 0; i < KPT; ++i) {
                const float p = s[r][i] == -INFINITY ? 0.f : exp2f(s[r][i] - m[r]);
                l[r] += p;                                            // this thread's keys; summed over the half warp at the end
                sp_[row + r][tx + 16 * i] = p;
            }
        }
        __syncwarp();
        // V rows hidden from both rows of the pair are not touched, and the key that only the second row sees has no part in the
        // first: 0 x Inf or 0 x NaN would reach the rows in front of it
        const int n_here = min(BN, n_keys - base), last = pre_n + r0 + row + 1 - base;
#pragma unroll 4
        for (int key = 0; key < min(n_here, last); ++key) {
            const float p0 = sp_[row][key], p1 = sp_[row + 1][key];
#pragma unroll
            for (int c = 0; c < CPT; ++c) {
                const float4 vx = *reinterpret_cast<const float4 *>(&sv[key][c * 64 + tx * 4]);
                o[0][c].x = fmaf(p0, vx.x, o[0][c].x); o[0][c].y = fmaf(p0, vx.y, o[0][c].y);
                o[0][c].z = fmaf(p0, vx.z, o[0][c].z); o[0][c].w = fmaf(p0, vx.w, o[0][c].w);
                o[1][c].x = fmaf(p1, vx.x, o[1][c].x); o[1][c].y = fmaf(p1, vx.y, o[1][c].y);
                o[1][c].z = fmaf(p1, vx.z, o[1][c].z); o[1][c].w = fmaf(p1, vx.w, o[1][c].w);
            }
        }
        if (last >= 0 && last < n_here) {
            const float p1 = sp_[row + 1][last];
#pragma unroll
            for (int c = 0; c < CPT; ++c) {
                const float4 vx = *reinterpret_cast<const float4 *>(&sv[last][c * 64 + tx * 4]);
                o[1][c].x = fmaf(p1, vx.x, o[1][c].x); o[1][c].y = fmaf(p1, vx.y, o[1][c].y);
                o[1][c].z = fmaf(p1, vx.z, o[1][c].z); o[1][c].w = fmaf(p1, vx.w, o[1][c].w);
            }
        }
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
#pragma unroll
        for (int d = 8; d > 0; d >>= 1) l[r] += __shfl_xor_sync(0xffffffffu, l[r], d);
        if (row + r >= n_rows) continue;
        const int64_t at = own_lo + r0 + row + r;
        const float inv = 1.f / l[r];
#pragma unroll
        for (int c = 0; c < CPT; ++c)
            *reinterpret_cast<float4 *>(a.out + (at * a.n_heads + h) * D + c * 64 + tx * 4) =
                make_float4(o[r][c].x * inv, o[r][c].y * inv, o[r][c].z * inv, o[r][c].w * inv);
        if (a.lse && tx == 0) a.lse[(int64_t)h * a.total_tokens + at] = (m[r] + log2f(l[r])) * kLn2P;
    }
}

int launch_prefill_simt(const void *q, const void *k, const void *v, const sp_layout *lay, const float *pos,
                        const float *slopes, int n_heads, int n_kv_heads, int head_dim, float scale, int rows,
                        void *out, float *lse, void *ws, cudaStream_t st)
{
    PrefillSimtArgs a;
    a.q = static_cast<const float *>(q); a.k = static_cast<const float *>(k); a.v = static_cast<const float *>(v);
    a.out = static_cast<float *>(out); a.lse = lse; a.status = static_cast<uint32_t *>(ws);
    a.ppo = lay->prompt_path_off; a.pre_start = lay->pre_start; a.pre_len = lay->pre_len;
    a.path_start = lay->path_start; a.doc_len = lay->doc_len; a.qry_len = lay->qry_len;
    a.n_prompts = lay->n_prompts; a.n_paths = lay->n_paths; a.n_heads = n_heads; a.n_kv_heads = n_kv_heads;
    a.max_pre_len = lay->max_pre_len; a.max_path_len = lay->max_path_len;
    a.rows_mode = rows; a.total_tokens = lay->total_tokens; a.scale_log2e = scale * kLog2eP;
    a.pos = pos; a.slopes = slopes;
    // No segment is longer than T, however loose the bounds; preambles and paths have a range of their own (one prefix of 1 000
    // rows beside hundreds of short paths: 63 tiles for every path otherwise).  What is too much for one grid takes several.
    const auto tiles = [&](int64_t n) { return (std::min<int64_t>(n, lay->total_tokens) + kSimtRows - 1) / kSimtRows; };
    const int64_t pre_tiles = rows == SP_ROWS_ALL ? tiles(lay->max_pre_len) : 0, path_tiles = tiles(lay->max_path_len);
    const int64_t step = std::max<int64_t>(1, kSimtMaxBlocks / ((int64_t)lay->n_prompts + lay->n_paths));
    for (int64_t t = 0; t == 0 || t < std::max(pre_tiles, path_tiles); t += step) {
        const int64_t n_pre = lay->n_prompts * std::clamp<int64_t>(pre_tiles - t, 0, step), n_path = lay->n_paths * std::clamp<int64_t>(path_tiles - t, 0, step);
        a.tile0 = (int)t; a.n_pre_blocks = (int)n_pre;
        const dim3 grid((unsigned)(n_pre + n_path + 1), n_heads);
        const int rc = head_dim == 64 ? launch(prefill_simt_kernel<64>, grid, kSimtThreads, 0, st, 1, a)
                                      : launch(prefill_simt_kernel<128>, grid, kSimtThreads, 0, st, 1, a);
        if (rc) return rc;
    }
    return SP_OK;
}

}  // namespace sp
