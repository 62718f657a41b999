// Tile list shared by the tensor-core prefill kernels: a one-block plan kernel turns the ragged
// fork-join layout (Section 3.2) into query tiles of a given height, each knowing its segment,
// its offset inside it and its prompt's fully visible preamble.
#pragma once
#include "common.cuh"

namespace sp {

struct TcTile {                       // one query tile (shared by all heads)
    int32_t q_row;                    // packed row of the tile's first query row
    int32_t n_rows;                   // valid rows in the tile (1..tile height)
    int32_t q_off;                    // offset of the first row inside its segment
    int32_t own_row;                  // packed row of the segment's first row
    int32_t pre_row, pre_len;         // fully visible prefix (the prompt's preamble), may be empty
    int32_t pad0, pad1;
};

constexpr int kPairKeys = 64;         // keys per key tile of a pair
struct alignas(16) TcPair {                       // one or two consecutive query tiles of a segment (shared by all heads)
    // Keys of the segment are numbered u: its fully visible prefix (the prompt's preamble, may be empty) at [0, pre_len),
    // its own rows from p16 = pre_len rounded up to 16.
    // Rows of consecutive paths: the "segment" starts with tile A's first path and ends with the last row of the item; what a row
    // sees of it starts with its own path.  p16 and steps_a follow from the rest there, and two other numbers take their place.
    int32_t own_base;                 // packed row of own key u is own_base + u
    int32_t q_u;                      // key number of tile A's first row
    int32_t pre_row, pre_len;
    int32_t p16;                      // rows of consecutive paths: index of tile A's first path (-1: one segment after all)
    int32_t rows_ab;                  // rows of tile A | rows of tile B, which follows it, << 16 (0: no tile B)
    int32_t steps_a;                  // key tiles of tile A; rows of consecutive paths: key number where tile B's first path starts
    int32_t steps;                    // key tiles of the item
};
static_assert(sizeof(TcPair) == sizeof(TcTile), "both lists use the same slots of the workspace");

struct TcHeader {                     // start of the workspace
    uint32_t status;
    uint32_t n_tiles;                 // entries of the list: tiles, or pairs of tiles
};

// Height of the query tiles of n rows in a row: as many tiles as it takes, of equal height in whole warps.
__host__ __device__ inline int even_height(int rows, int tile_rows)
{
    const int nt = (rows + tile_rows - 1) / tile_rows, even = nt > 1 ? ((rows + nt - 1) / nt + 31) & ~31 : tile_rows;
    return even < tile_rows ? even : tile_rows;
}

// ---- plan: ragged layout -> tile list ---------------------------------------------------
struct PlanArgs {
    const int32_t *ppo, *pre_start, *pre_len, *path_start, *doc_len, *qry_len;
    int n_prompts, n_paths, rows_mode;
    int tile_rows;                    // query rows per tile
    int max_pre_len, max_path_len;    // the host's bounds on the lengths (they sized the tile list)
    int64_t total_tokens;             // T: every segment must lie inside [0, T)
    int64_t max_tiles;                // capacity of the tile list
    int sort_from;                    // pairs: lists of at least so many records are sorted
    TcHeader *hdr;
    void *list;                       // TcTile or TcPair
};

// What the host cannot check, the plan kernel does: a segment whose device-side numbers
// contradict the host scalars (negative or oversized length, rows outside [0, T)) gets no tiles
// and the status word reports it, so nothing outside the caller's tensors is ever touched and
// the tile list cannot outgrow the workspace that was sized from those scalars.

// PAIRS: the tiles of a segment two by two from its end (an odd one stands alone at the front, where it has the
// fewest keys).  A segment that needs n tiles gets tiles of equal height, rounded up to the 32 rows of a warp:
// 184 rows as 96 + 88 instead of 128 + 56, which leaves tile A 32 keys less to look at.
//
// The attention kernel walks (record, head) with a stride of one item per block, so a block's share is a sample of the list.
// Runs of kSortWindow records are put in descending order of their work: a block then takes one of the large and one of the
// small items of every run, and the busiest block has 1 to 3 % more than the mean instead of 3 to 10 %; longer runs take
// records apart that share a prefix or a path in L2.  us unsorted / runs of 8 / 16 / 32 (launches far apart, so not at the power
// limit): 2 prompts x 400 documents 2170 / 2120 / 2086 / 2085, 64 x 17 behind a prefix 2350 / 2312 / 2306 / 2303, ALiBi 847 / 812 /
// 801 / 784; back to back 2491 / 2464 / 2447 / 2461, 2670 / 2668 / 2646 / 2657, 913 / 904 / 896 / 888, query rows only 609 / 596 /
// 590 / 597.
constexpr int kSortWindow = 16;
// ACROSS (pairs): tiles over the rows of consecutive paths.  A kernel of its own: what it has more costs a small launch 0.3 us.
template <bool PAIRS, bool ACROSS = false>
static __global__ void __launch_bounds__(1024) prefill_plan_kernel(const PlanArgs a)
{
    __shared__ int warp_tot[32];
    __shared__ int running;
    pdl_trigger();                    // the attention kernel sets itself up meanwhile
    pdl_wait();
    if (threadIdx.x == 0) { running = 0; a.hdr->status = STATUS_OK; }
    __syncthreads();
    const int n_seq = a.n_prompts + a.n_paths;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto prompt_of = [&](int i) {
        int lo = 0, hi = a.n_prompts - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (a.ppo[mid] <= i) lo = mid; else hi = mid - 1;
        }
        return lo;
    };
    bool across = ACROSS;
    if (across) {                     // what the host saw in its mirror, in the arrays themselves; otherwise segment by segment
        bool fit = true;
        for (int i = threadIdx.x; i < a.n_paths && fit; i += 1024) {
            const int b = prompt_of(i), n = a.doc_len[i] + a.qry_len[i];
            fit = a.ppo[b] >= 0 && a.ppo[b] <= i && i < a.ppo[b + 1] && a.ppo[b + 1] <= a.n_paths && a.pre_len[b] > 0 && n > 0 && n <= a.max_path_len &&
                  a.path_start[i] >= 0 && (int64_t)a.path_start[i] + n <= a.total_tokens &&
                  (i == a.ppo[b] || a.path_start[i] == a.path_start[i - 1] + a.doc_len[i - 1] + a.qry_len[i - 1]);
        }
        across = __syncthreads_and(fit);
    }
    for (int base = 0; base < n_seq; base += 1024) {
        const int s = base + threadIdx.x;
        int first = 0, rows = 0, own_row = 0, pre_row = 0, pre_n = 0;
        bool bad = false;
        if (s < a.n_prompts) {
            const int len = a.pre_len[s], row = a.pre_start[s];
            bad = len < 0 || len > a.max_pre_len || row < 0 || (int64_t)row + len > a.total_tokens;
            if (a.rows_mode == SP_ROWS_ALL && !bad) { rows = len; own_row = row; }
        } else if (s < n_seq) {
            const int i = s - a.n_prompts, lo = prompt_of(i);
            pre_row = a.pre_start[lo]; pre_n = a.pre_len[lo];
            own_row = a.path_start[i];
            const int dl = a.doc_len[i], ql = a.qry_len[i];
            bad = dl < 0 || ql < 0 || (int64_t)dl + ql > a.max_path_len || own_row < 0 ||
                  (int64_t)own_row + dl + ql > a.total_tokens ||
                  pre_n < 0 || pre_n > a.max_pre_len || pre_row < 0 || (int64_t)pre_row + pre_n > a.total_tokens;
#ifdef SP_DEBUG_BOUNDS
            // debug build: no other segment may share a row with this path (every pair is looked at)
            for (int o = 0; o < n_seq && !bad; ++o) {
                if (o == s) continue;
                const int orow = o < a.n_prompts ? a.pre_start[o] : a.path_start[o - a.n_prompts];
                const int olen = o < a.n_prompts ? a.pre_len[o] : a.doc_len[o - a.n_prompts] + a.qry_len[o - a.n_prompts];
                bad = olen > 0 && dl + ql > 0 && orow < own_row + dl + ql && own_row < orow + olen;
            }
#endif
            first = a.rows_mode == SP_ROWS_QUERY_ONLY ? dl : 0;
            rows = bad ? 0 : dl + ql - first;
        }
        if (bad) a.hdr->status = STATUS_BAD_LAYOUT;
        // Rows of consecutive paths: a prompt's rows behind its preamble are cut into pairs of tiles from the first to the last, and a
        // path writes the records of the pairs that start in it.
        const bool own = !(across && s >= a.n_prompts && rows > 0);
        int run0 = 0, run = rows, last = 0;                       // rows cut as one run, the first one's number; its last path
        if (ACROSS && !own) {
            const int b = prompt_of(s - a.n_prompts);
            last = a.ppo[b + 1] - 1;
            run0 = a.path_start[a.ppo[b]];
            run = a.path_start[last] + a.doc_len[last] + a.qry_len[last] - run0;
        }
        int nt = (rows + a.tile_rows - 1) / a.tile_rows, height = a.tile_rows;
        if (PAIRS && (nt > 1 || !own)) {
            height = even_height(run, a.tile_rows);
            nt = (rows + height - 1) / height;
        }
        const int at = own_row - run0;
        int w0 = 0, n_rec = PAIRS ? (nt + 1) / 2 : nt;
        if (ACROSS && !own) {
            w0 = (at + 2 * height - 1) / (2 * height);
            n_rec = (at + rows + 2 * height - 1) / (2 * height) - w0;
        }
        int incl = n_rec;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane == 31) warp_tot[warp] = incl;
        __syncthreads();
        int before = running;
        for (int w = 0; w < warp; ++w) before += warp_tot[w];
        const int off = before + incl - n_rec;
        for (int t = 0; t < n_rec && off + t < a.max_tiles; ++t) {
            if (ACROSS && !own) {
                const int q0 = (w0 + t) * 2 * height, rows_a = min(height, run - q0), rows_b = min(height, run - q0 - rows_a);
                TcPair pr;
                const int p16 = (pre_n + 15) & ~15;
                pr.own_base = own_row - p16;
                pr.q_u = p16 + q0 - at;
                pr.pre_row = pre_row; pr.pre_len = pre_n;
                pr.p16 = s - a.n_prompts;
                pr.rows_ab = rows_a | rows_b << 16;
                int lo = s - a.n_prompts, hi = last;              // the path of tile B's first row
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (a.path_start[mid] - run0 <= q0 + rows_a) lo = mid; else hi = mid - 1;
                }
                pr.steps_a = a.path_start[lo] - pr.own_base;
                pr.steps = (pr.q_u + rows_a + rows_b + kPairKeys - 1) / kPairKeys;
                static_cast<TcPair *>(a.list)[off + t] = pr;
            } else if (PAIRS) {
                const int t0 = max(2 * t - (nt & 1), 0);          // first tile of the record
                const bool two = !((nt & 1) && t == 0);
                const int rows_a = min(height, rows - t0 * height), rows_b = two ? min(height, rows - (t0 + 1) * height) : 0;
                TcPair pr;
                pr.p16 = (pre_n + 15) & ~15;
                pr.own_base = own_row - pr.p16;
                pr.q_u = pr.p16 + first + t0 * height;
                pr.pre_row = pre_row; pr.pre_len = pre_n;
                pr.rows_ab = rows_a | rows_b << 16;
                pr.steps_a = ACROSS ? 0 : (pr.q_u + rows_a + kPairKeys - 1) / kPairKeys;
                if (ACROSS) pr.p16 = -1;
                pr.steps = (pr.q_u + rows_a + rows_b + kPairKeys - 1) / kPairKeys;
                static_cast<TcPair *>(a.list)[off + t] = pr;
            } else {
                TcTile tl;
                tl.q_off = first + t * height;
                tl.q_row = own_row + tl.q_off;
                tl.n_rows = min(height, rows - t * height);
                tl.own_row = own_row;
                tl.pre_row = pre_row; tl.pre_len = pre_n; tl.pad0 = 0; tl.pad1 = 0;
                static_cast<TcTile *>(a.list)[off + t] = tl;
            }
        }
        __syncthreads();
        if (threadIdx.x == 1023) running = before + incl;
        __syncthreads();
    }
    const int n_list = (int)min((int64_t)running, a.max_tiles);
    if (threadIdx.x == 0) a.hdr->n_tiles = (uint32_t)n_list;
    if (PAIRS && n_list >= a.sort_from) {
        TcPair *list = static_cast<TcPair *>(a.list);
        const int at = lane & (kSortWindow - 1);
        for (int i = threadIdx.x; i - lane < n_list; i += 1024) {
            int4 *rec = reinterpret_cast<int4 *>(list + i);
            int4 lo, hi;
            int cost = -1;
            if (i < n_list) {
                lo = rec[0]; hi = rec[1];
                cost = hi.w * ((uint32_t)hi.y >> 16 ? 5 : 3);       // steps; a lone tile's takes 0.6 of a pair's
            }
            int rank = 0;
#pragma unroll
            for (int o = 0; o < kSortWindow; ++o) {
                const int other = __shfl_sync(0xffffffffu, cost, o, kSortWindow);
                rank += other > cost || (other == cost && o < at);
            }
            if (i < n_list) { rec += 2 * (rank - at); rec[0] = lo; rec[1] = hi; }
        }
    }
}

static inline int64_t plan_max_tiles(int n_prompts, int n_paths, int max_pre_len, int max_path_len, int tile_rows)
{
    return (int64_t)n_prompts * ((max_pre_len + tile_rows - 1) / tile_rows) +
           (int64_t)n_paths * ((max_path_len + tile_rows - 1) / tile_rows);
}

}  // namespace sp
