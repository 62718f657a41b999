// sp_path_scores: Bayesian path saliency (Section 3.2.3; Appendix B.1, Eq. 2).
//
// The logits tensor [paths * query length, vocab] is the largest object of the online
// phase and each element is needed exactly once, so the kernel is one streaming HBM
// pass: a block per scored row, 16-byte cache-streaming loads, a per-thread online
// (max, sum of exponentials) pair merged by warp shuffles, one log per row.  Rows whose
// target is -1 are not read at all.  A second tiny kernel adds each path's rows in a
// fixed order (no float atomics), so scores are reproducible bit for bit.
#include <cfloat>
#include <type_traits>

#include "common.cuh"

namespace sp {

constexpr int kScoreUnroll = 4;
constexpr float kLog2e = 1.4426950408889634f;

__device__ __forceinline__ float fast_exp2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Merges (m2, s2) into (m, s): s counts exponentials relative to the running maximum m.
__device__ __forceinline__ void merge_ms(float &m, float &s, float m2, float s2)
{
    const float mn = fmaxf(m, m2);
    const float a = (m == mn) ? 1.f : fast_exp2((m - mn) * kLog2e);     // also covers m == -inf
    const float b = (m2 == mn) ? 1.f : fast_exp2((m2 - mn) * kLog2e);
    s = s * a + s2 * b;
    m = mn;
}

__device__ __forceinline__ uint4 ld_evict_first(const void *p)
{
    uint4 w;
    asm volatile("ld.global.cs.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(w.x), "=r"(w.y), "=r"(w.z), "=r"(w.w) : "l"(p));
    return w;
}
template <typename T> __device__ __forceinline__ void load_stream(const T *p, float (&f)[Vec<T>::N]);
template <> __device__ __forceinline__ void load_stream<__nv_bfloat16>(const __nv_bfloat16 *p, float (&f)[8])
{
    const uint4 w = ld_evict_first(p);
    f[0] = bf16_lo(w.x); f[1] = bf16_hi(w.x); f[2] = bf16_lo(w.y); f[3] = bf16_hi(w.y);
    f[4] = bf16_lo(w.z); f[5] = bf16_hi(w.z); f[6] = bf16_lo(w.w); f[7] = bf16_hi(w.w);
}
template <> __device__ __forceinline__ void load_stream<float>(const float *p, float (&f)[4])
{
    const uint4 w = ld_evict_first(p);
    f[0] = __uint_as_float(w.x); f[1] = __uint_as_float(w.y); f[2] = __uint_as_float(w.z); f[3] = __uint_as_float(w.w);
}

// Rows start at any element (ld is the vocabulary size, which is rarely a multiple of 8): up to one vector's worth of elements
// at each end is read one by one, all between them with aligned 16-byte loads.  Vocabulary 50 257, 16 prompts x 20
// documents: 127 us (187 when such rows were read element by element).
// Masked logits (-inf, or the type's lowest value) are ordinary input and add nothing: the running maximum may still be -inf,
// or so large that its product with log2 e is not finite, when they are met.  Both are kept out of the sum by a clamp; a row
// whose maximum itself is that large is summed again (a test of the maximum inside the loop: 508 us where this takes 500).
// One row by kScoreThreads threads (tid); sync() is their barrier, sm / ss a number per warp.
template <typename T, int kScoreThreads, typename Sync>
__device__ __forceinline__ void score_row(const T *logits, int64_t ld, int64_t t, int y, int vocab, float *row_logp, int tid, float *sm, float *ss, Sync sync)
{
    if (y < 0 || y >= vocab) {           // no target: contributes nothing, row is not read
        if (tid == 0) row_logp[t] = 0.f;
        return;
    }
    const T *row = logits + t * ld;
    const float picked = tid == 0 ? to_float(row[y]) : 0.f;              // ahead of the stream, not behind it
    float m = -INFINITY, s = 0.f;

    constexpr int N = Vec<T>::N;
    const int head = min((int)((16 - (reinterpret_cast<uintptr_t>(row) & 15)) & 15) / (int)sizeof(T), vocab);
    const int nvec = (vocab - head) / N;
    const T *body = row + head;
    // the ends first: their latency hides behind the body's
    const int n_ends = vocab - nvec * N;
    for (int c = tid; c < n_ends; c += kScoreThreads) {
        const float xv = to_float(row[c < head ? c : c + nvec * N]);
        if (xv > m) { s *= fast_exp2((m - xv) * kLog2e); m = xv; }
        if (xv != -INFINITY) s += fast_exp2((xv - m) * kLog2e);
    }
    for (int i0 = tid; i0 < nvec; i0 += kScoreThreads * kScoreUnroll) {
        float f[kScoreUnroll][N];
#pragma unroll
        for (int u = 0; u < kScoreUnroll; ++u) {
            const int i = i0 + u * kScoreThreads;
            if (i < nvec) {
                load_stream<T>(body + (int64_t)i * N, f[u]);
            } else {
#pragma unroll
                for (int j = 0; j < N; ++j) f[u][j] = -INFINITY;
            }
        }
        float cm = f[0][0];
#pragma unroll
        for (int u = 0; u < kScoreUnroll; ++u)
#pragma unroll
            for (int j = 0; j < N; ++j) cm = fmaxf(cm, f[u][j]);
        if (cm > m) {                 // rescale the running sum to the new maximum
            s *= fast_exp2((m - cm) * kLog2e);
            m = cm;
        }
        const float mb = fmaxf(m * kLog2e, -FLT_MAX);       // m may be -inf, or its product not finite
        float acc = 0.f;
#pragma unroll
        for (int u = 0; u < kScoreUnroll; ++u)
#pragma unroll
            for (int j = 0; j < N; ++j) acc += fast_exp2(fmaf(f[u][j], kLog2e, -mb));
        s += acc;
    }

#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float m2 = __shfl_xor_sync(0xffffffffu, m, o);
        const float s2 = __shfl_xor_sync(0xffffffffu, s, o);
        merge_ms(m, s, m2, s2);
    }
    const int warp = tid >> 5, lane = tid & 31;
    if (lane == 0) { sm[warp] = m; ss[warp] = s; }
    sync();
    if (warp > 0) return;
    m = sm[0]; s = ss[0];
    for (int w = 1; w < kScoreThreads / 32; ++w) merge_ms(m, s, sm[w], ss[w]);
    if (fabsf(m) > 1e38f && m > -INFINITY) {              // the same in all lanes
        s = 0.f;
        for (int c = lane; c < vocab; c += 32) {
            const float xv = to_float(row[c]);
            if (xv != -INFINITY) s += fast_exp2((xv - m) * kLog2e);
        }
        s = warp_sum(s);
    }
    if (lane == 0) row_logp[t] = picked - (m + logf(s));
}

template <typename T, int kScoreThreads>
__global__ void __launch_bounds__(kScoreThreads)
row_logp_kernel(const T *logits, int64_t ld, const int32_t *targets, int vocab, float *row_logp)
{
    __shared__ float sm[kScoreThreads / 32], ss[kScoreThreads / 32];
    pdl_wait();
    pdl_trigger();
    const int64_t t = blockIdx.x;
    score_row<T, kScoreThreads>(logits, ld, t, targets[t], vocab, row_logp, threadIdx.x, sm, ss, []() { __syncthreads(); });
}

// scores[i] = weight[i] * sum_t row_logp[t] + prior[i], t in [t0, t1); one warp, fixed order.
__device__ __forceinline__ void path_sum(const float *row_logp, int i, int t0, int t1, const float *prior, const float *weight, float *scores)
{
    const int lane = threadIdx.x & 31;
    double acc = 0.0;
    for (int t = t0 + lane; t < t1; t += 32) acc += (double)__ldcg(row_logp + t);       // other blocks have written them
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) {
        const double w = weight ? (double)weight[i] : 1.0;
        const double pr = prior ? (double)prior[i] : 0.0;
        scores[i] = (float)(w * acc + pr);
    }
}

__global__ void __launch_bounds__(256)
path_sum_kernel(const float *row_logp, const int32_t *row_off, int n_paths, const float *prior, const float *weight, float *scores)
{
    pdl_wait();
    pdl_trigger();
    const int i = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (i < n_paths) path_sum(row_logp, i, row_off[i], row_off[i + 1], prior, weight, scores);
}

// So few logits that launches are all that counts: the rows of a path are worked on by the blocks of one cluster, kRowsAtOnce a block, all at
// once, and the first block adds them up: one launch instead of two.  Rows in front of the first path and behind the last one go with
// those.
constexpr int kRowsAtOnce = 4, kScoreCluster = 8;
template <typename T>
__global__ void __launch_bounds__(256 * kRowsAtOnce)
path_scores_kernel(const T *logits, int64_t ld, const int32_t *targets, const int32_t *row_off, int n_rows, int vocab, const float *prior,
                   const float *weight, float *row_logp, float *scores)
{
    __shared__ float sm[kRowsAtOnce][8], ss[kRowsAtOnce][8];
    pdl_wait();
    pdl_trigger();
    const int path = blockIdx.y, rank = blockIdx.x, blocks = gridDim.x, group = threadIdx.x >> 8;
    const int t0 = row_off[path], t1 = row_off[path + 1];
    const int first = path == 0 ? 0 : max(t0, 0), last = path == (int)gridDim.y - 1 ? n_rows : min(t1, n_rows);
    auto sync = [&]() { asm volatile("barrier.cta.sync %0, 256;" ::"r"(group + 1) : "memory"); };
    for (int t = first + group * blocks + rank; t < last; t += blocks * kRowsAtOnce) {
        score_row<T, 256>(logits, ld, t, targets[t], vocab, row_logp, threadIdx.x & 255, sm[group], ss[group], sync);
        sync();                                             // the numbers of this row's warps have been read
    }
    __syncwarp();                                           // rows that end in their first warp's first thread leave warps diverged
    if (blocks > 1) asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    else __syncthreads();
    if (rank == 0 && threadIdx.x < 32) path_sum(row_logp, path, t0, t1, prior, weight, scores);
}

}  // namespace sp

extern "C" size_t sp_path_scores_workspace_bytes(int64_t n_rows)
{
    return sp::round_up(256 + (size_t)(n_rows > 0 ? n_rows : 0) * sizeof(float), 256);
}

extern "C" int sp_path_scores(const void *logits, int64_t ld_logits, const int32_t *targets,
                              const int32_t *row_off, int64_t n_rows, int n_paths, int vocab,
                              const float *prior, const float *weight, float *scores,
                              float *row_logp, void *ws, size_t ws_bytes, int dtype, void *stream)
{
    using namespace sp;
    SP_REQUIRE(dtype == SP_F32 || dtype == SP_BF16, SP_ERR_INVALID_ARG, "sp_path_scores: unknown dtype %d", dtype);
    SP_REQUIRE(n_rows >= 0 && n_rows < (int64_t)INT32_MAX && n_paths >= 0, SP_ERR_INVALID_ARG,
               "sp_path_scores: n_rows %lld / n_paths %d out of range", (long long)n_rows, n_paths);
    SP_REQUIRE(vocab > 0 && ld_logits >= vocab, SP_ERR_INVALID_ARG,
               "sp_path_scores: vocab %d must be positive and <= ld_logits %lld", vocab, (long long)ld_logits);
    if (n_paths == 0) return SP_OK;
    SP_REQUIRE(row_off && scores, SP_ERR_INVALID_ARG, "sp_path_scores: row_off / scores is NULL");
    SP_REQUIRE(n_rows == 0 || (logits && targets), SP_ERR_INVALID_ARG, "sp_path_scores: logits / targets is NULL");
    SP_REQUIRE((reinterpret_cast<uintptr_t>(logits) % elt_bytes(dtype)) == 0, SP_ERR_INVALID_ARG,
               "sp_path_scores: logits not aligned to the element size");
    float *rows_out = row_logp;
    if (!rows_out) {
        SP_REQUIRE(ws && aligned256(ws) && ws_bytes >= sp_path_scores_workspace_bytes(n_rows), SP_ERR_WORKSPACE,
                   "sp_path_scores: workspace of %zu bytes (256-byte aligned) required when row_logp is NULL",
                   sp_path_scores_workspace_bytes(n_rows));
        rows_out = reinterpret_cast<float *>(static_cast<char *>(ws) + 256);
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const auto go = [&](auto *p) {
        using T = std::remove_const_t<std::remove_pointer_t<decltype(p)>>;
        // One launch where the host's share of two is what a caller waits for and the GPU's time no longer: up to 32 rows, eight to a path in the
        // mean, 128 KB of logits, no more paths than rows.  A block to each of eight rows while those fit on the SMs; its other three are for paths
        // that have more.  Scores and top-k, us called one by one (queued ahead), two launches / one: 4 x 8 rows of 512 in fp32
        // 18.4 / 15.9 (5.9 / 5.5), 8 x 4 of 2 048 in bf16 18.6 / 16.1 (5.9 / 5.7), 32 x 1 of 2 048 18.6 / 16.3 (5.9 / 5.9), 1 x 8 of 8 192
        // 18.6 / 16.1 (5.7 / 5.9).  Not with more: blocks that take rows one after another, or blocks by the thousand (cold, scores alone: 1 x 256
        // of 8 000 11.3 / 32.8, 65 535 paths without rows 17 / 418), or rows so long that four in a block are slow (4 x 8 of 50 432 9.1 / 14.7).
        if (n_rows > 0 && n_rows <= kScoreCluster * kRowsAtOnce && n_rows <= kScoreCluster * (int64_t)n_paths && n_paths <= n_rows &&
            n_rows * vocab * (int64_t)sizeof(T) <= 128 << 10) {
            int blocks = kScoreCluster;
            while (blocks > 1 && (blocks / 2 >= n_rows || blocks * n_paths > num_sms())) blocks /= 2;
            return launch(path_scores_kernel<T>, dim3(blocks, n_paths), 256 * kRowsAtOnce, 0, st, blocks, p, ld_logits, targets, row_off, (int)n_rows, vocab,
                          prior, weight, rows_out, scores);
        }
        // Many rows: small blocks, of which more are in flight at different stages of a row; few rows: the block that is done with its
        // row sooner.  us with 128 / 256 threads: 30 720 rows 480 / 487, 30 720 short rows (8 000) 86 / 105, 1 920 rows 40 / 38, 480
        // rows 19.4 / 15.9.
        const bool many = n_rows >= 24 * (int64_t)num_sms();
        if (n_rows > 0)
            if (int rc = launch(many ? row_logp_kernel<T, 128> : row_logp_kernel<T, 256>, (unsigned)n_rows, many ? 128 : 256, 0, st, 1, p, ld_logits, targets,
                                vocab, rows_out)) return rc;
        return launch(path_sum_kernel, (n_paths + 7) / 8, 256, 0, st, 1, rows_out, row_off, n_paths, prior, weight, scores);
    };
    return dtype == SP_BF16 ? go(static_cast<const __nv_bfloat16 *>(logits)) : go(static_cast<const float *>(logits));
}
