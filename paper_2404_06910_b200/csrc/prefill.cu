// sp_superpose_prefill entry point: argument checks and kernel selection.
#include <algorithm>

#include "common.cuh"

namespace sp {
int launch_prefill_simt(const void *q, const void *k, const void *v, const sp_layout *lay, const float *pos,
                        const float *slopes, int n_heads, int n_kv_heads, int head_dim, float scale, int rows,
                        void *out, float *lse, void *ws, cudaStream_t st);
size_t prefill_tc_workspace_bytes(int n_prompts, int n_paths, int max_pre_len, int max_path_len, int n_heads);
int launch_prefill_tc(const void *q, const void *k, const void *v, const sp_layout *lay, const float *pos,
                      const float *slopes, int n_heads, int n_kv_heads, int head_dim, float scale, int rows, void *out,
                      float *lse, void *ws, cudaStream_t st);
size_t prefill_tc_rope_workspace_bytes(int n_prompts, int n_paths, int max_pre_len, int max_path_len, int64_t total_tokens);
int launch_prefill_tc_rope(const void *q, const void *k, const void *v, const sp_layout *lay, const float *pos, double base,
                           int pairing, int n_heads, int n_kv_heads, float scale, void *out, float *lse, void *ws,
                           cudaStream_t st);
size_t prefill_qonly_workspace_bytes(int n_prompts, int n_paths, int max_pre_len, int max_path_len);
int launch_prefill_qonly(const void *q, const void *k, const void *v, const sp_layout *lay, const float *pos,
                         const float *slopes, int n_heads, int n_kv_heads, float scale, int longest, bool split, void *out,
                         float *lse, void *ws, cudaStream_t st);
}  // namespace sp

extern "C" size_t sp_prefill_workspace_bytes(int n_prompts, int n_paths, int max_pre_len,
                                             int max_path_len, int n_heads, int head_dim, int dtype)
{
    if (dtype == SP_BF16)                         // enough for either rows mode
        return std::max(sp::prefill_tc_workspace_bytes(n_prompts, n_paths, max_pre_len, max_path_len, n_heads),
                        sp::prefill_qonly_workspace_bytes(n_prompts, n_paths, max_pre_len, max_path_len));
    return 256;
}

namespace sp {
// Query rows only, head_dim 128: which of two kernels, and how P is carried in the one made for them (prefill_qonly.cu).
//  - An even number of query heads to a KV head: the kernel for all rows, whose tiles then hold the rows of several heads and load
//    K and V once for them.  us, that / prefill_qonly.cu, 32 rows of 8 x 100 documents behind 48 rows: 336 / 387 (two heads), 200 /
//    365 (four).
//  - More than 48 query rows in a path, which are two items there: the kernel for all rows.  64 rows 704 / 998, behind 400 rows 1521 / 2001.
//  - Otherwise prefill_qonly.cu.  8 x 100 documents, against what served them before (the tcgen05 kernel for few items and for more
//    than 32 rows, a warp-level one): 32 rows behind 48 610 / 470, behind 384 1162 / 724, behind 1 200 (4 x 100) 1334 / 860; 8 rows 549 / 416;
//    48 rows 734 / 553, behind 600 2270 / 1290; ALiBi 32 rows 762 / 480, 48 rows 792 / 718; 1 prompt x 20 documents 22.0 / 17.4.
// The number of query rows is known from the host mirror only; without one the kernel for all rows, but for many items behind a preamble
// from which on it loses more than the other one does with more than 48 rows.
// P as two bf16 numbers, but without a bias and with many items (path, head) of a few key tiles: there it is one number except for an
// item's first 32 keys, which is more exact than what served them before (of the norm from 64-bit results, 40 prompts of 10 or 20
// documents: 2.01e-3 to 2.14e-3, 2.09e-3 to 2.16e-3 before; two numbers 1.66e-3) and 0 to 3 % faster (documents of 32-64 rows 100.5 / 104.0 us); a
// probability is then off by 2^-9 of itself at most.
// With more key tiles the running maximum it needs costs more than the second number (behind 384 rows 836 / 721).  Under ALiBi the
// weight is on the nearest keys, which 32 fixed ones do not catch: 1.82e-3 to 1.89e-3 where it was 1.88e-3 before; two numbers 1.66e-3, at up
// to 3 % of the time (behind 48 rows 474 / 476, documents of 40 rows 259 / 267).
static int qonly_rows(const sp_layout *lay, bool alibi, int n_heads, int n_kv_heads)      // 0: the kernel for all rows
{
    if (n_heads / n_kv_heads % 2 == 0) return 0;
    if (!lay->host_mirror) return (int64_t)lay->n_paths * n_heads > 9 * (int64_t)num_sms() && lay->max_pre_len > (alibi ? 64 : 384) ? 48 : 0;
    int longest = 1;
    for (int i = 0; i < lay->n_paths; ++i) longest = std::max(longest, lay->host_mirror->qry_len[i]);
    return longest <= 48 ? longest : 0;
}
static bool qonly_split(const sp_layout *lay, bool alibi, int n_heads)
{
    return alibi || (int64_t)lay->n_paths * n_heads <= 9 * (int64_t)num_sms() || lay->max_pre_len > 128 || (int64_t)lay->max_pre_len + lay->max_path_len > 640;
}

static int prefill_entry(const void *q, const void *k, const void *v, const sp_layout *lay, const float *pos,
                         const float *slopes, int n_heads, int n_kv_heads, int head_dim, float scale, int rows,
                         void *out, float *lse, void *ws, size_t ws_bytes, int dtype, void *stream)
{
    SP_REQUIRE(dtype == SP_F32 || dtype == SP_BF16, SP_ERR_INVALID_ARG, "sp_superpose_prefill: unknown dtype %d", dtype);
    if (int rc = check_layout(lay)) return rc;
    SP_REQUIRE(head_dim == 64 || head_dim == 128, SP_ERR_UNSUPPORTED,
               "sp_superpose_prefill: head_dim %d (64 or 128 supported)", head_dim);
    SP_REQUIRE(n_heads > 0 && n_kv_heads > 0 && n_heads % n_kv_heads == 0 && n_heads <= 65535, SP_ERR_INVALID_ARG,
               "sp_superpose_prefill: n_heads %d must be a positive multiple of n_kv_heads %d", n_heads, n_kv_heads);
    SP_REQUIRE(rows == SP_ROWS_ALL || rows == SP_ROWS_QUERY_ONLY, SP_ERR_INVALID_ARG,
               "sp_superpose_prefill: unknown rows mode %d", rows);
    SP_REQUIRE(scale == scale && scale > 0.f, SP_ERR_INVALID_ARG, "sp_superpose_prefill: scale must be positive");
    if (lay->total_tokens == 0 || lay->n_prompts == 0) return SP_OK;
    SP_REQUIRE(q && k && v && out, SP_ERR_INVALID_ARG, "sp_superpose_prefill: NULL tensor");
    SP_REQUIRE(aligned16(q) && aligned16(k) && aligned16(v) && aligned16(out), SP_ERR_INVALID_ARG,
               "sp_superpose_prefill: tensors must be 16-byte aligned");
    const size_t need = sp_prefill_workspace_bytes(lay->n_prompts, lay->n_paths, lay->max_pre_len,
                                                   lay->max_path_len, n_heads, head_dim, dtype);
    SP_REQUIRE(ws && aligned256(ws) && ws_bytes >= need, SP_ERR_WORKSPACE,
               "sp_superpose_prefill: workspace of %zu bytes (256-byte aligned) required", need);

    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (dtype == SP_BF16 && head_dim == 128 && rows == SP_ROWS_QUERY_ONLY)
        if (const int longest = qonly_rows(lay, pos != nullptr, n_heads, n_kv_heads))
            return launch_prefill_qonly(q, k, v, lay, pos, slopes, n_heads, n_kv_heads, scale, longest, qonly_split(lay, pos != nullptr, n_heads), out, lse, ws, st);
    // bf16 goes to the tensor cores for both head sizes (head_dim 64, 8 prompts x 20 documents, 32 heads: 0.17 ms; the fp32
    // SIMT kernel, which served it before, took 9.4 ms)
    if (dtype == SP_BF16)
        return launch_prefill_tc(q, k, v, lay, pos, slopes, n_heads, n_kv_heads, head_dim, scale, rows, out, lse, ws, st);
    return launch_prefill_simt(q, k, v, lay, pos, slopes, n_heads, n_kv_heads, head_dim, scale, rows, out, lse, ws, st);
}
}  // namespace sp

extern "C" int sp_superpose_prefill(const void *q, const void *k, const void *v, const sp_layout *lay,
                                    int n_heads, int n_kv_heads, int head_dim, float scale, int rows,
                                    void *out, float *lse, void *ws, size_t ws_bytes, int dtype,
                                    void *stream)
{
    return sp::prefill_entry(q, k, v, lay, nullptr, nullptr, n_heads, n_kv_heads, head_dim, scale, rows, out, lse,
                             ws, ws_bytes, dtype, stream);
}

extern "C" int sp_superpose_prefill_alibi(const void *q, const void *k, const void *v, const sp_layout *lay,
                                          const float *pos, const float *slopes, int n_heads, int n_kv_heads,
                                          int head_dim, float scale, int rows, void *out, float *lse, void *ws,
                                          size_t ws_bytes, int dtype, void *stream)
{
    using namespace sp;
    SP_REQUIRE(lay == nullptr || lay->total_tokens == 0 || (pos && slopes), SP_ERR_INVALID_ARG,
               "sp_superpose_prefill_alibi: pos and slopes are required");
    return prefill_entry(q, k, v, lay, pos, slopes, n_heads, n_kv_heads, head_dim, scale, rows, out, lse, ws,
                         ws_bytes, dtype, stream);
}

extern "C" size_t sp_prefill_rope_workspace_bytes(int n_prompts, int n_paths, int max_pre_len, int max_path_len,
                                                  int64_t total_tokens, int n_heads, int head_dim, int dtype)
{
    (void)n_heads;
    if (dtype != SP_BF16 || head_dim != 128) return 256;
    return sp::prefill_tc_rope_workspace_bytes(n_prompts, n_paths, max_pre_len, max_path_len, total_tokens);
}

extern "C" int sp_superpose_prefill_rope(const void *q, const void *k, const void *v, const sp_layout *lay,
                                         const float *pos, double base, int pairing, int n_heads, int n_kv_heads,
                                         int head_dim, float scale, void *out, float *lse, void *ws, size_t ws_bytes,
                                         int dtype, void *stream)
{
    using namespace sp;
    SP_REQUIRE(dtype == SP_F32 || dtype == SP_BF16, SP_ERR_INVALID_ARG, "sp_superpose_prefill_rope: unknown dtype %d", dtype);
    if (int rc = check_layout(lay)) return rc;
    SP_REQUIRE(n_heads > 0 && n_kv_heads > 0 && n_heads % n_kv_heads == 0 && n_heads <= 65535, SP_ERR_INVALID_ARG,
               "sp_superpose_prefill_rope: n_heads %d must be a positive multiple of n_kv_heads %d", n_heads, n_kv_heads);
    SP_REQUIRE(pairing == SP_ROPE_HALF_SPLIT || pairing == SP_ROPE_INTERLEAVED, SP_ERR_INVALID_ARG,
               "sp_superpose_prefill_rope: unknown pairing %d", pairing);
    SP_REQUIRE(base > 0.0, SP_ERR_INVALID_ARG, "sp_superpose_prefill_rope: base must be positive");
    SP_REQUIRE(scale == scale && scale > 0.f, SP_ERR_INVALID_ARG, "sp_superpose_prefill_rope: scale must be positive");
    SP_REQUIRE(dtype == SP_BF16 && head_dim == 128, SP_ERR_UNSUPPORTED,
               "sp_superpose_prefill_rope: bf16 with head_dim 128 only (rotate with sp_rope_apply and call sp_superpose_prefill)");
    if (lay->total_tokens == 0 || lay->n_prompts == 0) return SP_OK;
    SP_REQUIRE(q && k && v && out && pos, SP_ERR_INVALID_ARG, "sp_superpose_prefill_rope: NULL pointer");
    SP_REQUIRE(aligned16(q) && aligned16(k) && aligned16(v) && aligned16(out), SP_ERR_INVALID_ARG,
               "sp_superpose_prefill_rope: tensors must be 16-byte aligned");
    const size_t need = sp_prefill_rope_workspace_bytes(lay->n_prompts, lay->n_paths, lay->max_pre_len, lay->max_path_len,
                                                        lay->total_tokens, n_heads, head_dim, dtype);
    SP_REQUIRE(ws && aligned256(ws) && ws_bytes >= need, SP_ERR_WORKSPACE,
               "sp_superpose_prefill_rope: workspace of %zu bytes (256-byte aligned) required", need);
    return launch_prefill_tc_rope(q, k, v, lay, pos, base, pairing, n_heads, n_kv_heads, scale, out, lse, ws,
                                  static_cast<cudaStream_t>(stream));
}
