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
                         const float *slopes, int n_heads, int n_kv_heads, float scale, void *out, float *lse,
                         void *ws, cudaStream_t st);
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
// Query rows only, head_dim 128: which of two kernels.  The tcgen05 kernel has a quarter of its tile's rows at work (32 of 128) and
// carries P as two bf16 numbers; the warp-level kernel (prefill_qonly.cu) works on 32 rows at a time.
//  - An even number of query heads to a KV head: tcgen05, whose tiles then hold the rows of several heads.  us, tcgen05 /
//    warp-level, 4 x 20 documents behind 1 200 rows: 193 / 302 (two heads), 114 / 303 (four); ALiBi 257 / 347, 155 / 343.
//  - Few items (a path's query rows and a head each): tcgen05; the warp-level kernel has too few warps to hide its latency.  1
//    prompt x 20 documents of 64-256 rows, 32 heads: 23.3 / 24.1 behind 32 rows, 43.4 / 52.6 behind 384; 2 prompts: 47 / 54
//    behind 128, 175 / 181 behind 1 200; ALiBi 61 / 66 behind 128, 83 / 83 behind 256, 110 / 105 behind 400.
//  - More than 32 query rows in a path: tcgen05; the warp-level kernel reads every key again for each 32 rows.  48 rows, 8 x 100
//    documents: 666 / 1216 behind 48 rows, 1825 / 3114 behind 600.
//  - Otherwise warp-level: 8 x 100 documents, back to back: 622 / 600 behind 16 rows, 689 / 655 behind 48, 839 / 769 behind 128,
//    1430 / 1202 behind 384; ALiBi 722 / 696 behind 16, 841 / 758 behind 64.
// The number of query rows is known from the host mirror only; without one tcgen05 up to the preamble behind which it loses
// less than the warp-level kernel does with 33 rows and more.
static bool query_rows_warp_level(const sp_layout *lay, bool alibi, int n_heads, int n_kv_heads)
{
    if (n_heads / n_kv_heads % 2 == 0) return false;
    if ((int64_t)lay->n_paths * n_heads <= 9 * (int64_t)num_sms() && (!alibi || lay->max_pre_len <= 256)) return false;
    if (!lay->host_mirror) return lay->max_pre_len > (alibi ? 64 : 384);
    int longest = 0;
    for (int i = 0; i < lay->n_paths; ++i) longest = std::max(longest, lay->host_mirror->qry_len[i]);
    return longest <= 32;
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
    if (dtype == SP_BF16 && head_dim == 128 && rows == SP_ROWS_QUERY_ONLY && query_rows_warp_level(lay, pos != nullptr, n_heads, n_kv_heads))
        return launch_prefill_qonly(q, k, v, lay, pos, slopes, n_heads, n_kv_heads, scale, out, lse, ws, st);
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
