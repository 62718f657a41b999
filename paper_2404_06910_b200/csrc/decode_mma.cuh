// One-token decode attention for query heads that share a KV head (bf16): both products on warp-level tensor-core
// instructions (mma.sync m16n8k16), fragments loaded straight from global memory.
//
// With g query heads per KV head a step still reads every K and V row once, but the SIMT kernel pays 2 g D multiply-adds a
// key, which bounds it long before HBM does (g = 4: 0.24 of the copy bandwidth).  Here a warp takes 16 keys at a time:
//   S [heads x keys] = Q K^T      A = Q, up to 8 heads in rows 0-7 of the fragment, B = K
//   O^T [d x heads] += V^T P^T    A = V^T, B = P^T, which is the S fragment as it is
// A contraction may run over its elements in any order and output rows may be any permutation, so every thread loads
// contiguous 16-byte pieces of K and V rows and uses them as fragments: no shared memory, no ldmatrix.  Only V needs a
// byte permute to pair two keys.  P is carried as the sum of two bf16 numbers (16 bits of mantissa), so the result is as
// good as with fp32 products, values that are not finite included.
#pragma once

namespace sp {

constexpr int kMmaHeads = 8;         // query heads per block at most
constexpr int kMmaKeys = 16;         // keys per warp and turn
constexpr int kMmaMaxWarps = 4;      // warps per block at most
// Warps resident per SM, by the registers that a warp's loads and accumulators take: 168 with head_dim 128, less than 128 with 64
// (64 prompts x 16 KV heads of 64: one warp to a block and 44.8 us with a budget of 12, two and 29.4 with 16).
constexpr int mma_warps_per_sm(int D) { return D == 64 ? 16 : 12; }

__device__ __forceinline__ void mma_16n8k16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

static __device__ const uint4 g_zero_row[16] = {};

// Grid (n_splits, KV heads x blocks of up to 8 query heads, prompts); the n_splits blocks of a (prompt, y) are a cluster.
template <int D, bool ALIBI, bool ROPE>
__global__ void __launch_bounds__(32 * kMmaMaxWarps, mma_warps_per_sm(D) / kMmaMaxWarps)
decode_mma_kernel(const __grid_constant__ DecodeArgs a, const __grid_constant__ DecodeRope rope, int rope_pairing)
{
    using T = __nv_bfloat16;
    constexpr int NC = D / 32;              // 16-byte pieces of a K row per thread (pieces tig + 4 c)
    constexpr int NV = D / 64;              // 16-byte pieces of a V row per thread (pieces gid + 8 c)
    constexpr int NM = D / 16;              // 16-row tiles of O^T
    constexpr int PS = D + 2;               // one partial: D outputs, max, sum

    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n_seg = a.k + 2;
    const DecodeSmem<T> sm(smem_raw, n_seg);
    const int split = blockIdx.x, b = blockIdx.z;
    const int group = a.n_heads / a.n_kv_heads, per_kv = (group + kMmaHeads - 1) / kMmaHeads;
    const int hk = blockIdx.y / per_kv, sub_group = blockIdx.y - hk * per_kv;
    const int h0 = hk * group + sub_group * kMmaHeads, nh = min(kMmaHeads, group - sub_group * kMmaHeads);
    const int64_t row_elems = (int64_t)a.n_kv_heads * D;
    const int W = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gid = lane >> 2, tig = lane & 3;
    float2 *cs = reinterpret_cast<float2 *>(sm.end);            // [D/2] (cos, sin), ROPE only
    float *red = reinterpret_cast<float *>(cs + D / 2);         // [W][nh][PS]
    float *part = red + W * nh * PS;                            // first block of the cluster: [n_splits][nh][PS]

    decode_cluster_begin(a);
    pdl_wait();
    uint4 qf[NC];                            // query head h0 + gid, unscaled bf16; on its way while the table is built
#pragma unroll
    for (int c = 0; c < NC; ++c) qf[c] = make_uint4(0u, 0u, 0u, 0u);
    if (gid < nh) {
        const uint4 *src = reinterpret_cast<const uint4 *>(static_cast<const T *>(a.q) + ((int64_t)b * a.n_heads + h0 + gid) * D);
#pragma unroll
        for (int c = 0; c < NC; ++c) qf[c] = src[tig + 4 * c];
    }
    decode_segments<T, ALIBI>(a, sm, n_seg, b, hk, D, row_elems);
    if (ROPE) decode_angles<D>(a, rope, b, cs);
    __syncthreads();
    decode_scan(sm, n_seg);
    __syncthreads();

    const int total = sm.lo[n_seg];
    const int chunk = ((total + a.n_splits - 1) / a.n_splits + kMmaKeys - 1) / kMmaKeys * kMmaKeys;
    const int lo = min(split * chunk, total), hi = min(lo + chunk, total);
    // ROPE: the newest tail row (the last key of the sequence, when there is a tail) is still unrotated
    const int j_new = (ROPE && sm.lo[n_seg] > sm.lo[n_seg - 1]) ? total - 1 : -1;
    const bool owns_new = j_new >= lo && j_new < hi;                 // block-uniform; j_new is then hi - 1
    const int hi_loop = owns_new ? hi - 1 : hi;                      // the new key is handled after the loop

    // rotates this thread's pieces tig + 4 c of a row: elements 8 (tig + 4 c) .. + 7
    auto rotate = [&](uint4 (&x)[NC]) {
        if (rope_pairing == SP_ROPE_HALF_SPLIT) {
#pragma unroll
            for (int c = 0; c < NC / 2; ++c) {
                uint32_t *lo_w = reinterpret_cast<uint32_t *>(&x[c]), *hi_w = reinterpret_cast<uint32_t *>(&x[c + NC / 2]);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float2 w0 = cs[8 * (tig + 4 * c) + 2 * e], w1 = cs[8 * (tig + 4 * c) + 2 * e + 1];
                    float n0, n1, n2, n3;
                    rope_rotate(bf16_lo(lo_w[e]), bf16_lo(hi_w[e]), w0.x, w0.y, n0, n2);
                    rope_rotate(bf16_hi(lo_w[e]), bf16_hi(hi_w[e]), w1.x, w1.y, n1, n3);
                    lo_w[e] = pack_bf16x2(n0, n1);
                    hi_w[e] = pack_bf16x2(n2, n3);
                }
            }
        } else {
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                uint32_t *wd = reinterpret_cast<uint32_t *>(&x[c]);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float2 w = cs[4 * (tig + 4 * c) + e];
                    float n0, n1;
                    rope_rotate(bf16_lo(wd[e]), bf16_hi(wd[e]), w.x, w.y, n0, n1);
                    wd[e] = pack_bf16x2(n0, n1);
                }
            }
        }
    };

    if (ROPE) rotate(qf);

    float m = -INFINITY, l = 0.f, o[NM][4];  // head gid: maximum, this thread's share of the sum; O^T rows, heads 2 tig, + 1
#pragma unroll
    for (int i = 0; i < NM; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
    const float q_pos = ALIBI ? a.q_pos[b] : 0.f;
    const float slope_l2 = (ALIBI && gid < nh) ? a.slopes[h0 + gid] * kLog2eD : 0.f;

    // 16 keys: kr = K rows gid, gid + 8; vr = V rows 2 tig, 2 tig + 1, 2 tig + 8, 2 tig + 9.  n: keys that exist.
    auto attend = [&](const uint4 (&kr)[2][NC], const uint4 (&vr)[4][NV], int n, float kpos) {
        float s[2][4];
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            s[t][0] = s[t][1] = s[t][2] = s[t][3] = 0.f;
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                mma_16n8k16(s[t], qf[c].x, 0u, qf[c].y, 0u, kr[t][c].x, kr[t][c].y);
                mma_16n8k16(s[t], qf[c].z, 0u, qf[c].w, 0u, kr[t][c].z, kr[t][c].w);
            }
        }
        float x[4];                          // keys 2 tig, 2 tig + 1, 2 tig + 8, 2 tig + 9
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int key = 2 * tig + (e & 1) + 8 * (e >> 1);
            x[e] = s[e >> 1][e & 1] * a.scale_log2e;
            if (ALIBI) x[e] -= slope_l2 * fabsf(q_pos - __shfl_sync(0xffffffffu, kpos, key));
            if (key >= n) x[e] = -INFINITY;
        }
        float mx = fmaxf(fmaxf(x[0], x[1]), fmaxf(x[2], x[3]));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        if (__any_sync(0xffffffffu, mx > m)) {
            const float m_new = fmaxf(m, mx), r = m == m_new ? 1.f : ex2f(m - m_new);      // n >= 1: m_new is a number
            m = m_new;
            l *= r;
            const float r0 = __shfl_sync(0xffffffffu, r, 8 * tig), r1 = __shfl_sync(0xffffffffu, r, 8 * tig + 4);
#pragma unroll
            for (int i = 0; i < NM; ++i) { o[i][0] *= r0; o[i][1] *= r1; o[i][2] *= r0; o[i][3] *= r1; }
        }
        float p[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) { p[e] = ex2f(x[e] - m); l += p[e]; }
        uint32_t ph0, ph1, pl0, pl1;
        split_bf16(p[0], p[1], ph0, pl0);
        split_bf16(p[2], p[3], ph1, pl1);
        // row gid of tile i is element 8 gid + i, row gid + 8 is element 8 gid + i + 64 (D = 64: 8 gid + i + 4)
#pragma unroll
        for (int i = 0; i < NM; ++i) {
            const int i1 = D == 128 ? i : i + 4;
            auto pair = [&](int k, int e, int c) {
                const uint32_t *w0 = reinterpret_cast<const uint32_t *>(&vr[k][c]), *w1 = reinterpret_cast<const uint32_t *>(&vr[k + 1][c]);
                return __byte_perm(w0[e >> 1], w1[e >> 1], (e & 1) ? 0x7632 : 0x5410);
            };
            const uint32_t a0 = pair(0, i, 0), a1 = pair(0, i1, NV - 1), a2 = pair(2, i, 0), a3 = pair(2, i1, NV - 1);
            mma_16n8k16(o[i], a0, a1, a2, a3, ph0, ph1);
            mma_16n8k16(o[i], a0, a1, a2, a3, pl0, pl1);
        }
    };

    const bool mine_new = ROPE && owns_new && warp == 0;
    const int64_t new_off = mine_new ? (int64_t)(j_new - sm.lo[n_seg - 1]) * row_elems : 0;
    if (mine_new && lane < 4)              // asked into L2 ahead of its use
        prefetch_l2((lane < 2 ? sm.k : sm.v)[n_seg - 1] + new_off + (lane & 1) * (D / 2));

    int seg = 0;
    for (int base = lo + warp * kMmaKeys; base < hi_loop; base += W * kMmaKeys) {
        const int n = min(kMmaKeys, hi_loop - base);
        // lane i (and i + 16) finds key i of the turn; keys that do not exist read the last one's K and get no weight, which is not
        // enough where V holds an Inf: they read a V row of zeros
        const int j = base + min(lane & 15, n - 1);
        while (j >= sm.lo[seg + 1]) ++seg;                  // keys ascend: segments only advance
        const int64_t off = (int64_t)(j - sm.lo[seg]) * row_elems;
        const float kpos = ALIBI ? sm.pos[seg][j - sm.lo[seg]] : 0.f;
        const unsigned long long kp = reinterpret_cast<unsigned long long>(sm.k[seg] + off), vp = reinterpret_cast<unsigned long long>((lane & 15) < n ? sm.v[seg] + off : reinterpret_cast<const T *>(g_zero_row));
        uint4 kr[2][NC], vr[4][NV];
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            const uint4 *src = reinterpret_cast<const uint4 *>(__shfl_sync(0xffffffffu, kp, gid + 8 * t));
#pragma unroll
            for (int c = 0; c < NC; ++c) kr[t][c] = ld_stream16(src + tig + 4 * c);
        }
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const uint4 *src = reinterpret_cast<const uint4 *>(__shfl_sync(0xffffffffu, vp, 2 * tig + (t & 1) + 8 * (t >> 1)));
#pragma unroll
            for (int c = 0; c < NV; ++c) vr[t][c] = ld_stream16(src + gid + 8 * c);
        }
        attend(kr, vr, n, kpos);
    }

    if (mine_new) {
        // The newest key: rotated, rounded and written back for the later steps, then one more turn with one key.
        uint4 *krow = reinterpret_cast<uint4 *>(const_cast<T *>(sm.k[n_seg - 1]) + new_off);
        const uint4 *vrow = reinterpret_cast<const uint4 *>(sm.v[n_seg - 1] + new_off);
        uint4 kr[2][NC], vr[4][NV];
#pragma unroll
        for (int c = 0; c < NC; ++c) kr[0][c] = krow[tig + 4 * c];
#pragma unroll
        for (int c = 0; c < NV; ++c) {                      // the key is number 0, of the threads with tig 0
            vr[1][c] = vr[2][c] = vr[3][c] = make_uint4(0u, 0u, 0u, 0u);
            vr[0][c] = tig == 0 ? vrow[gid + 8 * c] : vr[1][c];
        }
        rotate(kr[0]);
        __syncwarp();
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            if (gid == 0) krow[tig + 4 * c] = kr[0][c];
            kr[1][c] = kr[0][c];
        }
        attend(kr, vr, 1, 0.f);
    }

    // ---- combine the warps of this block (fixed order) --------------------------------
    l += __shfl_xor_sync(0xffffffffu, l, 1);
    l += __shfl_xor_sync(0xffffffffu, l, 2);
#pragma unroll
    for (int r = 0; r < 2; ++r)
        if (2 * tig + r < nh) {
            float *mine = red + (warp * nh + 2 * tig + r) * PS + 8 * gid;
#pragma unroll
            for (int i = 0; i < NM; ++i) { mine[i] = o[i][r]; mine[D == 128 ? i + 64 : i + 4] = o[i][2 + r]; }
        }
    if (tig == 0 && gid < nh) { red[(warp * nh + gid) * PS + D] = m; red[(warp * nh + gid) * PS + D + 1] = l; }
    __syncthreads();

    float *mine = decode_cluster_target(a, part, nh * PS);
    for (int idx = threadIdx.x; idx < nh * D; idx += blockDim.x) {
        const int r = idx / D, d = idx & (D - 1);
        float bm = -INFINITY, bl = 0.f, bo = 0.f;
        for (int i = 0; i < W; ++i) bm = fmaxf(bm, red[(i * nh + r) * PS + D]);
        for (int i = 0; i < W; ++i) {
            const float *rp = red + (i * nh + r) * PS;
            const float wgt = rp[D] == -INFINITY ? 0.f : ex2f(rp[D] - bm);
            bl += rp[D + 1] * wgt;
            bo += rp[d] * wgt;
        }
        if (a.n_splits == 1) {
            decode_store<T>(a, (int64_t)b * a.n_heads + h0 + r, D, d, bm, bl, bo);
        } else {
            mine[r * PS + d] = bo;
            if (d == 0) { mine[r * PS + D] = bm; mine[r * PS + D + 1] = bl; }
        }
    }
    decode_cluster_merge<T, D>(a, part, nh, (int64_t)b * a.n_heads + h0);
}

}  // namespace sp
