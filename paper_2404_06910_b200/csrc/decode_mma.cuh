// One-token decode attention in bf16: for query heads that share a KV head both products on warp-level tensor-core instructions
// (mma.sync m16n8k16), for single heads in fp32 arithmetic.
//
// With g query heads per KV head a step still reads every K and V row once, but the SIMT kernel pays 2 g D multiply-adds a
// key, which bounds it long before HBM does (g = 4: 0.24 of the copy bandwidth).  Here a warp takes 16 keys at a time:
//   S [heads x keys] = Q K^T      A = Q, up to 8 heads in rows 0-7 of the fragment, B = K
//   O^T [d x heads] += V^T P^T    A = V^T, B = P^T, which is the S fragment as it is
// A contraction may run over its elements in any order and output rows may be any permutation, so every thread uses
// contiguous 16-byte pieces of K and V rows as fragments: no ldmatrix.  Only V needs a byte permute to pair two keys.  P is carried as
// the sum of two bf16 numbers (16 bits of mantissa), so the result is as good as with fp32 products (1.6555e-3 of the norm from 64-bit
// results with either, the rounding of the output), values that are not finite included.
// Single heads, where the SIMT kernel's multiply-adds cost nothing that shows, keep its arithmetic: with the products above their
// log-sum-exp was up to 4.6e-6 from 64 bits where it is 1.9e-6 now and was before, and the output 3e-6 of its distance further off, at no better
// times (2 prompts x 32 heads, 8 kept of long documents 16.2 us with products, 16.0 so; 16 x 32 heads 23.2 / 22.7; D = 64 18.1 / 17.7).
// What bounds it is latency: a turn of 16 keys is a chain of 0.65 us for a warp (products, maximum, exponentials), and where loads go to
// registers nothing is in flight meanwhile.  So K and V rows run through a ring in shared memory (cp.async), two turns of 8 KB
// ahead of a warp's arithmetic: 8 warps per SM keep 128 KB in flight.  Two chains of products for S instead of one and fewer instructions per
// copy changed nothing.  Cold reads, 2 prompts x 32 heads, 8 kept of long documents 24.5 -> 21.6 us (14.5 at the copy bandwidth); which
// launches take which form, and the figures: mma_launch() in decode.cu.
#pragma once

namespace sp {

constexpr int kMmaHeads = 8;         // query heads per block at most
constexpr int kMmaKeys = 16;         // keys per warp and turn
constexpr int kMmaMaxWarps = 4;      // warps per block at most
constexpr int kMmaStages = 3;        // RING: turns of a warp in shared memory
// Warps resident per SM, by the registers that a warp's loads and accumulators take or (RING) the shared memory of its ring; held in
// registers: 64 prompts x 16 KV heads of 64: one warp to a block and 44.8 us with a budget of 12, two and 29.4 with 16.
constexpr int mma_warps_per_sm(int D, bool ring) { return D == 64 ? 16 : (ring ? 8 : 12); }
template <int D> struct MmaRing {    // a warp's: [stage]([K][V] rows of the turn's keys | positions)
    static constexpr int ROW = D * 2, V = kMmaKeys * ROW, POS = 2 * V, STAGE = POS + 128, BYTES = kMmaStages * STAGE;
};

// Start of the rings in shared memory: behind the segment table (whose size is no multiple of 16 with an odd number of segments), the
// angles and the cluster's partials, of partial_bytes each.  A multiple of 128: 16 bytes off a 32-byte sector, every copy is split (48
// units in 4 blocks of 4 warps each: 11.0 against 12.7 us).
template <int D> __host__ __device__ __forceinline__ size_t mma_ring_offset(const DecodeArgs &a, int partial_bytes)
{
    return round_up(decode_table_bytes(a.k + 2) + (D / 2) * sizeof(float2) + (a.n_splits > 1 ? (size_t)a.n_splits * partial_bytes : 0), 128);
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, bool valid)
{
    const int n = valid ? 16 : 0;        // 0: zero-filled, nothing is read
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const void *src) { asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory"); }
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ void mma_16n8k16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

static __device__ const uint4 g_zero_row[16] = {};

// Grid (n_splits, KV heads x blocks of up to 8 query heads, prompts); the n_splits blocks of a (prompt, y) are a cluster.
// RING: K and V rows go through a ring in shared memory, two turns ahead of the arithmetic; otherwise a turn's loads go to registers
// and nothing is in flight while a warp computes.
// SINGLE (with RING): one head to a KV head, in fp32 arithmetic: D / 8 lanes to a key, a running softmax per group of such lanes.
template <int D, bool ALIBI, bool ROPE, bool RING, bool SINGLE>
__global__ void __launch_bounds__(32 * kMmaMaxWarps, mma_warps_per_sm(D, RING) / kMmaMaxWarps)
decode_mma_kernel(const __grid_constant__ DecodeArgs a, const __grid_constant__ DecodeRope rope, int rope_pairing)
{
    using T = __nv_bfloat16;
    constexpr int NC = D / 32;              // 16-byte pieces of a K row per thread (pieces tig + 4 c)
    constexpr int NV = D / 64;              // 16-byte pieces of a V row per thread (pieces gid + 8 c)
    constexpr int NM = D / 16;              // 16-row tiles of O^T
    constexpr int PS = D + 2;               // one partial: D outputs, max, sum

    extern __shared__ __align__(128) unsigned char smem_raw[];
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
    unsigned char *rings = nullptr;                             // RING: behind `part`, and `red` takes their place in the end
    if constexpr (RING) {
        part = red;
        rings = smem_raw + mma_ring_offset<D>(a, min(group, kMmaHeads) * PS * (int)sizeof(float));
        red = reinterpret_cast<float *>(rings);
    }

    constexpr int LPK = D / 8, KG = 32 / LPK;                   // SINGLE: lanes to a key, groups of them
    const int sub = lane % LPK, kg = lane / LPK;

    decode_cluster_begin(a);
    pdl_wait();
    uint4 qf[NC];                            // query head h0 + gid, unscaled bf16; on its way while the table is built
    uint4 q1 = make_uint4(0u, 0u, 0u, 0u);   // SINGLE: its piece `sub`
#pragma unroll
    for (int c = 0; c < NC; ++c) qf[c] = make_uint4(0u, 0u, 0u, 0u);
    if (SINGLE) {
        q1 = reinterpret_cast<const uint4 *>(static_cast<const T *>(a.q) + ((int64_t)b * a.n_heads + h0) * D)[sub];
    } else if (gid < nh) {
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

    // SINGLE: the same for the eight elements of piece `sub`, rounded as they are stored
    auto rotate1 = [&](uint4 &x) {
        uint32_t *wd = reinterpret_cast<uint32_t *>(&x);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            float n0, n1;
            if (rope_pairing == SP_ROPE_HALF_SPLIT) {
                const bool upper = sub >= LPK / 2;
                const uint32_t other = __shfl_xor_sync(0xffffffffu, wd[e], LPK / 2), lo_w = upper ? other : wd[e], hi_w = upper ? wd[e] : other;
                const float2 w0 = cs[8 * (sub % (LPK / 2)) + 2 * e], w1 = cs[8 * (sub % (LPK / 2)) + 2 * e + 1];
                float n2, n3;
                rope_rotate(bf16_lo(lo_w), bf16_lo(hi_w), w0.x, w0.y, n0, n2);
                rope_rotate(bf16_hi(lo_w), bf16_hi(hi_w), w1.x, w1.y, n1, n3);
                if (upper) { n0 = n2; n1 = n3; }
            } else {
                const float2 w = cs[4 * sub + e];
                rope_rotate(bf16_lo(wd[e]), bf16_hi(wd[e]), w.x, w.y, n0, n1);
            }
            wd[e] = pack_bf16x2(n0, n1);
        }
    };

    if (ROPE && !SINGLE) rotate(qf);
    if (ROPE && SINGLE) rotate1(q1);
    uint64_t qs[4], acc[4];                  // SINGLE: the query's elements in log2 units, the group's output, two numbers each
    {
        float f[8];
        Raw16<T>::unpack(q1, f);
#pragma unroll
        for (int e = 0; e < 4; ++e) { qs[e] = ptx::pack_f32x2(f[2 * e] * a.scale_log2e, f[2 * e + 1] * a.scale_log2e); acc[e] = 0ull; }
    }

    float m = -INFINITY, l = 0.f, o[NM][4];  // head gid: maximum, this thread's share of the sum; O^T rows, heads 2 tig, + 1
#pragma unroll
    for (int i = 0; i < NM; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
    const float q_pos = ALIBI ? a.q_pos[b] : 0.f;
    const float slope_l2 = (ALIBI && (SINGLE || gid < nh)) ? a.slopes[h0 + (SINGLE ? 0 : gid)] * kLog2eD : 0.f;

    // SINGLE: LPK / 2 keys to a group of LPK lanes, their pieces `sub` in kr and vr; key u exists where u < n and is lanes 2 u's and 2 u + 1's (kpos)
    // once its products have been added up (half as many shuffles as if every lane had every sum, and one exponential a lane: with those, 25
    // prompts x 32 heads, 5 warps to an SM, took 114.5 us where this takes 112.2).
    constexpr int KEYS1 = LPK / 2;
    auto attend1 = [&](const uint4 (&kr)[KEYS1], const uint4 (&vr)[KEYS1], float kpos, int n) {
        auto pairs = [](const uint4 &w, uint64_t (&f)[4]) {
            const uint32_t x[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) f[e] = ptx::pack_f32x2(bf16_lo(x[e]), bf16_hi(x[e]));
        };
        float x[KEYS1];
#pragma unroll
        for (int u = 0; u < KEYS1; ++u) {
            uint64_t f[4], d = 0ull;
            pairs(kr[u], f);
#pragma unroll
            for (int e = 0; e < 4; ++e) d = ptx::fma_f32x2(qs[e], f[e], d);
            float d0, d1;
            ptx::unpack_f32x2(d, d0, d1);
            x[u] = d0 + d1;
        }
#pragma unroll
        for (int c = KEYS1 / 2, s = LPK / 2; s > 1; c /= 2, s /= 2) {          // halves of the keys change hands
            const bool up = sub & s;
#pragma unroll
            for (int u = 0; u < c; ++u) {
                const float keep = up ? x[u + c] : x[u], give = up ? x[u] : x[u + c];
                x[u] = keep + __shfl_xor_sync(0xffffffffu, give, s);
            }
        }
        x[0] += __shfl_xor_sync(0xffffffffu, x[0], 1);
        if (ALIBI) x[0] -= slope_l2 * fabsf(q_pos - kpos);
        if (sub / 2 >= n) x[0] = -INFINITY;
        float top = x[0];
#pragma unroll
        for (int s = LPK / 2; s > 1; s /= 2) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, s));
        if (top > m) {
            const float r = ex2f(m - top);
            l *= r;
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[e] = ptx::mul_f32x2(acc[e], ptx::pack_f32x2(r, r));
            m = top;
        }
        const float p = sub / 2 < n ? ex2f(x[0] - m) : 0.f;
        l += p;                                                                 // of this lane's keys
#pragma unroll
        for (int u = 0; u < KEYS1; ++u) {
            const float w = __shfl_sync(0xffffffffu, p, 2 * u, LPK);
            uint64_t f[4];
            pairs(vr[u], f);
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[e] = ptx::fma_f32x2(ptx::pack_f32x2(w, w), f[e], acc[e]);
        }
    };

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
    if constexpr (RING) {
        // Rows are stored in 16-byte pieces permuted so that the fragments' reads are free of conflicts: K by the row's parity, V by the
        // row pair.
        const unsigned char *ring = rings + warp * MmaRing<D>::BYTES;
        const uint32_t ring_s = (uint32_t)__cvta_generic_to_shared(ring);
        constexpr int PIECES = D / 8, PER = 32 / PIECES;             // of a row; rows per copy instruction
        const int piece = lane % PIECES, row0 = lane / PIECES;
        auto fetch = [&](int base, int stage) {
            if (base < hi_loop) {
                const int n = min(kMmaKeys, hi_loop - base), j = base + min(lane & 15, n - 1);
                while (j >= sm.lo[seg + 1]) ++seg;                  // lane i (and i + 16) finds key i of the turn; keys ascend: segments only advance
                const int64_t off = (int64_t)(j - sm.lo[seg]) * row_elems;
                const char *kp = reinterpret_cast<const char *>(sm.k[seg] + off), *vp = reinterpret_cast<const char *>(sm.v[seg] + off);
                const uint32_t dst = ring_s + stage * MmaRing<D>::STAGE;
                auto copy = [&](int r, const char *krow, const char *vrow, bool exists) {
                    cp_async16(dst + r * MmaRing<D>::ROW + ((piece ^ ((r & 1) << 2)) << 4), krow + piece * 16, true);
                    cp_async16(dst + MmaRing<D>::V + r * MmaRing<D>::ROW + ((piece ^ (r & 6)) << 4), vrow + piece * 16, exists);
                };
                if (n == kMmaKeys && __all_sync(0xffffffffu, seg == __shfl_sync(0xffffffffu, seg, 0))) {        // rows one after another
                    const char *k0 = reinterpret_cast<const char *>(__shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(kp), 0)) + row0 * row_elems * 2;
                    const char *v0 = reinterpret_cast<const char *>(__shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(vp), 0)) + row0 * row_elems * 2;
#pragma unroll
                    for (int i = 0; i < kMmaKeys / PER; ++i, k0 += PER * row_elems * 2, v0 += PER * row_elems * 2) copy(i * PER + row0, k0, v0, true);
                } else {
                    // keys that do not exist read the last one's K and get no weight, which is not enough where V holds an Inf: zeros for V
#pragma unroll 2
                    for (int i = 0; i < kMmaKeys / PER; ++i) {
                        const int r = i * PER + row0;
                        copy(r, reinterpret_cast<const char *>(__shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(kp), r)),
                             reinterpret_cast<const char *>(__shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(vp), r)), r < n);
                    }
                }
                if (ALIBI && lane < 16) cp_async4(dst + MmaRing<D>::POS + lane * 4, sm.pos[seg] + (j - sm.lo[seg]));
            }
            cp_async_commit();
        };
        int stage = 0;
#pragma unroll
        for (int i = 0; i < kMmaStages - 1; ++i) fetch(lo + (warp + i * W) * kMmaKeys, i);
        for (int base = lo + warp * kMmaKeys; base < hi_loop; base += W * kMmaKeys) {
            cp_async_wait<kMmaStages - 2>();
            __syncwarp();                                           // every lane's copies have landed, and the turn before this one has been read
            fetch(base + (kMmaStages - 1) * W * kMmaKeys, stage == 0 ? kMmaStages - 1 : stage - 1);
            const unsigned char *kt = ring + stage * MmaRing<D>::STAGE, *vt = kt + MmaRing<D>::V;
            if (++stage == kMmaStages) stage = 0;
            if constexpr (SINGLE) {                                 // group kg: rows kg, kg + KG, ..
                uint4 kr[KEYS1], vr[KEYS1];
#pragma unroll
                for (int u = 0; u < KEYS1; ++u) {
                    const int r = kg + u * KG;
                    kr[u] = *reinterpret_cast<const uint4 *>(kt + r * MmaRing<D>::ROW + ((sub ^ ((r & 1) << 2)) << 4));
                    vr[u] = *reinterpret_cast<const uint4 *>(vt + r * MmaRing<D>::ROW + ((sub ^ (r & 6)) << 4));
                }
                const float kpos = ALIBI ? *reinterpret_cast<const float *>(kt + MmaRing<D>::POS + (kg + sub / 2 * KG) * 4) : 0.f;
                attend1(kr, vr, kpos, (min(kMmaKeys, hi_loop - base) - kg + KG - 1) / KG);
            } else {
                uint4 kr[2][NC], vr[4][NV];
#pragma unroll
                for (int t = 0; t < 2; ++t)
#pragma unroll
                    for (int c = 0; c < NC; ++c) kr[t][c] = *reinterpret_cast<const uint4 *>(kt + (gid + 8 * t) * MmaRing<D>::ROW + (((tig + 4 * c) ^ ((gid & 1) << 2)) << 4));
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const int r = 2 * tig + (t & 1) + 8 * (t >> 1);
#pragma unroll
                    for (int c = 0; c < NV; ++c) vr[t][c] = *reinterpret_cast<const uint4 *>(vt + r * MmaRing<D>::ROW + (((gid + 8 * c) ^ (r & 6)) << 4));
                }
                attend(kr, vr, min(kMmaKeys, hi_loop - base), ALIBI ? *reinterpret_cast<const float *>(kt + MmaRing<D>::POS + (lane & 15) * 4) : 0.f);
            }
        }
        cp_async_wait<0>();
        __syncthreads();                                        // the rings are done with
    } else {
        for (int base = lo + warp * kMmaKeys; base < hi_loop; base += W * kMmaKeys) {
            const int n = min(kMmaKeys, hi_loop - base);
            // lane i (and i + 16) finds key i of the turn; keys that do not exist read the last one's K and get no weight, which is not
            // enough where V holds an Inf: they read a V row of zeros
            const int j = base + min(lane & 15, n - 1);
            while (j >= sm.lo[seg + 1]) ++seg;              // keys ascend: segments only advance
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
    }

    if (SINGLE && mine_new) {                                // as below; the key is the first group's first, all else zero: 0 x Inf is not
        uint4 *krow = reinterpret_cast<uint4 *>(const_cast<T *>(sm.k[n_seg - 1]) + new_off);
        uint4 kr[KEYS1], vr[KEYS1];
#pragma unroll
        for (int u = 0; u < KEYS1; ++u) kr[u] = vr[u] = make_uint4(0u, 0u, 0u, 0u);
        kr[0] = krow[sub];
        rotate1(kr[0]);
        __syncwarp();
        if (kg == 0) {
            krow[sub] = kr[0];
            vr[0] = reinterpret_cast<const uint4 *>(sm.v[n_seg - 1] + new_off)[sub];
        }
        attend1(kr, vr, 0.f, kg == 0 ? 1 : 0);
    } else if (mine_new) {
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
    if constexpr (SINGLE) {                                  // the groups of this warp first
        float top = m;
#pragma unroll
        for (int s = LPK; s < 32; s <<= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, s));
        const float r = m == -INFINITY ? 0.f : ex2f(m - top);
        m = top;
        l *= r;
#pragma unroll
        for (int s = 2; s < 32; s <<= 1) l += __shfl_xor_sync(0xffffffffu, l, s);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            float f[2];
            ptx::unpack_f32x2(ptx::mul_f32x2(acc[e], ptx::pack_f32x2(r, r)), f[0], f[1]);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
#pragma unroll
                for (int s = LPK; s < 32; s <<= 1) f[i] += __shfl_xor_sync(0xffffffffu, f[i], s);
                if (kg == 0) red[warp * PS + sub * 8 + 2 * e + i] = f[i];
            }
        }
        float *mine = red + warp * PS;
        if (lane == 0) { mine[D] = m; mine[D + 1] = l; }
    } else {
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
    }
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
