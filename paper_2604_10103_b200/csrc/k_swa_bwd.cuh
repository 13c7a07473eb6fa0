// Gradients of the block-sparse attention (Eq. 6) on the Blackwell tensor path, for the training rollout's step with gradient
// (Alg. 1): with respect to the queries here, to the current chunk's keys and values in the second half of this file.  128-token
// blocks.
//
// With p = softmax(s) over the kept keys of a query row, s = q k^T / sqrt(d), and g = dL/dO_local:
//     dq = (1 / sqrt(d)) * sum_c p_c (g . v_c - delta) k_c,     delta = g . o_local     (= sum_c p_c g . v_c)
// The forward pass leaves lse = log sum_c exp(s_c) per row (hf_sparse_swa), so p = exp(s - lse) needs no running maximum,
// and delta is formed per unit here, by k_rowdot for dK and dV; the block mask is the forward's (held fixed: the top-K choice is piecewise constant).
//
// Per (batch*head, query block) unit and kept key tile t, three tensor-core products:
//   S  = Q K_t^T          A = Q  (tensor memory),  B = K_t (smem, K-major)           -> TMEM [0, 128)
//   dP = dO V_t^T         A = dO (smem, K-major),  B = V_t (smem, K-major)           -> TMEM [128, 256)
//   dQ += dS K_t          A = dS (TMEM [448, 512), bf16),  B = K_t (MN-major)        -> TMEM [256, 256 + D)
// and between them, on the softmax warps (four per half g of the key columns, thread = query row):
//   dS = exp2(S c - lse log2 e) * (dP - delta) / sqrt(d)        (columns past a short block's end: 0)
// As in the forward kernel, the score buffers are free as soon as they are in registers, dS has slots of its own, dS K is
// issued per half as its four warps finish, and a warp each issues the scores and dS K: the tensor core forms the next
// tile's scores while the softmax warps work.  What bounds it: 1 536 clk of tensor time and about as much shared-memory
// operand traffic per tile (Q in tensor memory saves 256 clk of it).  12 heads of 128, 4 680 queries, 28 kept blocks: 153 us with
// one MMA warp, both score operands in shared memory and scalar softmax code, 128 with packed code, 109 like this.  (Score tiles of half
// the width, which leave room for more buffers, do not pay: a 128 x 64 product takes as long as a 128 x 128 one; 126 us.)
// A K tile is held from S to dS K (three stages), a V tile only until dP (two).  The output leaves through the tile Q came in
// by, once the next unit's Q has been copied out of it.  Every wait is bounded and reports through the device status word.
#pragma once
#include "k_swa_tc5.cuh"

// delta[r] = sum_d dO[r][d] * O[r][d].  D / 8 lanes per row (16 bytes of each tensor per lane), four rows per lane with all
// eight loads in flight: memory-bound (28.75 MB at 12 heads x 4 680 rows x 128: 11.5 us with one row per warp and four bytes
// per lane, 5.7 us like this).  grid: 1 + ceil(rows / (4 * 256 / (D / 8))), 256 threads; thread block 0 orders
// the units of the kernel that follows.
__device__ __forceinline__ float dot8(const uint4& x, const uint4& y) {
    const uint32_t xs[4] = {x.x, x.y, x.z, x.w}, ys[4] = {y.x, y.y, y.z, y.w};
    float acc = 0.f;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float2 u = unpack_bf16(xs[e]), v = unpack_bf16(ys[e]);
        acc = fmaf(u.x, v.x, fmaf(u.y, v.y, acc));
    }
    return acc;
}
template <int D>
struct RowDot { static constexpr int LPR = D / 8, RPB = 4 * 256 / LPR; };      // lanes per row; rows per thread block

// The units of the dK/dV kernel (key blocks of the current chunk) in descending order of the query blocks that keep them,
// written by one extra thread block of the k_rowdot launch before it.  Key blocks differ in popularity (9.4 +- 2.6 of 37 at 28 of
// 111 kept, i.i.d. or not): in natural order the busiest of 148 thread blocks has 49 pairs and unit ends against a mean of 37,
// in this order 38.
struct BwdOrder {
    const uint32_t* mask;    // [B*H, T_m, mask_words]
    int mask_words, first_block, n_b, Tm, BH;
    int2* order;             // [B*H * n_b]: unit, its pairs (-1: not counted)
};
constexpr int BWD_ORDER_MAX = 4096;              // units that are ordered; beyond that a thread block has dozens and balance comes by itself
__device__ __noinline__ void bwd_order_units(const BwdOrder& q) {
    __shared__ int cnt[BWD_ORDER_MAX];
    __shared__ int at[HF_MAX_TN + 2];            // units with fewer kept pairs come later: bin b holds count Tm - b
    const int n = q.BH * q.n_b, tid = threadIdx.x;
    if (n > BWD_ORDER_MAX || q.Tm > HF_MAX_TN) {
        for (int u = tid; u < n; u += 256) q.order[u] = make_int2(u, -1);
        return;
    }
    for (int u = tid; u < n; u += 256) cnt[u] = 0;
    for (int b = tid; b <= q.Tm + 1; b += 256) at[b] = 0;
    __syncthreads();
    // a thread takes mask rows tid, tid + 256, ..., four of them and two words of each in flight: a division per row.  (Three per word, the
    // words of all rows in one range: the launch took 13.1 us behind dq at 12 heads of 37 units, 10.0 like this; 6.7 without the ordering.)
    const int w0 = q.first_block >> 5, nw = ((q.first_block + q.n_b - 1) >> 5) - w0 + 1, rows = q.BH * q.Tm;
    for (int r0 = tid; r0 < rows; r0 += 4 * 256)
        for (int x0 = 0; x0 < nw; x0 += 2) {
            uint32_t bits[4][2];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int x = 0; x < 2; ++x)
                    bits[i][x] = r0 + 256 * i < rows && x0 + x < nw ? __ldg(q.mask + (size_t)(r0 + 256 * i) * q.mask_words + w0 + x0 + x) : 0u;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (r0 + 256 * i >= rows) break;
                int* mine = cnt + (r0 + 256 * i) / q.Tm * q.n_b;
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    const int j0 = (w0 + x0 + x) * 32 - q.first_block;
                    uint32_t left = bits[i][x];
                    while (left) {
                        const int j = j0 + __ffs(left) - 1;
                        left &= left - 1;
                        if (j >= 0 && j < q.n_b) atomicAdd(mine + j, 1);
                    }
                }
            }
        }
    __syncthreads();
    for (int u = tid; u < n; u += 256) atomicAdd(&at[q.Tm - cnt[u] + 1], 1);
    __syncthreads();
    if (tid < 32) {                              // at[b] = first position of bin b: running sums, 32 bins at a time
        int base = 0;
        for (int b0 = 0; b0 <= q.Tm + 1; b0 += 32) {
            const int b = b0 + tid;
            int v = b <= q.Tm + 1 ? at[b] : 0;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int x = __shfl_up_sync(0xffffffffu, v, off);
                if (tid >= off) v += x;
            }
            if (b <= q.Tm + 1) at[b] = base + v;
            base += __shfl_sync(0xffffffffu, v, 31);
        }
    }
    __syncthreads();
    for (int u = tid; u < n; u += 256) q.order[atomicAdd(&at[q.Tm - cnt[u]], 1)] = make_int2(u, cnt[u]);
}
template <int D>
__global__ void __launch_bounds__(256) k_rowdot(const bf16* __restrict__ a, const bf16* __restrict__ b, float* __restrict__ out, long long rows, BwdOrder ord) {
    typedef RowDot<D> C;
    pdl_wait();
    pdl_trigger();              // the backward kernel may set itself up; it waits for this grid before it reads delta
    if (blockIdx.x == 0) { bwd_order_units(ord); return; }      // (the first thread block: it starts first and ends last)
    const int block = blockIdx.x - 1;
    const int part = threadIdx.x % C::LPR;
    const long long r0 = (long long)block * C::RPB + threadIdx.x / C::LPR;
    uint4 x[4], y[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const long long r = r0 + i * (256 / C::LPR);
        x[i] = y[i] = make_uint4(0, 0, 0, 0);
        if (r < rows) {
            x[i] = __ldg(reinterpret_cast<const uint4*>(a + r * D) + part);
            y[i] = __ldg(reinterpret_cast<const uint4*>(b + r * D) + part);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float acc = dot8(x[i], y[i]);
#pragma unroll
        for (int off = C::LPR / 2; off >= 1; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        const long long r = r0 + i * (256 / C::LPR);
        if (part == 0 && r < rows) out[r] = acc;
    }
}

// dS = P (dP - delta) / sqrt(d) of 32 columns of a thread's row as bf16 pairs: packed fp32, two columns per instruction.  The factor
// 1 / sqrt(d) comes before the rounding to bf16 (at head dim 128 it is no power of two: after it, half of the values of dQ are
// other bf16 numbers); it rides in the fused multiply-add that takes delta off.  MASK: columns from nv on count nothing.
template <bool MASK>
__device__ __forceinline__ void bwd_ds(const uint32_t* s, const uint32_t* dp, int nv, float scale_log2, float scale, float neg_lse2, float delta, uint32_t (&pk)[16]) {
    const float2 c2 = make_float2(scale_log2, scale_log2), l2 = make_float2(neg_lse2, neg_lse2);
    const float2 f2 = make_float2(scale, scale), nd = make_float2(-delta * scale, -delta * scale);
#pragma unroll
    for (int e0 = 0; e0 < 32; e0 += 8) {
        float2 x[4], g[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int e = e0 + 2 * v;
            x[v] = ffma2(make_float2(__uint_as_float(s[e]), __uint_as_float(s[e + 1])), c2, l2);
            g[v] = ffma2(make_float2(__uint_as_float(dp[e]), __uint_as_float(dp[e + 1])), f2, nd);
        }
#pragma unroll
        for (int v = 0; v < 4; ++v) x[v] = make_float2(fast_exp2(x[v].x), fast_exp2(x[v].y));
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int e = e0 + 2 * v;
            x[v] = fmul2(x[v], g[v]);
            pk[e >> 1] = pack_bf16(MASK && e >= nv ? 0.f : x[v].x, MASK && e + 1 >= nv ? 0.f : x[v].y);
        }
    }
}

template <int D>
struct SwaBwd {
    static constexpr int BLK = 128;
    static constexpr int SUB = D / 64, SUB_BYTES = BLK * 128, TILE_BYTES = SUB * SUB_BYTES;
    static constexpr int KST = 3, VST = 2;
    static constexpr int OFF_Q = 0, OFF_DO = TILE_BYTES, OFF_K = 2 * TILE_BYTES, OFF_V = OFF_K + KST * TILE_BYTES;   // (Q: also the output's staging tile)
    static constexpr int OFF_BAR = OFF_V + VST * TILE_BYTES;
    static constexpr int OFF_DELTA = OFF_BAR + 384;      // [2 units][128 rows]
    static constexpr int USED_BYTES = OFF_DELTA + 2 * BLK * 4;
    // one CTA per SM (it takes all of TMEM); slack for the alignment of the tiles to 1 KB
    static constexpr int SMEM_BYTES = USED_BYTES + 1024 > 120 * 1024 ? USED_BYTES + 1024 : 120 * 1024;
    static constexpr int THREADS = 384;                  // warps 0-7: softmax (four per half of the key columns), 8: K loads, 9: V, Q, dO loads, 10: scores, 11: dS K
    static constexpr int WARP_LOAD_K = 8, WARP_LOAD_V = 9, WARP_S = 10, WARP_DQ = 11;
    static constexpr int COL_DQ = 256, COL_Q = 384, COL_DS = 448, TMEM_COLS = 512;
};

struct SwaBwdParams {
    const int32_t* idx;      // [B*H, T_m, keep]
    int keep, Tc, n_b, n_cached, ring_head, P, n_sink, Tm, n_units, Tn;
    uint32_t nb_magic;       // ceil(2^32 / n_b) (n_b > 1)
    float scale_log2, scale; // log2(e) / sqrt(d), 1 / sqrt(d)
    const float* lse;        // [B*H, T_c] natural log of the row's sum of exponentials (forward)
    const bf16 *d_o, *o;     // [B*H, T_c, D] g, o_local
    int* dev_status;
};

template <int D>
__global__ void __launch_bounds__(SwaBwd<D>::THREADS, 1)
k_swa_bwd_dq(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_do,
             const __grid_constant__ CUtensorMap tm_kring, const __grid_constant__ CUtensorMap tm_vring,
             const __grid_constant__ CUtensorMap tm_kcur, const __grid_constant__ CUtensorMap tm_vcur,
             const __grid_constant__ CUtensorMap tm_dq, const __grid_constant__ SwaBwdParams p) {
    using namespace tc5;
    typedef SwaBwd<D> C;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t s_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* s_gen = smem_raw + (s_base - smem_u32(smem_raw));
    const uint32_t sQ = s_base + C::OFF_Q, sDO = s_base + C::OFF_DO, sK = s_base + C::OFF_K, sV = s_base + C::OFF_V;
    const uint32_t bar0 = s_base + C::OFF_BAR;
    // Tile t of the thread block's stream.  K and V rings (kf, ke, vf, ve): index = stage, completion t / stages.  sd (both score
    // products of tile t complete) and se: completion t.  ds (dS written, four warps) and df: index = half of the key columns,
    // completion t.
    const uint32_t bar_kf = bar0, bar_ke = bar0 + 48, bar_vf = bar0 + 96, bar_ve = bar0 + 128, bar_sd = bar0 + 160, bar_ds = bar0 + 176,
                   bar_se = bar0 + 192,         // scores of tile t are in registers (eight warps)
                   bar_df = bar0 + 208,         // dS K of a half of tile t complete: its dS slot is free
                   bar_drain = bar0 + 224,      // two: each MMA warp's last operations complete
                   bar_qf = bar0 + 240,         // unit n: Q landed
                   bar_cp = bar0 + 248,         // unit n: ... and copied to tensor memory
                   bar_qe = bar0 + 256,         // unit n: its output, staged where Q of unit n + 1 had been, has left
                   bar_of = bar0 + 264, bar_oe = bar0 + 272,       // unit n: dO landed / read for the last time
                   bar_dqf = bar0 + 280, bar_dqe = bar0 + 288,
                   bar_x = bar0 + 304;          // four: unit n's delta, between the two warps that share 32 rows
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(s_gen + C::OFF_BAR + 296);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(s_gen + C::OFF_BAR + 300);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int keep = p.keep;
    const int my_units = (p.n_units - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;

    if (threadIdx.x == 0) {
        for (int s = 0; s < C::KST; ++s) { mbar_init(bar_kf + 8 * s, 1); mbar_init(bar_ke + 8 * s, 1); }
        for (int s = 0; s < C::VST; ++s) { mbar_init(bar_vf + 8 * s, 1); mbar_init(bar_ve + 8 * s, 1); }
        for (int s = 0; s < 2; ++s) { mbar_init(bar_ds + 8 * s, 4); mbar_init(bar_df + 8 * s, 1); mbar_init(bar_drain + 8 * s, 1); }
        for (int s = 0; s < 4; ++s) mbar_init(bar_x + 8 * s, 2);
        mbar_init(bar_sd, 1); mbar_init(bar_se, 8);
        mbar_init(bar_qf, 1); mbar_init(bar_cp, 1); mbar_init(bar_of, 1); mbar_init(bar_oe, 1); mbar_init(bar_qe, 8); mbar_init(bar_dqf, 1); mbar_init(bar_dqe, 8);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == C::WARP_S) {
        tmem_alloc(smem_u32(tmem_slot), C::TMEM_COLS);
        tmem_relinquish();
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    pdl_wait();

    auto wait_w = [&](uint32_t bar, uint32_t parity, int where) -> bool {
        return mbar_wait_warp<true>(bar, parity & 1u, abort_flag, p.dev_status, where);
    };

    if (warp == C::WARP_LOAD_K || warp == C::WARP_LOAD_V) {
        // ================================================================= TMA producers: K; V, Q and dO
        if (lane == 0) {
            const bool is_k = warp == C::WARP_LOAD_K;
            bool ok = true;
            RingPos<C::KST> rk;
            RingPos<C::VST> rv;
            int t = 0;
            const int Tn = p.Tn;
            auto load_q = [&](int m) {
                const int u = blockIdx.x + m * gridDim.x, bh = u / p.Tm, i = u - bh * p.Tm;
                mbar_expect_tx(bar_qf, C::TILE_BYTES);
#pragma unroll
                for (int s = 0; s < C::SUB; ++s) tma_load_4d(sQ + s * C::SUB_BYTES, &tm_q, s * 64, i * C::BLK, bh, 0, bar_qf);
            };
            if (!is_k && my_units > 0) load_q(0);
            for (int n = 0; ok && n < my_units; ++n) {
                const int u = blockIdx.x + n * gridDim.x;
                const int bh = u / p.Tm;
                const int32_t* my_idx = p.idx + (size_t)u * keep;
                if (!is_k) {
                    if (n >= 1 && !(ok = mbar_wait<true>(bar_oe, (n - 1) & 1, abort_flag, p.dev_status, 94))) break;
                    mbar_expect_tx(bar_of, C::TILE_BYTES);
#pragma unroll
                    for (int s = 0; s < C::SUB; ++s) tma_load_4d(sDO + s * C::SUB_BYTES, &tm_do, s * 64, (u - bh * p.Tm) * C::BLK, bh, 0, bar_of);
                }
                for (int j = 0; ok && j < keep; ++j, ++t) {
                    const int blk = checked_block(__ldg(my_idx + j), Tn, is_k ? p.dev_status : nullptr, u);
                    int c = 0, jb = blk;
                    while (jb >= p.n_b) { jb -= p.n_b; ++c; }
                    const bool cur = (c == p.n_sink + p.n_cached);
                    int slot = 0;
                    if (!cur) {
                        if (c < p.n_sink) slot = p.P + c;
                        else { slot = p.ring_head + c - p.n_sink; if (slot >= p.P) slot -= p.P; }
                    }
                    const CUtensorMap* m = is_k ? (cur ? &tm_kcur : &tm_kring) : (cur ? &tm_vcur : &tm_vring);
                    const int st = is_k ? rk.stage : rv.stage;
                    const uint32_t ph = is_k ? rk.phase : rv.phase;
                    const uint32_t full = (is_k ? bar_kf : bar_vf) + 8 * st, freed = (is_k ? bar_ke : bar_ve) + 8 * st;
                    if (t >= (is_k ? C::KST : C::VST) && !(ok = mbar_wait<true>(freed, ph ^ 1u, abort_flag, p.dev_status, is_k ? 82 : 83))) break;
                    mbar_expect_tx(full, C::TILE_BYTES);
#pragma unroll
                    for (int s = 0; s < C::SUB; ++s)
                        tma_load_4d((is_k ? sK : sV) + st * C::TILE_BYTES + s * C::SUB_BYTES, m, s * 64, jb * C::BLK, bh, slot, full);
                    if (is_k) rk.advance(); else rv.advance();
                    if (!is_k && ok && j == (keep > 2 ? 2 : keep - 1) && n + 1 < my_units) {
                        // Q of the next unit: its tile is free once this unit's has been copied out of it and the output of the
                        // unit before, staged there since, has left (said after this unit's first tile)
                        if (n == 0) ok = mbar_wait<true>(bar_cp, 0, abort_flag, p.dev_status, 81);
                        else ok = mbar_wait<true>(bar_qe, (n - 1) & 1, abort_flag, p.dev_status, 80);
                        if (!ok) break;
                        load_q(n + 1);
                    }
                }
            }
            if (!ok) {
                const long long t0 = clock64();
                while (clock64() - t0 < 400000) {}
            }
        }
    } else if (warp == C::WARP_S) {
        // ================================================================= scores (warp-uniform, one elected lane issues)
        constexpr uint32_t IDESC_S = idesc_bf16(128, false);
        constexpr uint32_t STEP = C::TILE_BYTES >> 4;             // descriptor address field counts 16-byte units
        const uint64_t dq0 = smem_desc_sw128(sQ, 16, 1024), dd0 = smem_desc_sw128(sDO, 16, 1024);
        const uint64_t dk0 = smem_desc_sw128(sK, 16, 1024), dv0 = smem_desc_sw128(sV, 16, 1024);
        const uint32_t hi_k = (uint32_t)(dk0 >> 32);
        bool ok = true;
        int t = 0;
        RingPos<C::KST> rk;
        RingPos<C::VST> rv;
        for (int n = 0; ok && n < my_units; ++n) {
            for (int j = 0; ok && j < keep; ++j, ++t) {
                if (j == 0) {
                    // Q moves to tensor memory, where the previous unit's last scores have read theirs by then
                    if (!(ok = wait_w(bar_qf, n, 84))) break;
                    if (t >= 1 && !(ok = wait_w(bar_sd, t - 1, 92))) break;
                    fence_after_sync();
                    if (elect_one()) {
#pragma unroll
                        for (int ks = 0; ks < D / 16; ++ks)                         // 16 features = 32 bytes of a row = 8 columns
                            tmem_cp_128x256b(tmem + C::COL_Q + 8 * ks, dq0 + (uint64_t)((ks >> 2) * (C::SUB_BYTES >> 4) + (ks & 3) * 2));
                        mma_commit(bar_cp);
                    }
                    __syncwarp();
                    if (!(ok = wait_w(bar_of, n, 95))) break;
                }
                if (!(ok = wait_w(bar_kf + 8 * rk.stage, rk.phase, 85))) break;
                if (!(ok = wait_w(bar_vf + 8 * rv.stage, rv.phase, 86))) break;
                if (t >= 1 && !(ok = wait_w(bar_se, t - 1, 91))) break;        // the tile before is in registers
                fence_after_sync();
                if (elect_one()) {
                    // dP first: V's stage, of which there are fewer, is free earlier
                    mma_ss_tile<D>(tmem + 128, (uint32_t)dd0, (uint32_t)dv0 + rv.stage * STEP, hi_k, IDESC_S);
                    mma_commit(bar_ve + 8 * rv.stage);
                    if (j == keep - 1) mma_commit(bar_oe);
                    mma_ts_kmajor<D>(tmem, tmem + C::COL_Q, (uint32_t)dk0 + rk.stage * STEP, hi_k, IDESC_S);
                    mma_commit(bar_sd);
                }
                __syncwarp();
                rk.advance();
                rv.advance();
            }
        }
        if (elect_one()) mma_commit(bar_drain);
        __syncwarp();
        {
            const long long t0 = clock64();
            while (!mbar_try_wait(bar_drain, 0) && clock64() - t0 < WAIT_LIMIT_CYCLES) {}
        }
    } else if (warp == C::WARP_DQ) {
        // ================================================================= dQ += dS K
        constexpr uint32_t IDESC_DQ = idesc_bf16(D, true);
        constexpr uint32_t STEP = C::TILE_BYTES >> 4, HALF = 64 * 128 >> 4;  // 64 rows of a tile, in 16-byte units
        const uint64_t dkm = smem_desc_sw128(sK, C::SUB_BYTES, 1024);        // the K tile again, as the MN-major operand
        const uint32_t hi_m = (uint32_t)(dkm >> 32);
        bool ok = true;
        int t = 0;
        RingPos<C::KST> rk;
        for (int n = 0; ok && n < my_units; ++n) {
            for (int j = 0; ok && j < keep; ++j, ++t) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (!(ok = wait_w(bar_ds + 8 * h, t, 87))) break;
                    // the accumulator of the previous unit has been read out before this unit's first product overwrites it
                    if (h == 0 && j == 0 && n >= 1 && !(ok = wait_w(bar_dqe, n - 1, 88))) break;
                    fence_after_sync();
                    if (elect_one()) {
                        mma_ts_half(tmem + C::COL_DQ, tmem + C::COL_DS + 32 * h, (uint32_t)dkm + rk.stage * STEP + h * HALF, hi_m, IDESC_DQ, j > 0 || h > 0);
                        mma_commit(bar_df + 8 * h);
                        if (h == 1) {
                            mma_commit(bar_ke + 8 * rk.stage);
                            if (j == keep - 1) mma_commit(bar_dqf);
                        }
                    }
                    __syncwarp();
                }
                rk.advance();
            }
        }
        if (elect_one()) mma_commit(bar_drain + 8);
        __syncwarp();
        {
            const long long t0 = clock64();
            while (!mbar_try_wait(bar_drain + 8, 0) && clock64() - t0 < WAIT_LIMIT_CYCLES) {}
        }
    } else {
        // ================================================================= softmax warps: dS from S and dP; dQ out at the unit's end
        const int grp = warp >> 2;                          // the half of every tile's key columns this warp turns; then a half of dQ's columns
        const int row = (warp & 3) * 32 + lane;
        const uint32_t lane_base = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        const bool lane0 = lane == 0, ragged = p.Tc % C::BLK != 0;
        bool ok = true;
        int t = 0;
        for (int n = 0; ok && n < my_units; ++n) {
            const int u = blockIdx.x + n * gridDim.x;
            const int bh = u / p.Tm, i = u - bh * p.Tm;
            const int32_t* my_idx = p.idx + (size_t)u * keep;
            const int q0 = i * C::BLK, nq = min(C::BLK, p.Tc - q0);
            const size_t g_row = (size_t)bh * p.Tc + q0 + row;
            const float neg_lse2 = row < nq ? -p.lse[g_row] * 1.4426950408889634f : 0.f;
            // delta = g . o_local of the unit's rows: a warp takes 16 rows, all its loads in flight, and the two warps of a row
            // exchange.  About 1 000 clk per unit, against a launch before this kernel: the step with gradient at 12 heads of 128,
            // 4 680 queries 363 -> 358 us, at 2 x 8 heads of 64, 1 300 queries 96.1 -> 94.6 us.
            float* delta_s = reinterpret_cast<float*>(s_gen + C::OFF_DELTA) + (n & 1) * C::BLK;
            {
                constexpr int LPR = D / 8, RPS = 32 / LPR, STEPS = 16 / RPS;        // lanes per row, rows per step
                const int r0 = (warp & 3) * 32 + grp * 16 + lane / LPR;
                uint4 x[STEPS], y[STEPS];
#pragma unroll
                for (int v = 0; v < STEPS; ++v) {
                    x[v] = y[v] = make_uint4(0, 0, 0, 0);
                    if (r0 + v * RPS < nq) {
                        const size_t at = ((size_t)bh * p.Tc + q0 + r0 + v * RPS) * D + (lane % LPR) * 8;
                        x[v] = __ldg(reinterpret_cast<const uint4*>(p.d_o + at));
                        y[v] = __ldg(reinterpret_cast<const uint4*>(p.o + at));
                    }
                }
#pragma unroll
                for (int v = 0; v < STEPS; ++v) {
                    float acc = dot8(x[v], y[v]);
#pragma unroll
                    for (int off = LPR / 2; off >= 1; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
                    if (lane % LPR == 0) delta_s[r0 + v * RPS] = acc;
                }
            }
            ok = mbar_meet_warp(bar_x + 8 * (warp & 3), n, lane0, abort_flag, p.dev_status, 97);
            if (!ok) break;
            const float delta = delta_s[row];           // (rows past the chunk's end: 0)
            uint32_t tails = 0;         // one bit per tile of the current 32: the block is a chunk's short last one
            for (int j = 0; j < keep; ++j, ++t) {
                if (ragged && (j & 31) == 0) {
                    const uint32_t e = j + lane < keep ? (uint32_t)__ldg(my_idx + j + lane) : 0u;
                    const uint32_t x1 = (e < (uint32_t)p.Tn ? e : 0u) + 1u;     // (an entry outside [0, T_n) is block 0, as for the loader)
                    tails = __ballot_sync(0xffffffffu, p.n_b == 1 || __umulhi(x1, p.nb_magic) * p.n_b == x1);
                }
                const bool tail = (tails >> (j & 31)) & 1u;
                ok = mbar_wait_warp(bar_sd, t & 1, abort_flag, p.dev_status, 89);
                if (!ok) break;
                fence_after_sync();
                const uint32_t tS = lane_base + 64 * grp;
                uint32_t s[2][32], dp[2][32];
                tmem_ld32(tS, s[0]);
                tmem_ld32(tS + 32, s[1]);
                tmem_ld32(tS + 128, dp[0]);
                tmem_ld32(tS + 160, dp[1]);
                tmem_wait_ld();
                fence_before_sync();
                mbar_arrive_if(bar_se, lane0);                  // the next tile's scores may be formed
                auto store_ds = [&](int c, const uint32_t (&pk)[16]) {
                    if (c == 0 && t >= 1) {                     // the half's dS slot: dS K of the tile before has read it
                        ok = mbar_wait_warp(bar_df + 8 * grp, (t - 1) & 1, abort_flag, p.dev_status, 96);
                        fence_after_sync();
                    }
                    tmem_st16(lane_base + C::COL_DS + 32 * grp + 16 * c, pk);
                };
                if (!tail) {
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        uint32_t pk[16];
                        bwd_ds<false>(s[c], dp[c], 32, p.scale_log2, p.scale, neg_lse2, delta, pk);
                        store_ds(c, pk);
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        uint32_t pk[16];
                        bwd_ds<true>(s[c], dp[c], p.Tc - (p.n_b - 1) * C::BLK - grp * 64 - c * 32, p.scale_log2, p.scale, neg_lse2, delta, pk);
                        store_ds(c, pk);
                    }
                }
                if (!ok) break;
                tmem_wait_st();
                fence_before_sync();
                mbar_arrive_if(bar_ds + 8 * grp, lane0);
                if (j == 0 && n >= 1) {         // the previous unit's output has long left its staging tile by now
                    if (lane0) bulk_wait_read();
                    __syncwarp();
                    mbar_arrive_if(bar_qe, lane0);
                }
            }
            if (!ok) break;
            ok = mbar_wait_warp(bar_dqf, n & 1, abort_flag, p.dev_status, 90);
            if (ok && n + 1 < my_units) ok = mbar_wait_warp(bar_cp, (n + 1) & 1, abort_flag, p.dev_status, 93);    // Q of the next unit has left the staging tile
            if (!ok) break;
            fence_after_sync();
            uint32_t out[D / 4];
#pragma unroll
            for (int c = 0; c < D / 64; ++c) {
                uint32_t o[32];
                tmem_ld32(lane_base + C::COL_DQ + grp * (D / 2) + c * 32, o);
                tmem_wait_ld();
#pragma unroll
                for (int e = 0; e < 32; e += 2) out[c * 16 + e / 2] = pack_bf16(__uint_as_float(o[e]), __uint_as_float(o[e + 1]));
            }
            fence_before_sync();
            mbar_arrive_if(bar_dqe, lane0);
            // out through shared memory and one bulk tensor store per warp (32 rows x half of the columns; the map clips)
            constexpr int RB = D;                           // bytes per staged row (D / 2 columns)
            const uint32_t off = C::OFF_Q + warp * 32 * RB;
            uint8_t* stage = s_gen + off + lane * RB;
            const int swz = D == 128 ? lane & 7 : (lane >> 1) & 3;
#pragma unroll
            for (int c = 0; c < D / 16; ++c)
                *reinterpret_cast<uint4*>(stage + ((c ^ swz) << 4)) = make_uint4(out[4 * c], out[4 * c + 1], out[4 * c + 2], out[4 * c + 3]);
            fence_proxy_async();
            __syncwarp();
            if (lane0 && q0 + (warp & 3) * 32 < p.Tc) {
                tma_store_4d(&tm_dq, s_base + off, grp * (D / 2), q0 + (warp & 3) * 32, bh, 0);
                bulk_commit();
            }
        }
        if (lane0) bulk_wait_all();
    }
    fence_before_sync();
    __syncthreads();
    if (warp == C::WARP_S) {
        fence_after_sync();
        tmem_dealloc(tmem, C::TMEM_COLS);
    }
}

// ------------------------------------------------------------------------------------------------------------
// dK and dV of the current chunk (the keys and values that carry gradient in the rollout: the cache holds clean chunks of
// earlier, gradient-free passes).  The transposed walk: unit = (batch*head, key block j of the current chunk); for every query
// block i that keeps j (read off the selection's bit mask), rows = keys, columns = queries:
//   S^T  = K_j Q_i^T      A = K_j (smem), B = Q_i (smem)                      -> TMEM [0, 128)
//   dP^T = V_j dO_i^T     A = V_j (smem), B = dO_i (smem)                     -> TMEM [128, 256)
//   P^T  = exp2(S^T c - lse_i log2 e)  (bf16, over S^T),   dS^T = P^T (dP^T - delta_i) / sqrt(d)  (bf16, over dP^T)
//   dV_j += P^T dO_i      A = P^T (TMEM), B = dO_i (MN-major)                  -> TMEM [256, 256 + D)
//   dK_j += dS^T Q_i      A = dS^T (TMEM), B = Q_i (MN-major)                  -> TMEM [384, 384 + D)
// Accumulators and one pair of score tiles fill tensor memory at head dim 128.  What keeps the tensor core busy all the same is
// the order in which the one MMA warp issues: dV(t), S(t + 1), dK(t), dP(t + 1) -- the softmax warps form dS(t) during the first
// two products and P(t + 1) during the last two.  A pair is 2 048 clk of tensor time and, with the tiles' arrival, somewhat
// more of shared-memory traffic.  lse and delta are per QUERY, i.e. per column here: a warp of its own finds the pairs and stages
// them a pair ahead; the others only need the number of a unit's pairs, which comes with the order.  A query row past the
// chunk's end gets lse = +inf, so its P and dS are zero, and key rows past the end only reach output rows that are not stored:
// no masks.
// 12 heads of 128, 4 680 queries, 28 kept blocks (28 pairs per thread block): whole tiles that alternate strictly between
// tensor core and (scalar) softmax 134 us; half-width score tiles, which overlap but take the tensor core twice as long (a
// 128 x 64 product costs as much as a 128 x 128 one), 94 us, 85 with the units in order of their pairs (BwdOrder); the order
// above 71 us.  (The two score regions as chains with an MMA warp each: 79 us, their products interleave and each region
// is late.  Walking the mask in every warp: 1 000 clk per pair of 4 000.)
// ------------------------------------------------------------------------------------------------------------
template <int D>
struct SwaBwdKV {
    static constexpr int BLK = 128;
    static constexpr int SUB = D / 64, SUB_BYTES = BLK * 128, TILE_BYTES = SUB * SUB_BYTES;
    static constexpr int STAGES = 2;
    static constexpr int OFF_K = 0, OFF_V = TILE_BYTES, OFF_Q = 2 * TILE_BYTES, OFF_DO = OFF_Q + STAGES * TILE_BYTES;
    static constexpr int OFF_OUT = OFF_DO + STAGES * TILE_BYTES;         // staging of the output tile, 32 rows x D / 2 columns per warp
    static constexpr int OFF_BAR = OFF_OUT + BLK * D * 2;
    static constexpr int OFF_ROW = OFF_BAR + 256;        // [2 pairs][2 halves of the queries][-lse log2 e, -delta / sqrt(d)][64] floats
    static constexpr int USED_BYTES = OFF_ROW + 2 * 2 * BLK * 4;
    // one CTA per SM (it takes all of TMEM); slack for the alignment of the tiles to 1 KB, as far as there is room (checked)
    static constexpr int WANT_BYTES = USED_BYTES + 1024 > 120 * 1024 ? USED_BYTES + 1024 : 120 * 1024, MAX_SMEM = 232448;
    static constexpr int SMEM_BYTES = WANT_BYTES < MAX_SMEM ? WANT_BYTES : MAX_SMEM;
    static_assert(USED_BYTES <= MAX_SMEM, "shared memory layout does not fit");
    static constexpr int THREADS = 352;                  // warps 0-7: softmax (two halves of the queries), 8: TMA, 9: MMA,
    static constexpr int WARP_TMA = 8, WARP_MMA = 9, WARP_ROW = 10;                 // 10: lse and delta of the queries
    static constexpr int COL_DV = 256, COL_DK = 384, TMEM_COLS = 512;
};

struct SwaBwdKVParams {
    const uint32_t* mask;    // [B*H, T_m, mask_words]: the forward's selection
    int mask_words, first_block;     // logical index of the current chunk's first key block
    int Tc, n_b, Tm, n_units;        // units = B*H x n_b
    const int2* order;       // [n_units]: the units, most pairs first, with the number of their pairs (-1: not counted)
    float scale_log2, scale;
    const float* lse;        // [B*H, T_c]
    const float* delta;      // [B*H, T_c]
    int* dev_status;
};

// The query blocks that keep a unit's key block, in ascending order: 32 mask rows at a time, one ballot each.  All calls by a
// whole warp.
struct PairWalk {
    int bh = 0, jb = 0, w = 0;
    uint32_t bits = 0;
    __device__ __forceinline__ uint32_t word(const SwaBwdKVParams& p, int w_) const {
        const int i = w_ * 32 + (threadIdx.x & 31), jlog = p.first_block + jb;
        const bool kept = i < p.Tm && ((__ldg(p.mask + ((size_t)bh * p.Tm + i) * p.mask_words + (jlog >> 5)) >> (jlog & 31)) & 1u);
        return __ballot_sync(0xffffffffu, kept);
    }
    __device__ __forceinline__ void open(const SwaBwdKVParams& p, int u) {
        bh = u / p.n_b; jb = u - bh * p.n_b; w = 0;
        bits = word(p, 0);
    }
    // the pairs of unit u: all of its mask words
    __device__ __forceinline__ int count(const SwaBwdKVParams& p, int u) {
        open(p, u);
        int n = __popc(bits);
        for (int x = 1; x * 32 < p.Tm; ++x) n += __popc(word(p, x));
        return n;
    }
    __device__ __forceinline__ int pop(const SwaBwdKVParams& p) {      // the next query block, or -1
        while (bits == 0) {
            if (++w * 32 >= p.Tm) return -1;
            bits = word(p, w);
        }
        const int i = w * 32 + __ffs(bits) - 1;
        bits &= bits - 1;
        return i;
    }
};

template <int D>
__global__ void __launch_bounds__(SwaBwdKV<D>::THREADS, 1)
k_swa_bwd_dkv(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_do,
              const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
              const __grid_constant__ CUtensorMap tm_dk, const __grid_constant__ CUtensorMap tm_dv,
              const __grid_constant__ SwaBwdKVParams p) {
    using namespace tc5;
    typedef SwaBwdKV<D> C;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t s_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    if (s_base - smem_u32(smem_raw) + C::USED_BYTES > C::SMEM_BYTES) {   // the window started too far off a 1 KB boundary
        if (threadIdx.x == 0) { atomicOr(p.dev_status, HF_DEV_TIMEOUT_FLAG); atomicExch(p.dev_status + 1, 97); }
        return;
    }
    uint8_t* s_gen = smem_raw + (s_base - smem_u32(smem_raw));
    const uint32_t sK = s_base + C::OFF_K, sV = s_base + C::OFF_V, sQ = s_base + C::OFF_Q, sDO = s_base + C::OFF_DO;
    const uint32_t bar0 = s_base + C::OFF_BAR;
    // pair t of the thread block: Q and dO rings, stage t & 1; pd: completion t; pr, ds: index = half of the queries, completion t
    const uint32_t bar_kvf = bar0, bar_kve = bar0 + 8,         // m-th unit with pairs: K and V landed / read for the last time
                   bar_qf = bar0 + 16, bar_qe = bar0 + 32, bar_of = bar0 + 48, bar_oe = bar0 + 64,
                   bar_sd = bar0 + 152, bar_pd = bar0 + 88,    // S of pair t complete and its lse and delta staged (index t & 1); dP complete
                   bar_pr = bar0 + 96, bar_ds = bar0 + 112,    // half of P, dS written (four warps)
                   bar_accf = bar0 + 128, bar_acce = bar0 + 136;       // unit n: dV and dK complete / read out
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(s_gen + C::OFF_BAR + 144);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(s_gen + C::OFF_BAR + 148);
    float* row_vals = reinterpret_cast<float*>(s_gen + C::OFF_ROW);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // Unit number n of this thread block: position n * grid + c of the order, with c running backwards in odd rounds.
    const int rounds = p.n_units / (int)gridDim.x, rest = p.n_units - rounds * (int)gridDim.x;
    auto place = [&](int n) -> int { return (n & 1) ? (int)gridDim.x - 1 - (int)blockIdx.x : (int)blockIdx.x; };
    const int my_units = rounds + (place(rounds) < rest ? 1 : 0);
    auto unit_of = [&](int n) -> int2 { return n < my_units ? __ldg(p.order + n * (int)gridDim.x + place(n)) : make_int2(0, 0); };
    auto pairs_of = [&](int2 u) -> int {
        PairWalk walk;
        return u.y >= 0 ? u.y : walk.count(p, u.x);
    };

    if (threadIdx.x == 0) {
        mbar_init(bar_kvf, 1); mbar_init(bar_kve, 1);
        for (int s = 0; s < 2; ++s) {
            mbar_init(bar_qf + 8 * s, 1); mbar_init(bar_qe + 8 * s, 1); mbar_init(bar_of + 8 * s, 1); mbar_init(bar_oe + 8 * s, 1);
            mbar_init(bar_pr + 8 * s, 4); mbar_init(bar_ds + 8 * s, 4);
        }
        mbar_init(bar_sd, 2); mbar_init(bar_sd + 8, 2); mbar_init(bar_pd, 1); mbar_init(bar_accf, 1); mbar_init(bar_acce, 8);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == C::WARP_MMA) {
        tmem_alloc(smem_u32(tmem_slot), C::TMEM_COLS);
        tmem_relinquish();
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    pdl_wait();

    auto wait_w = [&](uint32_t bar, uint32_t parity, int where) -> bool {
        return mbar_wait_warp<true>(bar, parity & 1u, abort_flag, p.dev_status, where);
    };

    if (warp == C::WARP_TMA) {
        // ================================================================= TMA producer: K_j, V_j per unit; Q_i, dO_i per kept pair
        bool ok = true;
        int t = 0, m = 0;                             // pairs; units that have any
        PairWalk walk;
        for (int n = 0; ok && n < my_units; ++n) {
            walk.open(p, unit_of(n).x);
            bool first = true;
            for (int i = walk.pop(p); ok && i >= 0; i = walk.pop(p), ++t) {
                if (first) {
                    if (m >= 1 && !(ok = wait_w(bar_kve, m - 1, 91))) break;
                    if (elect_one()) {
                        mbar_expect_tx(bar_kvf, 2 * C::TILE_BYTES);
#pragma unroll
                        for (int s = 0; s < C::SUB; ++s) {
                            tma_load_4d(sK + s * C::SUB_BYTES, &tm_k, s * 64, walk.jb * C::BLK, walk.bh, 0, bar_kvf);
                            tma_load_4d(sV + s * C::SUB_BYTES, &tm_v, s * 64, walk.jb * C::BLK, walk.bh, 0, bar_kvf);
                        }
                    }
                    __syncwarp();
                    first = false; ++m;
                }
                const int st = t & 1;
                // dO first: its stage is free half a pair before Q's
                if (t >= 2 && !(ok = wait_w(bar_oe + 8 * st, (t >> 1) - 1, 90))) break;
                if (elect_one()) {
                    mbar_expect_tx(bar_of + 8 * st, C::TILE_BYTES);
#pragma unroll
                    for (int s = 0; s < C::SUB; ++s)
                        tma_load_4d(sDO + st * C::TILE_BYTES + s * C::SUB_BYTES, &tm_do, s * 64, i * C::BLK, walk.bh, 0, bar_of + 8 * st);
                }
                __syncwarp();
                if (t >= 2 && !(ok = wait_w(bar_qe + 8 * st, (t >> 1) - 1, 92))) break;
                if (elect_one()) {
                    mbar_expect_tx(bar_qf + 8 * st, C::TILE_BYTES);
#pragma unroll
                    for (int s = 0; s < C::SUB; ++s)
                        tma_load_4d(sQ + st * C::TILE_BYTES + s * C::SUB_BYTES, &tm_q, s * 64, i * C::BLK, walk.bh, 0, bar_qf + 8 * st);
                }
                __syncwarp();
            }
        }
        if (!ok) {
            const long long t0 = clock64();
            while (clock64() - t0 < 400000) {}
        }
    } else if (warp == C::WARP_MMA) {
        // ================================================================= MMA issuer (warp-uniform, one elected lane issues)
        constexpr uint32_t IDESC_S = idesc_bf16(128, false);
        constexpr uint32_t IDESC_ACC = idesc_bf16(D, true);
        constexpr uint32_t TILE_STEP = C::TILE_BYTES >> 4, HALF = 64 * 128 >> 4;    // 64 rows of a tile, in 16-byte units
        const uint64_t kd = smem_desc_sw128(sK, 16, 1024), vd = smem_desc_sw128(sV, 16, 1024);
        const uint64_t qd = smem_desc_sw128(sQ, 16, 1024), od = smem_desc_sw128(sDO, 16, 1024);
        const uint64_t qm = smem_desc_sw128(sQ, C::SUB_BYTES, 1024), om = smem_desc_sw128(sDO, C::SUB_BYTES, 1024);     // as MN-major operands
        const uint32_t hi_k = (uint32_t)(kd >> 32), hi_m = (uint32_t)(qm >> 32);
        bool ok = true;
        // ---- the scores run one pair ahead, over unit boundaries too: a count of pairs of their own
        int n_s = -1, t_s = 0, m_s = -1, left_s = 0;  // left_s: pairs of the unit whose scores are still to be issued, the next one included
        bool first_s = false;
        int2 unit_s = unit_of(0);
        auto next_unit_s = [&]() {                    // the next unit that has pairs, if there is one
            while (left_s == 0 && ++n_s < my_units) {
                left_s = pairs_of(unit_s);
                unit_s = unit_of(n_s + 1);
                if (left_s > 0) { first_s = true; ++m_s; }
            }
        };
        auto issue_s = [&]() -> bool {                // S^T = K Q^T
            if (first_s && !wait_w(bar_kvf, m_s, 93)) return false;
            first_s = false;
            if (!wait_w(bar_qf + 8 * (t_s & 1), t_s >> 1, 94)) return false;
            fence_after_sync();
            if (elect_one()) {
                mma_ss_tile<D>(tmem, (uint32_t)kd, (uint32_t)qd + (t_s & 1) * TILE_STEP, hi_k, IDESC_S);
                mma_commit(bar_sd + 8 * (t_s & 1));
            }
            __syncwarp();
            return true;
        };
        auto issue_dp = [&]() -> bool {               // dP^T = V dO^T, and on to the next pair
            if (!wait_w(bar_of + 8 * (t_s & 1), t_s >> 1, 89)) return false;
            fence_after_sync();
            if (elect_one()) {
                mma_ss_tile<D>(tmem + 128, (uint32_t)vd, (uint32_t)od + (t_s & 1) * TILE_STEP, hi_k, IDESC_S);
                mma_commit(bar_pd);
                if (left_s == 1) mma_commit(bar_kve);                 // K_j and V_j have been read for the last time
            }
            __syncwarp();
            ++t_s;
            if (--left_s == 0) next_unit_s();
            return true;
        };
        next_unit_s();
        if (left_s > 0) ok = issue_s() && issue_dp();
        int t = 0;
        int2 unit = unit_of(0);
        for (int n = 0; ok && n < my_units; ++n) {
            const int pairs = pairs_of(unit);
            unit = unit_of(n + 1);
            if (pairs == 0) {
                // no pairs: the read-out of the unit before comes first, or this unit's completion could pass it by
                if (n >= 1 && !(ok = wait_w(bar_acce, n - 1, 97))) break;
                if (elect_one()) mma_commit(bar_accf);
                __syncwarp();
                continue;
            }
            for (int x = 0; ok && x < pairs; ++x, ++t) {
                const int st = t & 1;
                // the accumulators of the previous unit have been read out before this unit's first product overwrites them
                if (x == 0 && n >= 1 && !(ok = wait_w(bar_acce, n - 1, 96))) break;
                bool more = false;
#pragma unroll
                for (int c = 0; c < 2; ++c) {         // dV += P^T dO, scores of the next pair; dK += dS^T Q, dP of the next pair
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (!(ok = wait_w((c == 0 ? bar_pr : bar_ds) + 8 * h, t, 95))) break;
                        fence_after_sync();
                        if (elect_one()) {
                            mma_ts_half(tmem + (c == 0 ? C::COL_DV : C::COL_DK), tmem + 128 * c + 64 * h,
                                        (uint32_t)(c == 0 ? om : qm) + st * TILE_STEP + h * HALF, hi_m, IDESC_ACC, x > 0 || h > 0);
                            if (h == 1) {
                                mma_commit((c == 0 ? bar_oe : bar_qe) + 8 * st);      // (the pair's scores completed before P, dS were formed)
                                if (c == 1 && x == pairs - 1) mma_commit(bar_accf);   // everything of this unit has completed
                            }
                        }
                        __syncwarp();
                    }
                    if (!ok) break;
                    if (c == 0) more = left_s > 0;
                    if (more && !(ok = c == 0 ? issue_s() : issue_dp())) break;
                }
            }
        }
        if (!ok) {                                    // given up: nothing of this warp's is in flight when tensor memory is freed
            const long long t0 = clock64();
            while (clock64() - t0 < 400000) {}
        }
    } else if (warp == C::WARP_ROW) {
        // ================================================================= -lse log2 e and -delta / sqrt(d) of every pair's queries, a pair ahead
        bool ok = true;
        int t = 0;
        PairWalk walk;
        for (int n = 0; ok && n < my_units; ++n) {
            walk.open(p, unit_of(n).x);
            for (int i = walk.pop(p); i >= 0; i = walk.pop(p), ++t) {
                float nl[4], nd[4];
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const int r = i * C::BLK + x * 32 + lane;
                    const bool in = r < p.Tc;                         // rows past the chunk's end: weight zero
                    nl[x] = in ? -p.lse[(size_t)walk.bh * p.Tc + r] * 1.4426950408889634f : -INFINITY;
                    nd[x] = in ? -p.delta[(size_t)walk.bh * p.Tc + r] * p.scale : 0.f;
                }
                // dK of pair t - 2 has left the tensor core, so its values have been read
                if (t >= 2 && !(ok = wait_w(bar_qe + 8 * (t & 1), (t >> 1) - 1, 87))) break;
                float* slot = row_vals + (t & 1) * 256;
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    float* at = slot + (x >> 1) * 128 + (x & 1) * 32 + lane;
                    at[0] = nl[x];
                    at[64] = nd[x];
                }
                __syncwarp();
                mbar_arrive_if(bar_sd + 8 * (t & 1), lane == 0);
            }
        }
    } else {
        // ================================================================= softmax warps (rows = keys, columns = queries)
        const int grp = warp >> 2;                          // the half of every pair's queries this warp turns; then a half of the output columns
        const uint32_t lane_base = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        const bool lane0 = lane == 0;
        const float2 c2 = make_float2(p.scale_log2, p.scale_log2), f2 = make_float2(p.scale, p.scale);
        bool ok = true;
        int t = 0;
        int2 unit = unit_of(0);
        for (int n = 0; ok && n < my_units; ++n) {
            const int pairs = pairs_of(unit), bh = unit.x / p.n_b, k0 = (unit.x - bh * p.n_b) * C::BLK;
            const bool any = pairs > 0;
            unit = unit_of(n + 1);
            for (int x = 0; x < pairs; ++x) {
                const float* rv = row_vals + ((t & 1) * 2 + grp) * 128;
                // ---- P = exp2(S c - lse log2 e), kept in registers for dS
                ok = mbar_wait_warp(bar_sd + 8 * (t & 1), (t >> 1) & 1, abort_flag, p.dev_status, 98);
                if (!ok) break;
                fence_after_sync();
                const uint32_t tS = lane_base + 64 * grp, tP = tS + 128;
                float2 pe[32];
                {
                    uint32_t s[2][32];
                    tmem_ld32(tS, s[0]);
                    tmem_ld32(tS + 32, s[1]);
                    tmem_wait_ld();
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const float4* nl = reinterpret_cast<const float4*>(rv + c * 32);
                        uint32_t pk[16];
#pragma unroll
                        for (int e = 0; e < 32; e += 4) {
                            const float4 l4 = nl[e >> 2];
                            float2& x0 = pe[16 * c + e / 2];
                            float2& x1 = pe[16 * c + e / 2 + 1];
                            x0 = ffma2(make_float2(__uint_as_float(s[c][e]), __uint_as_float(s[c][e + 1])), c2, make_float2(l4.x, l4.y));
                            x1 = ffma2(make_float2(__uint_as_float(s[c][e + 2]), __uint_as_float(s[c][e + 3])), c2, make_float2(l4.z, l4.w));
                            x0 = make_float2(fast_exp2(x0.x), fast_exp2(x0.y));
                            x1 = make_float2(fast_exp2(x1.x), fast_exp2(x1.y));
                            pk[e / 2] = pack_bf16(x0.x, x0.y);
                            pk[e / 2 + 1] = pack_bf16(x1.x, x1.y);
                        }
                        tmem_st16(tS + 16 * c, pk);
                    }
                }
                tmem_wait_st();
                fence_before_sync();
                mbar_arrive_if(bar_pr + 8 * grp, lane0);
                // ---- dS = P (dP - delta) / sqrt(d)
                ok = mbar_wait_warp(bar_pd, t & 1, abort_flag, p.dev_status, 88);
                if (!ok) break;
                fence_after_sync();
                {
                    uint32_t dp[2][32];
                    tmem_ld32(tP, dp[0]);
                    tmem_ld32(tP + 32, dp[1]);
                    tmem_wait_ld();
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const float4* nd = reinterpret_cast<const float4*>(rv + 64 + c * 32);
                        uint32_t dk_[16];
#pragma unroll
                        for (int e = 0; e < 32; e += 4) {
                            const float4 d4 = nd[e >> 2];
                            const float2 g0 = ffma2(make_float2(__uint_as_float(dp[c][e]), __uint_as_float(dp[c][e + 1])), f2, make_float2(d4.x, d4.y));
                            const float2 g1 = ffma2(make_float2(__uint_as_float(dp[c][e + 2]), __uint_as_float(dp[c][e + 3])), f2, make_float2(d4.z, d4.w));
                            const float2 x0 = fmul2(pe[16 * c + e / 2], g0), x1 = fmul2(pe[16 * c + e / 2 + 1], g1);
                            dk_[e / 2] = pack_bf16(x0.x, x0.y);
                            dk_[e / 2 + 1] = pack_bf16(x1.x, x1.y);
                        }
                        tmem_st16(tP + 16 * c, dk_);
                    }
                }
                tmem_wait_st();
                fence_before_sync();
                mbar_arrive_if(bar_ds + 8 * grp, lane0);
                ++t;
            }
            if (!ok) break;
            ok = mbar_wait_warp(bar_accf, n & 1, abort_flag, p.dev_status, 99);
            if (!ok) break;
            fence_after_sync();
            // dV and dK of the unit as bf16 (zeros if no query block keeps the key block), out through shared memory and one bulk
            // tensor store per warp and tensor (32 rows x half of the columns; rows past the chunk's end are clipped by the map)
            uint32_t out[2][D / 4];
#pragma unroll
            for (int which = 0; which < 2; ++which)
#pragma unroll
                for (int c = 0; c < D / 64; ++c) {
                    uint32_t o[32];
                    tmem_ld32(lane_base + (which == 0 ? C::COL_DV : C::COL_DK) + grp * (D / 2) + c * 32, o);
                    tmem_wait_ld();
#pragma unroll
                    for (int e = 0; e < 32; e += 2)
                        out[which][c * 16 + e / 2] = any ? pack_bf16(__uint_as_float(o[e]), __uint_as_float(o[e + 1])) : 0u;
                }
            fence_before_sync();
            mbar_arrive_if(bar_acce, lane0);                // the accumulators may take the next unit
            constexpr int RB = D;                           // bytes per staged row (D / 2 columns)
            const uint32_t off = C::OFF_OUT + warp * 32 * RB;
            uint8_t* stage = s_gen + off + lane * RB;
            const int swz = D == 128 ? lane & 7 : (lane >> 1) & 3;
#pragma unroll
            for (int which = 0; which < 2; ++which) {
                if (lane0) bulk_wait_read();                // this warp's previous store has read its part
                __syncwarp();
#pragma unroll
                for (int c = 0; c < D / 16; ++c)
                    *reinterpret_cast<uint4*>(stage + ((c ^ swz) << 4)) = make_uint4(out[which][4 * c], out[which][4 * c + 1], out[which][4 * c + 2], out[which][4 * c + 3]);
                fence_proxy_async();
                __syncwarp();
                if (lane0 && k0 + (warp & 3) * 32 < p.Tc) {
                    tma_store_4d(which == 0 ? &tm_dv : &tm_dk, s_base + off, grp * (D / 2), k0 + (warp & 3) * 32, bh, 0);
                    bulk_commit();
                }
            }
        }
        if (lane0) bulk_wait_all();
    }
    fence_before_sync();
    __syncthreads();
    if (warp == C::WARP_MMA) {
        fence_after_sync();
        tmem_dealloc(tmem, C::TMEM_COLS);
    }
}
