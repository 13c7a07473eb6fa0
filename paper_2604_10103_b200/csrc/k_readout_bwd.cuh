// Backward of the history read-out (Eq. 4 with the Linear folded into the state) with respect to the queries.
//
// Forward, per query row r of a (batch, head):  f = phi(q_r),  den = f . z + eps,  y_r = (f S') / den + bias,
// S' = S W^T the folded state.  With g_r = dL/dy_r:
//     u   = S' g_r                      (u[a] = sum_c S'[a, c] g_r[c])           -- the one contraction: U = G S'^T
//     df  = (u - (f . u / den) z) / den
//     dq_r = df * phi'(q_r),            phi'(x) = 1 for x > 0, e^x otherwise
// The state itself comes from evicted chunks of earlier, gradient-free passes of the rollout (Alg. 1 back-propagates
// through the sampled step only), so nothing flows into S, z or the cached K / V here.
//
// Persistent kernel; a thread block takes a contiguous range of (batch*head, 128-row tile) units:
//   warp 8   TMA: the tile of G (bf16, K-major, 128-byte swizzle; two buffers), the tile of Q and the head's z (two buffers) and, the (batch,
//            head) changes, the hi and lo halves of S' ([a][c] bf16 -- as the B operand that is N = a by K = c, K-major)
//   warp 9   tcgen05.mma: U = G S'_hi^T + G S'_lo^T into one of two TMEM accumulators (D columns each)
//   warps 0-7  thread = half a row (two warps per TMEM lane quadrant): f and its part of f . z while the product runs, then
//            U once, its part of f . u; the two halves meet in shared memory; dq takes q's place in the tile and leaves by
//            bulk tensor store (rows past the chunk's end are clipped by the map)
// Memory-bound by its bytes (q, g, dq: 43 MB at 12 heads x 4 680 x 128 = 6.5 us) but short: three units per thread block, so
// start-up and the chain of one unit weigh most.  Four epilogue warps that read U twice and q and z through L1 23.4 us; 10.9 like this.
// Every wait is bounded; on expiry the thread block raises the device status word and leaves through the common exit.
#pragma once
#include "k_swa_tc5.cuh"

template <int D>
struct ReadoutBwd {
    static constexpr int ROWS = 128;
    static constexpr int SUB = D / 64;
    static constexpr int G_BYTES = ROWS * D * 2, S_BYTES = D * D * 2;
    static constexpr int GST = 2, QST = 2;
    static constexpr int OFF_G = 0, OFF_Q = GST * G_BYTES, OFF_S = OFF_Q + QST * G_BYTES, OFF_Z = OFF_S + 2 * S_BYTES;
    static constexpr int OFF_DOT = OFF_Z + QST * D * 4;            // [2 units][2 halves][128 rows] (f . u, f . z)
    static constexpr int OFF_BAR = OFF_DOT + 2 * 2 * ROWS * 8;
    static constexpr int USED_BYTES = OFF_BAR + 160;
    static constexpr int SMEM_BYTES = USED_BYTES + 1024;
    static constexpr int THREADS = 320, WARP_TMA = 8, WARP_MMA = 9;
    static constexpr int STORERS = SUB == 2 ? 8 : 4;               // warps that store: 64 columns each
    static constexpr int TMEM_COLS = 2 * D;
};

struct ReadoutBwdParams {
    const float* z;           // [B*H, D]
    int Tc, Tm, n_units;
    float eps;
    int* dev_status;
};

// tm_g, tm_q: [D, T_c, B*H, 1] box {64, 128}; tm_sh, tm_sl: [D, D, B*H, 1] box {64, D}; tm_dq: as tm_q, box {64, 32}; all
// 128-byte swizzle.
template <int D>
__global__ void __launch_bounds__(ReadoutBwd<D>::THREADS, 1)
k_readout_bwd_dq(const __grid_constant__ CUtensorMap tm_g, const __grid_constant__ CUtensorMap tm_q,
                 const __grid_constant__ CUtensorMap tm_sh, const __grid_constant__ CUtensorMap tm_sl,
                 const __grid_constant__ CUtensorMap tm_dq, const __grid_constant__ ReadoutBwdParams p) {
    using namespace tc5;
    typedef ReadoutBwd<D> C;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t s_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* s_gen = smem_raw + (s_base - smem_u32(smem_raw));
    const uint32_t bar0 = s_base + C::OFF_BAR;
    const uint32_t bar_gfull = bar0, bar_gfree = bar0 + 16, bar_ufull = bar0 + 32, bar_ufree = bar0 + 48, bar_sfull = bar0 + 64,
                   bar_qfull = bar0 + 72, bar_qfree = bar0 + 96,
                   bar_x = bar0 + 128;                             // four: the two warps that share 32 rows meet
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(s_gen + C::OFF_BAR + 120);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(s_gen + C::OFF_BAR + 124);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int upc = (p.n_units + (int)gridDim.x - 1) / (int)gridDim.x;
    const int u0 = min((int)blockIdx.x * upc, p.n_units);
    const int my_units = min(upc, p.n_units - u0);

    if (threadIdx.x == 0) {
        for (int s = 0; s < 2; ++s) {
            mbar_init(bar_gfull + 8 * s, 1); mbar_init(bar_gfree + 8 * s, 1);
            mbar_init(bar_ufull + 8 * s, 1); mbar_init(bar_ufree + 8 * s, 8);
        }
        for (int s = 0; s < C::QST; ++s) { mbar_init(bar_qfull + 8 * s, 1); mbar_init(bar_qfree + 8 * s, C::STORERS); }
        for (int s = 0; s < 4; ++s) mbar_init(bar_x + 8 * s, 2);
        mbar_init(bar_sfull, 1);
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
    pdl_trigger();

    if (warp == C::WARP_TMA) {
        if (lane == 0) {
            bool ok = true;
            int bh_prev = -1;
            RingPos<C::QST> rq;
            for (int n = 0; ok && n < my_units; ++n, rq.advance()) {
                const int u = u0 + n;
                const int bh = u / p.Tm, i = u - bh * p.Tm;
                const int s = n & 1;
                if (n >= 2 && !(ok = mbar_wait<true>(bar_gfree + 8 * s, ((n >> 1) & 1) ^ 1, abort_flag, p.dev_status, 62))) break;
                mbar_expect_tx(bar_gfull + 8 * s, C::G_BYTES);
#pragma unroll
                for (int v = 0; v < C::SUB; ++v)
                    tma_load_4d(s_base + C::OFF_G + s * C::G_BYTES + v * C::ROWS * 128, &tm_g, v * 64, i * C::ROWS, bh, 0, bar_gfull + 8 * s);
                if (bh != bh_prev) {
                    // the products of the previous unit (the last one of the other head) have read S'
                    if (n >= 1 && !(ok = mbar_wait<true>(bar_gfree + 8 * ((n - 1) & 1), ((n - 1) >> 1) & 1, abort_flag, p.dev_status, 61))) break;
                    bh_prev = bh;
                    mbar_expect_tx(bar_sfull, 2 * C::S_BYTES);
#pragma unroll
                    for (int v = 0; v < C::SUB; ++v) {
                        tma_load_4d(s_base + C::OFF_S + v * D * 128, &tm_sh, v * 64, 0, bh, 0, bar_sfull);
                        tma_load_4d(s_base + C::OFF_S + C::S_BYTES + v * D * 128, &tm_sl, v * 64, 0, bh, 0, bar_sfull);
                    }
                }
                if (n >= C::QST && !(ok = mbar_wait<true>(bar_qfree + 8 * rq.stage, rq.phase ^ 1u, abort_flag, p.dev_status, 67))) break;
                const uint32_t full = bar_qfull + 8 * rq.stage;
                mbar_expect_tx(full, C::G_BYTES + D * 4);
#pragma unroll
                for (int v = 0; v < C::SUB; ++v)
                    tma_load_4d(s_base + C::OFF_Q + rq.stage * C::G_BYTES + v * C::ROWS * 128, &tm_q, v * 64, i * C::ROWS, bh, 0, full);
                bulk_load(s_base + C::OFF_Z + rq.stage * D * 4, p.z + (size_t)bh * D, D * 4, full);
            }
            if (!ok) {   // gave up: let the copies already in flight land before the thread block leaves
                const long long t0 = clock64();
                while (clock64() - t0 < 400000) {}
            }
        }
    } else if (warp == C::WARP_MMA) {
        constexpr uint32_t IDESC = idesc_bf16(D, false);
        bool ok = true;
        int bh_prev = -1, epoch = -1;
        auto wait_w = [&](uint32_t bar, uint32_t parity, int where) -> bool {
            return mbar_wait_warp<true>(bar, parity & 1u, abort_flag, p.dev_status, where);
        };
        for (int n = 0; ok && n < my_units; ++n) {
            const int s = n & 1;
            const int bh = (u0 + n) / p.Tm;
            if (!(ok = wait_w(bar_gfull + 8 * s, n >> 1, 64))) break;
            if (bh != bh_prev) {
                bh_prev = bh; ++epoch;
                if (!(ok = wait_w(bar_sfull, epoch, 63))) break;
            }
            if (n >= 2 && !(ok = wait_w(bar_ufree + 8 * s, (n >> 1) - 1, 65))) break;
            fence_after_sync();
            if (elect_one()) {
                const uint32_t tU = tmem + s * D;
                const uint64_t dg = smem_desc_sw128(s_base + C::OFF_G + s * C::G_BYTES, 16, 1024);
                const uint64_t dsh = smem_desc_sw128(s_base + C::OFF_S, 16, 1024);
                const uint64_t dsl = smem_desc_sw128(s_base + C::OFF_S + C::S_BYTES, 16, 1024);
#pragma unroll
                for (int ks = 0; ks < D / 16; ++ks) {
                    // 16 contraction columns = 32 bytes inside a 128-byte row; the next 64-column sub-tile is ROWS (or D) rows on
                    const uint64_t og = (uint64_t)(((ks >> 2) * C::ROWS * 128 + (ks & 3) * 32) >> 4);
                    const uint64_t os = (uint64_t)(((ks >> 2) * D * 128 + (ks & 3) * 32) >> 4);
                    mma_ss(tU, dg + og, dsh + os, IDESC, ks > 0);
                    mma_ss(tU, dg + og, dsl + os, IDESC, true);
                }
                mma_commit(bar_ufull + 8 * s);
                mma_commit(bar_gfree + 8 * s);
            }
            __syncwarp();
        }
        if (!ok) {       // gave up: nothing of this warp's is in flight when tensor memory is freed
            const long long t0 = clock64();
            while (clock64() - t0 < 400000) {}
        }
    } else {
        const int half = warp >> 2, quad = warp & 3;
        const int row = quad * 32 + lane;
        const bool lane0 = lane == 0, storer = C::SUB == 2 || half == 0;
        constexpr int HC = D / 2;                                  // columns per thread
        bool ok = true;
        RingPos<C::QST> rq;
        int prev = 0;                                              // Q stage of the unit before
        uint32_t met = 0;                                          // meetings with the warp of the rows' other half
        auto meet = [&](int where) -> bool { return mbar_meet_warp(bar_x + 8 * quad, met++, lane0, abort_flag, p.dev_status, where); };
        for (int n = 0; ok && n < my_units; ++n, rq.advance()) {
            const int u = u0 + n;
            const int bh = u / p.Tm, i = u - bh * p.Tm;
            const uint32_t q_off = C::OFF_Q + rq.stage * C::G_BYTES + (C::SUB == 2 ? half * C::ROWS * 128 : 0);
            uint8_t* q_row = s_gen + q_off + row * 128;
            const int c0 = C::SUB == 2 ? 0 : half * 4;             // first 16-byte chunk of the row's half
            const float4* z4 = reinterpret_cast<const float4*>(s_gen + C::OFF_Z + rq.stage * D * 4) + half * (HC / 4);
            if (!(ok = mbar_wait_warp(bar_qfull + 8 * rq.stage, rq.phase, abort_flag, p.dev_status, 68))) break;
            float f[HC];
            float fz = 0.f;
#pragma unroll
            for (int c = 0; c < HC / 8; ++c) {
                const uint4 w = *reinterpret_cast<const uint4*>(q_row + (((c0 + c) ^ (row & 7)) << 4));
                const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
                const float4 z0 = z4[2 * c], z1 = z4[2 * c + 1];
                const float zz[8] = {z0.x, z0.y, z0.z, z0.w, z1.x, z1.y, z1.z, z1.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float2 x = unpack_bf16(ws[e]);
                    f[c * 8 + 2 * e] = phi_elu1(x.x);
                    f[c * 8 + 2 * e + 1] = phi_elu1(x.y);
                    fz = fmaf(f[c * 8 + 2 * e], zz[2 * e], fmaf(f[c * 8 + 2 * e + 1], zz[2 * e + 1], fz));
                }
            }
            if (n >= 1 && storer && lane0) {                       // the unit before has left its tile
                bulk_wait_read();
                mbar_arrive(bar_qfree + 8 * prev);
            }
            if (!(ok = mbar_wait_warp(bar_ufull + 8 * (n & 1), (n >> 1) & 1, abort_flag, p.dev_status, 66))) break;
            fence_after_sync();
            uint32_t uu[HC / 32][32];
#pragma unroll
            for (int c = 0; c < HC / 32; ++c) tmem_ld32(tmem + ((uint32_t)(quad * 32) << 16) + (n & 1) * D + half * HC + c * 32, uu[c]);
            tmem_wait_ld();
            fence_before_sync();
            mbar_arrive_if(bar_ufree + 8 * (n & 1), lane0);        // U is in registers: the accumulator may take the unit after the next
            float fu = 0.f;
#pragma unroll
            for (int e = 0; e < HC; e += 2)
                fu = fmaf(f[e], __uint_as_float(uu[e / 32][e % 32]), fmaf(f[e + 1], __uint_as_float(uu[e / 32][e % 32 + 1]), fu));
            // ---- the row's other half: f . u and f . z of all columns
            float2* dots = reinterpret_cast<float2*>(s_gen + C::OFF_DOT) + (n & 1) * 2 * C::ROWS + row;
            dots[half * C::ROWS] = make_float2(fu, fz);
            if (!(ok = meet(69))) break;
            const float2 d0 = dots[0], d1 = dots[C::ROWS];
            const float inv = 1.f / (d0.y + d1.y + p.eps);
            const float ratio = (d0.x + d1.x) * inv;
            // ---- df = (u - ratio z) / den, dq = df phi'(q);  phi'(x) = 1 above zero, e^x = phi(x) <= 1 at and below it: min(f, 1)
#pragma unroll
            for (int c = 0; c < HC / 8; ++c) {
                const float4 z0 = z4[2 * c], z1 = z4[2 * c + 1];
                const float zz[8] = {z0.x, z0.y, z0.z, z0.w, z1.x, z1.y, z1.z, z1.w};
                uint32_t w[4];
#pragma unroll
                for (int e = 0; e < 8; e += 2) {
                    const int at = c * 8 + e;
                    const float g0 = fmaf(-ratio, zz[e], __uint_as_float(uu[at / 32][at % 32])) * inv;
                    const float g1 = fmaf(-ratio, zz[e + 1], __uint_as_float(uu[at / 32][at % 32 + 1])) * inv;
                    w[e / 2] = pack_bf16(g0 * fminf(f[at], 1.f), g1 * fminf(f[at + 1], 1.f));
                }
                *reinterpret_cast<uint4*>(q_row + (((c0 + c) ^ (row & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
            }
            fence_proxy_async();
            if (C::SUB == 2) __syncwarp();
            else if (!(ok = meet(60))) break;                      // 64 columns are both halves' here
            if (storer && lane0) {
                if (i * C::ROWS + quad * 32 < p.Tc)
                    tma_store_4d(&tm_dq, s_base + q_off + quad * 32 * 128, C::SUB == 2 ? half * 64 : 0, i * C::ROWS + quad * 32, bh, 0);
                bulk_commit();
            }
            prev = rq.stage;
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
