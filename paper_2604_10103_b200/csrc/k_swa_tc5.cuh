// Block-sparse sliding-window attention (Eq. 6; Alg. 3 inner loops) on the Blackwell tensor path:
// TMA loads addressed by the kept-block lists, tcgen05.mma with S / P / Q / O in tensor memory, fp32 softmax against a
// reference exponent fixed per row and unit.  Blocks of 16, 64 or 128 tokens, head dim 64 or 128.  The HIST
// instantiation also forms the history term of Eq. 4 and adds it (Eq. 7) before the one rounding to bf16.
//
// Persistent kernel, one CTA per SM; a CTA walks its units (128 consecutive query rows of one batch*head) and their tiles
// of 128 keys as one stream of tiles t = 0, 1, ...
//   BLK = 128       unit = query block, tile = kept key block.
//   BLK = 16, 64    unit = G = 128 / BLK query blocks ("row groups") with a kept list each; tile = G key blocks side by side
//                   (G boxes of BLK rows, anywhere in the window).  The G lists are merged into one list of key blocks
//                   (k_union.cuh; in a forward call by the selection), each with the set of row groups that keep it; a (row
//                   group, key block) pair that is not kept is masked to -inf before the exponential.  k / |union| of the products are wanted: ~57 % for two lists
//                   that keep a random quarter each, ~100 % when neighbouring query blocks keep the same blocks.  A unit's
//                   first tile holds a kept block of every row group (with 16 tokens its first one), so that every row has a finite
//                   maximum there.
//
// Roles (12 warps, 20 with four column groups):
//   softmax warps       NG = two column groups of four warps (four at head dim 64, see swa_groups); thread (group g, row r) owns 128 / NG
//                       columns of S of row r (TMEM lane = row), from 128 g / NG on, and D / NG columns of O.  It takes its share of S into
//                       registers (the S buffer is free from then on), forms P = exp2(S c - m) and writes it as bf16 to the P buffer.
//   K loader, V loader  TMA: K tiles (ring of two), V tiles (ring of two), Q, and for HIST the folded state S W^T and z
//   S warp, P V warp    tcgen05.mma issue, one warp per product.
//       S_t = Q K_t^T      A = Q (tensor memory), B = K_t (smem, K-major, 128B swizzle)       -> S buffer t & 1
//       O  += P_t V_t      A = P (tensor memory), B = V_t (smem, MN-major, 128B swizzle)      -> O, in two halves of 64 keys
//       D_h = phi(Q) S W^T three products of bf16 hi / lo halves (HIST)                       -> S buffer of the unit's last tile
//
// What bounds it, and why it is cut this way (measured with clock stamps and with a loop of the same products alone, 148
// CTAs, head dim 128, per 128 x 128 tile; 1 024 clk is the tensor pipe's own time):
//   - one warp issuing both products: every barrier test in its loop is ~70-90 clk in which the pipe runs dry (1 170 clk per
//     tile without tests, 1 440 with four, 1 806 with eight); two warps cover each other's tests (1 136; with Q in tensor
//     memory 1 025).
//   - S = Q K^T with both operands in shared memory reads 64 KB per tile at 128 B/clk, which the TMA writes of the next tiles
//     also need: 1 334 clk with the tile traffic running, 1 240 with Q in tensor memory; and it costs power, which is what
//     limits a long run (with everything running 93 -> 82 us for 84 tiles per SM in a loop of seconds).
//   - the exponentials: 16 384 per tile at 16 per clk = 1 024 clk of the special-function unit, 1 200 with their loads.
//   - the softmax warps' serial path between two tiles' exponentials (three barrier tests, tensor-memory load and store, two
//     arrivals): every instruction the convergence unit has to serve costs, so waits are warp-uniform, arrivals predicated, a
//     tile's tail flag comes from one ballot over 32 list entries, and full, masked and empty tiles are separate code (selects in
//     every tile: +9 us of a 134 us forward).  Four groups of 32 columns instead of two (16 warps) cover more of it and pay it
//     twice as often: 132 against 130 us at head dim 128; at 64 they pay (swa_groups).
//   - power: back to back the kernel runs at the board's limit (990 W, SM clock 1 965 -> 1 610 MHz), where time follows energy;
//     packing P with one conversion instead of two adds and a permute is worth 2 % there.
// Measured against the version with one MMA warp, Q in shared memory, three S buffers and a second kernel (plus a separate
// history read-out) for blocks of 16 and 64 tokens, forward call at 12 heads, 4 680 queries, window 14 040 keys, 25 % kept:
// 128-token blocks 131.8 -> 129.5 us, 64-token blocks 208 -> 174 us; 16-token blocks (head dim 64, 1 300 queries) 73.6 -> 65 us.
//
// Range of the fixed reference, and what happens outside it.  Alg. 3 carries a running row maximum so that no input
// overflows; here the reference is fixed after the first tile (row maximum x 2^HEADROOM; softmax does not depend on it), which
// covers rows whose later tiles rise up to about 100 natural-log units above the first one.  A unit with a row beyond that
// (row sum not finite or above 2^100 at the unit's end -- a complete test: every P is a term of the row sum) is put on a list
// in shared memory, and when the thread block has finished its tile stream it computes those units again with the running
// maximum, rescaling l and O as Alg. 3 prints them (swa_redo_unit below: the warp-level code of k_swa_mma.cuh, plus the
// history term where this kernel forms it), overwriting the rows the fast path left.  The result is therefore the softmax of
// Eq. 6 for every finite input.
#pragma once
#include "tc5_common.cuh"
#include "k_swa_mma.cuh"
#include "k_union.cuh"

// NGROUPS: softmax column groups (four warps each), two or four.  At head dim 64 the products leave the softmax warps' chain between two
// tiles' exponentials as the bound, and four groups of 32 columns overlap more of it: 444 units of 12 heads, 28 kept blocks of 128
// tokens 85.6 -> 79.7 us, 10 kept 36.7 -> 34.4.  Below five tiles their meetings at a unit's ends weigh more.  Forward calls, two groups /
// four, us:                 one tile       three          four           five           eight
//   1 unit                  7.30 / 7.55    9.09 / 9.22    9.86 / 9.86   10.75 / 10.50   13.1 / 12.7
//   64 units                8.96 / 9.09    10.9 / 10.9    11.7 / 11.5   12.4 / 12.4     15.1 / 14.6
//   444 units               22.5 / 23.0    27.8 / 27.9    30.3 / 29.8   32.6 / 32.1     40.3 / 39.2
// The masked segments of 64-token blocks weigh more too (117 -> 119 us), blocks of 16 tokens have not been tried, and head dim 128 has no
// registers for it: two there.
inline constexpr int swa_groups(int d, int blk, int tiles) { return d == 64 && blk == 128 && tiles >= 5 ? 4 : 2; }

template <int D, int NGROUPS>
struct SwaTc5 {
    static constexpr int NG = NGROUPS, NSW = 4 * NG;   // softmax column groups; softmax warps
    static constexpr long long SKEW_CLK = NG == 2 ? 700 : 300;       // offset between the column groups, in clocks (see the softmax warps)
    static constexpr int SCOLS = 128 / NG;             // S columns per softmax thread
    static constexpr int OCOLS = D / NG;               // O columns per softmax thread
    static constexpr int SUB = D / 64;                 // 64-column (128-byte) sub-tiles per operand tile
    static constexpr int SUB_BYTES = 128 * 128;        // 16 KB
    static constexpr int TILE_BYTES = SUB * SUB_BYTES;
    static constexpr int HSUB_BYTES = D * 128;         // S W^T halves: D rows of 64-column sub-tiles
    static constexpr int H_BYTES = SUB * HSUB_BYTES;
    static constexpr float HEADROOM = 60.f;           // log2 distance of the softmax reference above the first tile's row maximum
    // Tensor memory: two S buffers, P, Q, O.  There is room for one P buffer at head dim 128.  Its halves (keys 0..63 from
    // the lower half of the column groups, keys 64..127 from the upper) are products and barriers of their own, so that a group waits only
    // for the product of its own last half, issued a whole tile earlier.
    static constexpr int COL_P = 256, COL_Q = COL_P + 64, COL_O = COL_Q + D / 2, TMEM_COLS = 512;
    static_assert(COL_O + D <= TMEM_COLS, "tensor memory layout");
    static constexpr int OFF_Q = 0, OFF_K = TILE_BYTES, OFF_V = OFF_K + 2 * TILE_BYTES;
    static constexpr int OFF_H = OFF_V + 2 * TILE_BYTES;       // S W^T, hi then lo; also the staging tile of the output
    // (the second pass keeps its fp32 history tile behind the operand tiles of swa_mma_unit, in front of the barriers)
    static constexpr int OFF_BAR = OFF_H + 2 * H_BYTES > SwaMma<128, D>::SMEM_BYTES + 128 * D * 4 ? OFF_H + 2 * H_BYTES
                                                                                                    : SwaMma<128, D>::SMEM_BYTES + 128 * D * 4;
    // units whose rows left the range of the fixed reference: count, last unit listed, up to REDO_CAP local unit numbers
    // (more than that: every unit of the thread block is computed again)
    static constexpr int OFF_REDO = OFF_BAR + 256, REDO_CAP = 8;
    static constexpr int OFF_Z = OFF_REDO + 64;        // z [D] of the unit's head
    static_assert((2 + REDO_CAP) * 4 <= OFF_Z - OFF_REDO, "the list must fit");
    static constexpr int OFF_XM = OFF_Z + 512;         // row maxima of the column groups [NG][128]
    static constexpr int USED_BYTES = OFF_XM + NG * 128 * 4;
    // row sums and shares of Eq. 4's denominator [2][NG][128] at a unit's end: beside the staging tile of the output
    static constexpr int OFF_XS = OFF_H + NSW * 32 * OCOLS * 2;
    static_assert(OFF_XS + 2 * NG * 128 * 4 <= OFF_BAR, "exchange buffers");
    static constexpr int MAX_SMEM = 232448;            // 227 KB: the most one thread block can have
    // Slack for the manual 1024-byte alignment of the operand tiles (the kernel checks that it was enough); more than
    // half an SM's shared memory so that one CTA owns the SM (it allocates all 512 TMEM columns)
    static constexpr int WANT_BYTES = (USED_BYTES + 1024) > 120 * 1024 ? (USED_BYTES + 1024) : 120 * 1024;
    static constexpr int SMEM_BYTES = WANT_BYTES < MAX_SMEM ? WANT_BYTES : MAX_SMEM;
    static_assert(USED_BYTES <= MAX_SMEM, "shared memory layout does not fit");
    static constexpr int THREADS = 32 * NSW + 128;
    static constexpr int WARP_LOAD_K = NSW, WARP_LOAD_V = NSW + 1, WARP_S = NSW + 2, WARP_PV = NSW + 3;
};

struct Tc5Params {
    const int32_t* idx;      // [B*H, T_m, keep]
    int keep, Tc, n_b, n_cached, ring_head, P;   // P: physical ring slots (one more than the window holds); the sink slots follow them
    int n_sink;              // sink chunks held (logical chunks 0 .. n_sink - 1)
    int Tn;                  // key blocks of the window: (n_sink + n_cached + 1) n_b
    uint32_t nb_magic;       // ceil(2^32 / n_b) (n_b > 1): x / n_b = high word of x * nb_magic for x <= 1024
    int Tm, n_units;         // query blocks per batch*head; units in all (unit u = bh * upb + i)
    int upb;                 // units per batch*head: T_m, or ceil(T_c / 128) with 16- / 64-token blocks
    const uint32_t* entries; // 16- / 64-token blocks: [units, max_tiles, G] merged lists (k_union.cuh) ...
    const int* tiles;        // ... and tiles per unit
    int max_tiles;
    float scale_log2;
    const float* hist;       // optional fp32 [B*H, T_c, D]: history term formed by another kernel, added in the epilogue
    // History term formed in the kernel (its HIST instantiation): z [B*H, D], bias [H, D] or nullptr, eps of Eq. 4's denominator
    int heads;
    float eps;
    const bf16* q;
    const float* z;
    const bf16* bias;
    const float* cos_q;      // rotation of Eq. 4's numerator, tables [D / 8][T_c][4], or nullptr: none
    const float* sin_q;
    bf16* o;
    float* lse;
    int* dev_status;
    // for the units that are computed again with a running maximum: the window as plain pointers, and the folded state
    ChunkTable tab;
    const bf16* sf_hi;       // [B*H, D, D] bf16 hi / lo halves of S W^T (HIST only)
    const bf16* sf_lo;
};

// Ring position of item i in a ring of N stages: stage i % N, completed-phase parity (i / N) & 1, kept incrementally.
template <int N>
struct RingPos {
    int stage = 0;
    uint32_t phase = 0;
    __device__ __forceinline__ void advance() { if (++stage == N) { stage = 0; phase ^= 1u; } }
};

// One unit again, the way Alg. 3 prints it (running maximum m, rescaling of l and O), by threads 0 .. 255 of the thread
// block, after the tile stream has drained (shared memory and the exchange buffers are free by then).  HIST: the history
// term of Eq. 4 for the unit's rows is formed first, in fp32 on the CUDA cores, into a shared-memory tile that the
// attention epilogue adds (Eq. 7).  Slow and rare by design.
template <int D, int BLK, int HIST>
__device__ __noinline__ void swa_redo_unit(uint8_t* s_gen, const Tc5Params& p, int u) {
    typedef SwaMma<128, D> M;          // its shared-memory window is the largest: the history tile sits behind it
    constexpr int ROWS = 128;
    const int bh = u / p.upb, i = u - bh * p.upb;
    const int q0 = i * ROWS, nq = min(ROWS, p.Tc - q0);
    const int tid = threadIdx.x;
    const float* hist_rows = p.hist ? p.hist + ((size_t)bh * p.Tc + q0) * D : nullptr;
    auto sync256 = [] { asm volatile("bar.sync 2, 256;\n" ::: "memory"); };
    sync256();                         // the previous unit's epilogue has read its history tile
    if constexpr (HIST) {
        constexpr int PS = D + 1;                                            // padded row of the phi(Q) tile
        float* phi_t = reinterpret_cast<float*>(s_gen + M::TILE_BYTES);     // [128][D + 1], in the K / V stages (not yet in use)
        float* den_t = phi_t + ROWS * PS;                                   // [128]
        float* hist_t = reinterpret_cast<float*>(s_gen + M::SMEM_BYTES);    // [128][D], behind the attention tiles
        static_assert(M::TILE_BYTES + (ROWS * PS + ROWS) * 4 <= M::SMEM_BYTES, "phi(Q) tile must fit in the K / V stages");
        static_assert(M::SMEM_BYTES + ROWS * D * 4 <= SwaTc5<D, 2>::OFF_BAR, "history tile must fit");
        {   // phi(q) of the unit's rows (zero past the chunk's end): thread = (row, half of the features)
            const int row = tid >> 1, f0 = (tid & 1) * (D / 2);
            const bf16* src = p.q + ((size_t)bh * p.Tc + q0 + row) * D + f0;
            for (int c = 0; c < D / 2; c += 8) {
                uint4 w = make_uint4(0, 0, 0, 0);
                if (row < nq) w = __ldg(reinterpret_cast<const uint4*>(src + c));
                const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float2 x = unpack_bf16(ws[e]);
                    phi_t[row * PS + f0 + c + 2 * e] = row < nq ? phi_elu1(x.x) : 0.f;
                    phi_t[row * PS + f0 + c + 2 * e + 1] = row < nq ? phi_elu1(x.y) : 0.f;
                }
            }
        }
        sync256();
        if (tid < ROWS) {       // Eq. 4's denominator phi(q).z + eps, one row per thread
            float dsum = 0.f;
            const float* zr = p.z + (size_t)bh * D;
            for (int a = 0; a < D; ++a) dsum = fmaf(phi_t[tid * PS + a], __ldg(zr + a), dsum);
            den_t[tid] = dsum + p.eps;
        }
        if constexpr (HIST == 2) {      // the numerator sees phi(q) rotated, the denominator above does not
            sync256();
            const int row = tid >> 1, f0 = (tid & 1) * (D / 2), r_tab = min(q0 + row, p.Tc - 1);
            for (int a = f0; a < f0 + D / 2; a += 2) {
                const size_t at = ((size_t)(a / 8) * p.Tc + r_tab) * 4 + a / 2 % 4;
                const float c = __ldg(p.cos_q + at), sn = __ldg(p.sin_q + at);
                const float x0 = phi_t[row * PS + a], x1 = phi_t[row * PS + a + 1];
                phi_t[row * PS + a] = fmaf(-x1, sn, x0 * c);
                phi_t[row * PS + a + 1] = fmaf(x0, sn, x1 * c);
            }
            sync256();
        }
        {   // numerator phi(q) S' : thread = (output column, group of rows); S' = hi + lo halves of the folded state
            constexpr int GROUPS = 256 / D, RPT = ROWS / GROUPS;
            const int c = tid % D, r0 = (tid / D) * RPT;
            const bf16* sh = p.sf_hi + (size_t)bh * D * D + c;
            const bf16* sl = p.sf_lo + (size_t)bh * D * D + c;
            float acc[RPT];
#pragma unroll
            for (int r = 0; r < RPT; ++r) acc[r] = 0.f;
            for (int a = 0; a < D; ++a) {
                const float sv = __bfloat162float(sh[(size_t)a * D]) + __bfloat162float(sl[(size_t)a * D]);
#pragma unroll
                for (int r = 0; r < RPT; ++r) acc[r] = fmaf(phi_t[(r0 + r) * PS + a], sv, acc[r]);
            }
            sync256();                                            // denominators written
            const float b = p.bias ? __bfloat162float(p.bias[(size_t)(bh % p.heads) * D + c]) : 0.f;
#pragma unroll
            for (int r = 0; r < RPT; ++r) hist_t[(r0 + r) * D + c] = acc[r] / den_t[r0 + r] + b;
        }
        sync256();                                                // tile complete; the K / V stages are free again
        hist_rows = hist_t;
    }
    if (tid >= SwaMma<BLK, D>::THREADS) return;
    for (int g = 0; g < 128 / BLK; ++g) {
        const int qb = i * (128 / BLK) + g, unit = bh * p.Tm + qb;
        if (qb >= p.Tm) break;
        if (tid == 0) atomicAdd(p.dev_status + 2, 1);             // count of query blocks that took this path
        swa_mma_unit<BLK, D>(s_gen, p.q, p.tab, p.idx + (size_t)unit * p.keep, p.keep, p.Tc, p.n_b, p.scale_log2,
                             hist_rows ? hist_rows + (size_t)g * BLK * D : nullptr, p.o, p.lse, p.dev_status, qb, bh, unit);
    }
}

// One thread's weights of W consecutive columns of its S row: P = exp2(S c - m) as bf16 pairs, and their fp32 sum into rsum.
// MASK: columns from nv on have weight zero (S taken as -inf).  Packed fp32: the scale-and-shift and the sum handle two columns
// per instruction.
template <int W, bool MASK>
__device__ __forceinline__ void swa_weights(const uint32_t* r, int nv, float scale_log2, float m, float2 (&rsum)[4], uint32_t* pk) {
    const float2 scale2 = make_float2(scale_log2, scale_log2), negm2 = make_float2(-m, -m);
#pragma unroll
    for (int e0 = 0; e0 < W; e0 += 8) {         // four column pairs at a time, stage by stage: independent work side by side
        float2 x[4], pe[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int e = e0 + 2 * v;
            x[v].x = __uint_as_float(MASK && e >= nv ? 0xff800000u : r[e]);
            x[v].y = __uint_as_float(MASK && e + 1 >= nv ? 0xff800000u : r[e + 1]);
            x[v] = ffma2(x[v], scale2, negm2);
        }
#pragma unroll
        for (int v = 0; v < 4; ++v) pe[v] = make_float2(fast_exp2(x[v].x), fast_exp2(x[v].y));
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            rsum[v] = fadd2(rsum[v], pe[v]);
            pk[(e0 >> 1) + v] = pack_bf16(pe[v].x, pe[v].y);
        }
    }
}
template <int W, bool MASK>
__device__ __forceinline__ float swa_max(const uint32_t* r, int nv) {
    float mx[2] = {-INFINITY, -INFINITY};
#pragma unroll
    for (int e = 0; e < W; e += 2) {            // three-input maximum: two values per instruction
        const float a = __uint_as_float(MASK && e >= nv ? 0xff800000u : r[e]);
        const float b = __uint_as_float(MASK && e + 1 >= nv ? 0xff800000u : r[e + 1]);
        mx[(e >> 1) & 1] = fmax3(mx[(e >> 1) & 1], a, b);
    }
    return fmaxf(mx[0], mx[1]);
}

// Persistent: CTA c processes units c, c + gridDim.x, ...
// HIST 1: the history term is formed here; 2: with its numerator rotated (code of its own: as a branch it cost the plain one
// 2 % of the call); 0: p.hist, if any, is added.
template <int D, int BLK, int HIST, int NGROUPS>
__global__ void __launch_bounds__(SwaTc5<D, NGROUPS>::THREADS, 1)
k_swa_tc5(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_kring,
          const __grid_constant__ CUtensorMap tm_vring, const __grid_constant__ CUtensorMap tm_kcur,
          const __grid_constant__ CUtensorMap tm_vcur, const __grid_constant__ CUtensorMap tm_sh,
          const __grid_constant__ CUtensorMap tm_sl, const __grid_constant__ CUtensorMap tm_o,
          const __grid_constant__ Tc5Params p) {
    using namespace tc5;
    typedef SwaTc5<D, NGROUPS> C;
    constexpr int G = 128 / BLK;                       // key blocks per tile = row groups per unit
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t s_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    if (s_base - smem_u32(smem_raw) + C::USED_BYTES > C::SMEM_BYTES) {   // the window started too far off a 1 KB boundary
        if (threadIdx.x == 0) { atomicOr(p.dev_status, HF_DEV_TIMEOUT_FLAG); atomicExch(p.dev_status + 1, 99); }
        return;
    }
    uint8_t* s_gen = smem_raw + (s_base - smem_u32(smem_raw));
    const uint32_t sQ = s_base + C::OFF_Q, sK = s_base + C::OFF_K, sV = s_base + C::OFF_V, sH = s_base + C::OFF_H;
    const uint32_t bar0 = s_base + C::OFF_BAR;
    // Barriers (pairs: index t & 1, completion t >> 1).  Whoever waits for item t of a pair cannot be passed by item t + 2:
    // producing that one needs the waiter's own step, so a parity test is exact.
    const uint32_t bar_kf = bar0, bar_vf = bar0 + 16,      // K / V tile t landed
                   bar_sf = bar0 + 32,                     // S_t complete (its K stage is free)
                   bar_se = bar0 + 48,                     // S_t is in the softmax warps' registers (all of them)
                   bar_pf = bar0 + 64,                     // two: a half of P_t written (half of the softmax warps); completion t
                   bar_pv = bar0 + 80,                     // P V of tile t complete, second half (so its V stage is free)
                   bar_ph = bar0 + 216,                    // ... first half
                   // unit n: Q landed / its shared-memory tile is free, which takes the word of both its readers: the copy to tensor
                   // memory (a commit behind it) and, for HIST, the phi pass of every softmax warp at the unit's last tile.  Neither
                   // implies the other: in a unit of one tile nothing else orders the phi pass behind the copy, which waits for K.
                   bar_qf = bar0 + 96, bar_qe = bar0 + 104,
                   bar_hf = bar0 + 112, bar_he = bar0 + 120,   // unit n: S W^T and z landed / free
                   bar_af = bar0 + 128,                    // unit n: phi(Q) operand written
                   bar_ud = bar0 + 136,                    // unit n: history products complete
                   bar_dr = bar0 + 144,                    // unit n: D_h (and O) read by the epilogue
                   bar_x = bar0 + 152,                     // four: exchange between the warps that share 32 rows
                   bar_drain = bar0 + 232;                 // two: each MMA warp's last operations complete
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(s_gen + C::OFF_BAR + 184);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(s_gen + C::OFF_BAR + 188);
    int* redo_cnt = reinterpret_cast<int*>(s_gen + C::OFF_REDO);
    int* redo_last = redo_cnt + 1;
    int* redo_list = redo_cnt + 2;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int my_units = (p.n_units - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
    auto tiles_of = [&](int n) -> int {               // tiles of local unit n
        if constexpr (BLK == 128) return p.keep;
        else return n < my_units ? __ldg(p.tiles + blockIdx.x + n * gridDim.x) : 0;
    };

    if (threadIdx.x == 0) {
        for (int s = 0; s < 2; ++s) {
            mbar_init(bar_kf + 8 * s, 1); mbar_init(bar_vf + 8 * s, 1); mbar_init(bar_sf + 8 * s, 1); mbar_init(bar_pv + 8 * s, 1);
            mbar_init(bar_se + 8 * s, C::NSW); mbar_init(bar_pf + 8 * s, C::NSW / 2); mbar_init(bar_ph + 8 * s, 1); mbar_init(bar_drain + 8 * s, 1);
        }
        for (int s = 0; s < 4; ++s) mbar_init(bar_x + 8 * s, C::NG);
        mbar_init(bar_qf, 1); mbar_init(bar_qe, HIST ? C::NSW + 1 : 1); mbar_init(bar_hf, 1); mbar_init(bar_he, C::NSW);
        mbar_init(bar_af, C::NSW); mbar_init(bar_ud, 1); mbar_init(bar_dr, C::NSW);
        *abort_flag = 0;
        *redo_cnt = 0; *redo_last = -1;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == C::WARP_S) {
        tmem_alloc(smem_u32(tmem_slot), C::TMEM_COLS);
        tmem_relinquish();
    }
    if (warp == C::WARP_LOAD_K && lane == 0) { tma_prefetch_map(&tm_kring); tma_prefetch_map(&tm_kcur); }
    if (warp == C::WARP_LOAD_V && lane == 0) {
        tma_prefetch_map(&tm_q); tma_prefetch_map(&tm_vring); tma_prefetch_map(&tm_vcur);
        if (HIST) { tma_prefetch_map(&tm_sh); tma_prefetch_map(&tm_sl); }
    }
    if (warp == 0 && lane == 0) tma_prefetch_map(&tm_o);
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    // Everything above (barriers, tensor memory) may overlap the tail of the kernel before this one in the stream when the
    // launch allows it; the lists it wrote are read from here on.
    pdl_wait();
    // The next kernel in the stream may be made resident on SMs this grid has left (it waits itself) -- only where a thread
    // block of this kernel takes all of an SM's shared memory, so that no waiting block of the dependent grid ever sits
    // beside a working block of this one.
    if (C::SMEM_BYTES > 200 * 1024) pdl_trigger();

    auto wait_w = [&](uint32_t bar, uint32_t parity, int where) -> bool {      // a warp's wait, warp-uniform result
        return mbar_wait_warp<true>(bar, parity & 1u, abort_flag, p.dev_status, where);
    };

    if (warp == C::WARP_LOAD_K || warp == C::WARP_LOAD_V) {
        // ================================================================= TMA producers
        // One lane copies a tile of a 128-token block; blocks of 16 or 64 tokens have a lane each (G boxes a tile: one after the other, with
        // their list entries' loads between them, they bounded the tile loop: 16-token blocks, 12 heads, 1 300 queries, 62 of 246 blocks
        // kept 53 -> 32.5 us at head dim 64, 69 -> 41 at 128).  The loops are the warp's.
        const bool is_k = (warp == C::WARP_LOAD_K);
        const int box = lane < G ? lane : 0;
        bool ok = true;
        int t = 0;
        const int Tn = p.Tn;
        const uint32_t tiles = is_k ? sK : sV, full = is_k ? bar_kf : bar_vf, freed = is_k ? bar_sf : bar_pv;
        auto list_of = [&](int u) -> const uint32_t* {
            if constexpr (BLK == 128) return reinterpret_cast<const uint32_t*>(p.idx + (size_t)u * p.keep);
            else return p.entries + (size_t)u * p.max_tiles * G + box;
        };
        uint32_t e_next = my_units > 0 ? __ldg(list_of(blockIdx.x)) : 0u;      // list entry, read one tile ahead
        for (int n = 0; ok && n < my_units; ++n) {
            const int u = blockIdx.x + n * gridDim.x;
            const int bh = u / p.upb, i = u - bh * p.upb;
            const int cnt = tiles_of(n);
            if (!is_k) {   // Q of this unit, once the softmax warps are done with the previous one
                if (n >= 1 && !(ok = wait_w(bar_qe, n - 1, 1))) break;
                if (lane == 0) {
                    mbar_expect_tx(bar_qf, C::TILE_BYTES);
#pragma unroll
                    for (int s = 0; s < C::SUB; ++s) tma_load_4d(sQ + s * C::SUB_BYTES, &tm_q, s * 64, i * 128, bh, 0, bar_qf);
                }
                __syncwarp();
            }
            const uint32_t* list = list_of(u);
            for (int j = 0; j < cnt; ++j, ++t) {
                const uint32_t st = t & 1, dst = tiles + st * C::TILE_BYTES + box * BLK * 128, bar = full + 8 * st;
                int blk;
                if constexpr (BLK == 128) blk = checked_block((int)e_next, Tn, is_k && lane == 0 ? p.dev_status : nullptr, u);
                else { blk = (int)(e_next & 1023u); if (blk >= Tn) blk = 0; }          // (the list builder has checked every entry already)
                e_next = __ldg(j + 1 < cnt ? list + (j + 1) * G : list_of(n + 1 < my_units ? u + (int)gridDim.x : u));
                int c = 0, jb = blk;
                while (jb >= p.n_b) { jb -= p.n_b; ++c; }          // at most HF_MAX_CHUNKS - 1 steps; no XU-pipe division
                // logical chunk order: sink chunks (slots P, P + 1, ...), cached chunks oldest first (ring), current chunk
                const bool cur = (c == p.n_sink + p.n_cached);
                int slot = 0;
                if (!cur) {
                    if (c < p.n_sink) slot = p.P + c;
                    else { slot = p.ring_head + c - p.n_sink; if (slot >= p.P) slot -= p.P; }
                }
                const CUtensorMap* m = is_k ? (cur ? &tm_kcur : &tm_kring) : (cur ? &tm_vcur : &tm_vring);
                if (t >= 2 && !(ok = wait_w(freed + 8 * st, (t >> 1) - 1, 2))) break;
                if (lane == 0) mbar_expect_tx(bar, C::TILE_BYTES);
                __syncwarp();
                if (lane < G) {
#pragma unroll
                    for (int s = 0; s < C::SUB; ++s) tma_load_4d(dst + s * C::SUB_BYTES, m, s * 64, jb * BLK, bh, slot, bar);
                }
                __syncwarp();
                if (HIST && !is_k && j == (cnt > 1 ? 1 : 0)) {
                    // For the history term at the unit's end: the head's folded state and z.  The buffer is free once the
                    // previous unit's output, which was staged in it, has been read by the bulk stores.  (Two V tiles of
                    // this unit are on their way by now; the third needs P V of the first, which comes after that.)
                    if (n >= 1 && !(ok = wait_w(bar_he, n - 1, 13))) break;
                    if (lane == 0) {
                        mbar_expect_tx(bar_hf, 2 * C::H_BYTES + D * 4);
#pragma unroll
                        for (int s = 0; s < C::SUB; ++s) {
                            tma_load_4d(sH + s * C::HSUB_BYTES, &tm_sh, s * 64, 0, bh, 0, bar_hf);
                            tma_load_4d(sH + C::H_BYTES + s * C::HSUB_BYTES, &tm_sl, s * 64, 0, bh, 0, bar_hf);
                        }
                        bulk_load(s_base + C::OFF_Z, p.z + (size_t)bh * D, D * 4, bar_hf);
                    }
                    __syncwarp();
                }
            }
        }
        if (!ok) {   // gave up: let the copies already in flight land before the CTA leaves
            const long long t0 = clock64();
            while (clock64() - t0 < 400000) {}
        }
    } else if (warp == C::WARP_S) {
        // ================================================================= S = Q K^T
        // The whole warp walks the loop (uniform control flow, so that descriptors and addresses can live in uniform
        // registers); one elected lane issues the tensor-core instructions.
        constexpr uint32_t IDESC_S = idesc_bf16(128, false);
        constexpr uint32_t TILE_STEP = C::TILE_BYTES >> 4;      // descriptor address field counts 16-byte units
        const uint64_t dq0 = smem_desc_sw128(sQ, 16, 1024), dk0 = smem_desc_sw128(sK, 16, 1024);
        const uint32_t k_lo = (uint32_t)dk0, k_hi = (uint32_t)(dk0 >> 32);
        bool ok = true;
        int x = 0;
        for (int n = 0; ok && n < my_units; ++n) {
            const int cnt = tiles_of(n);
            for (int j = 0; j < cnt; ++j, ++x) {
                const uint32_t st = x & 1;
                if (j == 0) {
                    // Q of the unit moves from shared to tensor memory, where the previous unit's last S has read it by then
                    if (!(ok = wait_w(bar_qf, n, 4))) break;
                    if (n >= 1 && !(ok = wait_w(bar_sf + 8 * ((x - 1) & 1), (x - 1) >> 1, 22))) break;
                }
                if (!(ok = wait_w(bar_kf + 8 * st, x >> 1, 5))) break;
                // The S buffer: free once the softmax warps hold S of two tiles ago in registers.  HIST: at a unit's start the
                // buffer holds the previous unit's phi(Q) operand, at its second tile the previous unit's D_h.
                if (HIST && n >= 1 && j == 0) { if (!(ok = wait_w(bar_ud, n - 1, 23))) break; }
                else if (HIST && n >= 1 && j == 1) { if (!(ok = wait_w(bar_dr, n - 1, 24))) break; }
                else if (x >= 2) { if (!(ok = wait_w(bar_se + 8 * st, (x >> 1) - 1, 25))) break; }
                fence_after_sync();
                if (elect_one()) {
                    if (j == 0) {
#pragma unroll
                        for (int ks = 0; ks < D / 16; ++ks)      // 16 features = 32 bytes of a row = 8 columns
                            tmem_cp_128x256b(tmem + C::COL_Q + 8 * ks, dq0 + (uint64_t)((ks >> 2) * (C::SUB_BYTES >> 4) + (ks & 3) * 2));
                        mma_commit(bar_qe);
                    }
                    mma_ts_kmajor<D>(tmem + st * 128, tmem + C::COL_Q, k_lo + st * TILE_STEP, k_hi, IDESC_S);
                    mma_commit(bar_sf + 8 * st);
                }
                __syncwarp();
            }
        }
        // drain: all operations issued by this warp have completed before TMEM is freed
        if (elect_one()) mma_commit(bar_drain);
        __syncwarp();
        {
            const long long t0 = clock64();
            while (!mbar_try_wait(bar_drain, 0) && clock64() - t0 < WAIT_LIMIT_CYCLES) {}
        }
    } else if (warp == C::WARP_PV) {
        // ================================================================= O += P V, history products
        constexpr uint32_t IDESC_PV = idesc_bf16(D, true);
        constexpr uint32_t TILE_STEP = C::TILE_BYTES >> 4, H_STEP = C::H_BYTES >> 4;
        const uint32_t tO = tmem + C::COL_O;
        const uint64_t dv0 = smem_desc_sw128(sV, C::SUB_BYTES, 1024);
        const uint64_t dh0 = smem_desc_sw128(sH, C::HSUB_BYTES, 1024);    // S W^T tiles: laid out like a V tile (rows = contraction index)
        const uint32_t v_lo = (uint32_t)dv0, v_hi = (uint32_t)(dv0 >> 32), h_lo = (uint32_t)dh0, h_hi = (uint32_t)(dh0 >> 32);
        bool ok = true;
        int t = 0;
        for (int n = 0; ok && n < my_units; ++n) {
            const int cnt = tiles_of(n);
            for (int j = 0; j < cnt; ++j, ++t) {
                const uint32_t st = t & 1;
                if (HIST && j == cnt - 1) {
                    // D_h = phi(Q) S W^T while the softmax warps work on the unit's last tile: into that tile's S buffer (already
                    // in registers), A from the other S buffer (quarter k of the features: hi half at column 32 k, lo half D / 8 on),
                    // B = the hi and lo tiles of S W^T; three products, the lo x lo one is below fp32 resolution
                    if (!(ok = wait_w(bar_hf, n, 14))) break;
                    if (!(ok = wait_w(bar_af, n, 15))) break;
                    if (!(ok = wait_w(bar_se + 8 * st, t >> 1, 26))) break;
                    fence_after_sync();
                    const uint32_t tD = tmem + st * 128, tA = tmem + (st ^ 1u) * 128;
                    if (elect_one()) {
                        mma_ts_groups<D>(tD, tA, h_lo, h_hi, IDESC_PV, false);                 // hi x hi
                        mma_ts_groups<D>(tD, tA + D / 8, h_lo, h_hi, IDESC_PV, true);          // lo x hi
                        mma_ts_groups<D>(tD, tA, h_lo + H_STEP, h_hi, IDESC_PV, true);         // hi x lo
                        mma_commit(bar_ud);
                    }
                    __syncwarp();
                }
                if (!(ok = wait_w(bar_vf + 8 * st, t >> 1, 7))) break;
                if (!(ok = wait_w(bar_pf, t, 6))) break;
                fence_after_sync();
                if (elect_one()) {
                    mma_ts_half(tO, tmem + C::COL_P, v_lo + st * TILE_STEP, v_hi, IDESC_PV, j > 0);
                    mma_commit(bar_ph + 8 * st);
                }
                __syncwarp();
                if (!(ok = wait_w(bar_pf + 8, t, 28))) break;
                fence_after_sync();
                if (elect_one()) {
                    mma_ts_half(tO, tmem + C::COL_P + 32, v_lo + st * TILE_STEP + (64 * 128 >> 4), v_hi, IDESC_PV, true);
                    mma_commit(bar_pv + 8 * st);
                }
                __syncwarp();
            }
        }
        if (elect_one()) mma_commit(bar_drain + 8);
        __syncwarp();
        {
            const long long t0 = clock64();
            while (!mbar_try_wait(bar_drain + 8, 0) && clock64() - t0 < WAIT_LIMIT_CYCLES) {}
        }
    } else {
        // ================================================================= softmax / epilogue
        const int grp = warp >> 2;                          // column group: key columns [SCOLS grp, SCOLS grp + SCOLS) of a tile
        const int half = grp * 2 / C::NG;                   // the half of P they are in
        const int row = (warp & 3) * 32 + lane;             // query row of the unit = TMEM lane
        const int rg = row / BLK;                           // row group (query block within the unit)
        const uint32_t lane_base = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        constexpr int EPT = BLK >= C::SCOLS ? 1 : C::SCOLS / BLK;  // list entries (key blocks) under this thread's columns
        const int col0 = grp * C::SCOLS % BLK;                     // first column within its key block (0 where it has several)
        const uint32_t bar_xw = bar_x + 8 * (warp & 3);     // partners: the warps with the same rows in the other groups
        float* x_m = reinterpret_cast<float*>(s_gen + C::OFF_XM);
        float* x_l = reinterpret_cast<float*>(s_gen + C::OFF_XS);
        float* x_d = x_l + C::NG * 128;
        const bool ragged = p.Tc % BLK != 0;                // every chunk's last block is short
        bool ok = true;
        int t = 0;
        auto wait_s = [&](uint32_t bar, uint32_t parity, int where) -> bool {
            return mbar_wait_warp(bar, parity & 1u, abort_flag, p.dev_status, where);
        };
        // One arrival per warp.  (Tensor-memory loads and stores are warp instructions, complete for all lanes after the warp's
        // wait: only hand-overs of shared memory need the __syncwarp.)
        const bool lane0 = lane == 0;
        auto arrive_t = [&](uint32_t bar) { mbar_arrive_if(bar, lane0); };
        auto arrive_w = [&](uint32_t bar) { __syncwarp(); mbar_arrive_if(bar, lane0); };
        // Exchange number e of the kernel between partner warps: what a caller wrote to shared memory before is visible to the
        // others after.  Two per unit (maxima, then sums): a buffer written at one is read by the partners before they arrive
        // at the next, so each buffer is free again one exchange later.
        auto exchange = [&](uint32_t e, int where) -> bool { arrive_w(bar_xw); return wait_s(bar_xw, e, where); };
        auto note_redo = [&](int n) {                       // list unit n once
            if (atomicMax(redo_last, n) < n) {
                const int slot = atomicAdd(redo_cnt, 1);
                if (slot < C::REDO_CAP) redo_list[slot] = n;
            }
        };
        // (batch*head, position) of a unit without a division per unit; the tile count and the first list entries of the next
        // unit are read during the current one
        const int dbh = gridDim.x / p.upb, di = gridDim.x - dbh * p.upb;
        int u = blockIdx.x, bh = u / p.upb, i = u - bh * p.upb, cnt_next = tiles_of(0);
        const uint32_t bar_own = half == 0 ? bar_ph : bar_pv;      // product of its half of P
        // BLK 16, 64: list entries, read one tile ahead.  BLK 128: all that matters here is whether a tile is a chunk's short last
        // block; one bit per tile from a ballot over 32 list entries at a time (lane = entry), read one window ahead.  An entry
        // outside [0, T_n) is block 0 here as for the loader, which reports it.
        auto entries_of = [&](int unit) -> const uint32_t* {
            if constexpr (BLK == 128) return reinterpret_cast<const uint32_t*>(p.idx + (size_t)unit * p.keep);
            else return p.entries + (size_t)unit * p.max_tiles * G + grp * C::SCOLS / BLK;
        };
        uint32_t e_next[EPT], tails = 0;
#pragma unroll
        for (int x = 0; x < EPT; ++x) e_next[x] = 0u;
        if (my_units > 0) {
            if constexpr (BLK == 128) { if (ragged && lane < p.keep) e_next[0] = __ldg(entries_of(u) + lane); }
            else {
#pragma unroll
                for (int x = 0; x < EPT; ++x) e_next[x] = __ldg(entries_of(u) + x);
            }
        }
        for (int n = 0; ok && n < my_units; ++n) {
            const int q0 = i * 128;
            const int nq = min(128, p.Tc - q0);
            const int cnt = cnt_next;
            cnt_next = n + 1 < my_units ? tiles_of(n + 1) : 0;
            float m_used = 0.f, l_run = 0.f, dsum = 0.f;    // l_run, dsum: this thread's shares
            const uint32_t* ent = entries_of(u);
            // The previous unit's output was staged where S W^T lives, and z where its denominators were exchanged: the loader
            // may refill both once this warp's bulk store has read its part.  (Said after the unit's first tile, when the store
            // has long done so; in a unit of one tile, before it.)
            auto release_h = [&] {
                if (lane == 0) bulk_wait_read();
                arrive_w(bar_he);
            };
            if (HIST && n >= 1 && cnt == 1) release_h();
            for (int j = 0; j < cnt; ++j, ++t) {
                const uint32_t st = t & 1;
                uint32_t e_cur[EPT];
                if constexpr (BLK == 128) {
                    if (ragged && (j & 31) == 0) {
                        const uint32_t x1 = (e_next[0] < (uint32_t)p.Tn ? e_next[0] : 0u) + 1u;     // last block of a chunk: its index + 1 is a multiple of n_b (no division)
                        tails = __ballot_sync(0xffffffffu, p.n_b == 1 || __umulhi(x1, p.nb_magic) * p.n_b == x1);
                        const int j2 = j + 32 < cnt ? j + 32 : 0;
                        if (j2 + lane < p.keep) e_next[0] = __ldg(entries_of(j2 || n + 1 >= my_units ? u : u + (int)gridDim.x) + j2 + lane);
                    }
                } else {
                    const uint32_t* src = j + 1 < cnt ? ent + (j + 1) * G : entries_of(n + 1 < my_units ? u + (int)gridDim.x : u);
#pragma unroll
                    for (int x = 0; x < EPT; ++x) { e_cur[x] = e_next[x]; e_next[x] = __ldg(src + x); }
                }
                if (HIST && j == cnt - 1) {
                    // ---- history term (Eq. 4): A = phi(q) as bf16 hi + lo, this group's share of the features, into the other
                    // S buffer: this thread's own S columns of it, which it has read (last tile's share).  In a unit of one tile
                    // the buffer holds the last unit's D_h instead, which other groups may still be reading at head dim 64.
                    // (columns: quarter k of the features at column 32 k, hi half first)
                    constexpr int FPT = D / 4;              // features per quarter
                    if (D == 64 && cnt == 1 && n >= 1) ok = wait_s(bar_dr, n - 1, 29);
                    ok = ok && wait_s(bar_qf, n, 21) && wait_s(bar_hf, n, 27);
                    if (!ok) break;
#pragma unroll 1
                    for (int k = grp * (4 / C::NG); k < (grp + 1) * (4 / C::NG); ++k) {
                        const uint8_t* qrow = s_gen + C::OFF_Q + (D == 128 ? (k >> 1) * C::SUB_BYTES : 0) + row * 128;
                        const float* zs = reinterpret_cast<const float*>(s_gen + C::OFF_Z) + k * FPT;
                        const uint32_t tA = lane_base + (st ^ 1u) * 128 + k * 32;
                        uint32_t hi[FPT / 2], lo[FPT / 2];
#pragma unroll
                        for (int c = 0; c < FPT / 8; ++c) {
                            const int ch = (D == 128 ? 4 * (k & 1) : 2 * k) + c;           // 16-byte chunk of the row, 128-byte swizzle
                            const uint4 qv = *reinterpret_cast<const uint4*>(qrow + ((ch ^ (row & 7)) << 4));
                            const float4 z0 = *reinterpret_cast<const float4*>(zs + c * 8), z1 = *reinterpret_cast<const float4*>(zs + c * 8 + 4);
                            const float zz[8] = {z0.x, z0.y, z0.z, z0.w, z1.x, z1.y, z1.z, z1.w};
                            const uint32_t ws[4] = {qv.x, qv.y, qv.z, qv.w};
                            float cs[4] = {1.f, 1.f, 1.f, 1.f}, sn[4] = {0.f, 0.f, 0.f, 0.f};
                            if constexpr (HIST == 2) {      // the pairs' angles belong to the query's row
                                const int at = (k * (FPT / 8) + c) * p.Tc + min(q0 + row, p.Tc - 1);
                                const float4 c4 = __ldg(reinterpret_cast<const float4*>(p.cos_q) + at), s4 = __ldg(reinterpret_cast<const float4*>(p.sin_q) + at);
                                cs[0] = c4.x; cs[1] = c4.y; cs[2] = c4.z; cs[3] = c4.w;
                                sn[0] = s4.x; sn[1] = s4.y; sn[2] = s4.z; sn[3] = s4.w;
                            }
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const float2 xq = unpack_bf16(ws[e]);
                                float f0 = phi_elu1(xq.x), f1 = phi_elu1(xq.y);
                                dsum = fmaf(f0, zz[2 * e], fmaf(f1, zz[2 * e + 1], dsum));      // (the denominator is not rotated)
                                if constexpr (HIST == 2) {
                                    const float r0 = fmaf(-f1, sn[e], f0 * cs[e]), r1 = fmaf(f0, sn[e], f1 * cs[e]);
                                    f0 = r0; f1 = r1;
                                }
                                const uint32_t hp = pack_bf16(f0, f1);
                                const float2 hf = unpack_bf16(hp);
                                hi[c * 4 + e] = hp;
                                lo[c * 4 + e] = pack_bf16(f0 - hf.x, f1 - hf.y);
                            }
                        }
                        if constexpr (D == 128) { tmem_st16(tA, hi); tmem_st16(tA + 16, lo); }
                        else { tmem_st8(tA, hi); tmem_st8(tA + 8, lo); }
                    }
                    tmem_wait_st();
                    fence_before_sync();
                    arrive_w(bar_af);
                    arrive_t(bar_qe);
                }
                ok = wait_s(bar_sf + 8 * st, t >> 1, 8);
                if (!ok) break;
                fence_after_sync();
                // ---- this thread's share of the S row in registers
                uint32_t r[C::SCOLS];
#pragma unroll
                for (int c = 0; c < C::SCOLS / 32; ++c) tmem_ld32(lane_base + st * 128 + grp * C::SCOLS + c * 32, *reinterpret_cast<uint32_t(*)[32]>(r + 32 * c));
                tmem_wait_ld();
                // ---- columns of this thread that count: all, or the first nv of a segment (a short block; 0: its row group does not
                // keep the block).  Full and masked segments are separate code: selects on 32 registers in every tile cost 9 us of
                // a 134 us forward.
                constexpr int W = C::SCOLS / EPT;
                int nv[EPT];
#pragma unroll
                for (int x = 0; x < EPT; ++x) {
                    nv[x] = W;
                    if constexpr (BLK == 128) {
                        if ((tails >> (j & 31)) & 1u) nv[0] = p.Tc - (p.n_b - 1) * BLK - col0;
                    } else {
                        const bool kept = (e_cur[x] >> (10 + rg)) & 1u;
                        nv[x] = kept ? (int)((e_cur[x] >> 18) & 127u) - col0 : 0;
                    }
                }
                if (j == 0) {
                    // ---- the reference exponent of the row for the whole unit: the maximum of its first tile plus HEADROOM.  No
                    // running maximum, no rescaling and no exchange between the column groups after this.  P of the first tile is
                    // <= 2^-60; a later tile may rise above the first one by a factor of up to ~2^150 (about 100 natural-log
                    // units) before the row sum passes 2^100, which the end of the unit detects (fp32 overflows at 2^128; rows
                    // that fall below the first tile lose nothing: what flushes to zero is 2^-66 of the largest term).  Floating
                    // point is scale invariant, so the result is the one the exact running maximum gives.
                    float mine = -INFINITY;
#pragma unroll
                    for (int x = 0; x < EPT; ++x) mine = fmaxf(mine, swa_max<W, true>(r + x * W, nv[x]));
                    x_m[grp * 128 + row] = mine;
                    ok = exchange(0, 11);
                    if (!ok) break;
                    float mrow = x_m[row];
#pragma unroll
                    for (int g = 1; g < C::NG; ++g) mrow = fmaxf(mrow, x_m[g * 128 + row]);
                    // rows of a row group past the last query block keep nothing at all: any finite reference will do
                    m_used = mrow == -INFINITY ? 0.f : fmaf(mrow, p.scale_log2, C::HEADROOM);
                    if (grp > 0) {
                        // The exchange has put the two warps that share a scheduler (same rows, different column groups) in step;
                        // they would run their exponentials at the same time and their waits at the same time, and the
                        // special-function unit would idle through the latter.  Set back by part of a tile, one group's waits
                        // fall into the other's exponentials.  Nothing couples the groups until the end of the unit.
                        const long long t_skew = clock64();
                        while (clock64() - t_skew < grp * C::SKEW_CLK) {}
                    }
                }
                // ---- P = exp2(S*c - m), row sum, bf16 pairs, 32 columns at a time
                float2 rsum[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
                auto store_p = [&](int c, const uint32_t (&pk)[16]) {
                    if (c == 0) {                           // S is in registers: its buffer is free (said here, off the critical path)
                        fence_before_sync();
                        arrive_t(bar_se + 8 * st);
                    }
                    if (c == 0 && t >= 1) {                 // its half of the P buffer: the product of the tile before has read it
                        ok = wait_s(bar_own + 8 * ((t - 1) & 1), (t - 1) >> 1, 9);
                        fence_after_sync();
                    }
                    tmem_st16(lane_base + C::COL_P + (C::SCOLS / 2) * grp + 16 * c, pk);
                };
                if constexpr (BLK == 16) {
#pragma unroll
                    for (int c = 0; c < C::SCOLS / 32; ++c) {
                        uint32_t pk[16];
#pragma unroll
                        for (int x = 2 * c; x < 2 * c + 2; ++x) {
                            if (__all_sync(0xffffffffu, nv[x] >= W)) swa_weights<W, false>(r + x * W, W, p.scale_log2, m_used, rsum, pk + (x & 1) * (W / 2));
                            else if (__any_sync(0xffffffffu, nv[x] > 0)) swa_weights<W, true>(r + x * W, nv[x], p.scale_log2, m_used, rsum, pk + (x & 1) * (W / 2));
                            else {
#pragma unroll
                                for (int e = 0; e < W / 2; ++e) pk[(x & 1) * (W / 2) + e] = 0u;
                            }
                        }
                        store_p(c, pk);
                    }
                } else if (nv[0] >= W) {                    // (the same for the whole warp)
#pragma unroll
                    for (int c = 0; c < C::SCOLS / 32; ++c) {
                        uint32_t pk[16];
                        swa_weights<32, false>(r + 32 * c, 32, p.scale_log2, m_used, rsum, pk);
                        store_p(c, pk);
                    }
                } else if (BLK == 128 || nv[0] > 0) {
#pragma unroll
                    for (int c = 0; c < C::SCOLS / 32; ++c) {
                        uint32_t pk[16];
                        swa_weights<32, true>(r + 32 * c, nv[0] - 32 * c, p.scale_log2, m_used, rsum, pk);
                        store_p(c, pk);
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < C::SCOLS / 32; ++c) {
                        uint32_t pk[16];
#pragma unroll
                        for (int e = 0; e < 16; ++e) pk[e] = 0u;
                        store_p(c, pk);
                    }
                }
                if (!ok) break;
                l_run += ((rsum[0].x + rsum[0].y) + (rsum[1].x + rsum[1].y)) + ((rsum[2].x + rsum[2].y) + (rsum[3].x + rsum[3].y));
                tmem_wait_st();
                fence_before_sync();
                arrive_t(bar_pf + 8 * half);
                if (HIST && n >= 1 && j == 0 && cnt > 1) release_h();
            }
            if (!ok) break;
            // (a thread block that leaves room beside it lets the next kernel in only now: that one waits, but its blocks take slots)
            if (C::SMEM_BYTES <= 200 * 1024 && n + 1 == my_units) pdl_trigger();
            // ---- end of the unit: row sums (and the shares of Eq. 4's denominator) of the column groups, range test, output
            const bf16* bias_row = (HIST && p.bias) ? p.bias + (size_t)(bh % p.heads) * D + grp * C::OCOLS : nullptr;
            uint4 bw[C::OCOLS / 8];
#pragma unroll
            for (int c = 0; c < C::OCOLS / 8; ++c) bw[c] = bias_row ? __ldg(reinterpret_cast<const uint4*>(bias_row) + c) : make_uint4(0, 0, 0, 0);
            if constexpr (HIST) {
                ok = wait_s(bar_ud, n, 19);                 // D_h complete: the buffer of S W^T is free
                if (!ok) break;
                x_d[grp * 128 + row] = dsum;
            }
            x_l[grp * 128 + row] = l_run;
            ok = exchange(1, 12);
            if (!ok) break;
            l_run = x_l[row];
            float den = HIST ? x_d[row] : 0.f;
#pragma unroll
            for (int g = 1; g < C::NG; ++g) { l_run += x_l[g * 128 + row]; if constexpr (HIST) den += x_d[g * 128 + row]; }
            const float inv = 1.f / l_run, inv_den = 1.f / (p.eps + den);
            const size_t g_row = (size_t)bh * p.Tc + q0 + row;
            if (grp == 0 && row < nq && p.lse) p.lse[g_row] = (m_used + log2f(l_run)) * 0.6931471805599453f;
            const uint32_t tl = t - 1;                      // the unit's last tile
            ok = wait_s(bar_pv + 8 * (tl & 1), tl >> 1, 10);
            if (!ok) break;
            fence_after_sync();
            // overflow (or NaN): a later tile rose too far above the first one.  (After the wait: P V of this unit's last tile
            // needed every warp, so all of them have listed the unit before this one.)
            if (!(l_run < 1e30f)) note_redo(n);
            // Output through shared memory and one bulk tensor store per warp (32 rows x its group's columns):
            // row-per-thread global stores would touch 32 lines per instruction.  The staging tile is the S W^T buffer (free: the
            // history products have completed, or were never asked for); in the map's swizzle of the row width.
            const uint32_t stage_off = C::OFF_H + warp * (32 * C::OCOLS * 2);
            uint8_t* stage = s_gen + stage_off + lane * (C::OCOLS * 2);
            const int swz = C::OCOLS == 64 ? lane & 7 : C::OCOLS == 32 ? (lane >> 1) & 3 : (lane >> 2) & 1;
            if (!HIST && n >= 1) {
                if (lane == 0) bulk_wait_read();            // this warp's previous store has read its part
                __syncwarp();
            }
#pragma unroll
            for (int c = 0; c < C::OCOLS / 16; ++c) {
                uint32_t o[16], dh[16];
                tmem_ld16(lane_base + C::COL_O + grp * C::OCOLS + c * 16, o);
                if constexpr (HIST) tmem_ld16(lane_base + (tl & 1) * 128 + grp * C::OCOLS + c * 16, dh);
                tmem_wait_ld();
                if (c == C::OCOLS / 16 - 1) {
                    // The next unit's first P V overwrites O.  It needs the lower half of P of that tile from all warps of the lower half
                    // of the groups, each of which first meets the warps of its rows in ALL groups in the exchange of the maxima: all
                    // of them are past these loads then.
                    fence_before_sync();
                    if constexpr (HIST) arrive_t(bar_dr);
                }
                const float* hsrc = !HIST && p.hist ? p.hist + g_row * D + grp * C::OCOLS + c * 16 : nullptr;
#pragma unroll
                for (int v = 0; v < 2; ++v) {
                    float x[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) x[e] = __uint_as_float(o[v * 8 + e]) * inv;
                    if constexpr (HIST) {
#pragma unroll
                        for (int e = 0; e < 8; ++e) x[e] = fmaf(__uint_as_float(dh[v * 8 + e]), inv_den, x[e]);
                        // Eq. 4's Linear: its matrix is folded into the state, its bias is added here
                        const uint4 b = bw[c * 2 + v];
                        const float2 b0 = unpack_bf16(b.x), b1 = unpack_bf16(b.y), b2 = unpack_bf16(b.z), b3 = unpack_bf16(b.w);
                        x[0] += b0.x; x[1] += b0.y; x[2] += b1.x; x[3] += b1.y;
                        x[4] += b2.x; x[5] += b2.y; x[6] += b3.x; x[7] += b3.y;
                    } else if (hsrc && row < nq) {
                        const float4 h0 = *reinterpret_cast<const float4*>(hsrc + v * 8);
                        const float4 h1 = *reinterpret_cast<const float4*>(hsrc + v * 8 + 4);
                        x[0] += h0.x; x[1] += h0.y; x[2] += h0.z; x[3] += h0.w;
                        x[4] += h1.x; x[5] += h1.y; x[6] += h1.z; x[7] += h1.w;
                    }
                    uint4 w;
                    w.x = pack_bf16(x[0], x[1]); w.y = pack_bf16(x[2], x[3]);
                    w.z = pack_bf16(x[4], x[5]); w.w = pack_bf16(x[6], x[7]);
                    *reinterpret_cast<uint4*>(stage + (((c * 2 + v) ^ swz) << 4)) = w;
                }
            }
            fence_proxy_async();
            __syncwarp();
            if (lane == 0 && q0 + (warp & 3) * 32 < p.Tc) {     // rows past the chunk's end are clipped by the map
                tma_store_4d(&tm_o, s_base + stage_off, grp * C::OCOLS, q0 + (warp & 3) * 32, bh, 0);
                bulk_commit();
            }
            u += gridDim.x; bh += dbh; i += di;
            if (i >= p.upb) { i -= p.upb; ++bh; }
        }
    }
    if (warp < C::NSW && lane == 0) bulk_wait_read();    // output tiles still on their way out of shared memory
    fence_before_sync();
    __syncthreads();
    if (warp == C::WARP_S) {
        fence_after_sync();
        tmem_dealloc(tmem, C::TMEM_COLS);
    }
    // ---- second pass (rare): the listed units again, with the running maximum.  Every copy and tensor-core operation
    // of the tile stream has completed (the roles above drain before the barrier), so shared memory is free.
    // Its rows have also been handed to bulk stores, which must not land behind its own: every warp that issued some (a bulk store
    // belongs to the thread that issued it) waits until they are complete, before a barrier that all threads of the pass are behind.
    const int n_redo = *redo_cnt;
    if (n_redo > 0 && *abort_flag == 0) {                     // (the same for all threads)
        if (warp < C::NSW && lane == 0) bulk_wait_all();
        __syncthreads();
        if (threadIdx.x >= 256) return;
        fence_proxy_async();
        const int total = n_redo > C::REDO_CAP ? my_units : n_redo;
        for (int r = 0; r < total; ++r) {
            const int n = n_redo > C::REDO_CAP ? r : redo_list[r];
            swa_redo_unit<D, BLK, HIST>(s_gen, p, (int)blockIdx.x + n * (int)gridDim.x);
        }
    }
}
