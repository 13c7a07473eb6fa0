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
// Roles (12 warps with column groups, 20 with teams):
//   softmax warps       Column groups: two of four warps; thread (group g, row r) owns columns 64 g .. 64 g + 63 of S of row r (TMEM lane = row) in every
//                       tile and D / 2 columns of O.  Teams: two of eight warps, tiles t = team, team + 2, ...; a team's two halves own 32 columns of
//                       either half of the tile each.  A thread takes its share of S into registers (the S buffer is free from then on), forms
//                       P = exp2(S c - m) and writes it as bf16 to a P buffer.
//   K loader, V loader  TMA: K tiles and V tiles (rings of two, of four at head dim 64), Q, and for HIST the folded state S W^T and z
//   S warp, P V warp    tcgen05.mma issue, one warp per product.
//       S_t = Q K_t^T      A = Q (tensor memory; a unit's first tile: shared memory), B = K_t (smem, K-major, 128B swizzle) -> S buffer t & 1
//       O  += P_t V_t      A = P (tensor memory), B = V_t (smem, MN-major, 128B swizzle)      -> O, in two halves of 64 keys
//       D_h = phi(Q) S W^T three products of bf16 hi / lo halves (HIST)                       -> S buffer of the unit's last tile
//
// Teams or column groups.  A softmax warp's way through a tile is exponentials (8 clk a warp instruction and scheduler) and about 600 clk of
// waits, tensor-memory loads and stores and arrivals.  With column groups every warp pays the latter in every tile: 1 640-1 830 clk
// a tile at head dim 128 with the special-function unit at 56-62 %.  A team pays them in every other one and has two tiles' time for it, four
// warps on a scheduler cover each other, and no warp of one team waits for the other inside a unit: 1 380-1 450 clk a tile.  A P half of 64
// keys is written by both halves of a team, so that its product starts in the middle of the tile (with 64 columns in a row for each
// half it started at the end, and where there is one P buffer the other team waited for it: 1 770 clk).  At a unit's end one team forms phi(Q)
// while the other has the last tile; that one writes the output while the first has gone on to the next unit's first tile.  Twenty warps leave 96 registers a
// thread; what is spilt lies outside the tile loop (132 units, 20 and 40 tiles alike: 52 loads and 40 to 80 stores of local memory a thread block).  Forward calls, two
// column groups (head dim 64 from five tiles on: four) / teams, us:
//   head dim 128, 128-token blocks, 444 units of 28 tiles 125.7 / 121.8 (at the power limit), 1 776 units of 130 tiles 1 929 / 1 770; 132 units
//   of 20 tiles 31.3 / 29.7, of 40 tiles 49.9 / 44.6; 320 units of 20 tiles 79.8 / 76.7, of 40 tiles 134.1 / 122.7
//   head dim 64, 128-token blocks, 132 units of 8, 20, 40 tiles 16.4 / 16.2, 26.4 / 25.4, 43.3 / 39.4; 320 units of 1, 8, 40 tiles
//   20.7 / 19.1, 35.8 / 33.7, 113.5 / 103.8; 64-token blocks, 320 units of 10 and 25 kept blocks 41.3 / 37.5, 60.1 / 53.2; 16-token blocks, 12 units
//   of 4 and 40 kept blocks 14.9 / 14.7, 23.9 / 22.2
// At head dim 128 the phi(Q) operand has to wait in an S buffer and a unit's ends weigh more than column groups' (all warps share them): those stay
// for short lists (swa_teams, hf_dispatch.h) and for blocks of 16 and 64 tokens (their masked segments leave the tensor pipe the bound:
// 64-token blocks, 12 heads, 4 680 queries 158 / 163 us, 16-token blocks 43 / 44).
//
// The first unit ahead.  A thread block waits for the lists for 2 us and more after it is resident (launched under the selection's tail), and q, the folded
// state and z are there all the while.  Column groups form their first unit's history term in that time (form_ahead; AHEAD): the chain behind
// the unit's last tile is shorter by phi(Q) and the products.  Where this pays: swa_history_ahead (hf_dispatch.h); 16 forwards of 8 heads of 128, 300 queries and
// their commit 242.6 -> 228.5 us.  With teams the same code cost the tile loop more registers than it had (132 units of 40 tiles 44.9 -> 47.2 us): not there.
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
//     every tile: +9 us of a 134 us forward).
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
#include "hf_dispatch.h"

template <int D, bool TEAMED>
struct SwaTc5 {
    static constexpr int NSW = TEAMED ? 16 : 8;        // softmax warps: two teams of two halves, or two column groups; four warps each
    static constexpr int OCOLS = D / 2;                // O columns per softmax warp
    static constexpr int SUB = D / 64;                 // 64-column (128-byte) sub-tiles per operand tile
    static constexpr int SUB_BYTES = 128 * 128;        // 16 KB
    static constexpr int TILE_BYTES = SUB * SUB_BYTES;
    static constexpr int HSUB_BYTES = D * 128;         // S W^T halves: D rows of 64-column sub-tiles
    static constexpr int H_BYTES = SUB * HSUB_BYTES;
    static constexpr float HEADROOM = 60.f;           // log2 distance of the softmax reference above the first tile's row maximum
    // Tensor memory: two S buffers (teams: one each), P (a buffer per team at head dim 64; at 128 there is room for one), Q, O.  The halves of a P
    // buffer (keys 0..63, 64..127) are products and barriers of their own.
    static constexpr int PBUF = D == 64 ? 2 : 1;
    // The phi(Q) operand of the history products (D columns): in the P buffer of the team that forms it where there are two, else in that
    // team's S buffer, where the next unit's first S has to wait for the products.
    static constexpr bool A_IN_P = PBUF == 2;
    static_assert(!TEAMED || A_IN_P || !swa_teams(D, 128, 1, true), "a unit of one tile would have its operand where the unit before has D_h");
    static constexpr int COL_P = 256, COL_Q = COL_P + 64 * PBUF, COL_O = COL_Q + D / 2, TMEM_COLS = 512;
    static_assert(COL_O + D <= TMEM_COLS, "tensor memory layout");
    static constexpr int KV_LOG = D == 64 ? 2 : 1, KV = 1 << KV_LOG;   // stages of the K and of the V ring
    static constexpr int OFF_Q = 0, OFF_K = TILE_BYTES, OFF_V = OFF_K + KV * TILE_BYTES;
    static constexpr int OFF_H = OFF_V + KV * TILE_BYTES;       // S W^T, hi then lo; also the staging tile of the output (teams without a history term: one each)
    static constexpr int END_H = OFF_H + (H_BYTES > TILE_BYTES ? 2 * H_BYTES : 2 * TILE_BYTES);
    // D_h of a thread block's first unit, formed ahead of the tiles (column groups), in place of S W^T: fp32 [OCOLS][32 rows] for each warp
    static constexpr int DH_WARP = OCOLS * 32 * 4;
    static_assert(TEAMED || OFF_H + 8 * DH_WARP <= END_H, "buffers of the history term");
    // (the second pass keeps its fp32 history tile behind the operand tiles of swa_mma_unit, in front of the barriers)
    static constexpr int END_REDO = SwaMma<128, D>::SMEM_BYTES + 128 * D * 4;
    static constexpr int OFF_BAR = END_H > END_REDO ? END_H : END_REDO;
    // units whose rows left the range of the fixed reference: count, last unit listed, up to REDO_CAP local unit numbers
    // (more than that: every unit of the thread block is computed again)
    static constexpr int OFF_REDO = OFF_BAR + 384 + (KV > 2 ? 128 : 0), REDO_CAP = 8;
    static constexpr int OFF_Z = OFF_REDO + 64;        // z [D] of the unit's head
    static_assert((2 + REDO_CAP) * 4 <= OFF_Z - OFF_REDO, "the list must fit");
    static constexpr int OFF_XM = OFF_Z + 512;         // row maxima of the two halves of a unit's first tile [2][128]
    static constexpr int OFF_XL = OFF_XM + 1024;       // one team's row sums [128] and Eq. 4's denominators [128], for the other
    static constexpr int USED_BYTES = OFF_XL + 1024;
    // row sums of the halves of the team that writes the output [2][128]: behind the staging tile; without a history term, which leaves
    // that to the other team's output, in the places of z and of the denominators
    __host__ __device__ static constexpr int off_xy(bool hist, int half) { return hist ? OFF_H + TILE_BYTES + 512 * half : half ? OFF_XL + 512 : OFF_Z; }
    static_assert(OFF_H + TILE_BYTES + 2048 <= OFF_BAR, "exchange buffers");
    static constexpr int MAX_SMEM = 232448;            // 227 KB: the most one thread block can have
    // The window of a kernel without static shared memory starts on a 1 KB boundary, as the operand tiles have to (the kernel checks it, with what slack there
    // is: 64 bytes at head dim 128).  With a static array it would not, but then the runtime refuses MAX_SMEM, and hf_create fails with its error.
    // More than half an SM's shared memory, so that one CTA owns the SM (it allocates all 512 TMEM columns).
    static constexpr int WANT_BYTES = (USED_BYTES + 1024) > 120 * 1024 ? (USED_BYTES + 1024) : 120 * 1024;
    static constexpr int SMEM_BYTES = WANT_BYTES < MAX_SMEM ? WANT_BYTES : MAX_SMEM;
    static_assert(USED_BYTES <= MAX_SMEM && (SMEM_BYTES == MAX_SMEM || SMEM_BYTES >= USED_BYTES + 1024), "shared memory layout does not fit");
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
        static_assert(M::SMEM_BYTES + ROWS * D * 4 <= SwaTc5<D, false>::OFF_BAR, "history tile must fit");
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
// AHEAD (column groups with a history term): the first unit's is formed ahead of the wait for the kernel before this one; q has to be older than that
// one (code of its own: as a branch it cost the other calls 2 %).
template <int D, int BLK, int HIST, bool TEAMED, bool AHEAD>
__global__ void __launch_bounds__(SwaTc5<D, TEAMED>::THREADS, 1)
k_swa_tc5(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_kring,
          const __grid_constant__ CUtensorMap tm_vring, const __grid_constant__ CUtensorMap tm_kcur,
          const __grid_constant__ CUtensorMap tm_vcur, const __grid_constant__ CUtensorMap tm_sh,
          const __grid_constant__ CUtensorMap tm_sl, const __grid_constant__ CUtensorMap tm_o,
          const __grid_constant__ Tc5Params p) {
    using namespace tc5;
    typedef SwaTc5<D, TEAMED> C;
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
    const uint32_t bar_kf = bar0 + (C::KV > 2 ? 368 : 0), bar_vf = bar0 + (C::KV > 2 ? 400 : 16),     // K / V tile t landed
                   bar_sf = bar0 + 32,                     // S_t complete
                   bar_se = bar0 + 48,                     // S_t is in its team's registers
                   bar_ph = bar0 + 64,                     // P V of tile t complete, first half
                   bar_pv = bar0 + 80,                     // ... second half
                   // the K / V stage of tile t is free: with two stages, S_t and P V of tile t complete
                   bar_ke = C::KV > 2 ? bar0 + 432 : bar_sf, bar_ve = C::KV > 2 ? bar0 + 464 : bar_pv,
                   bar_pf = bar0 + 96,                     // two per P buffer: a half of P_t written; completion t (two P buffers: t >> 1)
                   // unit n: Q landed / copied to tensor memory
                   bar_qf = bar0 + 128, bar_qe = bar0 + 136,
                   bar_hf = bar0 + 144, bar_he = bar0 + 152,   // unit n: S W^T and z landed / free
                   bar_af = bar0 + 160,                    // unit n: phi(Q) operand written
                   bar_ud = bar0 + 168,                    // unit n: history products complete
                   bar_drain = bar0 + 184,                 // two: each MMA warp's last operations complete
                   bar_x = bar0 + 200,                     // four (32 rows each), unit n: one team's sums for the other's epilogue
                   bar_m = bar0 + 232,                     // four, unit n: row maxima of its first tile written
                   bar_mr = bar0 + 264,                    // four, unit n: ... and read by all four warps of the rows
                   bar_h = bar0 + 296,                     // four, unit n: the upper half's sums for the lower half of the same team
                   bar_y = bar0 + 328;                     // four, unit n: the halves of the team that writes the output meet
    // unit n: O, D_h and the other team's sums read by the epilogue (two barriers, completion n >> 1: a head-dim-64 unit of one tile may be
    // through before the next one's first S asks for the unit in front of it)
    auto bar_dr = [&](int n) -> uint32_t { return bar0 + ((n & 1) ? (C::KV > 2 ? 496 : 368) : 176); };
    const uint32_t bar_d0 = bar0 + (C::KV > 2 ? 504 : 376);     // the first unit's D_h, formed ahead, has been read from O's columns
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(s_gen + C::OFF_BAR + 360);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(s_gen + C::OFF_BAR + 364);
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
            mbar_init(bar_sf + 8 * s, 1); mbar_init(bar_se + 8 * s, 8);
            mbar_init(bar_ph + 8 * s, 1); mbar_init(bar_pv + 8 * s, 1); mbar_init(bar_drain + 8 * s, 1);
        }
        for (int s = 0; s < C::KV; ++s) {
            mbar_init(bar_kf + 8 * s, 1); mbar_init(bar_vf + 8 * s, 1);
            if (C::KV > 2) { mbar_init(bar_ke + 8 * s, 1); mbar_init(bar_ve + 8 * s, 1); }
        }
        for (int s = 0; s < 4; ++s) {
            mbar_init(bar_pf + 8 * s, TEAMED ? 8 : 4); mbar_init(bar_x + 8 * s, TEAMED ? 1 : 2); mbar_init(bar_m + 8 * s, 2); mbar_init(bar_mr + 8 * s, 4);
            mbar_init(bar_h + 8 * s, 1); mbar_init(bar_y + 8 * s, 2);
        }
        mbar_init(bar_qf, 1); mbar_init(bar_qe, HIST && !TEAMED ? 9 : 1); mbar_init(bar_hf, 1); mbar_init(bar_he, 8);
        mbar_init(bar_af, 8); mbar_init(bar_ud, 1); mbar_init(bar_dr(0), 8); mbar_init(bar_dr(1), 8); mbar_init(bar_d0, 8);
        *abort_flag = 0;
        *redo_cnt = 0; *redo_last = -1;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    static_assert(!AHEAD || (HIST && !TEAMED), "column groups form a history term ahead");
    constexpr bool early = AHEAD;
    float* x_den = reinterpret_cast<float*>(s_gen + C::OFF_XL) + 128;      // ... its denominators [128]
    if (early && threadIdx.x < 128) x_den[threadIdx.x] = 0.f;
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
    // Everything above (barriers, tensor memory), and the first unit's history term, may overlap the tail of the kernel before this one in
    // the stream when the launch allows it: every role waits for that kernel itself, before it reads the lists that one wrote.

    auto wait_w = [&](uint32_t bar, uint32_t parity, int where) -> bool {      // a warp's wait, warp-uniform result
        return mbar_wait_warp<true>(bar, parity & 1u, abort_flag, p.dev_status, where);
    };

    if (warp == C::WARP_LOAD_K || warp == C::WARP_LOAD_V) {
        // ================================================================= TMA producers
        // One lane copies a tile of a 128-token block; blocks of 16 or 64 tokens have a lane each (G boxes a tile: one after the other, with
        // their list entries' loads between them, they bounded the tile loop: 16-token blocks, 12 heads, 1 300 queries, 62 of 246 blocks
        // kept 53 -> 32.5 us at head dim 64, 69 -> 41 at 128).  The loops are the warp's.
        const bool is_k = (warp == C::WARP_LOAD_K);
        auto load_h = [&](int bh) {                             // folded state and z of a head
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
        };
        const int box = lane < G ? lane : 0;
        bool ok = true;
        int t = 0;
        const int Tn = p.Tn;
        const uint32_t tiles = is_k ? sK : sV, full = is_k ? bar_kf : bar_vf, freed = is_k ? bar_ke : bar_ve;
        auto list_of = [&](int u) -> const uint32_t* {
            if constexpr (BLK == 128) return reinterpret_cast<const uint32_t*>(p.idx + (size_t)u * p.keep);
            else return p.entries + (size_t)u * p.max_tiles * G + box;
        };
        auto load_q = [&](int n) {
            const int u = blockIdx.x + n * gridDim.x, bh = u / p.upb, i = u - bh * p.upb;
            if (lane == 0) {
                mbar_expect_tx(bar_qf, C::TILE_BYTES);
#pragma unroll
                for (int s = 0; s < C::SUB; ++s) tma_load_4d(sQ + s * C::SUB_BYTES, &tm_q, s * 64, i * 128, bh, 0, bar_qf);
            }
            __syncwarp();
        };
        if (!is_k && early) { load_q(0); load_h(blockIdx.x / p.upb); }
        pdl_wait();
        // The next kernel in the stream may be made resident on SMs this grid has left (it waits itself) -- only where a thread
        // block of this kernel takes all of an SM's shared memory, so that no waiting block of the dependent grid ever sits
        // beside a working block of this one.
        if (is_k && C::SMEM_BYTES > 200 * 1024) pdl_trigger();
        uint32_t e_next = my_units > 0 ? __ldg(list_of(blockIdx.x)) : 0u;      // list entry, read one tile ahead
        for (int n = 0; ok && n < my_units; ++n) {
            const int u = blockIdx.x + n * gridDim.x;
            const int bh = u / p.upb;
            const int cnt = tiles_of(n);
            if (!is_k && n == 0 && !early) load_q(0);
           const uint32_t* list = list_of(u);
            for (int j = 0; j < cnt; ++j, ++t) {
                const uint32_t st = t & (C::KV - 1), dst = tiles + st * C::TILE_BYTES + box * BLK * 128, bar = full + 8 * st;
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
                if (t >= C::KV && !(ok = wait_w(freed + 8 * st, (t >> C::KV_LOG) - 1, 2))) break;
                if (lane == 0) mbar_expect_tx(bar, C::TILE_BYTES);
                __syncwarp();
                if (lane < G) {
#pragma unroll
                    for (int s = 0; s < C::SUB; ++s) tma_load_4d(dst + s * C::SUB_BYTES, m, s * 64, jb * BLK, bh, slot, bar);
                }
                __syncwarp();
                if (HIST && !is_k && !(early && n == 0) && j == (cnt >= C::KV ? C::KV - 1 : cnt - 1)) {
                    // For the history term at the unit's end: the head's folded state and z.  The buffer is free once the
                    // previous unit's output, which was staged in it, has been read by the bulk stores.  (Two V tiles of
                    // this unit are on their way by now; the third needs P V of the first, which comes after that.)
                    if (n >= 1 && !(ok = wait_w(bar_he, n - 1, 13))) break;
                    load_h(bh);
                }
                // The next unit's Q, once this unit's is in tensor memory
                if (!is_k && n + 1 < my_units && j == (cnt > C::KV && !(HIST && !TEAMED) ? C::KV : cnt - 1)) {
                    if (!(ok = wait_w(bar_qe, n, 1))) break;
                    load_q(n + 1);
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
        const uint32_t q_lo = (uint32_t)dq0, k_lo = (uint32_t)dk0, k_hi = (uint32_t)(dk0 >> 32);
        bool ok = true;
        int x = 0, cnt_prev = 0;
        auto copy_q = [&] {                                 // the unit's Q from shared to tensor memory
            fence_after_sync();
            if (elect_one()) {
#pragma unroll
                for (int ks = 0; ks < D / 16; ++ks)         // 16 features = 32 bytes of a row = 8 columns
                    tmem_cp_128x256b(tmem + C::COL_Q + 8 * ks, dq0 + (uint64_t)((ks >> 2) * (C::SUB_BYTES >> 4) + (ks & 3) * 2));
                mma_commit(bar_qe);
            }
            __syncwarp();
        };
        if (early && (ok = wait_w(bar_qf, 0, 4))) copy_q();
        pdl_wait();
        for (int n = 0; ok && n < my_units; ++n) {
            const int cnt = tiles_of(n);
            for (int j = 0; j < cnt; ++j, ++x) {
                const uint32_t st = x & 1, kv = x & (C::KV - 1);
                if (j == 0 && !(ok = wait_w(bar_qf, n, 4))) break;
                if (!(ok = wait_w(bar_kf + 8 * kv, x >> C::KV_LOG, 5))) break;
                // The S buffer: free once the softmax warps hold S of two tiles ago in registers.  HIST: the buffer of a unit's last tile holds
                // its D_h afterwards, and (head dim 128) the other one its phi(Q) operand; the first unit's, formed ahead, was in the second buffer.
                if (HIST && n >= 1 && j == 1) { if (!(ok = wait_w(bar_dr(n - 1), (n - 1) >> 1, 30))) break; }
                else if (HIST && !C::A_IN_P && n >= 1 && j == 0 && !(early && n == 1)) { if (!(ok = wait_w(bar_ud, n - 1, 23))) break; }
                else if (HIST && C::A_IN_P && n >= 2 && j == 0 && cnt_prev == 1) { if (!(ok = wait_w(bar_dr(n - 2), (n - 2) >> 1, 35))) break; }
                else if (x >= 2) { if (!(ok = wait_w(bar_se + 8 * st, (x >> 1) - 1, 25))) break; }
                else if (early && x == 1) { if (!(ok = wait_w(bar_ud, 0, 40))) break; }
                fence_after_sync();
                if (elect_one()) {
                    // a unit's first product takes Q from shared memory (unless it is in tensor memory already), the others from tensor memory
                    if (j == 0 && !(early && n == 0)) mma_ss_tile<D>(tmem + st * 128, q_lo, k_lo + kv * TILE_STEP, k_hi, IDESC_S);
                    else mma_ts_kmajor<D>(tmem + st * 128, tmem + C::COL_Q, k_lo + kv * TILE_STEP, k_hi, IDESC_S);
                    mma_commit(bar_sf + 8 * st);
                    if (C::KV > 2) mma_commit(bar_ke + 8 * kv);
                }
                __syncwarp();
                if (j == 0 && !(early && n == 0)) {
                    // Q moves to tensor memory once the previous unit's last product, and its phi pass, have read what is there
                    if (n >= 1 && !(ok = wait_w(bar_sf + 8 * ((x - 1) & 1), (x - 1) >> 1, 22))) break;
                    if (HIST && C::A_IN_P && n >= 1 && !(ok = wait_w(bar_af, n - 1, 36))) break;
                    copy_q();
                }
            }
            cnt_prev = cnt;
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
        // D_h = phi(Q) S W^T: A in quarters of the features (quarter k at column 32 k, hi half first; in a P buffer all of hi, then all of lo), B = the hi
        // and lo tiles of S W^T; three products, the lo x lo one is below fp32 resolution
        auto history = [&](uint32_t tD, uint32_t tA) {
            fence_after_sync();
            if (elect_one()) {
                if constexpr (C::A_IN_P) {
                    mma_ts_half(tD, tA, h_lo, h_hi, IDESC_PV, false);                  // hi x hi
                    mma_ts_half(tD, tA + D / 2, h_lo, h_hi, IDESC_PV, true);           // lo x hi
                    mma_ts_half(tD, tA, h_lo + H_STEP, h_hi, IDESC_PV, true);          // hi x lo
                } else {
                    mma_ts_groups<D>(tD, tA, h_lo, h_hi, IDESC_PV, false);
                    mma_ts_groups<D>(tD, tA + D / 8, h_lo, h_hi, IDESC_PV, true);
                    mma_ts_groups<D>(tD, tA, h_lo + H_STEP, h_hi, IDESC_PV, true);
                }
                mma_commit(bar_ud);
            }
            __syncwarp();
        };
        bool ok = true;
        int t = 0;
        if (early && (ok = wait_w(bar_hf, 0, 14) && wait_w(bar_af, 0, 15)))
            history(tO, tmem + 128);
        pdl_wait();
        for (int n = 0; ok && n < my_units; ++n) {
            const int cnt = tiles_of(n);
            for (int j = 0; j < cnt; ++j, ++t) {
                const uint32_t st = t & 1, kv = t & (C::KV - 1);
                // while the softmax warps work on the unit's last tile: into that tile's S buffer (already in registers), A from the other
                if (HIST && j == cnt - 1 && !(early && n == 0)) {
                    ok = wait_w(bar_hf, n, 14) && wait_w(bar_af, n, 15) && wait_w(bar_se + 8 * st, t >> 1, 26);
                    if (!ok) break;
                    history(tmem + st * 128, C::A_IN_P ? tmem + C::COL_P + 64 * (st ^ 1u) : tmem + (st ^ 1u) * 128);
                }
                if (early && t == 0 && !(ok = wait_w(bar_d0, 0, 41))) break;            // O: the first unit's D_h has been read
                if (TEAMED && n >= 1 && j == 0 && !(ok = wait_w(bar_dr(n - 1), (n - 1) >> 1, 24))) break;     // O: the previous unit's has been read
                if (!(ok = wait_w(bar_vf + 8 * kv, t >> C::KV_LOG, 7))) break;
                const uint32_t pb = C::PBUF == 2 ? st : 0u, p_par = C::PBUF == 2 ? t >> 1 : t;
                if (!(ok = wait_w(bar_pf + 16 * pb, p_par, 6))) break;
                fence_after_sync();
                if (elect_one()) {
                    mma_ts_half(tO, tmem + C::COL_P + 64 * pb, v_lo + kv * TILE_STEP, v_hi, IDESC_PV, j > 0);
                    mma_commit(bar_ph + 8 * st);
                }
                __syncwarp();
                if (!(ok = wait_w(bar_pf + 16 * pb + 8, p_par, 28))) break;
                fence_after_sync();
                if (elect_one()) {
                    mma_ts_half(tO, tmem + C::COL_P + 64 * pb + 32, v_lo + kv * TILE_STEP + (64 * 128 >> 4), v_hi, IDESC_PV, true);
                    mma_commit(bar_pv + 8 * st);
                    if (C::KV > 2) mma_commit(bar_ve + 8 * kv);
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
        // Teams: the team's tiles are t = team, team + 2, ...; the half's columns of a tile 32 half + [0, 32) and 64 on.  Column groups (half):
        // every tile, columns 64 half + [0, 64).
        const int team = TEAMED ? warp >> 3 : 0, half = (warp >> 2) & 1, wq = warp & 3;
        const int row = wq * 32 + lane;                     // query row of the unit = TMEM lane
        const int rg = row / BLK;                           // row group (query block within the unit)
        const uint32_t lane_base = tmem + ((uint32_t)(wq * 32) << 16);
        const uint32_t tS = lane_base + 128 * team, pb = C::PBUF == 2 ? team : 0, tP = lane_base + C::COL_P + 64 * pb;
        constexpr int EPT = BLK == 128 ? 1 : BLK == 64 ? (TEAMED ? 2 : 1) : 4;     // list entries (key blocks) under the warp's columns
        float* x_m = reinterpret_cast<float*>(s_gen + C::OFF_XM);
        const bool ragged = p.Tc % BLK != 0;                // every chunk's last block is short
        bool ok = true;
        auto wait_s = [&](uint32_t bar, uint32_t parity, int where) -> bool {
            return mbar_wait_warp(bar, parity & 1u, abort_flag, p.dev_status, where);
        };
        // One arrival per warp.  (Tensor-memory loads and stores are warp instructions, complete for all lanes after the warp's
        // wait: only hand-overs of shared memory need the __syncwarp.)
        const bool lane0 = lane == 0;
        auto arrive_t = [&](uint32_t bar) { mbar_arrive_if(bar, lane0); };
        auto arrive_w = [&](uint32_t bar) { __syncwarp(); mbar_arrive_if(bar, lane0); };
        auto note_redo = [&](int n) {                       // list unit n once
            if (atomicMax(redo_last, n) < n) {
                const int slot = atomicAdd(redo_cnt, 1);
                if (slot < C::REDO_CAP) redo_list[slot] = n;
            }
        };
        // (batch*head, position) of a unit without a division per unit; the tile count and the first list entries of the next
        // unit are read during the current one
        const int dbh = gridDim.x / p.upb, di = gridDim.x - dbh * p.upb;
        int u = blockIdx.x, bh = u / p.upb, i = u - bh * p.upb;
        // BLK 16, 64: list entries of the next tile.  BLK 128: all that matters here is whether a tile is a chunk's short last
        // block; one bit per tile from a ballot over 32 list entries at a time (lane = entry), read one window ahead.  An entry
        // outside [0, T_n) is block 0 here as for the loader, which reports it.
        auto entries_of = [&](int unit) -> const uint32_t* {
            if constexpr (BLK == 128) return reinterpret_cast<const uint32_t*>(p.idx + (size_t)unit * p.keep);
            else return p.entries + (size_t)unit * p.max_tiles * G;
        };
        uint32_t e_next[EPT], tails = 0;
#pragma unroll
        for (int x = 0; x < EPT; ++x) e_next[x] = 0u;
        auto read_entries = [&](const uint32_t* src) {
            if constexpr (BLK == 16) {
                const uint2* src2 = reinterpret_cast<const uint2*>(src) + (TEAMED ? half : 2 * half);
                const uint2 a = __ldg(src2), b = __ldg(src2 + (TEAMED ? 2 : 1));
                e_next[0] = a.x; e_next[1] = a.y; e_next[2] = b.x; e_next[3] = b.y;
            } else if constexpr (BLK == 64 && TEAMED) {
                const uint2 a = __ldg(reinterpret_cast<const uint2*>(src));
                e_next[0] = a.x; e_next[1] = a.y;
            } else if constexpr (BLK == 64) e_next[0] = __ldg(src + half);
        };
        auto first_entries = [&](int unit, int pj, int cnt) {      // of a unit: its first window, or the team's first tile
            if constexpr (BLK == 128) { if (ragged && lane < p.keep) e_next[0] = __ldg(entries_of(unit) + lane); }
            else if (pj < cnt) read_entries(entries_of(unit) + pj * G);
        };
        bool staged = false;                                // this warp's last output is on its way out of shared memory
        // The previous unit's output was staged where S W^T lives: the loader may refill it, and z, once every warp's bulk store has read
        // its part.  (Said after the warp's next tile, when the store has long done so, or before its phi pass.)
        auto release_h = [&] {
            if (HIST && staged) {
                if (lane == 0) bulk_wait_read();
                arrive_w(bar_he);
                staged = false;
            }
        };
        // one bit per tile of the window of 32 that starts at tile j: the short last block of a chunk
        auto next_tails = [&](const uint32_t* ent, int j, int cnt) {
            const uint32_t x1 = (e_next[0] < (uint32_t)p.Tn ? e_next[0] : 0u) + 1u;     // last block of a chunk: its index + 1 is a multiple of n_b (no division)
            tails = __ballot_sync(0xffffffffu, p.n_b == 1 || __umulhi(x1, p.nb_magic) * p.n_b == x1);
            const int j2 = (j | 31) + 1 + lane;
            if (j2 < cnt) e_next[0] = __ldg(ent + j2);
        };
        // The reference exponent of the row for the whole unit: the maximum of its first tile plus HEADROOM.  No running maximum and no
        // rescaling after this.  P of the first tile is <= 2^-60; a later tile may rise above the first one by a factor of up to ~2^150
        // (about 100 natural-log units) before the row sum passes 2^100, which the end of the unit detects (fp32 overflows at 2^128; rows
        // that fall below the first tile lose nothing: what flushes to zero is 2^-66 of the largest term).  Floating point is scale
        // invariant, so the result is the one the exact running maximum gives.  Rows of a row group past the last query block keep nothing
        // at all: any finite reference will do.
        auto reference = [&](const float* xm) -> float {
            const float mrow = fmaxf(xm[row], xm[128 + row]);
            return mrow == -INFINITY ? 0.f : fmaf(mrow, p.scale_log2, C::HEADROOM);
        };
        // History term (Eq. 4) of unit n: this warp's quarters of the features of A = phi(q), as bf16 hi + lo, to tensor memory from ta on (quarter k
        // at column 32 k, hi half first; in a P buffer all of hi, then all of lo); returns its share of the denominator in dsum.
        auto form_phi = [&](int n, int q0, uint32_t ta, float& dsum) -> bool {
            constexpr int FPT = D / 4;              // features per quarter
            // (S columns 32 k on are the warp's own: a half's, or a column group's)
            const int k0 = TEAMED ? half : 2 * half, dk = TEAMED ? 2 : 1;
            if (!wait_s(TEAMED ? bar_qe : bar_qf, n, 21) || !wait_s(bar_hf, n, 27)) return false;
            fence_after_sync();
            float2 ds = make_float2(0.f, 0.f);
#pragma unroll 1
            for (int k = k0; k < (TEAMED ? 4 : 2 * half + 2); k += dk) {
                uint32_t qw[FPT / 2];
                if constexpr (!TEAMED) {                    // q from shared memory
                    const uint8_t* qrow = s_gen + C::OFF_Q + (D == 128 ? (k >> 1) * C::SUB_BYTES : 0) + row * 128;
#pragma unroll
                    for (int c = 0; c < FPT / 8; ++c) {
                        const uint4 qv = *reinterpret_cast<const uint4*>(qrow + (((D == 128 ? 4 * (k & 1) + c : 2 * k + c) ^ (row & 7)) << 4));
                        qw[4 * c] = qv.x; qw[4 * c + 1] = qv.y; qw[4 * c + 2] = qv.z; qw[4 * c + 3] = qv.w;
                    }
                } else {                                    // q from tensor memory
                    if constexpr (D == 128) tmem_ld16(lane_base + C::COL_Q + k * (FPT / 2), qw);
                    else tmem_ld8(lane_base + C::COL_Q + k * (FPT / 2), qw);
                    tmem_wait_ld();
                }
                const float* zs = reinterpret_cast<const float*>(s_gen + C::OFF_Z) + k * FPT;
                const uint32_t tA = ta + k * (C::A_IN_P ? FPT / 2 : 32);
                uint32_t hi[FPT / 2], lo[FPT / 2];
#pragma unroll
                for (int c = 0; c < FPT / 8; ++c) {
                    const float4 z0 = *reinterpret_cast<const float4*>(zs + c * 8), z1 = *reinterpret_cast<const float4*>(zs + c * 8 + 4);
                    const float zz[8] = {z0.x, z0.y, z0.z, z0.w, z1.x, z1.y, z1.z, z1.w};
                    float cs[4] = {1.f, 1.f, 1.f, 1.f}, sn[4] = {0.f, 0.f, 0.f, 0.f};
                    if constexpr (HIST == 2) {      // the pairs' angles belong to the query's row
                        const int at = (k * (FPT / 8) + c) * p.Tc + min(q0 + row, p.Tc - 1);
                        const float4 c4 = __ldg(reinterpret_cast<const float4*>(p.cos_q) + at), s4 = __ldg(reinterpret_cast<const float4*>(p.sin_q) + at);
                        cs[0] = c4.x; cs[1] = c4.y; cs[2] = c4.z; cs[3] = c4.w;
                        sn[0] = s4.x; sn[1] = s4.y; sn[2] = s4.z; sn[3] = s4.w;
                    }
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        float2 f = phi_elu1(unpack_bf16(qw[4 * c + e]));
                        ds = ffma2(f, make_float2(zz[2 * e], zz[2 * e + 1]), ds);       // (the denominator is not rotated)
                        if constexpr (HIST == 2) f = make_float2(fmaf(-f.y, sn[e], f.x * cs[e]), fmaf(f.x, sn[e], f.y * cs[e]));
                        const uint32_t hp = pack_bf16(f.x, f.y);
                        const float2 r = ffma2(unpack_bf16(hp), make_float2(-1.f, -1.f), f);
                        hi[c * 4 + e] = hp;
                        lo[c * 4 + e] = pack_bf16(r.x, r.y);
                    }
                }
                if constexpr (D == 128) { tmem_st16(tA, hi); tmem_st16(tA + 16, lo); }
                else { tmem_st8(tA, hi); tmem_st8(tA + D / 2, lo); }
            }
            tmem_wait_st();
            fence_before_sync();
            arrive_w(bar_af);
            if (!TEAMED) arrive_t(bar_qe);
            dsum = ds.x + ds.y;
            return true;
        };
        // This warp's columns of the head's bias (read ahead of the waits at a unit's end: one at a time between them they are a trip to L2 each)
        auto read_bias = [&](uint4 (&bw)[C::OCOLS / 8]) {
            const uint4* b = HIST && p.bias ? reinterpret_cast<const uint4*>(p.bias + (size_t)(bh % p.heads) * D + half * C::OCOLS) : nullptr;
#pragma unroll
            for (int c = 0; c < C::OCOLS / 8; ++c) bw[c] = b ? __ldg(b + c) : make_uint4(0, 0, 0, 0);
        };
        // Output of unit n, D_h at tD, or in shared memory (first unit, formed ahead).
        auto write_output = [&](int n, int q0, uint32_t tD, float inv, float inv_den, const uint4 (&bw)[C::OCOLS / 8]) {
            // Output through shared memory and one bulk tensor store per warp (32 rows x half of the columns): row-per-thread global stores
            // would touch 32 lines per instruction.  The staging tile is the S W^T buffer (free: the history products have completed;
            // where there are none each team has its own), in the map's swizzle of the row width.
            const bool ahead = early && n == 0;
            // (D_h in shared memory: 8 KB a warp, the staging tile in front of it)
            const uint32_t dh_off = C::OFF_H + warp * C::DH_WARP;
            const uint32_t stage_off = ahead ? dh_off : C::OFF_H + (HIST ? 0 : team * C::TILE_BYTES) + (half * 4 + wq) * (32 * C::OCOLS * 2);
            const float* dh_s = reinterpret_cast<const float*>(s_gen + dh_off) + lane;
            uint32_t dh0[TEAMED ? 1 : 32];                  // D_h where the staging tile goes
            if constexpr (HIST != 0 && !TEAMED) {
                if (ahead) {
#pragma unroll
                    for (int e = 0; e < 32; ++e) dh0[e] = __float_as_uint(dh_s[e * 32]);
                    __syncwarp();
                }
            }
            uint8_t* stage = s_gen + stage_off + lane * (C::OCOLS * 2);
            const int swz = C::OCOLS == 64 ? lane & 7 : (lane >> 1) & 3;
            if (!HIST && staged) {
                if (lane == 0) bulk_wait_read();        // this warp's previous store has read its part
                __syncwarp();
            }
#pragma unroll
            for (int c = 0; c < C::OCOLS / 16; ++c) {
                uint32_t o[16], dh[16];
                tmem_ld16(lane_base + C::COL_O + half * C::OCOLS + c * 16, o);
                if constexpr (HIST != 0) {
                    if (ahead) {
#pragma unroll
                        for (int e = 0; e < 16; ++e) dh[e] = c < 2 ? dh0[(16 * c + e) % (TEAMED ? 1 : 32)] : __float_as_uint(dh_s[(16 * c + e) * 32]);
                    } else tmem_ld16(tD + half * C::OCOLS + c * 16, dh);
                }
                tmem_wait_ld();
                if (c == C::OCOLS / 16 - 1) {
                    fence_before_sync();
                    if (TEAMED) arrive_w(bar_dr(n)); else if (HIST) arrive_t(bar_dr(n));
                }
                const float* hsrc = !HIST && p.hist ? p.hist + ((size_t)bh * p.Tc + q0 + row) * D + half * C::OCOLS + c * 16 : nullptr;
#pragma unroll
                for (int v = 0; v < 2; ++v) {
                    float x[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) x[e] = __uint_as_float(o[v * 8 + e]) * inv;
                    if constexpr (HIST != 0) {
#pragma unroll
                        for (int e = 0; e < 8; ++e) x[e] = fmaf(__uint_as_float(dh[v * 8 + e]), inv_den, x[e]);
                        // Eq. 4's Linear: its matrix is folded into the state, its bias is added here
                        const uint4 b = bw[c * 2 + v];
                        const float2 b0 = unpack_bf16(b.x), b1 = unpack_bf16(b.y), b2 = unpack_bf16(b.z), b3 = unpack_bf16(b.w);
                        x[0] += b0.x; x[1] += b0.y; x[2] += b1.x; x[3] += b1.y;
                        x[4] += b2.x; x[5] += b2.y; x[6] += b3.x; x[7] += b3.y;
                    } else if (hsrc && q0 + row < p.Tc) {
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
            if (lane == 0 && q0 + wq * 32 < p.Tc) {     // rows past the chunk's end are clipped by the map
                tma_store_4d(&tm_o, s_base + stage_off, half * C::OCOLS, q0 + wq * 32, bh, 0);
                bulk_commit();
            }
            staged = true;
        };
        // The first unit's history term ahead of its tiles, and ahead of the wait for the kernel before this one (q, the folded state, z and
        // the bias are older than that one): phi(Q), its products into O's columns, D_h from there to shared memory, the denominators
        // to x_den (the groups' shares added to zero: the same sum in either order).  A thread block of a small grid is resident 2 us and more before
        // the lists are there, and the chain behind its unit's last tile is shorter by phi and the products (3 000-4 000 clk).
        auto form_ahead = [&]() -> bool {
            float ds;
            if (!form_phi(0, i * 128, lane_base + 128, ds)) return false;
            atomicAdd(x_den + row, ds);
            if (!wait_s(bar_ud, 0, 42)) return false;
            fence_after_sync();
            float* dh = reinterpret_cast<float*>(s_gen + C::OFF_H + warp * C::DH_WARP) + lane;
#pragma unroll
            for (int c = 0; c < C::OCOLS / 16; ++c) {
                uint32_t o[16];
                tmem_ld16(lane_base + C::COL_O + half * C::OCOLS + c * 16, o);
                tmem_wait_ld();
#pragma unroll
                for (int e = 0; e < 16; ++e) dh[(c * 16 + e) * 32] = __uint_as_float(o[e]);
            }
            fence_before_sync();
            arrive_w(bar_d0);
            return true;
        };
        if (early) ok = form_ahead();
        pdl_wait();
        int cnt_next = tiles_of(0);
        if (my_units > 0) first_entries(u, team, cnt_next);
        if constexpr (TEAMED) {
            float* x_l = reinterpret_cast<float*>(s_gen + C::OFF_XL);
            float* x_d = x_l + 128;
            int t0 = 0;                                         // first tile of the unit
            for (int n = 0; ok && n < my_units; ++n) {
                const int q0 = i * 128;
                const int nq = min(128, p.Tc - q0);
                const int cnt = cnt_next;
                cnt_next = n + 1 < my_units ? tiles_of(n + 1) : 0;
                const int pj = (t0 ^ team) & 1;                 // own tiles of the unit: pj, pj + 2, ...
                float m_used = 0.f, l_run = 0.f, dsum = 0.f;    // l_run, dsum: this thread's shares
                const uint32_t* ent = entries_of(u);
                for (int j = pj; j < cnt; j += 2) {
                    const int t = t0 + j;
                    uint32_t e_cur[EPT];
                    if constexpr (BLK == 128) {
                        if (ragged && (j & 31) == pj) {
                            next_tails(ent, j, cnt);
                        }
                    } else {
#pragma unroll
                        for (int x = 0; x < EPT; ++x) e_cur[x] = e_next[x];
                        if (j + 2 < cnt) read_entries(ent + (j + 2) * G);
                    }
                    // valid columns of entry x for this row: all, or the first nv (a short block; 0: its row group does not keep the block)
                    auto valid = [&](int x) -> int {
                        if constexpr (BLK == 128) return (tails >> (j & 31)) & 1u ? p.Tc - (p.n_b - 1) * BLK : BLK;
                        else return (e_cur[x] >> (10 + rg)) & 1u ? (int)((e_cur[x] >> 18) & 127u) : 0;
                    };
                    // ... of the 32 columns 64 c + 32 half on (blocks of 64 and 128 tokens)
                    auto valid32 = [&](int c) -> int { return BLK == 128 ? valid(0) - 64 * c - 32 * half : valid(c) - 32 * half; };
                    if (!(ok = wait_s(bar_sf + 8 * team, t >> 1, 8))) break;
                    fence_after_sync();
                    if (j == 0) {
                        // row maxima for the reference exponent
                        float mine = -INFINITY;
                        uint32_t r[2][32];
                        tmem_ld32(tS + 32 * half, r[0]);
                        tmem_ld32(tS + 64 + 32 * half, r[1]);
                        tmem_wait_ld();
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
                            if constexpr (BLK == 16) mine = fmaxf(mine, fmaxf(swa_max<16, true>(r[c], valid(2 * c)), swa_max<16, true>(r[c] + 16, valid(2 * c + 1))));
                            else if (valid32(c) >= 32) mine = fmaxf(mine, swa_max<32, false>(r[c], 32));
                            else if (valid32(c) > 0) mine = fmaxf(mine, swa_max<32, true>(r[c], valid32(c)));
                        }
                        if (n >= 1 && !(ok = wait_s(bar_mr + 8 * wq, n - 1, 32))) break;       // the unit before: read
                        x_m[half * 128 + row] = mine;
                        arrive_w(bar_m + 8 * wq);
                    }
                    if (j <= 1) {
                        if (!(ok = wait_s(bar_m + 8 * wq, n, 11))) break;
                        m_used = reference(x_m);
                        arrive_w(bar_mr + 8 * wq);
                    }
                    // ---- P = exp2(S*c - m), row sum, bf16 pairs
                    float2 rsum[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        uint32_t r[32], pk[16];
                        tmem_ld32(tS + 64 * c + 32 * half, r);
                        tmem_wait_ld();
                        if (c == 1) {                           // S is in registers: its buffer is free
                            fence_before_sync();
                            arrive_t(bar_se + 8 * team);
                        }
                        // Full, masked and empty segments are separate code: selects on 32 registers in every tile cost 9 us of a 134 us
                        // forward.  (BLK 64, 128: the same for the whole warp.)
                        if constexpr (BLK == 16) {
#pragma unroll
                            for (int x = 0; x < 2; ++x) {
                                const int nv = valid(2 * c + x);
                                if (__all_sync(0xffffffffu, nv >= 16)) swa_weights<16, false>(r + 16 * x, 16, p.scale_log2, m_used, rsum, pk + 8 * x);
                                else if (__any_sync(0xffffffffu, nv > 0)) swa_weights<16, true>(r + 16 * x, nv, p.scale_log2, m_used, rsum, pk + 8 * x);
                                else {
#pragma unroll
                                    for (int e = 0; e < 8; ++e) pk[8 * x + e] = 0u;
                                }
                            }
                        } else {
                            const int nv = valid32(c);
                            if (nv >= 32) swa_weights<32, false>(r, 32, p.scale_log2, m_used, rsum, pk);
                            else if (nv > 0) swa_weights<32, true>(r, nv, p.scale_log2, m_used, rsum, pk);
                            else {
#pragma unroll
                                for (int e = 0; e < 16; ++e) pk[e] = 0u;
                            }
                        }
                        if (HIST && C::A_IN_P && c == 0 && j == 0 && n >= 1) {      // the P buffer held the unit before's phi(Q) operand
                            if (!(ok = wait_s(bar_ud, n - 1, 37))) break;
                        }
                        if (t >= C::PBUF) {                     // its half of the P buffer: the product that last read it is complete
                            const int tr = t - C::PBUF;
                            if (!(ok = wait_s((c == 0 ? bar_ph : bar_pv) + 8 * (tr & 1), tr >> 1, 9))) break;
                            fence_after_sync();
                        }
                        tmem_st16(tP + 32 * c + 16 * half, pk);
                        tmem_wait_st();
                        fence_before_sync();
                        arrive_t(bar_pf + 16 * pb + 8 * c);
                    }
                    if (!ok) break;
                    l_run += ((rsum[0].x + rsum[0].y) + (rsum[1].x + rsum[1].y)) + ((rsum[2].x + rsum[2].y) + (rsum[3].x + rsum[3].y));
                    release_h();
                }
                if (!ok) break;
                if (n + 1 < my_units) first_entries(u + (int)gridDim.x, (t0 + cnt ^ team) & 1, cnt_next);
                if (((cnt - 1) & 1) != pj) {
                    // ---- the other team has the unit's last tile, and its output: this one hands over its row sums and goes on to the next unit
                    if constexpr (HIST != 0) {
                        release_h();
                        if constexpr (C::A_IN_P) {              // its P buffer: the product of its last tile is complete
                            const int tx = t0 + cnt - 2;
                            if (tx >= 0) ok = wait_s(bar_pv + 8 * (tx & 1), tx >> 1, 29);
                        }
                        if (!(ok = ok && form_phi(n, q0, C::A_IN_P ? tP : tS, dsum))) break;
                    }
                    if (cnt == 1) arrive_t(bar_mr + 8 * wq);                    // (nothing to read)
                    if (half == 1) {
                        if (n >= 1 && !(ok = wait_s(bar_dr(n - 1), (n - 1) >> 1, 31))) break; // the sums of the unit before have been read
                        x_l[row] = l_run;
                        if constexpr (HIST != 0) x_d[row] = dsum;
                        arrive_w(bar_h + 8 * wq);
                    } else {
                        if (!(ok = wait_s(bar_h + 8 * wq, n, 33))) break;
                        x_l[row] += l_run;
                        if constexpr (HIST != 0) x_d[row] += dsum;
                        arrive_w(bar_x + 8 * wq);
                    }
                } else {
                    // (a thread block that leaves room beside it lets the next kernel in only now: that one waits, but its blocks take slots)
                    if (C::SMEM_BYTES <= 200 * 1024 && n + 1 == my_units) pdl_trigger();
                    // ---- output of the unit
                    uint4 bw[C::OCOLS / 8];
                    read_bias(bw);
                    if constexpr (HIST != 0) {
                        if (!(ok = wait_s(bar_ud, n, 19))) break;           // D_h complete: the buffer of S W^T is free
                    }
                    if (!(ok = wait_s(bar_x + 8 * wq, n, 12))) break;
                    float* x_y = reinterpret_cast<float*>(s_gen + C::off_xy(HIST != 0, half));
                    x_y[row] = l_run;
                    arrive_w(bar_y + 8 * wq);
                    if (!(ok = wait_s(bar_y + 8 * wq, n, 34))) break;
                    {   // (the same order in both halves: the same bits)
                        const float other = reinterpret_cast<const float*>(s_gen + C::off_xy(HIST != 0, half ^ 1))[row];
                        l_run = x_l[row] + (half ? other + l_run : l_run + other);
                    }
                    const float inv = 1.f / l_run, inv_den = HIST ? 1.f / (p.eps + x_d[row]) : 0.f;
                    const size_t g_row = (size_t)bh * p.Tc + q0 + row;
                    if (half == 0 && row < nq && p.lse) p.lse[g_row] = (m_used + log2f(l_run)) * 0.6931471805599453f;
                    const uint32_t tl = t0 + cnt - 1;           // the unit's last tile
                    if (!(ok = wait_s(bar_pv + 8 * (tl & 1), tl >> 1, 10))) break;
                    fence_after_sync();
                    // overflow (or NaN): a later tile rose too far above the first one.  (The next unit's first P V waits for all of this team's
                    // warps below: a unit is listed before the next one can be.)
                    if (!(l_run < 1e30f)) note_redo(n);
                    write_output(n, q0, tS, inv, inv_den, bw);
                }
                t0 += cnt;
                u += gridDim.x; bh += dbh; i += di;
                if (i >= p.upb) { i -= p.upb; ++bh; }
            }
        } else {
            // ---- column groups: all warps on the same tile
            static_assert(TEAMED || C::PBUF == 1, "one P buffer");
            // Exchange number e of the kernel between partner warps: what a caller wrote to shared memory before is visible to the
            // others after.  Two per unit (maxima, then sums): a buffer written at one is read by the partners before they arrive
            // at the next, so each buffer is free again one exchange later.
            auto exchange = [&](uint32_t e, int where) -> bool { arrive_w(bar_x + 8 * wq); return wait_s(bar_x + 8 * wq, e, where); };
            float* x_l = reinterpret_cast<float*>(s_gen + C::off_xy(true, 0));      // [2][128], behind the staging tile of the output
            float* x_d = x_l + 256;
            const uint32_t bar_own = half == 0 ? bar_ph : bar_pv;      // product of its half of P
            const uint32_t tPh = tP + 32 * half;
            const int col0 = 64 * half % BLK;                   // first column within its key block (0 where it has several)
            int t = 0;
            for (int n = 0; ok && n < my_units; ++n) {
                const int q0 = i * 128;
                const int nq = min(128, p.Tc - q0);
                const int cnt = cnt_next;
                cnt_next = n + 1 < my_units ? tiles_of(n + 1) : 0;
                float m_used = 0.f, l_run = 0.f, dsum = 0.f;    // l_run, dsum: this thread's shares
                const uint32_t* ent = entries_of(u);
                if (cnt == 1) release_h();
                for (int j = 0; j < cnt; ++j, ++t) {
                    const uint32_t st = t & 1;
                    uint32_t e_cur[EPT];
                    if constexpr (BLK == 128) {
                        if (ragged && (j & 31) == 0) next_tails(ent, j, cnt);
                    } else {
#pragma unroll
                        for (int x = 0; x < EPT; ++x) e_cur[x] = e_next[x];
                        if (j + 1 < cnt) read_entries(ent + (j + 1) * G);
                    }
                    if (HIST && j == cnt - 1 && !(early && n == 0)) {
                        // history term's operand into the other S buffer: this thread's own S columns of it, which it has read (last tile's share),
                        // or its columns of the last unit's D_h
                        if (!(ok = form_phi(n, q0, lane_base + (st ^ 1u) * 128, dsum))) break;
                    }
                    if (!(ok = wait_s(bar_sf + 8 * st, t >> 1, 8))) break;
                    fence_after_sync();
                    // ---- this thread's share of the S row in registers
                    uint32_t r[64];
#pragma unroll
                    for (int c = 0; c < 2; ++c) tmem_ld32(lane_base + st * 128 + half * 64 + c * 32, *reinterpret_cast<uint32_t(*)[32]>(r + 32 * c));
                    tmem_wait_ld();
                    // ---- columns of this thread that count: all, or the first nv of a segment (a short block; 0: its row group does not
                    // keep the block)
                    constexpr int W = 64 / EPT;
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
                        float mine = -INFINITY;
#pragma unroll
                        for (int x = 0; x < EPT; ++x) mine = fmaxf(mine, swa_max<W, true>(r + x * W, nv[x]));
                        x_m[half * 128 + row] = mine;
                        if (!(ok = exchange(0, 11))) break;
                        m_used = reference(x_m);
                        if (half > 0) {
                            // The exchange has put the two warps that share a scheduler (same rows, different column groups) in step;
                            // they would run their exponentials at the same time and their waits at the same time, and the
                            // special-function unit would idle through the latter.  Set back by part of a tile, one group's waits
                            // fall into the other's exponentials.  Nothing couples the groups until the end of the unit.
                            const long long t_skew = clock64();
                            while (clock64() - t_skew < 700) {}
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
                        tmem_st16(tPh + 16 * c, pk);
                    };
                    if constexpr (BLK == 16) {
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
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
                        for (int c = 0; c < 2; ++c) {
                            uint32_t pk[16];
                            swa_weights<32, false>(r + 32 * c, 32, p.scale_log2, m_used, rsum, pk);
                            store_p(c, pk);
                        }
                    } else if (BLK == 128 || nv[0] > 0) {
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
                            uint32_t pk[16];
                            swa_weights<32, true>(r + 32 * c, nv[0] - 32 * c, p.scale_log2, m_used, rsum, pk);
                            store_p(c, pk);
                        }
                    } else {
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
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
                    if (cnt > 1) release_h();
                }
                if (!ok) break;
                if (n + 1 < my_units) first_entries(u + (int)gridDim.x, 0, cnt_next);
                // ---- end of the unit: row sums (and the shares of Eq. 4's denominator) of the column groups, range test, output
                uint4 bw[C::OCOLS / 8];
                read_bias(bw);
                // (first unit, history term formed ahead: D_h is where the sums go otherwise)
                const bool ahead = early && n == 0;
                float* l0 = ahead ? x_den - 128 : x_l;
                float* l1 = ahead ? reinterpret_cast<float*>(s_gen + C::OFF_Z) : x_l + 128;
                if (HIST && !ahead) {
                    if (!(ok = wait_s(bar_ud, n, 19))) break;   // D_h complete: the buffer of S W^T is free
                    x_d[half * 128 + row] = dsum;
                }
                (half ? l1 : l0)[row] = l_run;
                if (!(ok = exchange(1, 12))) break;
                l_run = l0[row] + l1[row];
                const float inv = 1.f / l_run, inv_den = HIST ? 1.f / (p.eps + (ahead ? x_den[row] : x_d[row] + x_d[128 + row])) : 0.f;
                if (half == 0 && row < nq && p.lse) p.lse[(size_t)bh * p.Tc + q0 + row] = (m_used + log2f(l_run)) * 0.6931471805599453f;
                const uint32_t tl = t - 1;                      // the unit's last tile
                if (!(ok = wait_s(bar_pv + 8 * (tl & 1), tl >> 1, 10))) break;
                fence_after_sync();
                if (!(l_run < 1e30f)) note_redo(n);
                write_output(n, q0, lane_base + (tl & 1) * 128, inv, inv_den, bw);
                u += gridDim.x; bh += dbh; i += di;
                if (i >= p.upb) { i -= p.upb; ++bh; }
            }
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
