// Block pooling (Eq. 5 "Mean"), cache append, block scores and the per-row top-K (Alg. 3, mask M_c).
//
// Canonical float32 order (the selection must be reproducible bit for bit):
//   block sum, per column: 16 chains, chain r adds tokens r, r+16, ... of the block in ascending order
//   from +0; the chains are then added in ascending r; mean = sum / float(n) with n the block's length.
//   score: 32 partials, partial l = sum over columns l, l+32, ... ascending of rounded products
//   (multiply and add rounded separately, never fused); partials folded as a butterfly +16, +8, +4, +2, +1.
#pragma once
#include "hf_common.cuh"
#include "k_union.cuh"
#include "hf_dispatch.h"

template <int VEC> struct VecLoad;
template <> struct VecLoad<8> {
    typedef uint4 T;
    static __device__ __forceinline__ void widen(const uint4& u, float* f) {
        float2 a = unpack_bf16(u.x), b = unpack_bf16(u.y), c = unpack_bf16(u.z), d = unpack_bf16(u.w);
        f[0] = a.x; f[1] = a.y; f[2] = b.x; f[3] = b.y; f[4] = c.x; f[5] = c.y; f[6] = d.x; f[7] = d.y;
    }
};
template <> struct VecLoad<4> {
    typedef uint2 T;
    static __device__ __forceinline__ void widen(const uint2& u, float* f) {
        float2 a = unpack_bf16(u.x), b = unpack_bf16(u.y);
        f[0] = a.x; f[1] = a.y; f[2] = b.x; f[3] = b.y;
    }
};

struct PoolJob {            // one tensor to pool (and optionally copy) per blockIdx.z
    const bf16* src;        // [B*H, T_c, d]
    bf16* copy_dst;         // same shape, or nullptr (may be src itself: every thread rewrites exactly what it read)
    float* pooled;          // [B*H, n_b, d] block means, or nullptr (copy only)
    // temporal rotation (ROT instantiation): frame f of the chunk is turned by rot_base + rot_per_frame * f index steps
    int rot_on, rot_base, rot_per_frame;
};
struct PoolJobs { PoolJob job[3]; };

// Relative temporal RoPE of the softmax branch (Eq. 8): pairs [first_pair, first_pair + n_pairs) of a token's features
// turn by (index steps) x (the pair's frequency); cosine and sine come from tables over integer steps 0 .. t0 (a backward
// turn uses the entry of |steps| with the sine negated).  The arithmetic order is fixed, because the rotated values feed
// the block selection: x0' = x0 c - x1 s, x1' = x0 s + x1 c, each product and each sum rounded separately in float32, the
// result rounded to bf16 (the cache and the attention operands are bf16).
struct TemporalRope {
    const float* cos_tab;   // [t0 + 1][n_pairs]
    const float* sin_tab;
    int first_pair, n_pairs, tokens_per_frame;
};

// The frame of the chunk that row r of a block of n tokens starting at token t0 belongs to, or -1: no such row (a chunk's last
// block may hold fewer tokens than there are rows of threads, and past the chunk's end the tables have no angles).
__host__ __device__ inline int turn_frame(int t0, int r, int n, int tokens_per_frame) {
    return r < n ? (t0 + r) / tokens_per_frame : -1;
}

// Turn of one thread's VEC features of a row: cosine and sine of those of its VEC / 2 pairs that turn.
template <int VEC>
struct PairTurn {
    float c[VEC / 2], s[VEC / 2];
    int frame = -1;             // of the chunk; the entries are reloaded when a row belongs to another one
};
template <int VEC>
__device__ __forceinline__ void load_turn(PairTurn<VEC>& t, int first_feature, int steps, const TemporalRope& tr) {
    const int a = steps < 0 ? -steps : steps;
#pragma unroll
    for (int e = 0; e < VEC / 2; ++e) {
        const int pr = first_feature / 2 + e - tr.first_pair;
        if (pr >= 0 && pr < tr.n_pairs) {
            t.c[e] = __ldg(tr.cos_tab + (size_t)a * tr.n_pairs + pr);
            const float sn = __ldg(tr.sin_tab + (size_t)a * tr.n_pairs + pr);
            t.s[e] = steps < 0 ? -sn : sn;
        }
    }
}
template <int VEC, typename V>
__device__ __forceinline__ V rotate_vec(const V& u, const PairTurn<VEC>& t, int first_feature, const TemporalRope& tr) {
    float f[VEC];
    VecLoad<VEC>::widen(u, f);
    uint32_t w[VEC / 2];
#pragma unroll
    for (int e = 0; e < VEC / 2; ++e) {
        const int pr = first_feature / 2 + e - tr.first_pair;
        float y0 = f[2 * e], y1 = f[2 * e + 1];
        if (pr >= 0 && pr < tr.n_pairs) {
            y0 = __fsub_rn(__fmul_rn(f[2 * e], t.c[e]), __fmul_rn(f[2 * e + 1], t.s[e]));
            y1 = __fadd_rn(__fmul_rn(f[2 * e], t.s[e]), __fmul_rn(f[2 * e + 1], t.c[e]));
        }
        w[e] = pack_bf16(y0, y1);
    }
    V out;
    if constexpr (VEC == 8) { out.x = w[0]; out.y = w[1]; out.z = w[2]; out.w = w[3]; }
    else { out.x = w[0]; out.y = w[1]; }
    return out;
}

// One block of one tensor: copy (optional) and per-column mean in the canonical order.  256 threads: 16 threads per token
// row, 16 rows per pass.
template <int D, bool ROT>
__device__ __forceinline__ void pool_copy_block(const PoolJob& jb, int Tc, int blk, int n_b, int b_idx, int bh, const TemporalRope& tr) {
    constexpr int VEC = D / 16;
    typedef typename VecLoad<VEC>::T V;
    const int t0 = b_idx * blk;
    const int n = min(blk, Tc - t0);
    const int r = threadIdx.x >> 4, cv = threadIdx.x & 15;
    const size_t base = ((size_t)bh * Tc + t0) * D + cv * VEC;
    // Two batches of four rows: the loads of a batch first, then its copies, then its chain adds in token order.  (Four
    // 16-byte loads in flight per thread at six thread blocks per SM keep ~100 KB in flight per SM; eight would cost the
    // registers that the sixth block needs.)
    constexpr int MAXR = 8, BATCH = 4;            // blk <= 128 -> at most 8 rows per chain
    float acc[VEC];
#pragma unroll
    for (int e = 0; e < VEC; ++e) acc[e] = 0.f;
    // ROT: this thread's pairs are the same in every row, and a block's rows span few frames: the angles stay in registers
    PairTurn<VEC> turn;
    int frame_end = 0;          // first row of the block that belongs to the frame after turn.frame
    bool turns = false;         // any of this thread's pairs turns at all
    if (ROT) {
        turn.frame = turn_frame(t0, r, n, tr.tokens_per_frame);
        turns = jb.rot_on && turn.frame >= 0 && cv * VEC / 2 < tr.first_pair + tr.n_pairs && (cv + 1) * VEC / 2 > tr.first_pair;
        if (turns) {
            frame_end = (turn.frame + 1) * tr.tokens_per_frame - t0;
            load_turn<VEC>(turn, cv * VEC, jb.rot_base + jb.rot_per_frame * turn.frame, tr);
        }
    }
#pragma unroll
    for (int i0 = 0; i0 < MAXR; i0 += BATCH) {
        V u[BATCH];
#pragma unroll
        for (int i = 0; i < BATCH; ++i) {
            const int t = r + 16 * (i0 + i);
            if (t < n) {
                // (the rotating instantiation may work in place: plain loads there, the read-only path elsewhere)
                if (ROT) u[i] = *reinterpret_cast<const V*>(jb.src + base + (size_t)t * D);
                else u[i] = __ldg(reinterpret_cast<const V*>(jb.src + base + (size_t)t * D));
            }
        }
        if (ROT) {
            if (turns) {
#pragma unroll
                for (int i = 0; i < BATCH; ++i) {
                    const int t = r + 16 * (i0 + i);
                    if (t < n) {
                        if (t >= frame_end) {
                            turn.frame = turn_frame(t0, t, n, tr.tokens_per_frame);
                            frame_end = (turn.frame + 1) * tr.tokens_per_frame - t0;
                            if (jb.rot_per_frame != 0) load_turn<VEC>(turn, cv * VEC, jb.rot_base + jb.rot_per_frame * turn.frame, tr);
                        }
                        u[i] = rotate_vec<VEC, V>(u[i], turn, cv * VEC, tr);
                    }
                }
            }
        }
        if (jb.copy_dst) {
#pragma unroll
            for (int i = 0; i < BATCH; ++i) {
                const int t = r + 16 * (i0 + i);
                if (t < n) *reinterpret_cast<V*>(jb.copy_dst + base + (size_t)t * D) = u[i];
            }
        }
#pragma unroll
        for (int i = 0; i < BATCH; ++i) {
            if (r + 16 * (i0 + i) < n) {
                float f[VEC];
                VecLoad<VEC>::widen(u[i], f);
#pragma unroll
                for (int e = 0; e < VEC; ++e) acc[e] = __fadd_rn(acc[e], f[e]);
            }
        }
    }
    if (jb.pooled == nullptr) return;
    __shared__ float part[16][D];
#pragma unroll
    for (int e = 0; e < VEC; ++e) part[r][cv * VEC + e] = acc[e];
    __syncthreads();
    if (threadIdx.x < D) {
        float tot = part[0][threadIdx.x];
#pragma unroll
        for (int rr = 1; rr < 16; ++rr) tot = __fadd_rn(tot, part[rr][threadIdx.x]);
        jb.pooled[((size_t)bh * n_b + b_idx) * D + threadIdx.x] = __fdiv_rn(tot, (float)n);
    }
}

// grid (n_b, B*H, jobs), 256 threads.
template <int D>
__global__ void __launch_bounds__(256, 6) k_pool_copy(PoolJobs jobs, int Tc, int blk, int n_b) {
    pdl_wait();                 // launched under the tail of the kernel before it: that kernel's reads and writes are done from here on
    pdl_trigger();              // a dependent kernel (the selection) may be made resident; it waits for this grid itself
    const PoolJob jb = blockIdx.z == 0 ? jobs.job[0] : blockIdx.z == 1 ? jobs.job[1] : jobs.job[2];   // (no indexed copy of the parameter block)
    TemporalRope none = {nullptr, nullptr, 0, 0, 1};
    pool_copy_block<D, false>(jb, Tc, blk, n_b, blockIdx.x, blockIdx.y, none);
}
// The same with the temporal rotation applied to the jobs that ask for it (before the copy and the means).  The angles of a
// thread's pairs stay in registers from row to row (22 -> 16 us for two 14 MB tensors turned and copied, against table loads
// and a division per row).
template <int D>
__global__ void __launch_bounds__(256, 4) k_pool_copy_rot(PoolJobs jobs, int Tc, int blk, int n_b, TemporalRope tr) {
    pdl_wait();
    pdl_trigger();
    const PoolJob jb = blockIdx.z == 0 ? jobs.job[0] : blockIdx.z == 1 ? jobs.job[1] : jobs.job[2];
    pool_copy_block<D, true>(jb, Tc, blk, n_b, blockIdx.x, blockIdx.y, tr);
}

// The cache commit of several layers in one launch (Alg. 2 "KV.append" for every layer of the model): per layer the
// clean chunk's K (copied, block means stored) and V (copied) go to the ring slot slot[l] of that layer.
// grid (n_b, B*H, 2 * layers): blockIdx.z = 2 * layer + (0: K, 1: V).
struct PoolLayersParams {
    const bf16* k_src[64];      // per layer of the call: [B*H, T_c, d]
    const bf16* v_src[64];
    int slot[64];               // target slot within the layer's ring
    bf16* ring_k;               // first layer of the call: [layers][slots_per_layer][B*H, T_c, d]
    bf16* ring_v;
    float* pooled;              // [layers][slots_per_layer][B*H, n_b, d]
    size_t chunk_elems, pooled_elems;
    int slots_per_layer;
};
template <int D>
__global__ void __launch_bounds__(256, 6) k_pool_copy_layers(const __grid_constant__ PoolLayersParams p, int Tc, int blk, int n_b) {
    pdl_wait();
    pdl_trigger();
    const int lay = blockIdx.z >> 1;
    const bool is_v = blockIdx.z & 1;
    const size_t s = (size_t)lay * p.slots_per_layer + p.slot[lay];
    PoolJob jb;
    jb.src = is_v ? p.v_src[lay] : p.k_src[lay];
    jb.copy_dst = (is_v ? p.ring_v : p.ring_k) + s * p.chunk_elems;
    jb.pooled = is_v ? nullptr : p.pooled + s * p.pooled_elems;
    jb.rot_on = 0; jb.rot_base = 0; jb.rot_per_frame = 0;
    TemporalRope none = {nullptr, nullptr, 0, 0, 1};
    pool_copy_block<D, false>(jb, Tc, blk, n_b, blockIdx.x, blockIdx.y, none);
}

// A[i][j] = Mean(q_i) . Mean(k_j) in the canonical order, and the top-K of every row under the total order (score descending,
// block index ascending): bit mask and ascending index list.  grid (ceil(T_m / R), B*H), 64 R threads: R = four query
// blocks of a head per thread block, or eight.
//
// Scores: one THREAD per (query block, key block).  The butterfly of the canonical order is a plain tree, so a thread that walks
// the columns in the order l, l + 16, l + 8, l + 24 (l = 0..3, then 4..7) needs four running values and no shuffle: 2 D - 1
// packed fp32 operations per pair of columns.  Key rows come from shared memory (padded rows: conflict-free 16-byte reads), each
// fetched from L2 once for four query blocks, the cached chunks' before the wait for the pooling kernel; query rows are
// broadcast reads.  Top-K: one WARP per row, score images in registers, the keep-th largest found bit by bit (count by
// redux; the search ends as soon as a threshold separates exactly `keep`), ties cut by ballot.
//
// What bounds it: latency (a trip to L2, 32 + 32 tree steps, ~16 count steps).  The form before (one warp per score with its
// five-step butterfly, one query block per thread block, ranking by counting or a bitonic sort of the whole block):
// pooling + selection as part of the forward, 12 heads of 128: 128-token blocks (T_n 111) 128.3 -> 125.5 us, 64-token blocks
// (T_n 222) 171 -> 164 us, 16-token blocks at head dim 64 (T_n 246) 64.6 -> 55.1 us; this kernel alone at T_n 259, batch 4:
// 76 -> 39 us.
// G: the query blocks that share a unit of the attention kernel (blocks of 64 tokens: 2, of 16: 8), whose merged list is formed here
// from the masks in shared memory, or 1: none is asked for.  A kernel of its own behind this one costs a launch (k_union.cuh).  G = 8
// takes eight query blocks, one unit, per thread block, with as many threads per score.
// KPL: key blocks per lane of a ranking warp (T_n <= 32 KPL).  Rows of more than 256 key blocks come in several passes of key rows, and their
// grids are mostly large: there, too, eight query blocks share a key row's trip through L2 (T_n 259, 48 heads, behind the pooling: 42 us
// with four query blocks and KPL 32, 24.5 like this).  One isolated call, pooling and selection, heads of 128, four / eight query blocks: T_n 296,
// 48 heads 56.6 / 43.2 us, 12 heads 26.2 / 27.4, 2 heads 18.3 / 20.5; T_n 512, 12 heads 52 / 39.4; T_n 1 024, 1 head 43.2 / 47.0, 12 heads
// 111 / 107.5.
// RQ: query blocks per thread block.  Rows of 129 to 256 key blocks (KPL 8) have all their key rows in shared memory at once and four scores per thread,
// so that a key row is read once for four query blocks (the scores are bound by shared-memory reads) and no pass waits for the next one's rows: from the
// pooled rows' arrival to the scores, 12 heads of 128, T_n 222 12 100 -> 8 300 clk, heads of 64, T_n 246 7 300 -> 5 300; with the ranking's two bits a step and its
// words before the stores the forward of 64-token blocks 158 -> 155 us, of 16-token blocks at head dim 64 35.6 -> 33.4, 12 heads of 16-token blocks, T_n 176 45.0 -> 40.5;
// four query blocks or eight: select_rows_of (hf_dispatch.h).
template <int D, int G, int KPL, int RQ>
struct Select {
    static constexpr int R = RQ, KT = KPL == 8 ? 256 : 128;       // query blocks per thread block; key rows per pass
    static constexpr int THREADS = 64 * R;
    static constexpr int LD = D + 4;            // floats per key row in shared memory
    static int smem_bytes(int Tn) { return select_smem_bytes(D, R, Tn < KT ? Tn : KT, Tn); }
};
struct Quad { float2 a, b; };                   // four neighbouring columns
__device__ __forceinline__ Quad quad_add(const Quad& x, const Quad& y) { return {fadd2(x.a, y.a), fadd2(x.b, y.b)}; }
// Products rounded separately: x y + (-0), which is the rounded product for every x y.  (The packed multiply would be contracted
// with the packed addition that follows it, explicit rounding or not.)  nz: (-0, -0), a run-time value for the same reason.
__device__ __forceinline__ Quad quad_mul(const float4& x, const float4& y, float2 nz) {
    return {ffma2(make_float2(x.x, x.y), make_float2(y.x, y.y), nz), ffma2(make_float2(x.z, x.w), make_float2(y.z, y.w), nz)};
}
// Scores of one key row against RPT query rows (rows of D floats in shared memory).
template <int D, int RPT>
__device__ __forceinline__ void canonical_scores(const float* kr, const float* qr, float2 nz, float (&out)[RPT]) {
    constexpr int M = D / 32;
    Quad c[RPT];
#pragma unroll
    for (int h = 0; h < 2; ++h) {               // l = 0..3, then 4..7
        Quad b[RPT];
#pragma unroll
        for (int g = 0; g < 2; ++g) {           // columns l and l + 16, then l + 8 and l + 24
            Quad a[RPT];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int x = 4 * h + 8 * g + 16 * e;
                float4 kv[M];
#pragma unroll
                for (int m = 0; m < M; ++m) kv[m] = *reinterpret_cast<const float4*>(kr + x + 32 * m);
#pragma unroll
                for (int r = 0; r < RPT; ++r) {
                    Quad part = quad_mul(*reinterpret_cast<const float4*>(qr + r * D + x), kv[0], nz);
#pragma unroll
                    for (int m = 1; m < M; ++m) part = quad_add(part, quad_mul(*reinterpret_cast<const float4*>(qr + r * D + x + 32 * m), kv[m], nz));
                    a[r] = e == 0 ? part : quad_add(a[r], part);
                }
            }
#pragma unroll
            for (int r = 0; r < RPT; ++r) b[r] = g == 0 ? a[r] : quad_add(b[r], a[r]);
        }
#pragma unroll
        for (int r = 0; r < RPT; ++r) c[r] = h == 0 ? b[r] : quad_add(c[r], b[r]);
    }
#pragma unroll
    for (int r = 0; r < RPT; ++r) {
        const float2 dd = fadd2(c[r].a, c[r].b);
        out[r] = __fadd_rn(dd.x, dd.y);
    }
}
// Order-preserving image of a score: ascending integers = ascending floats, -0 = +0, a NaN (anywhere in the query block or the
// key block) below every number, so that exactly `keep` blocks are kept whatever the inputs hold.
__device__ __forceinline__ uint32_t score_image(float s) {
    const uint32_t u = __float_as_uint(s);
    if (s != s) return 0u;
    if (u == 0x80000000u) return 0x80000000u;
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Where a selection goes: per layer, and copies a caller asks for.
struct SelectOut {
    uint32_t* mask;              // [B*H, T_m, mask_words]
    int32_t* idx;                // [B*H, T_m, keep]
    uint32_t *mask_out;          // (nullptr: not wanted)
    int32_t* idx_out;
    float* scores_out;
    int mask_words;
};
// Top-K of one row by one warp: the row's scores in shared memory; its mask and ascending list are stored, the mask's word number
// `lane` is returned.  KPL: key blocks per lane (T_n <= 32 KPL).
template <int KPL>
__device__ __forceinline__ uint32_t rank_row(const float* sc, size_t row, int Tn, int keep, const SelectOut& o) {
    const int lane = threadIdx.x & 31;
    // lane l holds the images of blocks l, l + 32, ... (padding: 0, and behind every block)
    uint32_t key[KPL];
#pragma unroll
    for (int x = 0; x < KPL; ++x) {
        const int j = x * 32 + lane;
        key[x] = j < Tn ? score_image(sc[j]) : 0u;
    }
    // Few keys: every lane counts the images in front of its own (greater, or equal with a lower index; no image is 2^32 - 1, so one more
    // does not wrap).  Sixty-four shuffles at most, against a chain of ten to twenty votes: a forward of two heads of 64 queries, 16-token
    // blocks 9.3 -> 8.9 us; 16 forwards of 8 heads of 128, 300 queries and their commit 258.8 -> 253.6.
    int ahead[KPL <= 2 ? KPL : 1];
    uint32_t thr = 0;           // more keys: largest value with at least `keep` images at or above it
    int ties = Tn;              // ... and blocks at the threshold still to be kept, lowest index first
    bool exact = false;
    if constexpr (KPL <= 2) {
#pragma unroll
        for (int x = 0; x < KPL; ++x) ahead[x] = 0;
#pragma unroll
        for (int y = 0; y < KPL; ++y) {
            const int n = min(32, Tn - 32 * y);
#pragma unroll 8
            for (int l = 0; l < n; ++l) {
                const uint32_t other = __shfl_sync(0xffffffffu, key[y], l);
#pragma unroll
                for (int x = 0; x < KPL; ++x) ahead[x] += other + (32 * y + l < 32 * x + lane ? 1u : 0u) > key[x];
            }
        }
    } else {
        // Two bits a step, the three counts of a step side by side in one word (T_n <= 512; two words above): a step is a chain, mostly the sum
        // over the warp (3 300 -> 2 300 clk with 222 key blocks; votes and population counts instead 3 400).  Pooling and selection with a bit a step and the
        // stores between the words' votes / like this, us: T_n 72 and 120 in one launch 5.3 / 5.1, 6.1 / 5.9; T_n 80 9.6 / 9.0; 370 30.3 / 29.9, 400 22.7 / 22.1; in two words 592,
        // 720 (head dim 128, 64) 31.6 / 28.0, 70.7 / 64.1, 30.3 / 25.6.
        exact = keep >= Tn;         // exactly `keep` images at or above the threshold: no ties to cut (all blocks kept: every image counts)
        for (int sh = 30; sh >= 0 && !exact; sh -= 2) {
            const uint32_t c1 = thr | (1u << sh), c2 = thr | (2u << sh), c3 = thr | (3u << sh);
            uint32_t a1[2] = {0, 0}, a2[2] = {0, 0}, a3[2] = {0, 0};
#pragma unroll
            for (int x = 0; x < KPL; ++x) { a1[x & 1] += key[x] >= c1; a2[x & 1] += key[x] >= c2; a3[x & 1] += key[x] >= c3; }
            uint32_t n = a1[0] + a1[1] + ((a2[0] + a2[1]) << (KPL < 32 ? 10 : 16)), m = a3[0] + a3[1];
            if (KPL < 32) n += m << 20;
            n = __reduce_add_sync(0xffffffffu, n);
            const int n3 = (int)(KPL < 32 ? n >> 20 : __reduce_add_sync(0xffffffffu, m));
            const int n1 = (int)(n & (KPL < 32 ? 1023u : 65535u)), n2 = (int)(KPL < 32 ? n >> 10 & 1023u : n >> 16);
            if (n3 >= keep) { thr = c3; exact = n3 == keep; }
            else if (n2 >= keep) { thr = c2; exact = n2 == keep; }
            else if (n1 >= keep) { thr = c1; exact = n1 == keep; }
        }
        if (!exact) {
            int n = 0;
#pragma unroll
            for (int x = 0; x < KPL; ++x) n += key[x] > thr;
            ties = keep - __reduce_add_sync(0xffffffffu, n);
        }
    }
    const uint32_t below = (1u << lane) - 1u;
    uint32_t word[KPL];             // the row's mask
    if (KPL <= 2 || exact) {
#pragma unroll
        for (int x = 0; x < KPL; ++x) word[x] = __ballot_sync(0xffffffffu, x * 32 + lane < Tn && (KPL <= 2 ? ahead[x % (KPL <= 2 ? KPL : 1)] < keep : key[x] >= thr));
    } else {
#pragma unroll
        for (int x = 0; x < KPL; ++x) {
            const uint32_t eq = __ballot_sync(0xffffffffu, x * 32 + lane < Tn && key[x] == thr);
            word[x] = __ballot_sync(0xffffffffu, x * 32 + lane < Tn && (key[x] > thr || (key[x] == thr && __popc(eq & below) < ties)));
            ties -= __popc(eq);
        }
    }
    int pos = 0;
    uint32_t my_word = 0;
    int32_t* list = o.idx + row * keep;
#pragma unroll
    for (int x = 0; x < KPL; ++x) {
        if (lane == x) my_word = word[x];
        const int at = pos + __popc(word[x] & below);
        if ((word[x] >> lane & 1u) && at < keep) {      // (always true under the total order above; the store never leaves the row)
            list[at] = x * 32 + lane;
            if (o.idx_out) o.idx_out[row * keep + at] = x * 32 + lane;
        }
        pos += __popc(word[x]);
    }
    if (lane < o.mask_words) {
        o.mask[row * o.mask_words + lane] = my_word;
        if (o.mask_out) o.mask_out[row * o.mask_words + lane] = my_word;
    }
    return my_word;
}

// Scores of n key rows of a pass (key_row(j): their D floats in shared memory) against `rows` query rows, sc[r * Tn + j].  R: query rows
// a thread block may have; 512 threads for eight and for one, otherwise 256.
template <int D, int R, typename KeyRow>
__device__ __forceinline__ void score_pass(KeyRow key_row, int n, const float* s_q, int rows, float* sc, int Tn, float2 nz) {
    constexpr int THREADS = R == 8 || R == 1 ? 512 : 256, W = THREADS / R < 128 ? THREADS / R : 128;
    if (n <= W) {               // few keys: one score per thread
        const int j = threadIdx.x % W, r = threadIdx.x / W;
        if (j < n && r < rows) {
            float v[1];
            canonical_scores<D, 1>(key_row(j), s_q + r * D, nz, v);
            sc[r * Tn + j] = v[0];
        }
    } else {                    // two scores per thread: query blocks 2 h, 2 h + 1 (rows past T_m: stale shared memory, not stored)
        const int j = threadIdx.x & 127, r = (threadIdx.x >> 7) * 2;
        if (j < n && r < rows) {
            float v[2];
            canonical_scores<D, 2>(key_row(j), s_q + r * D, nz, v);
            sc[r * Tn + j] = v[0];
            if (r + 1 < rows) sc[(r + 1) * Tn + j] = v[1];
        }
    }
}
// ... of up to 256 key rows, four scores per thread (64 threads a query row).
template <int D>
__device__ __forceinline__ void score_quads(const float* s_k, int ld, int n, const float* s_q, int rows, float* sc, int Tn, float2 nz) {
    const int j = threadIdx.x & 255, r = (threadIdx.x >> 8) * 4;
    if (j < n && r < rows) {
        float v[4];
        canonical_scores<D, 4>(s_k + j * ld, s_q + r * D, nz, v);      // (rows past T_m: stale shared memory, not stored)
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (r + e < rows) sc[(r + e) * Tn + j] = v[e];
    }
}
// The end of a selection: scores out, top-K of every row, and (G > 1, lists.entries set) the merged lists of the units of these rows.
template <int KPL, int G, int R>
__device__ __forceinline__ void finish_rows(const float* s_sc, uint32_t (*s_mask)[32], int bh, int i0, int rows, int Tm, int Tn, int n_b, int keep,
                                            const SelectOut& o, const UnionOut& lists) {
    constexpr int THREADS = R == 8 || R == 1 ? 512 : 256;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (o.scores_out)
        for (int e = threadIdx.x; e < rows * Tn; e += THREADS) o.scores_out[((size_t)bh * Tm + i0) * Tn + e] = s_sc[e];
    if (warp < R) {
        const uint32_t word = warp < rows ? rank_row<KPL>(s_sc + warp * Tn, (size_t)bh * Tm + i0 + warp, Tn, keep, o) : 0u;
        if constexpr (G > 1) s_mask[warp][lane] = word;         // (query blocks past T_m, lanes past the words of T_n: 0)
    }
    if constexpr (G > 1) {
        if (lists.entries == nullptr) return;
        constexpr int UNITS = R / G, WPU = THREADS / 32 / UNITS;
        __syncthreads();
        const int x = warp / WPU, mt = i0 / G + x, upb = (Tm + G - 1) / G;
        if (mt < upb) union_lists<G>(s_mask + x * G, warp % WPU, WPU, Tn, n_b, bh * upb + mt, lists);
    }
}

template <int D, int KPL, int G, int RQ>
__global__ void __launch_bounds__(Select<D, G, KPL, RQ>::THREADS) k_select(ChunkTable tab, const float* __restrict__ pooled_q,
                                                int n_b, int Tm, int Tn, int keep, float neg_zero, SelectOut o, UnionOut lists) {
    typedef Select<D, G, KPL, RQ> C;
    const float2 nz = make_float2(neg_zero, neg_zero);
    extern __shared__ __align__(16) float sel_smem[];
    const int kt = min(Tn, C::KT);
    float* s_k = sel_smem;                      // [kt][LD]
    float* s_q = s_k + kt * C::LD;              // [R][D]
    float* s_sc = s_q + C::R * D;               // [R][Tn]
    __shared__ uint32_t s_mask[G > 1 ? C::R : 1][32];
    const int i0 = blockIdx.x * C::R, bh = blockIdx.y;
    const int rows = min(C::R, Tm - i0);
    const uint32_t s_k_addr = smem_u32(s_k);
    // key rows [j0, j1) of the pass that starts at `base`, sixteen bytes per thread and step
    auto load_keys = [&](int base, int j0, int j1) {
        constexpr int V = D / 4;
        for (int e = threadIdx.x; e < (j1 - j0) * V; e += C::THREADS) {
            const int j = j0 + e / V, part = e % V;
            int c = 0, jb = j;
            while (jb >= n_b) { jb -= n_b; ++c; }
            cp_async16(s_k_addr + ((j - base) * C::LD + part * 4) * 4, tab.pooled[c] + ((size_t)bh * n_b + jb) * D + part * 4, true);
        }
        cp_async_commit();
    };
    pdl_trigger();              // the attention kernel may be made resident as blocks of this grid leave
    // The cached chunks' rows are older than the pooling kernel before this one (which has itself waited for what came before it).
    const int old = min((tab.n_chunks - 1) * n_b, kt);
    load_keys(0, 0, old);
    pdl_wait();                 // the pooled rows of the queries and of the current chunk come from the kernel before
    for (int e = threadIdx.x; e < rows * (D / 4); e += C::THREADS)
        cp_async16(smem_u32(s_q) + e * 16, pooled_q + ((size_t)bh * Tm + i0) * D + e * 4, true);
    load_keys(0, old, kt);
    for (int base = 0; base < Tn; base += C::KT) {
        const int n = min(C::KT, Tn - base);
        if (base > 0) {
            __syncthreads();    // the pass before has been read
            load_keys(base, base, base + n);
        }
        cp_async_wait<0>();
        __syncthreads();
        if constexpr (KPL == 8) score_quads<D>(s_k, C::LD, n, s_q, rows, s_sc + base, Tn, nz);
        else score_pass<D, C::R>([&](int j) { return s_k + j * C::LD; }, n, s_q, rows, s_sc + base, Tn, nz);
    }
    __syncthreads();
    finish_rows<KPL, G, C::R>(s_sc, s_mask, bh, i0, rows, Tm, Tn, n_b, keep, o, lists);
}

// Pooling and selection of one call in one launch, for heads of few blocks: latency alone.  Against k_pool_copy + k_select it spares a launch
// and the means' way through L2 (two heads of 64 queries, 16-token blocks 11.65 -> 10.5 us a forward; 8 heads of 128, 300 queries,
// selection alone 7.0 -> 4.9).  With more blocks a head the thread blocks are too few for the pooling, which the other form spreads
// over the device (dispatch: pools_and_selects).  512 threads, and little code, which a thread block runs once, so that fetching it
// counts: with 256 threads that took a block of queries and one of keys each, and one kernel for both block sizes, 16 forwards of that
// shape and their commit took 253 us (1 300 clk from the rows' arrival to their sums), 242.5 like this; the two heads 9.2 -> 8.9.
struct PoolSelect {
    static constexpr int THREADS = 512;
    // key rows, query rows, scores, chains (128-token blocks: of one query block and one key block)
    static int smem_bytes(int d, int block, int Tn) {
        const int rows = block == 16 ? 8 : 1, part = block == 16 ? 0 : 2 * 16 * d;
        return (Tn * (d + 4) + rows * d + rows * Tn + part) * (int)sizeof(float);
    }
};
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory"); }
// A float into the same place of thread block `rank`'s shared memory.
__device__ __forceinline__ void cluster_store(uint32_t addr, int rank, float v) {
    asm volatile("{\n.reg .b32 a;\nmapa.shared::cluster.u32 a, %0, %1;\nst.shared::cluster.f32 [a], %2;\n}\n" ::"r"(addr), "r"(rank), "f"(v) : "memory");
}

// The cached chunks' key means of a head, rows of LD floats, on their way to shared memory.
template <int D, int LD>
__device__ __forceinline__ void load_cached_keys(float* s_k, const ChunkTable& tab, int n_old, int n_b, int bh) {
    for (int e = threadIdx.x; e < n_old * (D / 4); e += PoolSelect::THREADS) {
        const int j = e / (D / 4), part = e % (D / 4);
        int c = 0, jb = j;
        while (jb >= n_b) { jb -= n_b; ++c; }
        cp_async16(smem_u32(s_k) + (j * LD + part * 4) * 4, tab.pooled[c] + ((size_t)bh * n_b + jb) * D + part * 4, true);
    }
    cp_async_commit();
}

// 128-token blocks, at most sixteen a head (KPL 2: T_n <= 64, 4: <= 128).  grid (T_m, B*H), cluster (T_m): a thread block pools its query block (threads 0 .. 255) and the key
// block of the same number (the others), hands the key mean round the cluster through distributed shared memory, and ranks its row.
template <int D, int KPL>
__global__ void __launch_bounds__(PoolSelect::THREADS) k_pool_select(ChunkTable tab, const bf16* __restrict__ q, const bf16* __restrict__ k, int Tc,
                                                                     int Tm, int Tn, int keep, float neg_zero, SelectOut o) {
    constexpr int VEC = D / 16, MAXR = 8, LD = D + 4;       // MAXR: rows per chain
    typedef typename VecLoad<VEC>::T V;
    extern __shared__ __align__(16) float sel_smem[];
    float* s_k = sel_smem;                      // [T_n][LD]: key rows, cached chunks' first
    float* s_q = s_k + Tn * LD;                 // [D]
    float* s_part = s_q + D;                    // [2][16][D]: chains of the two blocks
    float* s_sc = s_part + 2 * 16 * D;          // [Tn]
    const int b = blockIdx.x, bh = blockIdx.y, n_old = Tn - Tm, n = min(128, Tc - b * 128);
    if (Tm > 1) cluster_arrive();               // (no thread block writes to another's shared memory before that one has started)
    pdl_wait();
    pdl_trigger();              // the attention kernel may be made resident as blocks of this grid leave
    const int x = threadIdx.x >> 8, r = (threadIdx.x & 255) >> 4, cv = threadIdx.x & 15;
    const bf16* src = (x == 0 ? q : k) + ((size_t)bh * Tc + (size_t)b * 128 + r) * D + cv * VEC;
    V u[MAXR];
#pragma unroll
    for (int i = 0; i < MAXR; ++i)
        if (r + 16 * i < n) u[i] = __ldg(reinterpret_cast<const V*>(src + (size_t)(16 * i) * D));
    load_cached_keys<D, LD>(s_k, tab, n_old, Tm, bh);
    // ---- the block's mean in the canonical order
    float acc[VEC];
#pragma unroll
    for (int e = 0; e < VEC; ++e) acc[e] = 0.f;
#pragma unroll
    for (int i = 0; i < MAXR; ++i) {
        if (r + 16 * i < n) {
            float f[VEC];
            VecLoad<VEC>::widen(u[i], f);
#pragma unroll
            for (int e = 0; e < VEC; ++e) acc[e] = __fadd_rn(acc[e], f[e]);
        }
    }
    float* part = s_part + (x * 16 + r) * D + cv * VEC;
#pragma unroll
    for (int e = 0; e < VEC; e += 4) *reinterpret_cast<float4*>(part + e) = make_float4(acc[e], acc[e + 1], acc[e + 2], acc[e + 3]);
    __syncthreads();
    if (Tm > 1) cluster_wait();
    if (threadIdx.x < 2 * D) {
        const int y = threadIdx.x / D, col = threadIdx.x % D;
        float tot = s_part[y * 16 * D + col];
#pragma unroll
        for (int rr = 1; rr < 16; ++rr) tot = __fadd_rn(tot, s_part[(y * 16 + rr) * D + col]);
        const float mean = __fdiv_rn(tot, (float)n);
        float* key = s_k + (n_old + b) * LD + col;
        if (y == 0) s_q[col] = mean;
        else if (Tm == 1) *key = mean;
        else for (int z = 0; z < Tm; ++z) cluster_store(smem_u32(key), z, mean);
    }
    cp_async_wait<0>();
    if (Tm > 1) { cluster_arrive(); cluster_wait(); }       // every key mean is in place in every thread block
    else __syncthreads();
    score_pass<D, 1>([&](int j) { return s_k + j * LD; }, Tn, s_q, 1, s_sc, Tn, make_float2(neg_zero, neg_zero));
    __syncthreads();
    finish_rows<KPL, 1, 1>(s_sc, nullptr, bh, b, 1, Tm, Tn, Tm, keep, o, UnionOut{nullptr, nullptr, 0, Tc});      // (T_n <= 8 chunks of 16 blocks)
}

// 16-token blocks, at most eight a head (one unit of the attention kernel).  grid (1, B*H).  Sixteen chains of one token: a thread takes a
// block's pair of columns, sixteen loads in flight.
template <int D>
__global__ void __launch_bounds__(PoolSelect::THREADS) k_pool_select16(ChunkTable tab, const bf16* __restrict__ q, const bf16* __restrict__ k, int Tc,
                                                                       int Tm, int Tn, int keep, float neg_zero, SelectOut o, UnionOut lists) {
    constexpr int R = 8, BLK = 16, LD = D + 4, TPB = D / 2, BPS = PoolSelect::THREADS / TPB;
    extern __shared__ __align__(16) float sel_smem[];
    float* s_k = sel_smem;                      // [T_n][LD]: key rows, cached chunks' first
    float* s_q = s_k + Tn * LD;                 // [R][D]
    float* s_sc = s_q + R * D;                  // [R][Tn]
    __shared__ uint32_t s_mask[R][32];
    const int n_old = Tn - Tm, bh = blockIdx.y;
    pdl_wait();
    pdl_trigger();
    load_cached_keys<D, LD>(s_k, tab, n_old, Tm, bh);
#pragma unroll 1
    for (int w = threadIdx.x / TPB; w < 2 * Tm; w += BPS) {         // query blocks, then key blocks
        const int b = w < Tm ? w : w - Tm, n = min(BLK, Tc - b * BLK), col = (threadIdx.x % TPB) * 2;
        const bf16* src = (w < Tm ? q : k) + ((size_t)bh * Tc + (size_t)b * BLK) * D + col;
        uint32_t u[16];
#pragma unroll
        for (int t = 0; t < 16; ++t) u[t] = t < n ? __ldg(reinterpret_cast<const uint32_t*>(src + (size_t)t * D)) : 0u;
        float2 tot;
#pragma unroll
        for (int t = 0; t < 16; ++t) {
            const float2 f = unpack_bf16(u[t]);
            const float x0 = __fadd_rn(0.f, f.x), x1 = __fadd_rn(0.f, f.y);
            tot.x = t == 0 ? x0 : __fadd_rn(tot.x, x0);
            tot.y = t == 0 ? x1 : __fadd_rn(tot.y, x1);
        }
        float* at = w < Tm ? s_q + b * D + col : s_k + (n_old + b) * LD + col;
        at[0] = __fdiv_rn(tot.x, (float)n);
        at[1] = __fdiv_rn(tot.y, (float)n);
    }
    cp_async_wait<0>();
    __syncthreads();
    score_pass<D, R>([&](int j) { return s_k + j * LD; }, Tn, s_q, Tm, s_sc, Tn, make_float2(neg_zero, neg_zero));
    __syncthreads();
    finish_rows<2, 8, R>(s_sc, s_mask, bh, 0, Tm, Tm, Tn, Tm, keep, o, lists);
}
