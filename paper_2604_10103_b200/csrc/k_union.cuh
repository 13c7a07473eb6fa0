// Merged kept lists of the query blocks that share a 128-row unit of the attention kernel (blocks of 16 or 64 tokens): which
// key blocks the unit walks, in which order, and which of its row groups keep each.  Formed by the selection kernel for the lists
// it has just made, by a kernel of its own for lists that come from the caller: behind the selection that one costs its launch and
// a trip through L2 (forward call, 12 heads: 16-token blocks at head dim 64, 1 300 queries 53.5 -> 50.9 us; 64-token blocks, 4 680 queries
// 161.0 -> 157.6 us; two heads of 64 queries 12.8 -> 11.7 us, all with the lists formed in the selection kernel).
#pragma once
#include "hf_common.cuh"

// One list entry: key block index (10 bits) | row groups that keep it (8 bits) << 10 | valid tokens in the block << 18.
__host__ __device__ __forceinline__ uint32_t union_entry(int blk, uint32_t rows, int nv) { return (uint32_t)blk | (rows << 10) | ((uint32_t)nv << 18); }

struct UnionOut {
    uint32_t* entries;       // [B*H * units, max_tiles, G], or nullptr: not wanted
    int* tiles;              // [B*H * units]
    int max_tiles, Tc;
};

// Where entry number i of class x goes in a unit's list; slots that stay empty get a padding entry.
//   G = 8: class 0 = some row group's lowest kept block, class 1 = the rest; class after class.  (A unit's first tile has to hold a
//          kept block of every row group: there are at most eight of class 0.)
//   G = 2: class 0 = kept by both row groups, 1 and 2 = kept by the first or the second alone.  The blocks of class 0 come first, two
//          to a tile, then one of class 1 beside one of class 2: in such a tile every row has one key block to weigh instead of two
//          or none, and the four schedulers have the same share of it.  In ascending order three of four tiles have a row group
//          that keeps both blocks, and the tile takes as long as a full one.  An odd block of class 0 has the first of what is left over
//          beside it, if the classes differ in length (one row group alone past the last query block, or a caller's list with repeats).
template <int G>
struct UnionOrder {
    int n0, n1, n2;
    __host__ __device__ int odd() const { return G == 2 ? n0 & 1 : 0; }
    __host__ __device__ int pairs() const { return n1 < n2 ? n1 : n2; }
    __host__ __device__ int rest() const { return n1 < n2 ? n2 - n1 : n1 - n2; }
    __host__ __device__ int slots() const {
        if (G != 2) return n0 + n1;
        return n0 + odd() + 2 * pairs() + (rest() > 0 ? rest() - odd() : 0);
    }
    __host__ __device__ int slot(int x, int i) const {
        if (G != 2) return x == 0 ? i : n0 + i;
        if (x == 0) return i;
        const int m = pairs(), c = n0 + odd();
        if (i < m) return c + 2 * i + x - 1;
        return odd() && i == m ? n0 : c + 2 * m + i - m - odd();
    }
    // padding inside the list (G = 2 only), or -1
    __host__ __device__ int hole() const { return odd() && rest() == 0 ? n0 : -1; }
};

// One unit's list, by nw warps of which the calling one is number w.  m [G][32]: the row groups' kept blocks as bit masks in shared
// memory (complete for all warps).  A padding entry repeats the unit's first block with no row group: it is loaded -- every box of
// a tile must hold finite numbers -- and fully masked.
template <int G>
__device__ __forceinline__ void union_lists(const uint32_t (*m)[32], int w, int nw, int Tn, int n_b, int unit, const UnionOut& u) {
    constexpr int BLK = 128 / G;
    const int lane = threadIdx.x & 31;
    uint32_t a0 = 0, a1 = 0, a2 = 0;            // lane l: word l of the classes
    if constexpr (G == 2) {
        const uint32_t x = m[0][lane], y = m[1][lane];
        a0 = x & y; a1 = x & ~y; a2 = y & ~x;
    } else {
        uint32_t all = 0;
#pragma unroll
        for (int r = 0; r < G; ++r) {
            const uint32_t x = m[r][lane];
            const int first = __ffs(__ballot_sync(0xffffffffu, x != 0)) - 1;
            if (lane == first) a0 |= x & (0u - x);
            all |= x;
        }
        a1 = all & ~a0;
    }
    const uint32_t all = a0 | a1 | a2;
    UnionOrder<G> ord;
    ord.n0 = __reduce_add_sync(0xffffffffu, __popc(a0));
    ord.n1 = __reduce_add_sync(0xffffffffu, __popc(a1));
    ord.n2 = G == 2 ? __reduce_add_sync(0xffffffffu, __popc(a2)) : 0;
    uint32_t* out = u.entries + (size_t)unit * u.max_tiles * G;
    const uint32_t below = (1u << lane) - 1u;
    for (int x = w; x < (Tn + 31) / 32; x += nw) {
        const uint32_t w0 = __shfl_sync(0xffffffffu, a0, x), w1 = __shfl_sync(0xffffffffu, a1, x), w2 = __shfl_sync(0xffffffffu, a2, x);
        const int b0 = __reduce_add_sync(0xffffffffu, lane < x ? __popc(a0) : 0), b1 = __reduce_add_sync(0xffffffffu, lane < x ? __popc(a1) : 0);
        const int b2 = G == 2 ? __reduce_add_sync(0xffffffffu, lane < x ? __popc(a2) : 0) : 0;
        if (((w0 | w1 | w2) >> lane) & 1u) {
            const int j = 32 * x + lane;
            uint32_t rows = 0;
#pragma unroll
            for (int r = 0; r < G; ++r) rows |= ((m[r][x] >> lane) & 1u) << r;
            int jb = j;
            while (jb >= n_b) jb -= n_b;
            const int nv = jb == n_b - 1 ? u.Tc - jb * BLK : BLK;
            const int at = (w0 >> lane) & 1u ? ord.slot(0, b0 + __popc(w0 & below))
                         : (w1 >> lane) & 1u ? ord.slot(1, b1 + __popc(w1 & below)) : ord.slot(2, b2 + __popc(w2 & below));
            out[at] = union_entry(j, rows, nv);
        }
    }
    if (w == 0) {
        const int fl = __ffs(__ballot_sync(0xffffffffu, all != 0)) - 1;      // (a list has at least one block)
        const int pad = 32 * fl + __ffs(__shfl_sync(0xffffffffu, all, fl)) - 1;
        const int slots = ord.slots(), n_tiles = (slots + G - 1) / G;
        if (lane < n_tiles * G - slots) out[slots + lane] = union_entry(pad, 0u, BLK);
        if (lane == 0 && ord.hole() >= 0) out[ord.hole()] = union_entry(pad, 0u, BLK);
        if (lane == 0) u.tiles[unit] = n_tiles;
    }
}

// Lists from a caller.  grid (units per batch*head, B*H), 256 threads.  idx: [B*H, T_m, keep].
template <int BLK>
__global__ void __launch_bounds__(256) k_union_tiles(const int32_t* __restrict__ idx, int keep, int Tm, int Tn, int n_b, UnionOut u, int* dev_status) {
    constexpr int G = 128 / BLK;
    __shared__ uint32_t m[G][32];
    const int mt = blockIdx.x, bh = blockIdx.y;
    if (threadIdx.x < G * 32) m[threadIdx.x >> 5][threadIdx.x & 31] = 0;
    __syncthreads();
    pdl_wait();                 // the lists come from the selection kernel launched before this one
    pdl_trigger();
    for (int e = threadIdx.x; e < G * keep; e += 256) {
        const int r = e / keep, jj = e - r * keep, qb = mt * G + r;
        if (qb < Tm) {
            const int j = checked_block(__ldg(idx + ((size_t)bh * Tm + qb) * keep + jj), Tn, dev_status, bh * Tm + qb);
            atomicOr(&m[r][j >> 5], 1u << (j & 31));
        }
    }
    __syncthreads();
    union_lists<G>(m, threadIdx.x >> 5, 8, Tn, n_b, bh * gridDim.x + mt, u);
}
