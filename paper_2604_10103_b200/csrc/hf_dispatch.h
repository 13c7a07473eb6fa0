// Which of two forms a call takes, where that is a function of numbers alone (host code without CUDA).
#pragma once

// Pooling and selection of a head's blocks in one launch: sixteen-token blocks, at most eight a head, by one thread block (faster on any
// grid: 12 to 1 024 heads 1.11 to 1.38 times); 128-token blocks, at most sixteen a head, by a cluster with a thread block for each (a single
// block: a thread block alone, faster on any grid).
//
// The cluster form spares a launch and the means' way through L2 as long as the clusters of all heads are resident at a time.  Behind
// the first wave it loses: the two-launch form has shorter thread blocks and spreads the pooling evenly.  `clusters` is how many of T_m thread
// blocks the device holds by its own count, `clusters16` how many of sixteen (hf_create asks; 0: none fits, as on a partition with small
// groups of SMs).  The last tenth of the count is not reached in one wave, and clusters of 11 to 15 get little more than the room of 16: heads
// of 128 lose from 15 to 17 heads on where the count says 21 to 14, heads of 64 at about four fifths of it.  Forward calls, three chunks
// cached, two launches / one, up to the line and past it (B200: 148 SMs):
//   heads of 128, T_m 3  (93 clusters)  81 heads 26.0 / 22.8 us,  94 heads 26.8 / 27.0     384 heads 73.0 / 80.1
//                 T_m 5  (56)           49 heads 28.2 / 25.5,     52 heads 28.3 / 28.3    1 024 heads 371 / 431
//                 T_m 8  (33)           28 heads 30.9 / 27.9,     33 heads 31.9 / 32.0    55 heads 43.3 / 43.9
//                 T_m 10 (26)           22 heads 34.2 / 32.1,     24 heads 35.3 / 35.7
//                 T_m 13 (as 16: 14)    14 heads 37.8 / 34.6,     16 heads 38.0 / 39.2    34 heads 54.0 / 58.9
//                 T_m 16 (14)           14 heads 41.7 / 38.9,     15 heads 42.8 / 43.5    27 heads 59.8 / 60.4
//   heads of 64,  T_m 11 (21)           17 heads 27.5 / 26.0,     19 heads 27.7 / 28.6
//                 T_m 12 (21)           17 heads 27.7 / 27.0,     19 heads 28.0 / 29.7
inline bool pool_select_one_launch(int block, int d, int Tm, int BH, int clusters, int clusters16) {
    if (block == 16) return Tm <= 8;
    if (block != 128 || Tm > 16) return false;
    if (Tm <= 10) return Tm == 1 || 10 * BH <= 9 * clusters;
    return BH <= clusters16 || (d == 64 && 5 * BH <= 4 * clusters);
}

// Whether a call that could be a copy may launch a kernel instead.  A copy takes any memory that the runtime can copy between; a kernel
// runs on the calling thread's current device, and reaches for certain only memory of its own.  (A copy also takes a stream of another device.
// A launch refuses that, which a caller of this has to answer with the copy: the runtime's question for a stream's device may not be
// asked while it is being captured.)
struct CallerMemory { bool given, aligned, device_memory; int device; };
inline bool kernel_instead_of_copy(int context_device, int current_device, const CallerMemory& m) {
    return current_device == context_device && (!m.given || (m.aligned && m.device_memory && m.device == context_device));
}

// Registers of the selection's ranking warps: T_n / 32 images per lane, in steps.
inline int select_kpl(int Tn) { return Tn <= 128 ? 4 : Tn <= 256 ? 8 : Tn <= 512 ? 16 : 32; }
// Whether a context whose windows have n_b .. max_Tn key blocks ever launches the step's kernel.
inline bool select_uses(int kpl, int n_b, int max_Tn) { return select_kpl(n_b) <= kpl && kpl <= select_kpl(max_Tn); }

// Query blocks that a thread block of the selection takes: eight where they share a unit's list (G 8: 16-token blocks) and for more than 256 key
// blocks; with 129 to 256, which are all in shared memory at once, eight where four would give more thread blocks than SMs ...
inline int select_rows(int kpl, int G, int Tm, int BH, int sms) {
    if (G == 8 || kpl > 8) return 8;
    return kpl == 8 && (Tm + 3) / 4 * BH > sms ? 8 : 4;
}
inline constexpr int select_smem_bytes(int d, int rows, int key_rows, int Tn) { return (key_rows * (d + 4) + rows * d + rows * Tn) * 4; }
// ... unless those are through in fewer rounds: an SM holds up to three thread blocks of four by registers (72 or 80 of 256 threads), by shared memory
// three at head dim 64 and up to 136 key blocks at 128, two up to 208, then one; of eight it holds one (76 or 86 registers of 512 threads).
// Pooling and selection of 64-token blocks, four / eight, us (forward calls: the same differences):
//   head dim 64, thread blocks of four in one round, of eight in two: T_n 130, 24 heads 12.0 / 15.6; 148, 16 heads 10.9 / 13.1; 180, 16 heads 12.3 / 15.6;
//   208, 12 and 16 heads 12.4 / 15.3, 13.9 / 17.1; 222, 16 heads 12.3 / 14.1; 250, 12 heads 13.9 / 17.1; two rounds, three of eight: 208, 24 heads 21.2 / 24.1;
//   250, 24 heads 25.3 / 26.7; as many: 130, 8, 12, 16 heads 7.7 / 8.0, 8.7 / 8.8, 10.2 / 9.5; 180, 8, 12, 24 heads 9.3 / 9.0, 11.2 / 9.8, 19.0 / 17.9; 222, 8, 12, 24
//   heads 9.8 / 9.0, 10.8 / 9.6, 17.6 / 17.5; 250, 8, 16 heads 11.5 / 10.3, 19.8 / 18.7
//   head dim 128, one round, two: 130, 24 heads 17.2 / 21.1; as many: 130, 12, 16 heads 13.5 / 11.8, 14.7 / 12.7; 148, 8 to 24 heads 11.2 / 11.4, 12.6 / 12.7, 18.3 / 18.0,
//   22.7 / 22.5; 180 13.0 / 12.2, 14.6 / 13.4, 21.4 / 21.6, 27.0 / 25.0; 208 14.1 / 13.0, 21.4 / 21.6, 23.7 / 23.5, 35.8 / 34.7; fewer of eight: 222 16.8 / 11.9, 18.8 / 13.5,
//   26.1 / 19.8, 35.0 / 24.2; 250 19.8 / 14.7, 28.8 / 23.8, 37.8 / 26.3, 56.9 / 40.7
// (The form with its key rows in two passes had three thread blocks to an SM at head dim 128 too: where that was one round and this is two, 148 to 250 key
// blocks with 304 to 416 thread blocks of four, pooling and selection alone take up to 1.07 times as long as they did, a forward call as long.)
inline int select_rows_of(int kpl, int G, int d, int Tn, int Tm, int BH, int sms) {
    const int rows = select_rows(kpl, G, Tm, BH, sms);
    if (G == 8 || kpl != 8 || rows == 4) return rows;
    const int fit = (228 << 10) / (select_smem_bytes(d, 4, Tn, Tn) + (G > 1 ? 512 : 128) + 1024), resident = fit < 3 ? fit : 3;
    const int rounds4 = ((Tm + 3) / 4 * BH + resident * sms - 1) / (resident * sms), rounds8 = ((Tm + 7) / 8 * BH + sms - 1) / sms;
    return rounds8 <= rounds4 ? 8 : 4;
}
// Whether some window of a context, n_b, 2 n_b .. max_Tn key blocks, launches the step's kernel with that many.
inline bool select_uses_rows(int kpl, int rows, int G, int d, int n_b, int max_Tn, int Tm, int BH, int sms) {
    for (int Tn = n_b; Tn <= max_Tn && select_uses(kpl, n_b, max_Tn); Tn += n_b)
        if (select_kpl(Tn) == kpl && select_rows_of(kpl, G, d, Tn, Tm, BH, sms) == rows) return true;
    return false;
}

// Softmax warps of the tcgen05 attention kernel in teams that take turns at the tiles, or in column groups on the same one (k_swa_tc5.cuh).  Head
// dim 64: teams.  Several units a thread block, 1 to 40 tiles: 1.01 to 1.13 times as fast.  One unit of few tiles has none to take turns at and pays for
// the hand-overs; two column groups (from five tiles on: four) / teams, forward calls (softmax branch alone), us:
//   12 units, 1, 3, 6 tiles 7.5 / 7.5, 9.3 / 9.2, 11.3 / 11.4  (5.8 / 6.1, 7.4 / 7.4, 9.6 / 9.6)
//   36 units, 1, 3, 6, 12 tiles 8.3 / 8.5, 10.1 / 10.1, 12.4 / 12.4, 16.9 / 16.5  (6.0 / 6.1, 7.6 / 7.5, 9.8 / 9.5, 14.0 / 13.6)
//   132 units, 1, 3, 6, 12, 16 tiles 9.9 / 10.3, 11.8 / 12.1, 14.1 / 14.3, 19.0 / 19.0, 22.4 / 22.2  (6.1 / 6.6, 7.8 / 8.1, 10.0 / 10.5, 14.5 / 15.3, 17.4 / 18.3)
//   156 units, 1, 3, 8 tiles 13.0 / 12.4, 16.2 / 15.3, 23.5 / 22.2  (8.2 / 7.3, 11.5 / 10.5, 18.6 / 17.7)
// The line cannot lie at the number of units: the two forms add a row's weights in another order, and the same head would not have the same bits in a call
// with other heads beside it.  Head dim 128, 128-token blocks: teams from 14 tiles on, from
// 8 without the history term, whose operand they keep in an S buffer; column groups / teams, forward calls (softmax branch alone), us:
//   132 units, 10 tiles 22.1 / 22.2, 12 tiles 23.9 / 23.7, 14 tiles 25.8 / 25.2, 24 tiles 34.7 / 32.7  (8 tiles 14.4 / 14.4, 12 tiles 18.3 / 16.8)
//   448 units, 10 tiles 67.1 / 69.3, 12 tiles 73.9 / 75.4, 14 tiles 81.0 / 80.9, 24 tiles 119.9 / 114.8  (8 tiles 44.6 / 41.0, 4 tiles 29.7 / 29.0)
// and column groups for its blocks of 16 and 64 tokens (0.90 to 0.98 times as fast with teams).
inline constexpr bool swa_teams(int d, int block, int tiles, bool history) { return d == 64 || (block == 128 && tiles >= (history ? 14 : 8)); }

// Whether the attention kernel's column groups form their first unit's history term ahead of the selection's end.  It is for nothing where the
// thread block is resident early, which takes an SM that the selection leaves free, and on the chain in front of the first tile where it is not.  What
// counts are the thread blocks of the last round, the first on the device and the last to finish.  Forward calls, heads of 128, behind / ahead, us:
//   128-token blocks, 12 units (12 selection blocks) of 1, 3, 8 tiles 10.8 / 10.0, 12.6 / 11.6, 16.6 / 15.6; 132 units (36) 14.5 / 15.1, 16.3 / 16.9,
//   20.5 / 21.1; 320 units, 24 in the last round (80) 29.1 / 27.1, 33.8 / 33.4, 47.0 / 46.6; 444 units, 148 in the last round 30.7 / 31.2, 35.6 / 36.8,
//   50.1 / 50.5
//   64-token blocks, 132 units of 2, 8, 20 kept blocks, T_n 84 (72) 18.4 / 17.4, 22.2 / 21.2, 28.3 / 27.5; 444 units 46.4 / 47.2, 62.3 / 63.1, 80.2 / 81.3; 1 776
//   units, T_n 74 141.6 / 145.5
//   16-token blocks (a thread block of the selection for each unit), 2 units of 2 and 8 kept blocks 12.8 / 11.5, 13.7 / 12.4; 12 units 13.3 / 12.1, 14.5 / 13.2; 36 units of 2,
//   8, 30 16.3 / 15.2, 20.9 / 20.4, 24.6 / 24.0; 132 units 22.8 / 23.3, 28.9 / 30.3, 42.8 / 44.3; 320 units 43.9 / 44.3, 57.0 / 57.3, 81.9 / 82.4
// No selection in front (selection_blocks 0: attention on lists that are there before the call): nothing to wait for, the term is only in the way of
// the first tile, and behind k_union_tiles there is less time than it takes.  hf_sparse_swa_merged, behind / ahead, us:
//   128-token blocks, 12 units of 1, 3, 8 tiles 8.4 / 9.3, 9.9 / 10.9, 14.0 / 15.1; 300 units 19.9 / 20.9, 22.6 / 23.9, 35.6 / 36.8
//   64-token blocks, 12 units of 2 and 8 kept blocks 9.7 / 10.0, 13.1 / 13.6; 156 units of 2, 8, 20 16.0 / 16.6, 23.9 / 24.9, 39.0 / 40.2
//   16-token blocks, 12 units of 4 and 30 kept blocks 12.0 / 12.5, 18.5 / 19.1; 132 units 14.7 / 14.0, 36.9 / 36.4
inline bool swa_history_ahead(int block, int units, int selection_blocks, int sms) {
    if (selection_blocks == 0) return false;
    const int last = units % sms ? units % sms : sms;
    return last + selection_blocks <= sms || (block == 64 && units < sms);
}
