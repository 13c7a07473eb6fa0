// Which of two forms a call takes, where that is a function of numbers alone (host code without CUDA).
#pragma once

// Whether pooling and selection are one launch: where a head's blocks are few, so that a thread block per query block (128 tokens; a cluster
// has sixteen, above eight by its kernel's attribute) or one for all (16 tokens) has little to pool, and the launch it spares weighs more.  From six blocks a head on, a grid well
// above the SMs is slower than the other form, which spreads the pooling evenly.  Forward calls without and with it, 3 chunks cached: 128-token
// blocks, 12 heads of 128, 700 queries (T_m 6) 16.7 / 14.7 us, 1 024 (T_m 8) 18.6 / 17.2, 1 300 (T_m 11) 25.2 / 22.3, 2 048 (T_m 16) 42.2 / 39.1; 24 heads of 64, 1 024 queries 23.0 / 20.8, 48
// heads 32.1 / 32.8; 16-token blocks, 2 heads of 64 queries 11.8 / 11.0, 12 heads of 300 queries (T_m 19) 28.1 / 29.1.
// clusters: how many clusters of T_m thread blocks the device holds at a time.  None (a partition with small groups of SMs): two launches.
inline bool pool_select_one_launch(int block, int Tm, int BH, int sm_count, int clusters) {
    if (block == 16) return Tm <= 8;
    if (block != 128 || (Tm > 1 && clusters < 1)) return false;
    return Tm <= 5 || (Tm <= 16 && 2 * BH * Tm <= 3 * sm_count);
}
