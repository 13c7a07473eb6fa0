// Head dim 128, blocks of 16 and 64 tokens: column groups.
#include "hf_swa_tc5.h"
#include "k_swa_tc5.cuh"

template <int BLK>
static const void* kernel(int history, bool ahead) {
    if (ahead) return history == 0 ? nullptr : history == 1 ? (const void*)k_swa_tc5<128, BLK, 1, false, true> : (const void*)k_swa_tc5<128, BLK, 2, false, true>;
    return history == 0 ? (const void*)k_swa_tc5<128, BLK, 0, false, false>
         : history == 1 ? (const void*)k_swa_tc5<128, BLK, 1, false, false> : (const void*)k_swa_tc5<128, BLK, 2, false, false>;
}
const void* swa_tc5_kernel_d128_small(int block, int history, bool teams, bool ahead) {
    return teams ? nullptr : block == 64 ? kernel<64>(history, ahead) : kernel<16>(history, ahead);
}
