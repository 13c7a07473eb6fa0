// Head dim 64: teams.
#include "hf_swa_tc5.h"
#include "k_swa_tc5.cuh"

template <int BLK>
static const void* kernel(int history) {
    return history == 0 ? (const void*)k_swa_tc5<64, BLK, 0, true, false>
         : history == 1 ? (const void*)k_swa_tc5<64, BLK, 1, true, false> : (const void*)k_swa_tc5<64, BLK, 2, true, false>;
}
const void* swa_tc5_kernel_d64(int block, int history, bool teams) {
    if (!teams) return nullptr;
    return block == 128 ? kernel<128>(history) : block == 64 ? kernel<64>(history) : kernel<16>(history);
}
