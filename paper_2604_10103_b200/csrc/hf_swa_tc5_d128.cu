// Head dim 128, 128-token blocks: teams and column groups.
#include "hf_swa_tc5.h"
#include "k_swa_tc5.cuh"

const void* swa_tc5_kernel_d128(int history, bool teams, bool ahead) {
    if (teams)
        return ahead ? nullptr : history == 0 ? (const void*)k_swa_tc5<128, 128, 0, true, false>
                               : history == 1 ? (const void*)k_swa_tc5<128, 128, 1, true, false> : (const void*)k_swa_tc5<128, 128, 2, true, false>;
    if (ahead) return history == 0 ? nullptr : history == 1 ? (const void*)k_swa_tc5<128, 128, 1, false, true> : (const void*)k_swa_tc5<128, 128, 2, false, true>;
    return history == 0 ? (const void*)k_swa_tc5<128, 128, 0, false, false>
         : history == 1 ? (const void*)k_swa_tc5<128, 128, 1, false, false> : (const void*)k_swa_tc5<128, 128, 2, false, false>;
}
