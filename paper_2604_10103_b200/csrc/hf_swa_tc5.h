// The instantiations of the tcgen05 attention kernel (k_swa_tc5.cuh), as handles for the runtime's launch and attribute calls.  They are compiled in files of
// their own, a device module each, which the runtime loads when a context first touches a kernel in it.  The first context of a process pays for modules by their
// size, and these kernels are more than half of the device code; a context reaches those of one file.  First context of a process, one module / four, ms:
// head dim 128, 128-token blocks 34.7 / 22.8, 64-token blocks 33.4 / 22.7; head dim 64, 128-token blocks 34.3 / 21.8, 16-token blocks 33.9 / 23.1 (compressed for size
// 28.8-31.1).
#pragma once

// history: 0 none (or another kernel's, added), 1 formed here, 2 with a rotated numerator.  nullptr: no such form.
const void* swa_tc5_kernel_d64(int block, int history, bool teams);
const void* swa_tc5_kernel_d128(int history, bool teams, bool ahead);                       // 128-token blocks
const void* swa_tc5_kernel_d128_small(int block, int history, bool teams, bool ahead);      // blocks of 16 and 64 tokens
inline const void* swa_tc5_kernel(int d, int block, int history, bool teams, bool ahead) {
    if (d == 64) return ahead ? nullptr : swa_tc5_kernel_d64(block, history, teams);
    return block == 128 ? swa_tc5_kernel_d128(history, teams, ahead) : swa_tc5_kernel_d128_small(block, history, teams, ahead);
}
