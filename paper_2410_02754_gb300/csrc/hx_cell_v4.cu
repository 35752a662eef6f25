// FP32 cell apply, variant 4: 4 vectors per item, 512 threads, one CTA per SM, paired FP32 multiply-adds
// (p = 2..7, nq = p + 2).
// The gather reads 32 contiguous bytes per node row and spin.
#include "hx_cell.cuh"

cudaError_t launch_cell_f32_v4(const CellJob* jobs, int n, cudaStream_t s) {
  return gbc::launch_cell_group<4, 512, 1, true>(jobs, n, s);
}

GBC_CHECK_WORD_ACCESSOR(gbc_check_word_cell4)
