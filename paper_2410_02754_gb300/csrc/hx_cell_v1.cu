// FP32 cell apply, variant 1: 2 vectors per item, 256 threads, registers sized for 3 CTAs per SM,
// paired FP32 multiply-adds
// (p = 2..5, nq = p + 2).
#include "hx_cell.cuh"

cudaError_t launch_cell_f32_v1(const CellJob* jobs, int n, cudaStream_t s) {
  return gbc::launch_cell_group<2, 256, 3, true>(jobs, n, s);
}

GBC_CHECK_WORD_ACCESSOR(gbc_check_word_cell1)
