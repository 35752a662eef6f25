// Dispatch of the FP32 cell apply over its compiled variants (chosen per
// context by the autotuner, gbc_tune).
#include "gbc_internal.h"

cudaError_t launch_cell_f32_v0(const CellJob* jobs, int n, cudaStream_t s);
cudaError_t launch_cell_f32_v1(const CellJob* jobs, int n, cudaStream_t s);
cudaError_t launch_cell_f32_v2(const CellJob* jobs, int n, cudaStream_t s);
cudaError_t launch_cell_f32_v3(const CellJob* jobs, int n, cudaStream_t s);
cudaError_t launch_cell_f32_v4(const CellJob* jobs, int n, cudaStream_t s);

CellVariant cell_variant(int v) {
  static const CellVariant tab[GBC_CELL_VARIANTS] = {{2, 256, 2, 1}, {2, 256, 3, 1},
                                                     {2, 256, 2, 0}, {2, 256, 3, 0},
                                                     {4, 512, 1, 1}};
  return tab[(v >= 0 && v < GBC_CELL_VARIANTS) ? v : 0];
}

// Registers for 3 CTAs per SM (80 a thread) hold no pencil of p = 6 or 7: 110 to 250 bytes spilled, and at
// p = 6 shared memory lets two CTAs in.  Variants 1 and 3 are there 0 and 2 (64 vectors, k != 0: p = 6 on
// 10^3 cells 593 -> 508 us a launch for variant 1, p = 7 on 11 x 9 x 8 cells 840 -> 709).
cudaError_t launch_cell_f32(const CellJob* jobs, int n, int variant, cudaStream_t s) {
  if ((variant == 1 || variant == 3) && jobs[0].c->mesh.p >= 6) --variant;
  switch (variant) {
    case 1: return launch_cell_f32_v1(jobs, n, s);
    case 2: return launch_cell_f32_v2(jobs, n, s);
    case 3: return launch_cell_f32_v3(jobs, n, s);
    case 4: return launch_cell_f32_v4(jobs, n, s);
    default: return launch_cell_f32_v0(jobs, n, s);
  }
}
