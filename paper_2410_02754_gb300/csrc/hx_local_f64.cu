// FP64 instantiations of the matrix-free cell apply (p = 2..7, nq = p + 2).
#include "hx_local.cuh"

// dispatch on p (nq = p + 2)
static cudaError_t launch_hx_group(const HxJob* jobs, int n, cudaStream_t s) {
  switch (jobs[0].c->mesh.p) {
    case 2: return gbc::launch_hx_group_p<3>(jobs, n, s);
    case 3: return gbc::launch_hx_group_p<4>(jobs, n, s);
    case 4: return gbc::launch_hx_group_p<5>(jobs, n, s);
    case 5: return gbc::launch_hx_group_p<6>(jobs, n, s);
    case 6: return gbc::launch_hx_group_p<7>(jobs, n, s);
    case 7: return gbc::launch_hx_group_p<8>(jobs, n, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_hx_local_group_f64(const HxJob* jobs, int n, cudaStream_t s) {
  return launch_hx_group(jobs, n, s);
}

cudaError_t launch_cell_gather_f64(const gbc_ctx* c, const double2* Ycell, double2* Y, int nvec,
                                   int ldx, cudaStream_t s) {
  const long long n = c->mesh.M * 2 * (long long)nvec;
  if (n <= 0) return cudaSuccess;
  const unsigned grid = (unsigned)std::min<long long>((n + 255) / 256, 64LL * gbc_sm_count());
  gbc::k_cell_gather<double><<<grid, 256, 0, s>>>(Y, Ycell, c->mesh, nvec, ldx);
  return cudaGetLastError();
}

GBC_CHECK_WORD_ACCESSOR(gbc_check_word_hx64)
