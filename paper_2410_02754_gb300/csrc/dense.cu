// Small dense FP64 complex linear algebra on the device (n <= 512):
// Cholesky S = L L^H, L^-H, and a parallel-order Jacobi Hermitian eigensolver.
//
// Paper: Sec. III.B.2 (the T x T projected problems of Rayleigh-Ritz); the
// Cholesky factor is the Cholesky-Gram-Schmidt orthonormalisation of X_s in the
// M_D inner product.
//
// Jacobi: round-robin ("circle") ordering makes n/2 disjoint (p, q) rotations
// per round; one launch applies all of them at once, A' = J^H A J, V' = V J, reading A and
// writing a second buffer, so a round needs no grid-wide synchronisation.  n - 1 rounds form
// a sweep; sweeps repeat until the off-diagonal Frobenius norm falls below 1e-14 ||A||_F.
// A thread owns the 2 x 2 block of two pairs: with J = diag(1, conj(ph)) [[c, s], [-s, c]] that
// is 12 FP64 operations an element (24 for an element at a time), which counts at 2 per clock
// and SM, and a block of 8 x 8 pairs computes its 16 rotations once.  A 200 x 200 matrix:
// 31.5 us a round with every element computing its own two rotations, 7.7 us with 2 x 2 blocks,
// 6.8 us with the rotation from two dependent roots (75 x 75: 18.3, 7.5, 6.8 us).
#include <cmath>

#include "gbc_internal.h"

namespace {

// ---- Cholesky, one column per launch ---------------------------------------
// For column j: L[i][j] = A[i][j] / sqrt(A[j][j]) (i >= j) and the trailing
// update A[i][k] -= A[i][j] conj(A[k][j]) / A[j][j] (i >= k > j).  Column j
// and A[j][j] are only read in this launch.
__global__ void k_chol_col(double2* A, double2* L, int n, int j, int* flag) {
  const int m = n - j;                       // rows j..n-1
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= (long long)m * m) return;
  const int i = j + (int)(t / m), k = j + (int)(t % m);
  if (k > i) return;
  const double d = A[(size_t)j * n + j].x;
  if (i == j && k == j) {
    if (!(d > 0.0)) *flag = 1;
  }
  if (!(d > 0.0)) return;
  if (k == j) {
    const double s = 1.0 / sqrt(d);
    const double2 a = A[(size_t)i * n + j];
    L[(size_t)i * n + j] = make_double2(a.x * s, a.y * s);
    return;
  }
  const double2 aij = A[(size_t)i * n + j], akj = A[(size_t)k * n + j];
  // aij conj(akj / d): the quotient first, whose size is that of column k over column j (the product
  // of the two entries leaves the range for columns 2^-256 of the largest)
  const double kx = akj.x / d, ky = akj.y / d;
  const double re = aij.x * kx + aij.y * ky;
  const double im = aij.y * kx - aij.x * ky;
  double2* a = &A[(size_t)i * n + k];
  a->x -= re;
  a->y -= im;
}

// Linv = L^-1 by forward substitution, one block per column c
__global__ void k_tri_inv(const double2* __restrict__ L, double2* Linv, int n) {
  __shared__ double2 y[512];
  __shared__ double2 red[256];
  const int c = blockIdx.x;
  for (int i = threadIdx.x; i < n; i += blockDim.x) y[i] = make_double2(0, 0);
  __syncthreads();
  for (int i = c; i < n; ++i) {
    // sum_{k=c}^{i-1} L[i][k] y[k]
    double2 acc = make_double2(0, 0);
    for (int k = c + threadIdx.x; k < i; k += blockDim.x) {
      const double2 l = L[(size_t)i * n + k], v = y[k];
      acc.x += l.x * v.x - l.y * v.y;
      acc.y += l.x * v.y + l.y * v.x;
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
      if (threadIdx.x < s) {
        red[threadIdx.x].x += red[threadIdx.x + s].x;
        red[threadIdx.x].y += red[threadIdx.x + s].y;
      }
      __syncthreads();
    }
    if (threadIdx.x == 0) {
      const double rhs_re = (i == c ? 1.0 : 0.0) - red[0].x;
      const double rhs_im = -red[0].y;
      const double2 d = L[(size_t)i * n + i];   // real positive diagonal
      y[i] = make_double2(rhs_re / d.x, rhs_im / d.x);
    }
    __syncthreads();
  }
  for (int i = threadIdx.x; i < n; i += blockDim.x) Linv[(size_t)i * n + c] = y[i];
}

// Q = Linv^H (upper triangular)
__global__ void k_conj_transpose(const double2* __restrict__ A, double2* B, int n) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= (long long)n * n) return;
  const int i = (int)(t / n), j = (int)(t % n);
  const double2 a = A[(size_t)j * n + i];
  B[(size_t)i * n + j] = make_double2(a.x, -a.y);
}

__global__ void k_hermitize(double2* A, int n) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= (long long)n * n) return;
  const int i = (int)(t / n), j = (int)(t % n);
  if (j < i) return;
  if (i == j) {
    A[(size_t)i * n + i].y = 0.0;
    return;
  }
  // the Gram kernels compute the upper triangle; the lower one is its mirror
  const double2 a = A[(size_t)i * n + j];
  A[(size_t)j * n + i] = make_double2(a.x, -a.y);
}

// ---- Jacobi --------------------------------------------------------------------
// pair k of round r, p < q (q >= n: p has no partner)
__device__ __forceinline__ void pair_of(int k, int r, int npad, int& p, int& q) {
  const int m = npad - 1;
  int a = m, b = r;
  if (k > 0) {
    a = r + k < m ? r + k : r + k - m;
    b = r - k >= 0 ? r - k : r - k + m;
  }
  p = min(a, b);
  q = max(a, b);
}

// rotation of a pair (p, q), both < n: J = [[c, s], [-s conj(ph), c conj(ph)]]
struct Rot { double c, s; double2 ph; };

__device__ __forceinline__ Rot make_rot(const double2* A, int n, int p, int q) {
  Rot r{1.0, 0.0, make_double2(1.0, 0.0)};
  if (q >= n) return r;
  const double2 apq = A[(size_t)p * n + q];
  const double app = A[(size_t)p * n + p].x, aqq = A[(size_t)q * n + q].x;
  const double del = 0.5 * (aqq - app), ad = fabs(del);
  const double m2 = apq.x * apq.x + apq.y * apq.y, d2 = del * del + m2;
  if (m2 > 1e-250 && d2 < 1e250) {   // no square overflows or loses bits
    // t = m / (del + sgn sqrt(del^2 + m^2)) with w = |del| + sqrt: c = w / sqrt(w^2 + m^2), s = c t;
    // two dependent roots instead of five roots and quotients (the round is bound by this chain)
    const double im = rsqrt(m2), mag = m2 * im;
    if (mag < 1e-18 * (fabs(app) + fabs(aqq))) return r;
    const double w = ad + sqrt(d2);
    const double h = rsqrt(w * w + m2);
    r.c = w * h;
    r.s = del >= 0 ? mag * h : -mag * h;
    r.ph = make_double2(apq.x * im, apq.y * im);
    return r;
  }
  const double mag = hypot(apq.x, apq.y);
  if (mag <= 1e-300 || mag < 1e-18 * (fabs(app) + fabs(aqq))) return r;
  r.ph = make_double2(apq.x / mag, apq.y / mag);
  const double tau = del / mag;
  const double t = (tau >= 0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
  r.c = 1.0 / sqrt(1.0 + t * t);
  r.s = t * r.c;
  return r;
}

// (a, b) <- (c a - s b', s a + c b'), b' = b ph or b conj(ph)
template <bool CONJ>
__device__ __forceinline__ void rot_pair(const Rot& R, double2& a, double2& b) {
  const double py = CONJ ? -R.ph.y : R.ph.y;
  const double2 d = make_double2(b.x * R.ph.x - b.y * py, b.x * py + b.y * R.ph.x);
  const double2 u = a;
  a = make_double2(R.c * u.x - R.s * d.x, R.c * u.y - R.s * d.y);
  b = make_double2(R.s * u.x + R.c * d.x, R.s * u.y + R.c * d.y);
}

constexpr int kJB = 8;   // pairs per block and direction
__global__ void __launch_bounds__(kJB* kJB)
k_jacobi_round(const double2* __restrict__ A, double2* __restrict__ Aout,
               const double2* __restrict__ V, double2* __restrict__ Vout, int n, int npad, int r) {
  __shared__ Rot rot[2][kJB];
  const int tid = threadIdx.x, lx = tid % kJB, ly = tid / kJB;
  const int np2 = npad / 2;
  const int k = blockIdx.y * kJB + ly, l = blockIdx.x * kJB + lx;
  int pk = 0, qk = n, pl = 0, ql = n;
  if (k < np2) pair_of(k, r, npad, pk, qk);
  if (l < np2) pair_of(l, r, npad, pl, ql);
  const bool act = k < np2 && l < np2;
  // this thread's inputs, loaded before the rotations are waited for
  double2 a00 = make_double2(0, 0), a01 = a00, a10 = a00, a11 = a00, v[2][2] = {{a00, a00}, {a00, a00}};
  if (act) {
    a00 = A[(size_t)pk * n + pl];
    if (ql < n) a01 = A[(size_t)pk * n + ql];
    if (qk < n) a10 = A[(size_t)qk * n + pl];
    if (qk < n && ql < n) a11 = A[(size_t)qk * n + ql];
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if (2 * k + i < n) {
        v[i][0] = V[(size_t)(2 * k + i) * n + pl];
        if (ql < n) v[i][1] = V[(size_t)(2 * k + i) * n + ql];
      }
  }
  if (tid < 2 * kJB) {
    const int i = (tid < kJB ? blockIdx.y : blockIdx.x) * kJB + tid % kJB;
    int p = 0, q = n;
    if (i < np2) pair_of(i, r, npad, p, q);
    rot[tid / kJB][tid % kJB] = make_rot(A, n, p, q);
  }
  __syncthreads();
  if (!act) return;
  const Rot Rk = rot[0][ly], Rl = rot[1][lx];
  rot_pair<true>(Rl, a00, a01);    // columns: A J
  rot_pair<true>(Rl, a10, a11);
  rot_pair<false>(Rk, a00, a10);   // rows: J^H (A J)
  rot_pair<false>(Rk, a01, a11);
  Aout[(size_t)pk * n + pl] = a00;
  if (ql < n) Aout[(size_t)pk * n + ql] = a01;
  if (qk < n) Aout[(size_t)qk * n + pl] = a10;
  if (qk < n && ql < n) Aout[(size_t)qk * n + ql] = a11;
#pragma unroll
  for (int i = 0; i < 2; ++i)
    if (2 * k + i < n) {
      rot_pair<true>(Rl, v[i][0], v[i][1]);
      Vout[(size_t)(2 * k + i) * n + pl] = v[i][0];
      if (ql < n) Vout[(size_t)(2 * k + i) * n + ql] = v[i][1];
    }
}

// off-diagonal and total squared Frobenius norms
__global__ void k_offnorm(const double2* __restrict__ A, int n, double* out) {
  __shared__ double r1[256], r2[256];
  double off = 0, tot = 0;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < (long long)n * n;
       t += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(t / n), j = (int)(t % n);
    const double2 a = A[t];
    const double m = a.x * a.x + a.y * a.y;
    tot += m;
    if (i != j) off += m;
  }
  r1[threadIdx.x] = off;
  r2[threadIdx.x] = tot;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
      r1[threadIdx.x] += r1[threadIdx.x + s];
      r2[threadIdx.x] += r2[threadIdx.x + s];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    atomicAdd(&out[0], r1[0]);
    atomicAdd(&out[1], r2[0]);
  }
}

// ascending eigenvalues (stable rank sort, one block) and column permutation of V
__global__ void k_sort_eig(const double2* __restrict__ A, const double2* __restrict__ V,
                           double* evals, double2* Q, int n) {
  __shared__ double w[512];
  __shared__ int rank[512];
  for (int i = threadIdx.x; i < n; i += blockDim.x) w[i] = A[(size_t)i * n + i].x;
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    int r = 0;
    for (int k = 0; k < n; ++k) r += (w[k] < w[i]) || (w[k] == w[i] && k < i);
    rank[i] = r;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += blockDim.x) evals[rank[i]] = w[i];
  for (long long t = threadIdx.x; t < (long long)n * n; t += blockDim.x) {
    const int row = (int)(t / n), col = (int)(t % n);
    Q[(size_t)row * n + rank[col]] = V[t];
  }
}

__global__ void k_identity(double2* V, int n) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= (long long)n * n) return;
  const int i = (int)(t / n), j = (int)(t % n);
  V[t] = make_double2(i == j ? 1.0 : 0.0, 0.0);
}

inline unsigned nb(long long n, int t = 256) { return (unsigned)((n + t - 1) / t); }

}  // namespace

cudaError_t launch_hermitize(double2* A, int n, cudaStream_t s) {
  k_hermitize<<<nb((long long)n * n), 256, 0, s>>>(A, n);
  return cudaGetLastError();
}

// S (n x n, Hermitian positive definite, destroyed) -> Q = L^-H.  Scratch: the
// context's small buffer holds L and L^-1.
gbc_status dense_cholesky_inv_h(gbc_ctx* c, double2* S, int n, double2* Q, cudaStream_t s) {
  const size_t nn = (size_t)n * n;
  GBC_TRY(gbc_ensure_small(c, sizeof(double2) * 3 * nn + 64));
  double2* L = (double2*)c->d_small;
  double2* Linv = L + nn;
  GBC_CU(c, cudaMemsetAsync(L, 0, sizeof(double2) * nn, s));
  GBC_CU(c, cudaMemsetAsync(c->d_flag, 0, sizeof(int), s));
  for (int j = 0; j < n; ++j) {
    const long long m = (long long)(n - j) * (n - j);
    k_chol_col<<<nb(m), 256, 0, s>>>(S, L, n, j, c->d_flag);
  }
  GBC_CU(c, cudaGetLastError());
  int flag[2] = {0, 0};
  GBC_CU(c, cudaMemcpyAsync(flag, c->d_flag, sizeof flag, cudaMemcpyDeviceToHost, s));
  GBC_CU(c, cudaStreamSynchronize(s));
  if (flag[1]) return gbc_fail(c, GBC_ETIMEOUT, kSplitExpired);
  if (flag[0]) return gbc_fail(c, GBC_ENOTPD, "Cholesky: non-positive pivot (overlap not positive definite)");
  k_tri_inv<<<n, 256, 0, s>>>(L, Linv, n);
  GBC_CU(c, cudaGetLastError());
  k_conj_transpose<<<nb(nn), 256, 0, s>>>(Linv, Q, n);
  GBC_CU(c, cudaGetLastError());
  return GBC_OK;
}

// A (n x n Hermitian, destroyed) -> ascending evals (device, n doubles) and the
// unitary Q whose columns are the eigenvectors.
gbc_status dense_eigh(gbc_ctx* c, double2* A, int n, double* evals_dev, double2* Q,
                      cudaStream_t s) {
  const size_t nn = (size_t)n * n;
  GBC_TRY(gbc_ensure_small(c, sizeof(double2) * 3 * nn + 64));
  double2* A2 = (double2*)c->d_small;
  double2* V = A2 + nn;
  double2* V2 = V + nn;
  double* norms = (double*)(V2 + nn);
  k_identity<<<nb(nn), 256, 0, s>>>(V, n);
  GBC_CU(c, cudaGetLastError());
  const int npad = (n % 2) ? n + 1 : n;
  const unsigned jb = (unsigned)((npad / 2 + kJB - 1) / kJB);
  double2 *a = A, *b = A2, *v = V, *w = V2;
  bool converged = (n <= 1);
  const int max_sweeps = 40;
  double prev_off = -1.0;
  for (int sweep = 0; sweep < max_sweeps && !converged; ++sweep) {
    for (int r = 0; r < npad - 1; ++r) {
      k_jacobi_round<<<dim3(jb, jb), kJB * kJB, 0, s>>>(a, b, v, w, n, npad, r);
      double2* t = a; a = b; b = t;
      t = v; v = w; w = t;
    }
    GBC_CU(c, cudaGetLastError());
    double hn[2] = {0, 0};
    int expired = 0;
    GBC_CU(c, cudaMemsetAsync(norms, 0, 2 * sizeof(double), s));
    k_offnorm<<<64, 256, 0, s>>>(a, n, norms);
    GBC_CU(c, cudaMemcpyAsync(hn, norms, 2 * sizeof(double), cudaMemcpyDeviceToHost, s));
    if (sweep == 0) GBC_CU(c, cudaMemcpyAsync(&expired, c->d_flag + 1, sizeof(int), cudaMemcpyDeviceToHost, s));
    GBC_CU(c, cudaStreamSynchronize(s));
    if (expired) return gbc_fail(c, GBC_ETIMEOUT, kSplitExpired);
    if (!(std::isfinite(hn[0]) && std::isfinite(hn[1])))
      return gbc_fail(c, GBC_EINVAL, "eigensolver: non-finite matrix entries");
    // converged when the off-diagonal part is at rounding level, or when it has
    // stopped shrinking while already tiny (the rounding floor of large n)
    const double off = std::sqrt(hn[0]), tot = std::sqrt(hn[1]);
    converged = off <= 1e-14 * tot || tot == 0.0 ||
                (off <= 1e-11 * tot && prev_off >= 0.0 && off >= 0.25 * prev_off);
    prev_off = off;
  }
  if (!converged) return gbc_fail(c, GBC_ETIMEOUT, "Jacobi eigensolver hit its sweep cap");
  k_sort_eig<<<1, 512, 0, s>>>(a, v, evals_dev, Q, n);
  GBC_CU(c, cudaGetLastError());
  return GBC_OK;
}
