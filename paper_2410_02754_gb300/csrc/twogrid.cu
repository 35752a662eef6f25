// Two-grid transfer of a spinor block from FE order p_c to p_f (p_f = p_c or
// p_c + 1) on the same mesh (Sec. IV.A, Eq. FEWfnsCMesh: the first SCF
// iterations use N^{h,p-1}, the later ones N^{h,p}).  The order-p_c space lies
// in the order-p_f space, so the coarse FE function is carried over exactly by
// nodal interpolation at the fine GLL nodes:
//
//   X_f[J] = sum_I N^{p_c}_I(r_J) X_c[I],
//
// per cell a tensor product of the 1-D matrix T[j][i] = l^{p_c}_i(x^{p_f}_j),
// applied in three sum-factorised stages.  The first and last rows of T are unit rows (the GLL nodes
// share their end points): those values are copied.  The other rows are dense products: with the
// ends copied these take 30 paired multiply-adds a pencil at p = 5 -> 6, the even-odd form 33
// instructions, and even-odd sums of entries that are close to 0 and 1 lose accuracy (relative error
// on uniform random blocks 1.01e-7 at p = 5 -> 6, 8.0e-8 dense).  p_f = p_c is the identity: a copy.
//
// One CTA per (cell, tile of kLanes 16-byte elements a node row: 8 FP32 or 4 FP64 vectors), the
// tiles of a cell next to each other so that they share its node rows' sectors in L2.  A thread
// owns a pencil of one element (two FP32 vectors or one FP64 vector), so shared-memory accesses
// are 16 bytes and FP32 products paired multiply-adds on (re, im).  Per spin: stage the coarse
// cell in shared memory with asynchronous copies (every load of the cell in flight at once,
// zero-fill for absent nodes), x stage -> B, y stage -> A, z stage -> global.  Neighbouring
// pencils are an odd number of points apart in every stage, so a quarter-warp's accesses (4
// elements x 2 pencils) cover all banks.  A cell writes only the fine nodes it owns (local
// index < p_f in every direction); with the periodic wrap and the Dirichlet faces this writes
// every free fine node exactly once, with no atomics.  HBM-bound in the limit (the coarse block
// read and the fine block written once).  Measured on one GB300, 16^3 cells, p = 5 -> 6, 256 FP32
// vectors: 2.91 ms with scalar products of every row on 8-byte elements (issue-bound), 1.53 ms with
// even-odd products on 16-byte elements, 1.37 ms now.  FP64, 64 vectors: p = 3 -> 4 on 20^3 cells 4.13,
// 3.88, 2.63 ms; p = 6 -> 7 on 12^3 cells 6.98, 5.76, 6.10 ms.
#include "hx_cell.cuh"

namespace {

using namespace gbc;

constexpr int kLanes = 4;       // 16-byte elements of a node row per CTA
constexpr int kThreads = 192;

template <typename T> __host__ __device__ constexpr int vecs_per_elem() { return sizeof(T) == 4 ? 2 : 1; }
// rows 1 .. NF-2 of T; FP32: every entry twice, the multiplier of a paired multiply-add on (re, im)
template <typename T, int NC, int NF> struct TwoGridTab {
  typename std::conditional<sizeof(T) == 4, float2, double>::type t[NF - 2][NC];
};

// asynchronous global -> shared copy of N bytes, of which src_bytes are read and the rest zero
template <int N> __device__ __forceinline__ void cp_async_n(void* dst, const void* src, int src_bytes) {
  static_assert(N == 8 || N == 16, "8- or 16-byte copies");
  if (N == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(src_bytes)
                 : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(src_bytes)
                 : "memory");
}

__device__ __forceinline__ float4 t_mul(float2 m, float4 x) {
  return cat2(p_mul(m, lo2(x)), p_mul(m, hi2(x)));
}
__device__ __forceinline__ float4 t_fma(float2 m, float4 x, float4 a) {
  return cat2(p_fma(m, lo2(x), lo2(a)), p_fma(m, hi2(x), hi2(a)));
}
__device__ __forceinline__ double2 t_mul(double m, double2 x) { return make_double2(m * x.x, m * x.y); }
__device__ __forceinline__ double2 t_fma(double m, double2 x, double2 a) {
  return make_double2(fma(m, x.x, a.x), fma(m, x.y, a.y));
}

// one 1-D product: ld(j) -> the NC inputs, st(row, value) for the NF outputs
template <typename T, int NC, int NF, typename L, typename S>
__device__ __forceinline__ void line(const TwoGridTab<T, NC, NF>& tb, L ld, S st) {
  using E = decltype(ld(0));
  E in[NC];
#pragma unroll
  for (int j = 0; j < NC; ++j) in[j] = ld(j);
  st(0, in[0]);
#pragma unroll
  for (int i = 1; i < NF - 1; ++i) {
    E a = t_mul(tb.t[i - 1][0], in[0]);
#pragma unroll
    for (int j = 1; j < NC; ++j) a = t_fma(tb.t[i - 1][j], in[j], a);
    st(i, a);
  }
  st(NF - 1, in[NC - 1]);
}

template <int NC> __host__ __device__ constexpr int odd_stride() { return NC | 1; }   // of A's x pencils
template <int NC, int NF> __host__ __device__ constexpr int points_a() {
  return NC * NC * odd_stride<NC>() > NF * NF * NC ? NC * NC * odd_stride<NC>() : NF * NF * NC;
}

// al_in / al_out: the node rows of Xc / Xf are 16-byte aligned
template <typename T, int NC, int NF>
__global__ void __launch_bounds__(kThreads)
k_prolongate(const __grid_constant__ MeshDev mc, const __grid_constant__ MeshDev mf, const cplx<T>* __restrict__ Xc, int ldxc,
             cplx<T>* __restrict__ Xf, int ldxf, int nvec, int ntiles, int al_in, int al_out,
             const __grid_constant__ TwoGridTab<T, NC, NF> tb) {
  using E = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
  constexpr int VE = vecs_per_elem<T>();
  constexpr int RS = odd_stride<NC>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  E* A = reinterpret_cast<E*>(smem_raw);               // [points_a][kLanes]
  E* B = A + points_a<NC, NF>() * kLanes;              // [NF NC NC][kLanes]
  __shared__ long long off[3][8];                      // coarse node offsets, < 0: no free node
  const int e = blockIdx.x / ntiles;
  const int vec0 = (blockIdx.x % ntiles) * kLanes * VE;
  const int cx = e % mc.ncell[0], cy = (e / mc.ncell[0]) % mc.ncell[1], cz = e / (mc.ncell[0] * mc.ncell[1]);
  if (threadIdx.x < 3 * NC) {
    const int d = threadIdx.x / NC, i = threadIdx.x % NC;
    const int g = (d == 0 ? cx : d == 1 ? cy : cz) * mc.p + i;
    int f;
    if (mc.periodic[d]) f = g >= mc.period[d] ? g - mc.period[d] : g;
    else f = (g == 0 || g == mc.period[d]) ? -1 : g - 1;
    const long long scale = d == 0 ? 1 : d == 1 ? mc.nfree[0] : (long long)mc.nfree[0] * mc.nfree[1];
    off[d][i] = f < 0 ? -(1LL << 60) : f * scale;
  }
  __syncthreads();
  for (int s = 0; s < 2; ++s) {
    // coarse cell nodes (x pencils) -> A
    for (int u = threadIdx.x; u < NC * NC * kLanes; u += kThreads) {
      const int l = u % kLanes, pid = u / kLanes;
      const long long Iyz = off[1][pid % NC] + off[2][pid / NC];
      const int v = vec0 + l * VE;
      const int have = max(0, min(VE, nvec - v));      // vectors of the element
#pragma unroll
      for (int x = 0; x < NC; ++x) {
        const long long I = Iyz + off[0][x];
        const bool ok = I >= 0 && have > 0;
        const cplx<T>* src = ok ? Xc + (I * 2 + s) * ldxc + v : Xc;
        E* dst = &A[(pid * RS + x) * kLanes + l];
        if (sizeof(T) == 8 || al_in) {
          cp_async_n<16>(dst, src, ok ? have * (int)sizeof(cplx<T>) : 0);
        } else {
          cp_async_n<8>(dst, src, ok ? 8 : 0);
          cp_async_n<8>(reinterpret_cast<char*>(dst) + 8, ok && have > 1 ? src + 1 : Xc, ok && have > 1 ? 8 : 0);
        }
      }
    }
    asm volatile("cp.async.commit_group;\ncp.async.wait_all;" ::: "memory");
    __syncthreads();
    // x: A [z][y][x] (NC^3) -> B [z][y][xq] (NC^2 NF)
    for (int u = threadIdx.x; u < NC * NC * kLanes; u += kThreads) {
      const int l = u % kLanes, pid = u / kLanes;
      line(tb, [&](int j) { return A[(pid * RS + j) * kLanes + l]; },
           [&](int q, E r) { B[(pid * NF + q) * kLanes + l] = r; });
    }
    __syncthreads();
    // y: B [z][y][xq] -> A [z][yq][xq] (NC NF^2)
    for (int u = threadIdx.x; u < NF * NC * kLanes; u += kThreads) {
      const int l = u % kLanes, xq = (u / kLanes) % NF, z = u / (kLanes * NF);
      line(tb, [&](int j) { return B[((z * NC + j) * NF + xq) * kLanes + l]; },
           [&](int q, E r) { A[((z * NF + q) * NF + xq) * kLanes + l] = r; });
    }
    __syncthreads();
    // z: A [z][yq][xq] -> owned fine nodes (xq, yq, zq < p_f); no wrap there, so the nodes of a
    // z pencil are a constant distance apart
    for (int u = threadIdx.x; u < (NF - 1) * (NF - 1) * kLanes; u += kThreads) {
      const int l = u % kLanes, xq = (u / kLanes) % (NF - 1), yq = u / (kLanes * (NF - 1));
      const int fx = cx * mf.p + xq - (mf.periodic[0] ? 0 : 1);
      const int fy = cy * mf.p + yq - (mf.periodic[1] ? 0 : 1);
      const int fz = cz * mf.p - (mf.periodic[2] ? 0 : 1);
      const int v = vec0 + l * VE;
      const bool in = fx >= 0 && fy >= 0 && v < nvec;
      const long long row = ((long long)fz * mf.nfree[1] + fy) * mf.nfree[0] + fx;
      cplx<T>* dst = Xf + (row * 2 + s) * ldxf + v;
      const long long step = (long long)mf.nfree[0] * mf.nfree[1] * 2 * ldxf;
      line(tb, [&](int j) { return A[((j * NF + yq) * NF + xq) * kLanes + l]; },
           [&](int q, E r) {
             if (q == NF - 1 || !in || fz + q < 0) return;
             cplx<T>* o = dst + q * step;
             if constexpr (sizeof(T) == 8) {
               *o = r;
             } else if (al_out && v + 1 < nvec) {
               *reinterpret_cast<float4*>(o) = r;
             } else {
               o[0] = make_float2(r.x, r.y);
               if (v + 1 < nvec) o[1] = make_float2(r.z, r.w);
             }
           });
    }
    __syncthreads();   // A is restaged by the next spin
  }
}

// p -> p: columns 0 .. nvec-1 of every row
template <typename T>
__global__ void k_copy_cols(const cplx<T>* __restrict__ X, int ldx, cplx<T>* __restrict__ Out, int ldo,
                            long long rows, int nvec) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < rows * nvec;
       i += (long long)gridDim.x * blockDim.x) {
    const long long r = i / nvec;
    const int v = (int)(i - r * nvec);
    Out[r * ldo + v] = X[r * ldx + v];
  }
}

template <typename T, int NC, int NF>
cudaError_t launch_prolongate_t(const gbc_ctx* cc, const gbc_ctx* cf, const cplx<T>* Xc, int ldxc,
                                cplx<T>* Xf, int ldxf, int nvec, cudaStream_t s) {
  TwoGridTab<T, NC, NF> tb;   // coarse Lagrange basis at the fine GLL nodes
  const std::vector<double>& xc = cc->tab.gll_x;
  const std::vector<double>& xf = cf->tab.gll_x;
  for (int j = 1; j < NF - 1; ++j)
    for (int i = 0; i < NC; ++i) {
      double l = 1.0;
      for (int k = 0; k < NC; ++k)
        if (k != i) l *= (xf[j] - xc[k]) / (xc[i] - xc[k]);
      if constexpr (sizeof(T) == 4) tb.t[j - 1][i] = make_float2((float)l, (float)l);
      else tb.t[j - 1][i] = l;
    }
  constexpr size_t smem = 16 * (size_t)kLanes * (points_a<NC, NF>() + NF * NC * NC);
  auto k = k_prolongate<T, NC, NF>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  constexpr int VT = kLanes * vecs_per_elem<T>();
  const long long ntiles = (nvec + VT - 1) / VT, blocks = (long long)cf->mesh.E * ntiles;
  if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
  auto aligned = [](const void* p, int ld) { return ((uintptr_t)p & 15) == 0 && (ld & 1) == 0; };
  k<<<(unsigned)blocks, kThreads, smem, s>>>(cc->mesh, cf->mesh, Xc, ldxc, Xf, ldxf, nvec, (int)ntiles,
                                             aligned(Xc, ldxc), aligned(Xf, ldxf), tb);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_prolongate(const gbc_ctx* cc, const gbc_ctx* cf, const void* Xc, int ldxc,
                              void* Xf, int ldxf, int nvec, cudaStream_t s) {
  const int pc = cc->mesh.p, pf = cf->mesh.p;
  const cplx<T>* xc = (const cplx<T>*)Xc;
  cplx<T>* xf = (cplx<T>*)Xf;
  if (pc == pf) {
    const long long n = 2 * cf->mesh.M * nvec;
    const unsigned grid = (unsigned)std::min<long long>((n + 255) / 256, 64LL * gbc_sm_count());
    k_copy_cols<T><<<grid, 256, 0, s>>>(xc, ldxc, xf, ldxf, 2 * cf->mesh.M, nvec);
    return cudaGetLastError();
  }
#define GBC_TG(PC) \
  if (pc == PC && pf == PC + 1) \
    return launch_prolongate_t<T, PC + 1, PC + 2>(cc, cf, xc, ldxc, xf, ldxf, nvec, s);
  GBC_TG(2) GBC_TG(3) GBC_TG(4) GBC_TG(5) GBC_TG(6)
#undef GBC_TG
  return cudaErrorInvalidValue;
}

}  // namespace

extern "C" gbc_status gbc_prolongate(gbc_ctx* coarse, gbc_ctx* fine, const void* Xc, int ldxc,
                                     void* Xf, int ldxf, int nvec, void* stream) {
  if (!coarse || !fine) return GBC_EINVAL;
  if (!Xc || !Xf) return gbc_fail(fine, GBC_EINVAL, "null block pointer");
  if (Xc == Xf) return gbc_fail(fine, GBC_EINVAL, "Xc and Xf must be distinct");
  if (!gbc_is_device_ptr(Xc) || !gbc_is_device_ptr(Xf))
    return gbc_fail(fine, GBC_EINVAL, "Xc and Xf must be device memory");
  if (nvec < 1 || ldxc < nvec || ldxf < nvec)
    return gbc_fail(fine, GBC_EINVAL, "need 1 <= nvec <= ldxc, ldxf");
  if (!coarse->mesh_set || !fine->mesh_set) return gbc_fail(fine, GBC_ESTATE, "mesh not set");
  if (coarse->dev != fine->dev) return gbc_fail(fine, GBC_EINVAL, "contexts on different devices");
  if (coarse->prec != fine->prec) return gbc_fail(fine, GBC_EINVAL, "precisions differ");
  for (int d = 0; d < 3; ++d)
    if (coarse->mesh.ncell[d] != fine->mesh.ncell[d] || coarse->h[d] != fine->h[d] ||
        coarse->mesh.periodic[d] != fine->mesh.periodic[d])
      return gbc_fail(fine, GBC_EINVAL, "coarse and fine contexts must share the mesh");
  const int pc = coarse->mesh.p, pf = fine->mesh.p;
  if (pf != pc && pf != pc + 1)
    return gbc_fail(fine, GBC_EUNSUPPORTED, "this build transfers p -> p or p -> p + 1");
  if (coarse->tab.gll_x.size() != (size_t)pc + 1 || fine->tab.gll_x.size() != (size_t)pf + 1)
    return gbc_fail(fine, GBC_ESTATE, "GLL tables not built");
  GBC_CU(fine, cudaSetDevice(fine->dev));
  cudaStream_t s = (cudaStream_t)stream;
  if (fine->prec == GBC_FP64)
    GBC_CU(fine, launch_prolongate<double>(coarse, fine, Xc, ldxc, Xf, ldxf, nvec, s));
  else
    GBC_CU(fine, launch_prolongate<float>(coarse, fine, Xc, ldxc, Xf, ldxf, nvec, s));
  return GBC_OK;
}
