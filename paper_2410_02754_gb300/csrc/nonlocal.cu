// Nonlocal spin-orbit part of H.X over compact projector supports.
//
// Paper: Eq. FEHnloc and the cell-level step 3 of Sec. IV.B.2,
//   Y += sum_a P_a Delta_a sum P_a^H X,
// done as three batched small contractions on the atom-support node lists:
//   C   = P_a^H X        (per atom: npj x 2 x nvec, reduction over the support)
//   C'  = Delta_a C      (2npj x 2npj times 2npj x nvec)
//   Y  += P_a C'         (FP64: atom by atom with atomics, both contractions as split
//                         products where they are large (split_gemm.cu); deterministic mode and the
//                         FP32 SIMT engine: node-centric, every support node sums its
//                         atoms' terms, a plain read-modify-write of Y)
// P_a is the node-based projector table (one row per distinct free node of the
// support, so nodes shared by several support cells are stored once).
#include <algorithm>
#include <type_traits>

#include "gbc_internal.h"

namespace {

// acc += conj(p) x and acc += p x, two multiply-adds per part (written out: the sum of two
// products added to acc compiles to three operations, which the FP64 pipe feels)
template <typename C> __device__ __forceinline__ void cmac_conj(C& acc, C p, C x) {
  acc.x = fma(p.x, x.x, fma(p.y, x.y, acc.x));
  acc.y = fma(p.x, x.y, fma(-p.y, x.x, acc.y));
}
template <typename C> __device__ __forceinline__ void cmac(C& acc, C p, C x) {
  acc.x = fma(p.x, x.x, fma(-p.y, x.y, acc.x));
  acc.y = fma(p.x, x.y, fma(p.y, x.x, acc.y));
}
// the same with a real p
__device__ __forceinline__ void cmac_conj(double2& acc, double p, double2 x) {
  acc.x += p * x.x;
  acc.y += p * x.y;
}
__device__ __forceinline__ void cmac(double2& acc, double p, double2 x) { cmac_conj(acc, p, x); }
// the part of a table entry that a kernel multiplies with
template <typename PT, typename C> __device__ __forceinline__ PT p_entry(C p) {
  if constexpr (std::is_same<PT, double>::value) return p.x;
  else return p;
}
__device__ __forceinline__ void catomic(float2* p, float2 v) { atomicAdd(p, v); }
__device__ __forceinline__ void catomic(double2* p, double2 v) {
  atomicAdd(&p->x, v.x);
  atomicAdd(&p->y, v.y);
}

constexpr int kStage = 64;      // support nodes staged in shared memory at a time
constexpr int kCols = 128;      // threads per block

// One block of the projection and of the atom-major expansion: kCols threads = CT
// columns (a column is one spin of one vector) x NG node groups, over rows [j0, j0 + cnt)
// of one atom's support.  Both kernels are bound by the FP64 pipe (about 2 FMAs per clock
// and SM: 4 npj per column and node against one 16-byte load of X), so what matters is
// that every lane has a column and every SM several blocks: with few columns the lanes go
// to further nodes, and the grid splits a 1024-node chunk into nsub parts when chunks x
// column tiles do not fill the SMs.  P rows are staged with an odd row stride, so the NG
// rows a warp reads at once sit in distinct bank groups.  Measured on one GB300: the FP64
// pipe is 85% busy in both; projection + expansion on 6 atoms x 18 projectors in 6^3 cells
// at p = 6 with 64 vectors, k != 0: 20.0 -> 6.6 ms, with the multiply-adds written as FMAs
// 4.0 ms; on 24 atoms in 16^3 cells with one vector, k = 0: 10.5 -> 0.59 ms, with real tables
// 0.29 ms (before: one chunk per block with all lanes as columns, and an expansion that walked
// each shared node's incidence list).
struct NlTile {
  int atom, npj, j0, cnt, noff;
  __device__ __forceinline__ NlTile(const int4* chunks, const int* atom_npj, int nsub) {
    const int4 ch = chunks[blockIdx.x];    // (atom, first position, count, node offset of atom)
    const int per = (ch.z + nsub - 1) / nsub;
    const int o = min(ch.z, (int)blockIdx.z * per);
    atom = ch.x;
    npj = atom_npj[atom];
    j0 = ch.y + o;
    cnt = min(per, ch.z - o);
    noff = ch.w;
  }
};

// C[(c_off + 2chi + s) * nvec + v] += sum_j conj(P[j][chi]) X[node_j][s][v]: each thread
// sums its nodes in registers, then the NG groups of a column are added by shuffles and
// through shared memory in a fixed order, and one thread per (chi, column) adds the
// block's sum to C (or stores it to Cpart, deterministic mode).
// REALP: the table's imaginary parts are zero (k = 0: no Bloch phases), half the FP64 work.
template <typename T, int MAXPJ, int CT, bool REALP>
__global__ void __launch_bounds__(kCols)
nl_project(const cplx<T>* __restrict__ X, int ldx, int nvec, int nsub,
           const int4* __restrict__ chunks, const long long* __restrict__ nodes,
           const cplx<T>* __restrict__ P, const int* __restrict__ atom_npj,
           const int* __restrict__ atom_pv_off, const int* __restrict__ atom_c_off,
           cplx<T>* __restrict__ Cbuf, long long M, cplx<T>* __restrict__ Cpart) {
  using C = cplx<T>;
  constexpr int NG = kCols / CT, RS = MAXPJ | 1, NW = kCols / 32, RC = 8;
  constexpr int NPS = kStage * RS, NRED = NW * CT * RC;
  using PT = typename std::conditional<REALP, double, C>::type;
  // staged P rows, then the partial sums
  __shared__ __align__(16) unsigned char sh_raw[NPS * sizeof(PT) > NRED * sizeof(C) ? NPS * sizeof(PT)
                                                                                     : NRED * sizeof(C)];
  PT* ps = reinterpret_cast<PT*>(sh_raw);
  C* sh = reinterpret_cast<C*>(sh_raw);
  __shared__ long long Ns[kStage];
  const NlTile t(chunks, atom_npj, nsub);
  const C* Pa = P + atom_pv_off[t.atom];
  const int lc = threadIdx.x % CT, grp = threadIdx.x / CT;
  const int col = blockIdx.y * CT + lc;
  const bool ok = col < 2 * nvec;
  const int s = ok ? col / nvec : 0, v = ok ? col % nvec : 0;
  C acc[MAXPJ];
#pragma unroll
  for (int c = 0; c < MAXPJ; ++c) acc[c] = cmake<C>(0, 0);
  for (int jb = 0; jb < t.cnt; jb += kStage) {
    const int nb = min(kStage, t.cnt - jb);
    for (int i = threadIdx.x; i < nb * t.npj; i += kCols) {
      const int jj = i / t.npj, c = i % t.npj;
      ps[jj * RS + c] = p_entry<PT>(Pa[(size_t)(t.j0 + jb + jj) * t.npj + c]);
    }
    for (int i = threadIdx.x; i < nb; i += kCols) Ns[i] = nodes[t.noff + t.j0 + jb + i];
    __syncthreads();
    if (ok) {
      for (int i = grp; i < nb; i += 4 * NG) {
        C x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int jj = i + u * NG;
          x[u] = (jj < nb && GBC_IN_RANGE(GBC_SITE_NL_NODE, Ns[jj], M))
                     ? X[(Ns[jj] * 2 + s) * ldx + v] : cmake<C>(0, 0);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int jj = i + u * NG;
          if (jj >= nb) break;
#pragma unroll
          for (int c = 0; c < MAXPJ; ++c)
            if (c < t.npj) cmac_conj(acc[c], ps[jj * RS + c], x[u]);
        }
      }
    }
    __syncthreads();
  }
  // add the node groups of each column: lanes of a warp, then the warps, RC projectors
  // at a time
  const int r0 = atom_c_off[t.atom];
#pragma unroll
  for (int c0 = 0; c0 < MAXPJ; c0 += RC) {
    if (c0 >= t.npj) break;
#pragma unroll
    for (int c = c0; c < (c0 + RC < MAXPJ ? c0 + RC : MAXPJ); ++c) {
      C a = acc[c];
#pragma unroll
      for (int o = 16; o >= CT; o >>= 1) {
        a.x += __shfl_xor_sync(0xffffffffu, a.x, o);
        a.y += __shfl_xor_sync(0xffffffffu, a.y, o);
      }
      if ((threadIdx.x & 31) < CT) sh[((threadIdx.x >> 5) * CT + lc) * RC + c - c0] = a;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < CT * RC; i += kCols) {
      const int c = c0 + i / CT, gc = blockIdx.y * CT + i % CT;
      if (c >= t.npj || gc >= 2 * nvec) continue;
      C a = cmake<C>(0, 0);
#pragma unroll
      for (int w = 0; w < NW; ++w) {
        const C b = sh[(w * CT + i % CT) * RC + c - c0];
        a.x += b.x;
        a.y += b.y;
      }
      const int row = 2 * c + gc / nvec, gv = gc % nvec;
      if (Cpart)   // this block's sums (k_nl_chunk_sum adds them in order)
        Cpart[((size_t)(blockIdx.x * nsub + blockIdx.z) * 2 * MAXPJ + row) * nvec + gv] = a;
      else
        catomic(&Cbuf[(size_t)(r0 + row) * nvec + gv], a);
    }
    __syncthreads();
  }
}

// Y[node][s][v] += sum_chi P[pos][chi] Cp[2chi+s][v], one atom's rows per block with FP64
// atomics (the cell apply adds to the same rows the same way): the block's C' columns stay
// in registers, and a node held by several atoms is updated once per atom instead of
// walking its incidence list through dependent loads.
template <int MAXPJ, int CT, bool REALP>
__global__ void __launch_bounds__(kCols)
nl_expand_add(double2* __restrict__ Y, int ldx, int nvec, int nsub,
              const int4* __restrict__ chunks, const long long* __restrict__ nodes,
              const double2* __restrict__ P, const int* __restrict__ atom_npj,
              const int* __restrict__ atom_pv_off, const int* __restrict__ atom_c_off,
              const double2* __restrict__ Cp, long long M) {
  constexpr int NG = kCols / CT, RS = MAXPJ | 1;
  using PT = typename std::conditional<REALP, double, double2>::type;
  __shared__ PT sh[kStage * RS];
  __shared__ long long Ns[kStage];
  const NlTile t(chunks, atom_npj, nsub);
  const double2* Pa = P + atom_pv_off[t.atom];
  const int lc = threadIdx.x % CT, grp = threadIdx.x / CT;
  const int col = blockIdx.y * CT + lc;
  const bool ok = col < 2 * nvec;
  const int s = ok ? col / nvec : 0, v = ok ? col % nvec : 0;
  const double2* Ca = Cp + (size_t)(atom_c_off[t.atom] + s) * nvec + v;
  double2 cp[MAXPJ];
#pragma unroll
  for (int c = 0; c < MAXPJ; ++c)
    cp[c] = (ok && c < t.npj) ? Ca[(size_t)(2 * c) * nvec] : make_double2(0, 0);
  for (int jb = 0; jb < t.cnt; jb += kStage) {
    const int nb = min(kStage, t.cnt - jb);
    for (int i = threadIdx.x; i < nb * t.npj; i += kCols) {
      const int jj = i / t.npj, c = i % t.npj;
      sh[jj * RS + c] = p_entry<PT>(Pa[(size_t)(t.j0 + jb + jj) * t.npj + c]);
    }
    for (int i = threadIdx.x; i < nb; i += kCols) Ns[i] = nodes[t.noff + t.j0 + jb + i];
    __syncthreads();
    if (ok) {
#pragma unroll 2
      for (int jj = grp; jj < nb; jj += NG) {
        double2 a = make_double2(0, 0);
#pragma unroll
        for (int c = 0; c < MAXPJ; ++c)
          if (c < t.npj) cmac(a, sh[jj * RS + c], cp[c]);
        if (GBC_IN_RANGE(GBC_SITE_NL_NODE, Ns[jj], M)) catomic(&Y[(Ns[jj] * 2 + s) * ldx + v], a);
      }
    }
    __syncthreads();
  }
}

// C[(c_off + r) * nvec + v] = sum over the atom's chunk parts k, in order, of Cpart[k][r][v]
template <typename T, int MAXPJ>
__global__ void k_nl_chunk_sum(const cplx<T>* __restrict__ Cpart, cplx<T>* __restrict__ Cbuf,
                               const int* __restrict__ chunk_off, const int* __restrict__ atom_npj,
                               const int* __restrict__ atom_c_off, int nvec, int nsub) {
  const int atom = blockIdx.x, r = blockIdx.y;
  const int v = blockIdx.z * blockDim.x + threadIdx.x;
  if (r >= 2 * atom_npj[atom] || v >= nvec) return;
  cplx<T> acc = cmake<cplx<T>>(0, 0);
  for (int k = chunk_off[atom] * nsub; k < chunk_off[atom + 1] * nsub; ++k) {
    const cplx<T> p = Cpart[((size_t)k * 2 * MAXPJ + r) * nvec + v];
    acc.x += p.x;
    acc.y += p.y;
  }
  Cbuf[(size_t)(atom_c_off[atom] + r) * nvec + v] = acc;
}

// Cp[(c_off + r) * nvec + v] = sum_c Delta[r][c] C[(c_off + c) * nvec + v]
template <typename T>
__global__ void nl_couple(const cplx<T>* __restrict__ Cbuf, cplx<T>* __restrict__ Cp,
                          const cplx<T>* __restrict__ delta, const int* __restrict__ atom_npj,
                          const int* __restrict__ atom_delta_off, const int* __restrict__ atom_c_off,
                          int nvec) {
  using C = cplx<T>;
  const int atom = blockIdx.x, r = blockIdx.y;
  const int n2 = 2 * atom_npj[atom];
  if (r >= n2) return;
  const int v = blockIdx.z * blockDim.x + threadIdx.x;
  if (v >= nvec) return;
  const C* D = delta + atom_delta_off[atom] + (size_t)r * n2;
  const size_t base = (size_t)atom_c_off[atom] * nvec + v;
  C acc = cmake<C>(0, 0);
#pragma unroll 12   // the loads of 12 terms in flight (36 at 18 projectors: latency is all it takes)
  for (int c = 0; c < n2; ++c) cmac(acc, D[c], Cbuf[base + (size_t)c * nvec]);
  Cp[base + (size_t)r * nvec] = acc;
}

// Node-major expansion (deterministic mode, and the overwrite mode of the FP32 SIMT engine):
// Y[node][s][v] += sum over atoms whose support holds node of sum_chi P[pos][chi] Cp[2chi+s][v].
// Every distinct support node is owned by the lowest-index atom whose support
// holds it; the owner's block writes it once (plain read-modify-write, no
// atomics) and adds the other atoms' terms from their incidence list.  The
// owner's C' column stays in registers, the staged P rows in shared memory.
constexpr int kExpStage = 32;
template <typename T, int MAXPJ>
__global__ void __launch_bounds__(kCols)
nl_expand(cplx<T>* __restrict__ Y, int ldx, int nvec, const int4* __restrict__ chunks,
          const long long* __restrict__ own_node, const int* __restrict__ own_pos,
          const int* __restrict__ own_xptr, const int2* __restrict__ own_xinc,
          const cplx<T>* __restrict__ P, const int* __restrict__ atom_npj,
          const int* __restrict__ atom_pv_off, const int* __restrict__ atom_c_off,
          const cplx<T>* __restrict__ Cp, int overwrite, long long M) {
  using C = cplx<T>;
  __shared__ C Ps[kExpStage][MAXPJ];
  const int4 ch = chunks[blockIdx.x];       // (atom, first owned index, count, -)
  const int atom = ch.x, u0 = ch.y, cnt = ch.z;
  const int npj = atom_npj[atom];
  const C* Pa = P + atom_pv_off[atom];
  const int col = blockIdx.y * kCols + threadIdx.x;
  const bool ok = col < 2 * nvec;
  const int s = ok ? col / nvec : 0, v = ok ? col % nvec : 0;
  C cp[MAXPJ];
  const C* Ca = Cp + (size_t)(atom_c_off[atom] + s) * nvec + v;
#pragma unroll
  for (int c = 0; c < MAXPJ; ++c) cp[c] = (ok && c < npj) ? Ca[(size_t)(2 * c) * nvec] : cmake<C>(0, 0);
  for (int jb = 0; jb < cnt; jb += kExpStage) {
    const int nb = min(kExpStage, cnt - jb);
    for (int t = threadIdx.x; t < nb * npj; t += kCols) {
      const int jj = t / npj, c = t % npj;
      Ps[jj][c] = Pa[(size_t)own_pos[u0 + jb + jj] * npj + c];
    }
    __syncthreads();
    if (ok) {
      for (int t = 0; t < nb; ++t) {
        const int u = u0 + jb + t;
        C acc = cmake<C>(0, 0);
#pragma unroll
        for (int c = 0; c < MAXPJ; ++c)
          if (c < npj) cmac(acc, Ps[t][c], cp[c]);
        for (int k = own_xptr[u]; k < own_xptr[u + 1]; ++k) {
          const int2 inc = own_xinc[k];
          const int nb2 = atom_npj[inc.x];
          const C* Pr = P + atom_pv_off[inc.x] + (size_t)inc.y * nb2;
          const C* Cr = Cp + (size_t)(atom_c_off[inc.x] + s) * nvec + v;
          for (int c = 0; c < nb2; ++c) cmac(acc, Pr[c], Cr[(size_t)(2 * c) * nvec]);
        }
        if (!GBC_IN_RANGE(GBC_SITE_NL_NODE, own_node[u], M)) continue;
        C* y = &Y[(own_node[u] * 2 + s) * ldx + v];
        if (overwrite) {
          *y = acc;
        } else {
          C o = *y;
          o.x += acc.x;
          o.y += acc.y;
          *y = o;
        }
      }
    }
    __syncthreads();
  }
}

// column tile (a power of two, at most a warp) and the parts a chunk is split into: about
// eight blocks per SM, at least 64 nodes per part
inline int nl_col_tile(int nvec) {
  int ct = 2;
  while (ct < 32 && ct < 2 * nvec) ct *= 2;
  return ct;
}
inline int nl_parts(const ProjDev& pj, int nvec) {
  const int ct = nl_col_tile(nvec);
  const long long blocks = (long long)pj.nchunks * ((2 * nvec + ct - 1) / ct);
  const long long want = (8LL * gbc_sm_count() + blocks - 1) / blocks;
  return (int)std::max<long long>(1, std::min<long long>(16, want));
}
// the FP64 tables are real (e^{-ik.r} = 1)
inline bool real_tables(const gbc_ctx* c) { return c->k[0] == 0.0 && c->k[1] == 0.0 && c->k[2] == 0.0; }
// f(std::integral_constant<int, CT>) for the column tile of nvec vectors
template <typename F> inline void nl_with_tile(int nvec, F f) {
  switch (nl_col_tile(nvec)) {
    case 2: return f(std::integral_constant<int, 2>());
    case 4: return f(std::integral_constant<int, 4>());
    case 8: return f(std::integral_constant<int, 8>());
    case 16: return f(std::integral_constant<int, 16>());
    default: return f(std::integral_constant<int, 32>());
  }
}

template <typename T, int MAXPJ>
cudaError_t run_project(gbc_ctx* c, const cplx<T>* X, int nvec, int ldx, cplx<T>* Cbuf,
                        cudaStream_t s) {
  const ProjDev& pj = c->proj;
  const cplx<T>* P = std::is_same<T, double>::value ? (const cplx<T>*)pj.d_P64
                                                    : (const cplx<T>*)pj.d_P32;
  const int nsub = nl_parts(pj, nvec);
  // deterministic mode: per-part sums, then each atom's parts added in order
  cplx<T>* Cpart = nullptr;
  if (c->deterministic) {
    if (gbc_ensure_work(c, 11, sizeof(cplx<T>) * pj.nchunks * nsub * 2 * MAXPJ * (size_t)nvec) != GBC_OK)
      return cudaErrorMemoryAllocation;
    Cpart = (cplx<T>*)c->work[11];
  }
  nl_with_tile(nvec, [&](auto ct) {
    constexpr int CT = decltype(ct)::value;
    dim3 grid(pj.nchunks, (2 * nvec + CT - 1) / CT, nsub);
    auto run = [&](auto kern) {
      kern<<<grid, kCols, 0, s>>>(X, ldx, nvec, nsub, pj.d_chunks, pj.d_nodes, P, pj.d_atom_npj,
                                  pj.d_atom_pv_off, pj.d_atom_c_off, Cbuf, c->mesh.M, Cpart);
    };
    if constexpr (std::is_same<T, double>::value) {
      if (real_tables(c)) return run(nl_project<T, MAXPJ, CT, true>);
    }
    run(nl_project<T, MAXPJ, CT, false>);
  });
  cudaError_t e = cudaGetLastError();
  if (!Cpart || e != cudaSuccess) return e;
  dim3 g2(pj.natoms, 2 * pj.max_npj, (nvec + kCols - 1) / kCols);
  k_nl_chunk_sum<T, MAXPJ><<<g2, kCols, 0, s>>>(Cpart, Cbuf, pj.d_chunk_off, pj.d_atom_npj,
                                                pj.d_atom_c_off, nvec, nsub);
  return cudaGetLastError();
}

template <int MAXPJ>
cudaError_t run_expand_add(const gbc_ctx* c, double2* Y, int nvec, int ldx, const double2* Cp,
                           cudaStream_t s) {
  const ProjDev& pj = c->proj;
  const int nsub = nl_parts(pj, nvec);
  nl_with_tile(nvec, [&](auto ct) {
    constexpr int CT = decltype(ct)::value;
    dim3 grid(pj.nchunks, (2 * nvec + CT - 1) / CT, nsub);
    auto run = [&](auto kern) {
      kern<<<grid, kCols, 0, s>>>(Y, ldx, nvec, nsub, pj.d_chunks, pj.d_nodes, pj.d_P64, pj.d_atom_npj,
                                  pj.d_atom_pv_off, pj.d_atom_c_off, Cp, c->mesh.M);
    };
    if (real_tables(c)) run(nl_expand_add<MAXPJ, CT, true>);
    else run(nl_expand_add<MAXPJ, CT, false>);
  });
  return cudaGetLastError();
}

// FP64 contractions as split products on the tensor cores (split_gemm.cu), with their workspace in
// place, where that is faster.  The direct kernels run at the FP64 rate (578 FMAs per ns at 95% of
// it; padded columns count), the split ones take, per support node, writing and reading its
// digits and the MMAs of one 64-wide tile of projectors, whatever their number.  Times in ns, the
// constants fitted to H.X of 122,514 and 329,884 support nodes (18 projectors, p = 6) and of 25,476
// and 1458 nodes (3 and 18).  Direct / split H.X, cell apply included, k != 0:
//   122,514 nodes: 8 vectors 1.05 / 1.20 ms, 16 2.01 / 1.70, 64 7.52 / 4.82, 200 23.7 / 14.1
//   329,884 nodes: 8 vectors 3.54 / 3.61 ms, 16 6.86 / 5.70, 64 27.0 / 18.9, 200 82.5 / 58.4
//   122,514 nodes at k = 0 (half the FP64 work): 16 vectors 1.36 / 1.59, 64 5.08 / 4.37 ms
//   25,476 nodes x 3 projectors, 64 vectors 1.71 / 1.84; 1458 nodes, 64 vectors 0.18 / 0.32 ms
// Where the workspace cannot be had (no memory left, or it would have to grow while the stream is
// captured) the direct kernels run.
bool use_split(gbc_ctx* c, int nvec, cudaStream_t s) {
  if (c->deterministic) return false;
  const ProjDev& pj = c->proj;
  const double np = (double)pj.nnodes_total;
  const int ct = nl_col_tile(nvec), dcols = (2 * nvec + ct - 1) / ct * ct, scols = (4 * nvec + 127) / 128 * 128;
  const double direct = (double)pj.pv_off.back() * dcols * (real_tables(c) ? 4 : 8) / 578.0;
  const double split = 120e3 + np * (4.0 + 0.02 * scols);
  if (direct < split) return false;
  const size_t bytes = nl_split_bytes(c, nvec);
  if (c->work_bytes[14] >= bytes) return true;
  cudaStreamCaptureStatus cap;
  if (cudaStreamIsCapturing(s, &cap) == cudaSuccess) {
    if (cap != cudaStreamCaptureStatusNone) return false;
    if (gbc_ensure_work(c, 14, bytes) == GBC_OK) return true;
  }
  cudaGetLastError();   // not left for the next launch's check
  return false;
}
bool use_tc(const gbc_ctx* c) { return c->nl_engine == GBC_NL_TENSOR && tc_nonlocal_supported(c->proj); }

}  // namespace

template <typename T>
cudaError_t launch_nonlocal(gbc_ctx* c, const cplx<T>* X, cplx<T>* Y, int nvec, int ldx,
                            cplx<T>* Cbuf, cplx<T>* Cpbuf, cudaStream_t s, bool overwrite,
                            void* bpre, bool may_alloc) {
  const ProjDev& pj = c->proj;
  if (pj.natoms == 0 || nvec == 0 || pj.nchunks == 0 || pj.nexp_chunks == 0) return cudaSuccess;
  const bool split = std::is_same<T, double>::value && may_alloc && !overwrite && use_split(c, nvec, s);
  cudaError_t e = cudaSuccess;
  if constexpr (std::is_same<T, double>::value) {
    if (split) {
      e = cudaMemsetAsync(Cbuf, 0, sizeof(cplx<T>) * (size_t)pj.rows_total * nvec, s);
      if (e == cudaSuccess) e = nl_split_project(c, X, nvec, ldx, Cbuf, s);
    }
  }
  if (!split) e = launch_nl_project<T>(c, X, nvec, ldx, Cbuf, s);
  if (e != cudaSuccess) return e;
  const cplx<T>* D = std::is_same<T, double>::value ? (const cplx<T>*)pj.d_delta64
                                                    : (const cplx<T>*)pj.d_delta32;
  dim3 g2(pj.natoms, 2 * pj.max_npj, (nvec + kCols - 1) / kCols);
  nl_couple<T><<<g2, kCols, 0, s>>>(Cbuf, Cpbuf, D, pj.d_atom_npj, pj.d_atom_delta_off,
                                   pj.d_atom_c_off, nvec);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if constexpr (std::is_same<T, float>::value) {
    if (use_tc(c)) return launch_tc_expand(pj, Y, nvec, ldx, Cpbuf, s, overwrite, bpre, c->d_cell_ctr);
  } else if (split) {
    return nl_split_expand(c, Y, nvec, ldx, Cpbuf, s);
  } else if (!overwrite && !c->deterministic) {
    if (pj.max_npj <= 4) return run_expand_add<4>(c, Y, nvec, ldx, Cpbuf, s);
    if (pj.max_npj <= 8) return run_expand_add<8>(c, Y, nvec, ldx, Cpbuf, s);
    if (pj.max_npj <= 18) return run_expand_add<18>(c, Y, nvec, ldx, Cpbuf, s);
    return run_expand_add<GBC_MAX_NPJ>(c, Y, nvec, ldx, Cpbuf, s);
  }
  const cplx<T>* P = std::is_same<T, double>::value ? (const cplx<T>*)pj.d_P64
                                                    : (const cplx<T>*)pj.d_P32;
  dim3 g3((unsigned)pj.nexp_chunks, (2 * nvec + kCols - 1) / kCols);
#define GBC_EXPAND(MP)                                                                        \
  nl_expand<T, MP><<<g3, kCols, 0, s>>>(Y, ldx, nvec, pj.d_exp_chunks, pj.d_own_node,           \
                                        pj.d_own_pos, pj.d_own_xptr, pj.d_own_xinc, P,         \
                                        pj.d_atom_npj, pj.d_atom_pv_off, pj.d_atom_c_off, Cpbuf, \
                                        overwrite ? 1 : 0, c->mesh.M)
  if (pj.max_npj <= 4) GBC_EXPAND(4);
  else if (pj.max_npj <= 8) GBC_EXPAND(8);
  else if (pj.max_npj <= 18) GBC_EXPAND(18);
  else GBC_EXPAND(GBC_MAX_NPJ);
#undef GBC_EXPAND
  return cudaGetLastError();
}

// C = (P_a x I2)^H X for every atom (rows c_off + 2chi + s), C zeroed first
template <typename T>
cudaError_t launch_nl_project(gbc_ctx* c, const cplx<T>* X, int nvec, int ldx, cplx<T>* Cbuf,
                              cudaStream_t s) {
  const ProjDev& pj = c->proj;
  if (pj.natoms == 0 || nvec == 0 || pj.nchunks == 0) return cudaSuccess;
  cudaError_t e = cudaMemsetAsync(Cbuf, 0, sizeof(cplx<T>) * (size_t)pj.rows_total * nvec, s);
  if (e != cudaSuccess) return e;
  if constexpr (std::is_same<T, float>::value) {
    if (use_tc(c)) return launch_tc_project(pj, c->mesh.M, X, nvec, ldx, Cbuf, s);
  }
  if (pj.max_npj <= 4) return run_project<T, 4>(c, X, nvec, ldx, Cbuf, s);
  if (pj.max_npj <= 8) return run_project<T, 8>(c, X, nvec, ldx, Cbuf, s);
  if (pj.max_npj <= 18) return run_project<T, 18>(c, X, nvec, ldx, Cbuf, s);
  return run_project<T, GBC_MAX_NPJ>(c, X, nvec, ldx, Cbuf, s);
}
template cudaError_t launch_nl_project<float>(gbc_ctx*, const float2*, int, int, float2*,
                                              cudaStream_t);
template cudaError_t launch_nl_project<double>(gbc_ctx*, const double2*, int, int, double2*,
                                               cudaStream_t);

template cudaError_t launch_nonlocal<float>(gbc_ctx*, const float2*, float2*, int, int, float2*,
                                            float2*, cudaStream_t, bool, void*, bool);
template cudaError_t launch_nonlocal<double>(gbc_ctx*, const double2*, double2*, int, int,
                                             double2*, double2*, cudaStream_t, bool, void*, bool);

size_t nl_work_bytes(const gbc_ctx* c, int nvec, int ldx, size_t el, size_t* bpre_off) {
  const size_t cb = el * (size_t)c->proj.rows_total * (size_t)nvec;
  const size_t off = (2 * cb + 255) & ~(size_t)255;
  const size_t xb = el == sizeof(float2) ? tc_expand_bpre_bytes(c->proj, nvec, ldx) : 0;
  if (bpre_off) *bpre_off = xb ? off : 0;
  return std::max<size_t>(64, xb ? off + xb : 2 * cb);
}

GBC_CHECK_WORD_ACCESSOR(gbc_check_word_nl)
