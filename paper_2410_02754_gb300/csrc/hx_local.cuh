// Cell-level apply of the local spinor Hamiltonian for FP64 blocks (matrix-free, sum
// factorisation), with atomic assembly into the global block or a per-cell result, and the
// even-odd 1-D tables that the FP32 form (hx_cell.cuh) shares.
//
// Paper: Sec. IV.B.2 (extract X^(e) = R^(e) X, cell products, assemble
// Y = sum_e R^(e)T Y^(e)) with the cell operator of Eq. FEHlocEl plus the
// k-terms of Eq. FEHloc in per-cell Hermitian form.  The dense cell matrix
// (N o V^eff) N^T of Sec. IV.B.1 is applied in factored form, as in hx_cell.cuh:
//   a  = N'_x^T X,  t1 = B_x X,  t2 = G_x X                      x pencils
//   u  = N'_y^T a;  c  = G_y t1 + B_y t2                          y pencils
//   w  = N'_z F N'_z^T u + G'_z u;  k = B_z c                     z pencils
//   Y^(e) = N'_x N'_y w + k                                       y, then x pencils
// N' = N diag(sqrt(w_q)), G_d = 1/2 A_d - (i/2) k_d (C^ - C^T), G'_z = (h_x h_y / 4) G_z,
// F = J [(V + |k|^2/2) I + B . sigma].
//
// Bound by the FP64 pipe (2 FMAs per clock and SM), so what counts is the number of FP64
// instructions and that no lane of one is idle: a warp's instruction takes its 16 cycles
// whether 2 or 32 lanes have a pencil.  A group of threads works on two (cell, vector) pairs
// at a time, one thread per pencil and spin; with the two pairs and two spins side by side
// the n_p^2 pencils of a stage fill 6.1 of 7 warps (p = 6; one pair a CTA filled 3.1 of 4), and
// the pairs may be of different cells, so a block of one vector fills the lanes as well.  Two
// independent groups per CTA (more at small p) keep the pipe busy across each other's
// barriers; at p = 5 and 6 a warp owns whole z planes and only the z stage is between group
// barriers.  Measured on one GB300 against one pair a CTA in seven stages: 6^3 cells, p = 6,
// 64 vectors, k != 0: 4.84 -> 3.46 ms a launch; 16^3 cells, one vector, k = 0: 1.21 -> 0.92 ms.
#pragma once

#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "gbc_internal.h"

namespace gbc {

// One system of a launch: its blocks, fields, mesh and the first global work item.
struct SysDesc {
  const double2* X;
  double2* Y;
  double2* Ycell;        // non-null: per-cell results [E][n_p^3][2][nvec] instead of assembly
  const double* fields;  // [E][NQ^3][4] J (V + |k|^2/2), J B_x, J B_y, J B_z
  int ldx, nvec;
  long long item0;       // work items (per (cell, vector)s each): [item0, item0 + ceil(E nvec / per))
  MeshDev mesh;
};

// A launch covers up to GBC_MAX_BATCH systems that share p, the cell edges and
// the k-point (hence the 1-D tables); items run over all systems.
struct LocalArgs {
  SysDesc sys[GBC_MAX_BATCH];
  int nsys;
  long long nitems;
};

__device__ __forceinline__ void atomic_add_c(double2* p, double2 v) {
  atomicAdd(&p->x, v.x);
  atomicAdd(&p->y, v.y);
}

// ---------------------------------------------------------------------------
// even-odd form of the 1-D operators
//
// GLL nodes and Gauss points are symmetric about the cell centre, so every 1-D
// matrix used here is centro-symmetric (M[no-1-i][ni-1-j] = M[i][j]: mass,
// stiffness, interpolation) or centro-antisymmetric (= -M[i][j]: C^ - C^T).
// With e_j = x_j + x_{ni-1-j}, o_j = x_j - x_{ni-1-j} (j < ni/2) and the
// middle entry x_mid when ni is odd,
//   y_i          =      (E e)_i + (O o)_i + Mid_i x_mid
//   y_{no-1-i}   = S * ((E e)_i - (O o)_i + Mid_i x_mid),   i < (no+1)/2,
// E = (M_ij + M_i,ni-1-j)/2, O = (M_ij - M_i,ni-1-j)/2: about half the
// multiply-adds of the dense product.
// ---------------------------------------------------------------------------
template <typename T, int NO, int NI> struct EO {
  static constexpr int HO = (NO + 1) / 2;
  static constexpr int HI = NI / 2 > 0 ? NI / 2 : 1;
  T E[HO][HI];
  T O[HO][HI];
  T Mid[HO];
};

template <typename T, int NP, int NQ> struct TablesEO {
  EO<T, NP, NP> B[3];    // 1-D Gauss mass h_d/2 B^               (symmetric)
  EO<T, NP, NP> Gr[3];   // 1/2 A_d (z: times h_x h_y / 4)          (symmetric)
  EO<T, NP, NP> Gi[3];   // -1/2 k_d (C^ - C^T) (z: the same)       (antisymmetric)
  EO<T, NQ, NP> Ni;      // N'^T: interpolation times sqrt(w_q), or s_q (FP32: gq_s)   (symmetric)
  EO<T, NP, NQ> Nt;      // N': times w_q over that factor                             (symmetric)
};

// host: even-odd split of a dense row-major NO x NI matrix (checks the symmetry)
template <typename T, int NO, int NI>
inline bool make_eo(const std::vector<double>& M, int S, EO<T, NO, NI>* out) {
  double mx = 0;
  for (double v : M) mx = std::max(mx, std::fabs(v));
  for (int i = 0; i < NO; ++i)
    for (int j = 0; j < NI; ++j)
      if (std::fabs(M[i * NI + j] - S * M[(NO - 1 - i) * NI + (NI - 1 - j)]) > 1e-10 * (mx + 1e-300))
        return false;
  for (int i = 0; i < EO<T, NO, NI>::HO; ++i) {
    for (int j = 0; j < EO<T, NO, NI>::HI; ++j) {
      out->E[i][j] = (T)0;
      out->O[i][j] = (T)0;
      if (j < NI / 2) {
        out->E[i][j] = (T)(0.5 * (M[i * NI + j] + M[i * NI + NI - 1 - j]));
        out->O[i][j] = (T)(0.5 * (M[i * NI + j] - M[i * NI + NI - 1 - j]));
      }
    }
    out->Mid[i] = (NI & 1) ? (T)M[i * NI + NI / 2] : (T)0;
  }
  return true;
}

template <typename T, int NP, int NQ>
inline bool make_tables_eo(const gbc_ctx* c, TablesEO<T, NP, NQ>* t) {
  const HostTables& h = c->tab;
  bool ok = true;
  for (int d = 0; d < 3; ++d) {
    // the mass products of N' leave out the edges, which the z operators carry for x and y
    const double hd = c->h[d], f = d == 2 ? 0.25 * c->h[0] * c->h[1] : 1.0;
    std::vector<double> B(NP * NP), Gr(NP * NP), Gi(NP * NP);
    for (int i = 0; i < NP; ++i)
      for (int j = 0; j < NP; ++j) {
        B[i * NP + j] = 0.5 * hd * h.Bh[i * NP + j];
        Gr[i * NP + j] = f * 0.5 * (2.0 / hd) * h.Ah[i * NP + j];
        Gi[i * NP + j] = -f * 0.5 * c->k[d] * (h.Ch[i * NP + j] - h.Ch[j * NP + i]);
      }
    ok = ok && make_eo<T, NP, NP>(B, 1, &t->B[d]) && make_eo<T, NP, NP>(Gr, 1, &t->Gr[d]) &&
         make_eo<T, NP, NP>(Gi, -1, &t->Gi[d]);
  }
  std::vector<double> Ni(NQ * NP), Nt(NP * NQ);
  for (int i = 0; i < NP; ++i)
    for (int q = 0; q < NQ; ++q) {
      const bool f32 = std::is_same<T, float>::value;
      const double s = f32 ? h.gq_s[q] : std::sqrt(h.gq_w[q]);
      Ni[q * NP + i] = h.N1[i * NQ + q] * s;
      Nt[i * NQ + q] = h.N1[i * NQ + q] * (f32 ? h.gq_w[q] / s : s);
    }
  ok = ok && make_eo<T, NQ, NP>(Ni, 1, &t->Ni) && make_eo<T, NP, NQ>(Nt, 1, &t->Nt);
  return ok;
}


// ---------------------------------------------------------------------------
// layout and grouping shared with the FP32 form (16-byte elements: here one spin of one
// (cell, vector), there both spins of one vector)
// ---------------------------------------------------------------------------
// Point strides (y, z) of the n_p^3 buffers (A, T2) and of T1 (up to n_q x n_q x n_p
// points).  A quarter-warp's 16-byte accesses (VB vectors, then neighbouring pencils) fall
// in the 8 distinct bank groups when neighbouring pencils are an odd number of points
// apart, which these strides give in every stage's pencil direction, and the vectors
// start 8 / VB groups apart (cell_vpoints).
template <int NP> struct CellLayout;
template <> struct CellLayout<3> { static constexpr int AY = 3, AZ = 9, QY = 5, QZ = 23; };
template <> struct CellLayout<4> { static constexpr int AY = 5, AZ = 21, QY = 5, QZ = 25; };
template <> struct CellLayout<5> { static constexpr int AY = 5, AZ = 25, QY = 7, QZ = 43; };
template <> struct CellLayout<6> { static constexpr int AY = 7, AZ = 43, QY = 7, QZ = 51; };
template <> struct CellLayout<7> { static constexpr int AY = 7, AZ = 49, QY = 9, QZ = 73; };
template <> struct CellLayout<8> { static constexpr int AY = 9, AZ = 72, QY = 9, QZ = 81; };
template <int NP> __host__ __device__ constexpr int cell_bufa() {   // points of A / T2
  return (NP - 1) * (1 + CellLayout<NP>::AY + CellLayout<NP>::AZ) + 1;
}
template <int NP> __host__ __device__ constexpr int cell_bufq() {   // points of T1
  return NP * (1 + CellLayout<NP>::QY) + (NP - 1) * CellLayout<NP>::QZ + 1;
}
template <int NP, int VB> __host__ __device__ constexpr int cell_vpoints() {
  // points per vector: [A | T2 | T1], padded to 8 / VB mod 8
  static_assert(VB == 2 || VB == 4, "VB");
  constexpr int n = 2 * cell_bufa<NP>() + cell_bufq<NP>(), r = 8 / VB;
  return n + ((8 + r - n % 8) % 8);
}
// Threads of a group: about one per pencil of a vector's x stage.  At p = 3 and 4 small
// groups are worth more than full rounds (12^3 cells, p = 4, 96 vectors: 446 us a launch at
// 128 threads, 642 at 256).
// At p = 7 two groups of 128 threads and 2 vectors each are 115 KB of shared memory, one CTA per SM;
// one group of 256 lets two CTAs in (11 x 9 x 8 cells, degree-6 filter without atoms: 150 vectors 15.10
// -> 13.26 ms at k = 0, 14.79 -> 13.83 at k != 0; 3 vectors 0.46 -> 0.43 and 0.50 -> 0.46).
template <int NP, int VB> __host__ __device__ constexpr int cell_group_threads() {
  constexpr int g4[9] = {0, 0, 0, 64, 128, 128, 256, 256, 256};
  constexpr int g2[9] = {0, 0, 0, 32, 64, 64, 128, 128, 256};
  return VB == 4 ? g4[NP] : g2[NP];
}
// Whether each warp owns whole z planes of a cell (see cell_body): where a plane's pencils
// fill a warp and a warp is left over (p = 6, 4 vectors: 28 to 32 lanes, 8.34 -> 7.62 ms a
// launch on 16^3 cells, 256 vectors; p = 5: 872 -> 815 us on 12^3 cells, 96 vectors).  At
// p = 7 a plane has 36 pencils a vector quad and every warp a plane (1048 -> 1090 us), at
// p <= 4 it leaves lanes idle (460 -> 575 us).
template <int NP> __host__ __device__ constexpr bool cell_planes() { return NP == 6 || NP == 7; }
// Whether a thread of the FP32 kernel's last stage has one spin of a pencil in recurrence mode: at p = 7
// and 2 vectors 128 pencils are half of the group, and the update's loads wait for each other.  11 x 9 x 8
// cells, k = 0: 7 vectors 112.9 -> 108.3 us a launch, 64 vectors 854 -> 852 (variant 2: 914 -> 885).  Without
// the update the shared-memory accesses of half a point each cost more (64 vectors 654 -> 693).
template <int NP, int VB> __host__ __device__ constexpr bool cell_split_spins() { return NP == 8 && VB == 2; }
constexpr int kNoNode = -(1 << 29);   // offset of a direction with no free node (Dirichlet face)

// ---------------------------------------------------------------------------
// the FP64 kernel
// ---------------------------------------------------------------------------
// even and odd parts (and the middle point of an odd count) of a pencil of NI points
template <int NI> struct PartsD {
  static constexpr int HI = NI / 2;
  double2 e[HI], o[HI], m;
};
template <int NI> __device__ __forceinline__ void set_part(PartsD<NI>& s, int j, double2 a, double2 b) {
  s.e[j] = make_double2(a.x + b.x, a.y + b.y);
  s.o[j] = make_double2(a.x - b.x, a.y - b.y);
}
template <int NI, typename F> __device__ __forceinline__ void load_parts(PartsD<NI>& s, F ld) {
#pragma unroll
  for (int j = 0; j < NI / 2; ++j) set_part(s, j, ld(j), ld(NI - 1 - j));
  if (NI & 1) s.m = ld(NI / 2);
}
// rows i and NO-1-i of a product: y_i = e + o, y_{NO-1-i} = e - o (the middle row is e)
struct AccD { double2 e, o; };
template <bool FIRST, int NO, int NI>
__device__ __forceinline__ void row_sym(const EO<double, NO, NI>& M, int i, const PartsD<NI>& s, AccD& a) {
#pragma unroll
  for (int j = 0; j < NI / 2; ++j) {
    if (FIRST && j == 0) {
      a.e = make_double2(M.E[i][j] * s.e[j].x, M.E[i][j] * s.e[j].y);
      if (NO - 1 - i != i) a.o = make_double2(M.O[i][j] * s.o[j].x, M.O[i][j] * s.o[j].y);
    } else {
      a.e.x += M.E[i][j] * s.e[j].x;
      a.e.y += M.E[i][j] * s.e[j].y;
      if (NO - 1 - i != i) {
        a.o.x += M.O[i][j] * s.o[j].x;
        a.o.y += M.O[i][j] * s.o[j].y;
      }
    }
  }
  if (NI & 1) {
    a.e.x += M.Mid[i] * s.m.x;
    a.e.y += M.Mid[i] * s.m.y;
  }
}
// a += i M x for a centro-antisymmetric M (the odd chain feeds the even accumulator and the
// even chain the odd one)
template <int NO, int NI>
__device__ __forceinline__ void row_anti(const EO<double, NO, NI>& M, int i, const PartsD<NI>& s, AccD& a) {
#pragma unroll
  for (int j = 0; j < NI / 2; ++j) {
    a.e.x -= M.O[i][j] * s.o[j].y;
    a.e.y += M.O[i][j] * s.o[j].x;
    if (NO - 1 - i != i) {
      a.o.x -= M.E[i][j] * s.e[j].y;
      a.o.y += M.E[i][j] * s.e[j].x;
    }
  }
  if ((NI & 1) && NO - 1 - i != i) {
    a.o.x -= M.Mid[i] * s.m.y;
    a.o.y += M.Mid[i] * s.m.x;
  }
}
template <int NO, typename F> __device__ __forceinline__ void put_rows(int i, const AccD& a, F st) {
  if (NO - 1 - i == i) {
    st(i, a.e);
  } else {
    st(i, make_double2(a.e.x + a.o.x, a.e.y + a.o.y));
    st(NO - 1 - i, make_double2(a.e.x - a.o.x, a.e.y - a.o.y));
  }
}
__device__ __forceinline__ void cp_async16z(void* dst, const void* src, int src_bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(src_bytes)
               : "memory");
}

constexpr int kHxThreads = 512;
// one group: 4 lane vectors (two (cell, vector)s x two spins) of [A | T2 | T1], the node
// offsets and records of three items
struct HxItem { int q, e[2], v[2], pad[3]; };   // system, cells (negative: none), vectors
constexpr int kHxSlots = 3;
template <int NP> __host__ __device__ constexpr size_t hx_group_smem() {
  return sizeof(double2) * 4 * (size_t)cell_vpoints<NP, 4>() + kHxSlots * (sizeof(HxItem) + 2 * 24 * sizeof(int));
}
template <int NP> __host__ __device__ constexpr int hx_groups() { return kHxThreads / cell_group_threads<NP, 4>(); }

// Whether items of one (cell, vector) are there too, for launches that leave SMs idle or one pair ahead of
// the others: at p = 4 and 7 half of the units is a round of the group's threads less (z stage: 144 on
// 128 threads, 324 on 256), so an SM with one or three single items is done before one with one or two
// pairs.  27 to 135 (cell, vector)s: p = 4 46 -> 36 us a launch, p = 7 141 -> 82; 400 to 420: p = 4 72 ->
// 59, p = 7 148 -> 120 (one pair a CTA in seven stages: 46, 138, 67 and 148).  Two single items an SM are
// no faster than one pair; at the other orders half of the units saves nothing (p = 5 at 420: 109 -> 152).
template <int NP> __host__ __device__ constexpr bool hx_single_items() { return NP == 5 || NP == 8; }

// PER: (cell, vector)s of an item
template <int NP, int NQ, bool KPT, int PER>
__global__ void __launch_bounds__(kHxThreads, 1)
hx_local_kernel(const __grid_constant__ LocalArgs a, const __grid_constant__ TablesEO<double, NP, NQ> tb) {
  constexpr int GT = cell_group_threads<NP, 4>(), NW = GT / 32;
  constexpr int BA = cell_bufa<NP>(), VS = cell_vpoints<NP, 4>();
  constexpr int NQ3 = NQ * NQ * NQ, HP = (NP + 1) / 2, HQ = (NQ + 1) / 2;
  using L = CellLayout<NP>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int group = threadIdx.x / GT;
  double2* sm = reinterpret_cast<double2*>(smem_raw + group * hx_group_smem<NP>());
  // lane vector w = 2 * slot + spin: point pidx at Buf(w)[pidx]
  auto Ab = [&](int w) { return sm + w * VS; };
  auto T2b = [&](int w) { return sm + w * VS + BA; };
  auto T1b = [&](int w) { return sm + w * VS + 2 * BA; };
  HxItem* rec0 = reinterpret_cast<HxItem*>(sm + 4 * VS);
  int* noff0 = reinterpret_cast<int*>(rec0 + kHxSlots);
  auto pa = [](int x, int y, int z) { return x + y * L::AY + z * L::AZ; };
  auto pq = [](int x, int y, int z) { return x + y * L::QY + z * L::QZ; };
  // odd groups number their warps backwards, so partly filled rounds fall on other schedulers
  const int tid0 = threadIdx.x % GT;
  const int tid = (group & 1) == 0 ? tid0 : ((NW - 1 - tid0 / 32) * 32 + (tid0 & 31));
  const int lane = tid & 31, warp = tid / 32;
  auto sync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "n"(GT) : "memory"); };
  constexpr bool PL = cell_planes<NP>();
  constexpr int PZW = PL ? (NP + NW - 1) / NW : NP;
  const int z0 = PL ? min(NP, warp * PZW) : 0, nz = PL ? min(NP - z0, PZW) : NP;
  constexpr int US = PL ? 32 : GT;
  const int ut = PL ? lane : tid;
  auto psync = [&]() {
    if (PL) __syncwarp();
    else sync();
  };
  // lane vectors of an item: unit u is lane vector u & lm of pencil u >> lb
  constexpr int lb = PER, lm = 2 * PER - 1;
  const long long ngroups = (long long)gridDim.x * hx_groups<NP>();
  // a CTA's groups take items gridDim.x apart, so few items spread over the SMs
  const long long first = (long long)group * gridDim.x + blockIdx.x;

  auto rec = [&](int n) -> HxItem& { return rec0[n % kHxSlots]; };
  auto noff = [&](int n, int slot) { return noff0 + (n % kHxSlots) * 48 + slot * 24; };
  // the group's last warp: record and node coordinates of the group's n-th item: node
  // (ix, iy, iz) is (no[8 + iy] + no[16 + iz]) * nfree[0] + no[ix], negative terms on a
  // Dirichlet face (a mesh may have more nodes than an int counts)
  auto post = [&](int n) {
    const long long it = first + n * ngroups;
    HxItem r{0, {-1, -1}, {0, 0}, {0, 0, 0}};
    if (it < a.nitems) {
      for (int k = 1; k < a.nsys; ++k)
        if (it >= a.sys[k].item0) r.q = k;
      const SysDesc& g = a.sys[r.q];
      const long long li = PER * (it - g.item0), n2 = (long long)g.mesh.E * g.nvec;
      for (int i = 0; i < PER; ++i)
        if (li + i < n2) {
          r.e[i] = (int)((li + i) / g.nvec);
          r.v[i] = (int)((li + i) - (long long)r.e[i] * g.nvec);
        }
    }
    if (lane == 0) rec(n) = r;
    if (lane < 3 * NP) {
      const MeshDev& m = a.sys[r.q].mesh;
      const int dd = lane / NP, i = lane % NP;
      for (int sl = 0; sl < 2; ++sl) {
        const int e = r.e[sl];
        if (e < 0) continue;
        const int c = dd == 0 ? e % m.ncell[0] : dd == 1 ? (e / m.ncell[0]) % m.ncell[1] : e / (m.ncell[0] * m.ncell[1]);
        const int gc = c * m.p + i;
        int f;
        if (m.periodic[dd]) f = gc >= m.period[dd] ? gc - m.period[dd] : gc;
        else f = (gc == 0 || gc == m.period[dd]) ? -1 : gc - 1;
        const int scale = dd < 2 ? 1 : m.nfree[1];
        noff(n, sl)[dd * 8 + i] = f < 0 ? kNoNode : f * scale;
      }
    }
  };
  // asynchronous gather of the thread's planes of item n into A, one (lane vector, x pencil)
  // at a time; zeros on Dirichlet faces and for an absent second (cell, vector)
  auto gather = [&](int n) {
    const HxItem it = rec(n);
    const SysDesc& g = a.sys[it.q];
    for (int i = ut; i < (NP * nz) << lb; i += US) {
      const int w = i & lm, pen = i >> lb, sl = w >> 1;
      const int y = pen % NP, z = z0 + pen / NP;
      const int* no = noff(n, sl);
      const bool have = (sl ? it.e[1] : it.e[0]) >= 0;
      const int Iyz = have ? no[8 + y] + no[16 + z] : kNoNode;
      double2* dst = &Ab(w)[pa(0, y, z)];
      const double2* src = g.X + (long long)(w & 1) * g.ldx + (sl ? it.v[1] : it.v[0]);
      const long long I0 = (long long)Iyz * g.mesh.nfree[0];
#pragma unroll
      for (int x = 0; x < NP; ++x) {
        const bool ok = Iyz >= 0 && no[x] >= 0 && GBC_IN_RANGE(GBC_SITE_HX64, I0 + no[x], g.mesh.M);
        cp_async16z(dst + x, ok ? src + 2 * (I0 + no[x]) * g.ldx : g.X, ok ? 16 : 0);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  const bool helper = warp == NW - 1;
  if (helper) {
    post(0);
    post(1);
  }
  sync();
  if (rec(0).e[0] >= 0) gather(0);
#pragma unroll 1
  for (int n = 0;; ++n) {
    const HxItem item = rec(n);
    if (item.e[0] < 0) break;
    const SysDesc& d = a.sys[item.q];
    asm volatile("cp.async.wait_all;" ::: "memory");
    psync();

    // ---- x pencils: T1 = N'^T X, A = B_x X (in place), T2 = G_x X
    for (int u = ut; u < (NP * nz) << lb; u += US) {
      const int w = u & lm, pen = u >> lb;
      const int y = pen % NP, z = z0 + pen / NP;
      double2 *A = Ab(w) + pa(0, y, z), *K = T2b(w) + pa(0, y, z), *Q = T1b(w) + pq(0, y, z);
      PartsD<NP> s;
      load_parts(s, [&](int j) { return A[j]; });
#pragma unroll
      for (int i = 0; i < HQ; ++i) {
        AccD r;
        row_sym<true, NQ>(tb.Ni, i, s, r);
        put_rows<NQ>(i, r, [&](int k, double2 v) { Q[k] = v; });
      }
#pragma unroll
      for (int i = 0; i < HP; ++i) {
        AccD r;
        row_sym<true, NP>(tb.B[0], i, s, r);
        put_rows<NP>(i, r, [&](int k, double2 v) { A[k] = v; });
        row_sym<true, NP>(tb.Gr[0], i, s, r);
        if (KPT) row_anti<NP>(tb.Gi[0], i, s, r);
        put_rows<NP>(i, r, [&](int k, double2 v) { K[k] = v; });
      }
    }
    psync();

    // ---- y pencils (in place): T1 = N'^T T1; T2 = G_y A + B_y T2
    for (int u = ut; u < (NQ * nz) << lb; u += US) {
      double2* Q = T1b(u & lm) + pq((u >> lb) % NQ, 0, z0 + (u >> lb) / NQ);
      PartsD<NP> s;
      load_parts(s, [&](int j) { return Q[j * L::QY]; });
#pragma unroll
      for (int i = 0; i < HQ; ++i) {
        AccD r;
        row_sym<true, NQ>(tb.Ni, i, s, r);
        put_rows<NQ>(i, r, [&](int k, double2 v) { Q[k * L::QY] = v; });
      }
    }
    for (int u = (ut + US - ((NQ * nz) << lb) % US) % US; u < (NP * nz) << lb; u += US) {
      const int w = u & lm, o = pa((u >> lb) % NP, 0, z0 + (u >> lb) / NP);
      const double2* A = Ab(w) + o;
      double2* K = T2b(w) + o;
      PartsD<NP> s1, s2;
      load_parts(s1, [&](int j) { return A[j * L::AY]; });
      load_parts(s2, [&](int j) { return K[j * L::AY]; });
#pragma unroll
      for (int i = 0; i < HP; ++i) {
        AccD r;
        row_sym<true, NP>(tb.Gr[1], i, s1, r);
        if (KPT) row_anti<NP>(tb.Gi[1], i, s1, r);
        row_sym<false, NP>(tb.B[1], i, s2, r);
        put_rows<NP>(i, r, [&](int k, double2 v) { K[k * L::AY] = v; });
      }
    }
    psync();
    // the planes of A are free: start the next item's gather behind the remaining stages
    if (rec(n + 1).e[0] >= 0) gather(n + 1);
    if (PL) sync();

    // ---- z pencils (in place): T1 = N' F N'^T T1 + G'_z T1; the two spins of a pencil are on
    // neighbouring lanes and swap their values by shuffle
    constexpr int UZ = (NQ * NQ) << lb;
#pragma unroll 1
    for (int rd = 0; rd < UZ; rd += GT) {
      const int uu = tid + rd;
      const bool act = uu < UZ;
      const int u = act ? uu : (uu & 1);
      const int w = u & lm, x = (u >> lb) % NQ, y = (u >> lb) / NQ;
      double2* Q = T1b(w) + pq(x, y, 0);
      const int e = max(0, (w >> 1) ? item.e[1] : item.e[0]);
      const double2* __restrict__ fld = reinterpret_cast<const double2*>(d.fields) + 2 * (size_t)e * NQ3;
      PartsD<NP> s;
      load_parts(s, [&](int j) { return Q[j * L::QZ]; });
      // up:   (V + bz) u + (bx - i by) d
      // down: (V - bz) d + (bx + i by) u
      auto spin_op = [&](int q, double2 own) {
        const double2 oth = make_double2(__shfl_xor_sync(0xffffffffu, own.x, 1),
                                         __shfl_xor_sync(0xffffffffu, own.y, 1));
        const double2 f0 = __ldg(fld + 2 * ((q * NQ + y) * NQ + x)), f1 = __ldg(fld + 2 * ((q * NQ + y) * NQ + x) + 1);
        const double dg = (w & 1) ? f0.x - f1.y : f0.x + f1.y, by = (w & 1) ? -f1.x : f1.x;
        return make_double2(dg * own.x + f0.y * oth.x + by * oth.y, dg * own.y + f0.y * oth.y - by * oth.x);
      };
      PartsD<NQ> t;
#pragma unroll
      for (int i = 0; i < HQ; ++i) {
        AccD r;
        double2 r0, r1;
        row_sym<true, NQ>(tb.Ni, i, s, r);
        put_rows<NQ>(i, r, [&](int k, double2 v) {
          if (k == i) r0 = spin_op(k, v);
          else r1 = spin_op(k, v);
        });
        if (NQ - 1 - i == i) t.m = r0;
        else set_part(t, i, r0, r1);
      }
#pragma unroll
      for (int i = 0; i < HP; ++i) {
        AccD r;
        row_sym<true, NP>(tb.Nt, i, t, r);
        row_sym<false, NP>(tb.Gr[2], i, s, r);
        if (KPT) row_anti<NP>(tb.Gi[2], i, s, r);
        if (act) put_rows<NP>(i, r, [&](int k, double2 v) { Q[k * L::QZ] = v; });
      }
    }
    // T2 = B_z T2 (the threads left idle by the last round above take the first units)
    for (int u = (tid + GT - UZ % GT) % GT; u < (NP * NP) << lb; u += GT) {
      double2* K = T2b(u & lm) + pa((u >> lb) % NP, (u >> lb) / NP, 0);
      PartsD<NP> s;
      load_parts(s, [&](int j) { return K[j * L::AZ]; });
#pragma unroll
      for (int i = 0; i < HP; ++i) {
        AccD r;
        row_sym<true, NP>(tb.B[2], i, s, r);
        put_rows<NP>(i, r, [&](int k, double2 v) { K[k * L::AZ] = v; });
      }
    }
    if (helper) post(n + 2);   // read after the group barrier that follows
    sync();

    // ---- y pencils (in place): T1 = N' T1
    for (int u = ut; u < (NQ * nz) << lb; u += US) {
      double2* Q = T1b(u & lm) + pq((u >> lb) % NQ, 0, z0 + (u >> lb) / NQ);
      PartsD<NQ> s;
      load_parts(s, [&](int j) { return Q[j * L::QY]; });
#pragma unroll
      for (int i = 0; i < HP; ++i) {
        AccD r;
        row_sym<true, NP>(tb.Nt, i, s, r);
        put_rows<NP>(i, r, [&](int k, double2 v) { Q[k * L::QY] = v; });
      }
    }
    psync();

    // ---- x pencils: N' T1 + T2, assembled
    for (int u = ut; u < (NP * nz) << lb; u += US) {
      const int w = u & lm, pen = u >> lb, sl = w >> 1, sp = w & 1;
      const int y = pen % NP, z = z0 + pen / NP;
      const int e = sl ? item.e[1] : item.e[0], vec = sl ? item.v[1] : item.v[0];
      if (e < 0) continue;
      const double2 *Q = T1b(w) + pq(0, y, z), *K = T2b(w) + pa(0, y, z);
      const int* no = noff(n, sl);
      const int Iyz = no[8 + y] + no[16 + z];
      PartsD<NQ> s;
      load_parts(s, [&](int j) { return Q[j]; });
#pragma unroll
      for (int i = 0; i < HP; ++i) {
        AccD r;
        row_sym<true, NP>(tb.Nt, i, s, r);
        put_rows<NP>(i, r, [&](int x, double2 v) {
          const double2 k = K[x];
          const double2 o = make_double2(v.x + k.x, v.y + k.y);
          const long long I = (long long)Iyz * d.mesh.nfree[0] + no[x];
          if (Iyz < 0 || no[x] < 0 || !GBC_IN_RANGE(GBC_SITE_HX64, I, d.mesh.M)) return;
          if (d.Ycell)
            d.Ycell[(((long long)e * (NP * NP * NP) + x + NP * (y + NP * z)) * 2 + sp) * d.nvec + vec] = o;
          else
            atomic_add_c(&d.Y[(I * 2 + sp) * d.ldx + vec], o);
        });
      }
    }
  }
}

template <int NP>
cudaError_t launch_hx_group_p(const HxJob* jobs, int n, cudaStream_t s) {
  constexpr int NQ = NP + 1;   // nq = p + 2
  if (n < 1 || n > GBC_MAX_BATCH) return cudaErrorInvalidValue;
  LocalArgs a;
  long long all = 0;
  for (int i = 0; i < n; ++i) all += (long long)jobs[i].c->mesh.E * jobs[i].nvec;
  const long long nsm = gbc_sm_count(), ones = (all + nsm - 1) / nsm, twos = (all + 2 * nsm - 1) / (2 * nsm);
  const int per = hx_single_items<NP>() && ones <= 3 && ones < 2 * twos ? 1 : 2;
  long long item = 0;
  for (int i = 0; i < GBC_MAX_BATCH; ++i) {
    SysDesc& d = a.sys[i];
    if (i >= n) {
      d = a.sys[0];
      d.item0 = 0x7fffffffffffffffLL;
      continue;
    }
    const gbc_ctx* c = jobs[i].c;
    d.X = (const double2*)jobs[i].X;
    d.Y = (double2*)jobs[i].Y;
    d.Ycell = (double2*)jobs[i].Ycell;
    d.fields = c->d_fields64;
    d.ldx = jobs[i].ldx;
    d.nvec = jobs[i].nvec;
    d.item0 = item;
    d.mesh = c->mesh;
    item += ((long long)c->mesh.E * d.nvec + per - 1) / per;
  }
  a.nsys = n;
  a.nitems = item;
  if (item <= 0) return cudaSuccess;
  const gbc_ctx* c0 = jobs[0].c;
  TablesEO<double, NP, NQ> tb;
  if (!make_tables_eo<double, NP, NQ>(c0, &tb)) return cudaErrorInvalidValue;
  const bool kpt = (c0->k[0] != 0.0 || c0->k[1] != 0.0 || c0->k[2] != 0.0);
  constexpr size_t smem = hx_groups<NP>() * hx_group_smem<NP>();
  static_assert(smem <= 227 * 1024, "shared memory of the FP64 cell apply");
  auto run = [&](auto kern) -> cudaError_t {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const long long nblk = std::min<long long>(item, gbc_sm_count());
    kern<<<(unsigned)nblk, kHxThreads, smem, s>>>(a, tb);
    return cudaGetLastError();
  };
  if constexpr (hx_single_items<NP>()) {
    if (per == 1) return kpt ? run(hx_local_kernel<NP, NQ, true, 1>) : run(hx_local_kernel<NP, NQ, false, 1>);
  }
  return kpt ? run(hx_local_kernel<NP, NQ, true, 2>) : run(hx_local_kernel<NP, NQ, false, 2>);
}

// Deterministic assembly: Y[I][s][v] += the results of every cell holding node I, added
// in a fixed order (cells by direction z, y, x, lower neighbour first).  Along each
// direction a node at grid index g is interior to cell g / p (local g % p), or, when
// g % p == 0, shared by cell g / p - 1 (local p; periodic wrap at 0) and cell g / p
// (local 0).
template <typename T>
__global__ void k_cell_gather(cplx<T>* __restrict__ Y, const cplx<T>* __restrict__ Ycell,
                              const MeshDev m, int nvec, int ldx) {
  const int np = m.p + 1;
  const long long np3 = (long long)np * np * np;
  const long long n = m.M * 2 * (long long)nvec;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x) {
    const int v = (int)(t % nvec);
    const long long rs = t / nvec;
    const int s = (int)(rs & 1);
    const long long I = rs >> 1;
    const long long f[3] = {I % m.nfree[0], (I / m.nfree[0]) % m.nfree[1],
                            I / ((long long)m.nfree[0] * m.nfree[1])};
    int cell[3][2], loc[3][2], cnt[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int g = (int)f[d] + (m.periodic[d] ? 0 : 1);
      const int q = g / m.p, r = g % m.p;
      if (r != 0) {
        cell[d][0] = q;
        loc[d][0] = r;
        cnt[d] = 1;
      } else {
        cnt[d] = 0;
        if (q > 0 || m.periodic[d]) {
          cell[d][cnt[d]] = q > 0 ? q - 1 : m.ncell[d] - 1;
          loc[d][cnt[d]++] = m.p;
        }
        if (q < m.ncell[d]) {
          cell[d][cnt[d]] = q;
          loc[d][cnt[d]++] = 0;
        }
      }
    }
    cplx<T> acc = cmake<cplx<T>>(0, 0);
    for (int a = 0; a < cnt[2]; ++a)
      for (int b = 0; b < cnt[1]; ++b)
        for (int c = 0; c < cnt[0]; ++c) {
          const long long e = cell[0][c] + (long long)m.ncell[0] * (cell[1][b] + (long long)m.ncell[1] * cell[2][a]);
          const long long l = loc[0][c] + np * (loc[1][b] + np * loc[2][a]);
          const cplx<T> y = Ycell[((e * np3 + l) * 2 + s) * nvec + v];
          acc.x += y.x;
          acc.y += y.y;
        }
    cplx<T>& o = Y[(I * 2 + s) * ldx + v];
    o.x += acc.x;
    o.y += acc.y;
  }
}

}  // namespace gbc
