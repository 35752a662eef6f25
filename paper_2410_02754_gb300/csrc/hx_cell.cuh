// Cell-level apply of the local spinor Hamiltonian for FP32 blocks, with an
// optional fused Chebyshev recurrence epilogue.
//
// Paper: Sec. IV.B.2 (extract X^(e) = R^(e) X, cell products, assemble
// Y = sum_e R^(e)T Y^(e)) for the cell operator of Eq. FEHlocEl plus the k-terms
// of Eq. FEHloc (per-cell Hermitian form), and Eq. chebfilt for the recurrence.
//
// Algorithm: with N' = N diag(sqrt(w_q)) (nodes x Gauss points, so that the 1-D mass is
// (h/2) N' N'^T; the tables split w_q unevenly, so that they round best to FP32) and the 1-D kinetic / k operators G_d,
//   a  = N'_x^T X,  t1 = B_x X,  t2 = G_x X                      x pencils (n_p^2)
//   u  = N'_y^T a;  c  = G_y t1 + B_y t2                          y pencils (n_q n_p; n_p^2)
//   w  = N'_z F N'_z^T u + G'_z u;  k = B_z c                     z pencils (n_q^2; n_p^2)
//   Y^(e) = N'_x N'_y w + k                                       y, then x pencils
// where F = J [(V + |k|^2/2) I + B . sigma] at the Gauss points and G'_z = (h_x h_y / 4) G_z:
// the z part of the kinetic term rides on the interpolated field (N'_x N'_y of G'_z u is
// B_x B_y G_z X), so five stages and five kinetic 1-D products do what the separate kinetic
// and potential passes of the dense form need seven for.  Every 1-D product is in even-odd
// form, the products of one input sharing its even and odd parts and the products of one
// output one accumulator.
//
// Mapping:
//  * a thread owns a pencil of one vector, both spins: shared memory holds (up, down) of a
//    point side by side, so every access is 16 bytes, the spin operator needs no exchange
//    between lanes, and a table entry is used four times per load; complex values are
//    float2 and a product is one paired multiply-add (or two scalar ones; both compiled);
//  * per vector three buffers used in place: A (gathered X^(e), then t1), T2 (t2, c, k) and
//    T1 (a, u, w);
//  * the gather of the next work item (cp.async) starts when A is free, after the second
//    stage, and hides behind the other three;
//  * a CTA is several independent groups of threads, each with its own work items, buffers
//    and named barrier, so one group's arithmetic fills the other's barrier waits at 128
//    registers a thread; at p = 5 and 6 a warp owns whole z planes of the cell, which leaves
//    two group barriers an item, both around the z stage; a helper warp takes the items from
//    the work counter two ahead, so neither the atomic's latency nor the index divisions are
//    waited for.
//
// Bounds at p = 6, k != 0 per cell and vector: 123,000 FP32 lane operations (960 cycles of
// an SM's 128 lanes) and 103 KB of shared-memory traffic (806 cycles at 128 bytes).  Measured
// on one GB300, 16^3 cells, p = 6, 256 vectors, k != 0, recurrence mode: 11.30 -> 7.62 ms a
// launch (2290 cycles; the L1 data pipe is 73% busy, issue 54%), from 12.3 -> 6.6 thousand
// warp instructions per cell and vector pair.  The steps: five stages and 16-byte two-spin
// pencils 9.29, index work once per pencil 9.07, items decoded once and fields staged 8.34,
// planes owned by warps 7.62.  Other sizes: 12^3 cells, p = 5, 96 vectors 1144 -> 815 us;
// p = 4 812 -> 460; 10^3 cells, p = 3, 128 vectors 460 -> 212; p = 7, 64 vectors 1167 -> 1048
// (in recurrence mode, tuned, 11 x 9 x 8 cells, k = 0: 3, 7 and 64 vectors 1.26, 1.58 and 6.63 ms a degree-6
// filter in seven stages, 1.24, 1.59 and 6.48 now).
//
// Assembly modes (per system):
//  * accumulate: Y += H^loc X with FP32 atomics on every node;
//  * recurrence: for nodes interior to the cell (owned by it alone) the cell
//    holds the complete local row, so the Chebyshev update is applied here:
//      X_out = a (M_D^-1 (Y + y_loc) - c X) - b X_prev
//    (Y holds the nonlocal term P C' of that row, written before this kernel,
//    or zero); nodes on cell faces are accumulated into Y with atomics and
//    finished by a separate row pass (launch_cheb_rows).
#pragma once

#include "hx_local.cuh"

namespace gbc {

// 1-D operator in even-odd form with every entry duplicated into a float2, the
// multiplier of a paired multiply-add on (re, im)
template <int NO, int NI> struct EO2 {
  static constexpr int HO = (NO + 1) / 2;
  static constexpr int HI = NI / 2 > 0 ? NI / 2 : 1;
  float2 E[HO][HI];
  float2 O[HO][HI];
  float2 Mid[HO];
};

// PACKED: entries duplicated for paired multiply-adds; otherwise plain FP32
// entries for two scalar multiply-adds (re, im) that take the entry straight
// from the constant bank
template <int NP, int NQ, bool PACKED> struct CellTables {
  template <int NO, int NI>
  using M = typename std::conditional<PACKED, EO2<NO, NI>, EO<float, NO, NI>>::type;
  M<NP, NP> B[3];    // 1-D Gauss mass
  M<NP, NP> Gr[3];   // 1/2 A_d (z: times h_x h_y / 4)
  M<NP, NP> Gi[3];   // -1/2 k_d (C^ - C^T) (z: times h_x h_y / 4)
  M<NQ, NP> Ni;      // N'^T: interpolation to the Gauss points times s_q (gq_s)
  M<NP, NQ> Nt;      // N': times w_q / s_q
};

// One system of a launch.
struct CellSys {
  const float2* X;      // block applied to
  float2* Y;            // accumulator
  const float* fields;  // [E][NQ^3][4] J (V + |k|^2/2), J B_x, J B_y, J B_z
  float2* Xout;         // recurrence mode: X_{k+1} (may alias Xprev)
  const float2* Xprev;  // recurrence mode: X_{k-1}, or null on the first step
  const float* invmd;   // recurrence mode: 1 / M_D per node
  float ca, cc, cb;     // recurrence mode: X_{k+1} = ca (M_D^-1 Y - cc X) - cb X_{k-1}
  int ldx, nvec, vchunks, cheb;
  long long item0;      // work items [item0, item0 + E * vchunks)
  MeshDev mesh;
};

struct CellArgs {
  CellSys sys[GBC_MAX_SYS];
  int nsys;
  long long nitems;
};

__device__ __forceinline__ float2 p_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
// a - b, exactly (the fused product -1 * b is exact)
__device__ __forceinline__ float2 p_sub(float2 a, float2 b) {
  return __ffma2_rn(make_float2(-1.f, -1.f), b, a);
}
__device__ __forceinline__ float2 p_mul(float2 m, float2 x) { return __fmul2_rn(m, x); }
__device__ __forceinline__ float2 p_fma(float2 m, float2 x, float2 acc) {
  return __ffma2_rn(m, x, acc);
}
__device__ __forceinline__ float2 dup(float v) { return make_float2(v, v); }

// 8-byte asynchronous global -> shared copy; src_bytes = 0 writes zeros
__device__ __forceinline__ void cp_async8(void* dst, const void* src, int src_bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(src_bytes)
               : "memory");
}
// 16-byte asynchronous global -> shared copy (both addresses 16-byte aligned)
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// products and sums of complex values held as float2: paired instructions for a duplicated
// table entry (float2), scalar ones for a plain entry
__device__ __forceinline__ float2 m_mul(float2 m, float2 x) { return p_mul(m, x); }
__device__ __forceinline__ float2 m_fma(float2 m, float2 x, float2 a) { return p_fma(m, x, a); }
__device__ __forceinline__ float2 m_mul(float m, float2 x) { return make_float2(m * x.x, m * x.y); }
__device__ __forceinline__ float2 m_fma(float m, float2 x, float2 a) {
  return make_float2(fmaf(m, x.x, a.x), fmaf(m, x.y, a.y));
}
template <bool PACKED> __device__ __forceinline__ float2 c_add(float2 a, float2 b) {
  return PACKED ? p_add(a, b) : make_float2(a.x + b.x, a.y + b.y);
}
template <bool PACKED> __device__ __forceinline__ float2 c_sub(float2 a, float2 b) {
  return PACKED ? p_sub(a, b) : make_float2(a.x - b.x, a.y - b.y);
}
__device__ __forceinline__ float2 lo2(float4 v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(float4 v) { return make_float2(v.z, v.w); }
__device__ __forceinline__ float4 cat2(float2 a, float2 b) { return make_float4(a.x, a.y, b.x, b.y); }

// even and odd parts (and the middle point of an odd count) of a pencil of NI points, both
// spins: e_j = x_j + x_{NI-1-j}, o_j = x_j - x_{NI-1-j}
template <int NI> struct Parts {
  static constexpr int HI = NI / 2;
  float2 e[2][HI], o[2][HI], m[2];
};
template <bool PACKED, int NI>
__device__ __forceinline__ void set_part(Parts<NI>& s, int j, float4 a, float4 b) {
  s.e[0][j] = c_add<PACKED>(lo2(a), lo2(b));
  s.o[0][j] = c_sub<PACKED>(lo2(a), lo2(b));
  s.e[1][j] = c_add<PACKED>(hi2(a), hi2(b));
  s.o[1][j] = c_sub<PACKED>(hi2(a), hi2(b));
}
template <bool PACKED, int NI, typename F>
__device__ __forceinline__ void load_parts(Parts<NI>& s, F ld) {
#pragma unroll
  for (int j = 0; j < NI / 2; ++j) set_part<PACKED>(s, j, ld(j), ld(NI - 1 - j));
  if (NI & 1) {
    const float4 c = ld(NI / 2);
    s.m[0] = lo2(c);
    s.m[1] = hi2(c);
  }
}

// rows i and NO-1-i of a product, as even and odd accumulators of both spins:
// y_i = ae + ao, y_{NO-1-i} = ae - ao (the middle row of an odd NO is ae alone)
struct Acc { float2 e[2], o[2]; };
// FIRST: a = M x, else a += M x, for a centro-symmetric M
template <bool FIRST, int NO, int NI, typename MT>
__device__ __forceinline__ void row_sym(const MT& M, int i, const Parts<NI>& s, Acc& a) {
  constexpr int HI = NI / 2;
#pragma unroll
  for (int j = 0; j < HI; ++j)
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      a.e[q] = (FIRST && j == 0) ? m_mul(M.E[i][j], s.e[q][j]) : m_fma(M.E[i][j], s.e[q][j], a.e[q]);
      if (NO - 1 - i != i)
        a.o[q] = (FIRST && j == 0) ? m_mul(M.O[i][j], s.o[q][j]) : m_fma(M.O[i][j], s.o[q][j], a.o[q]);
    }
  if (NI & 1) {
#pragma unroll
    for (int q = 0; q < 2; ++q) a.e[q] = m_fma(M.Mid[i], s.m[q], a.e[q]);
  }
}
// a += i M x for a centro-antisymmetric M (its odd chain feeds the even accumulator and the
// even chain the odd one)
template <int NO, int NI, typename MT>
__device__ __forceinline__ void row_anti(const MT& M, int i, const Parts<NI>& s, Acc& a) {
  constexpr int HI = NI / 2;
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    float2 te = m_mul(M.E[i][0], s.e[q][0]), to = m_mul(M.O[i][0], s.o[q][0]);
#pragma unroll
    for (int j = 1; j < HI; ++j) {
      te = m_fma(M.E[i][j], s.e[q][j], te);
      to = m_fma(M.O[i][j], s.o[q][j], to);
    }
    if (NI & 1) te = m_fma(M.Mid[i], s.m[q], te);
    a.e[q].x -= to.y;
    a.e[q].y += to.x;
    if (NO - 1 - i != i) {
      a.o[q].x -= te.y;
      a.o[q].y += te.x;
    }
  }
}
// st(row, both spins) for the two rows of a
template <bool PACKED, int NO, typename F>
__device__ __forceinline__ void put_rows(int i, const Acc& a, F st) {
  if (NO - 1 - i == i) {
    st(i, cat2(a.e[0], a.e[1]));
  } else {
    st(i, cat2(c_add<PACKED>(a.e[0], a.o[0]), c_add<PACKED>(a.e[1], a.o[1])));
    st(NO - 1 - i, cat2(c_sub<PACKED>(a.e[0], a.o[0]), c_sub<PACKED>(a.e[1], a.o[1])));
  }
}

// a work item: system, cell, first vector; e < 0: none
struct alignas(16) CellItem { int q, e, v0, pad; };
constexpr int kCellSlots = 4;    // item records and offset tables in flight
// one group: vector buffers, the cell's fields (FS), the item records and node offsets
template <int NP, int VB, bool FS> __host__ __device__ constexpr size_t cell_group_smem() {
  return sizeof(float4) * ((size_t)VB * cell_vpoints<NP, VB>() +
                           (FS ? (NP + 1) * (NP + 1) * (NP + 1) : 0)) +
         kCellSlots * (sizeof(CellItem) + sizeof(int) * 3 * 8);
}
// 1 / M_D of a cell's interior nodes: one table per CTA
template <int NP> __host__ __device__ constexpr size_t cell_mass_smem() {
  return (sizeof(float) * (NP - 2) * (NP - 2) * (NP - 2) + 15) / 16 * 16;
}
// the fields are staged in shared memory where MINB CTAs per SM still fit with them
template <int NP, int VB, int NT, int MINB> __host__ __device__ constexpr bool cell_stage_fields() {
  return MINB * (NT / cell_group_threads<NP, VB>() * cell_group_smem<NP, VB, true>() +
                 cell_mass_smem<NP>() + 1024) <= 228 * 1024;
}
template <int NP, int VB, int NT, int MINB> __host__ __device__ constexpr size_t cell_smem() {
  return NT / cell_group_threads<NP, VB>() * cell_group_smem<NP, VB, cell_stage_fields<NP, VB, NT, MINB>()>() +
         cell_mass_smem<NP>();
}

// The work items [0, nitems) of the systems sys[0 .. nsys) (item0 ascending), after each
// group's first taken from the counter *ctr (zero at launch) one at a time, so groups that
// finish early take more and the items in flight stay close to each other in
// the order (cell-major, vector chunks of a cell adjacent).  GT: threads of a group.
template <int NP, int NQ, bool KPT, int VB, int GT, bool PACKED, bool FS>
__device__ __forceinline__ void cell_body(const CellSys* __restrict__ sys, int nsys,
                                          long long nitems, const CellTables<NP, NQ, PACKED>& tb,
                                          unsigned long long* __restrict__ ctr) {
  constexpr int BA = cell_bufa<NP>();
  constexpr int NQ3 = NQ * NQ * NQ;
  constexpr int VS = cell_vpoints<NP, VB>();
  constexpr int HP = (NP + 1) / 2, HQ = (NQ + 1) / 2;   // row pairs
  using L = CellLayout<NP>;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  const int group = threadIdx.x / GT;
  float4* sm = reinterpret_cast<float4*>(sm_raw + group * cell_group_smem<NP, VB, FS>());
  // both spins of point pidx of vector v: Buf(v)[pidx]
  auto Ab = [&](int v) { return sm + v * VS; };
  auto T2b = [&](int v) { return sm + v * VS + BA; };
  auto T1b = [&](int v) { return sm + v * VS + 2 * BA; };
  auto pa = [](int x, int y, int z) { return x + y * L::AY + z * L::AZ; };
  auto pq = [](int x, int y, int z) { return x + y * L::QY + z * L::QZ; };
  // odd groups number their warps backwards: a stage's last, partly filled round then falls
  // on other schedulers than the even groups'
  const int tid0 = threadIdx.x % GT;
  const int tid = (group & 1) == 0 ? tid0 : ((GT / 32 - 1 - tid0 / 32) * 32 + (tid0 & 31));
  auto sync = [&]() {   // the group's own barrier
    if (GT == 32) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "n"(GT) : "memory");
  };
  // the work item with index ``it``
  auto decode = [&](long long it) {
    CellItem r{0, -1, 0, 0};
    if (it >= nitems) return r;
    if (nsys > 1) {   // one system: skip the scan over the descriptor slots
#pragma unroll
      for (int k = 1; k < GBC_MAX_SYS; ++k)
        if (k < nsys && it >= sys[k].item0) r.q = k;
    }
    const long long li = it - sys[r.q].item0;
    r.e = (int)(li / sys[r.q].vchunks);
    r.v0 = (int)(li - (long long)r.e * sys[r.q].vchunks) * VB;
    return r;
  };

  // records of the items in flight, item n in slot n % kCellSlots, with the node offsets of
  // its cell: local node (ix, iy, iz) is noff[0][ix] + noff[1][iy] + noff[2][iz], negative
  // where the node is on a Dirichlet face
  float4* fsm = sm + VB * VS;
  CellItem* rec = reinterpret_cast<CellItem*>(fsm + (FS ? NQ3 : 0));
  int* noff0 = reinterpret_cast<int*>(rec + kCellSlots);
  auto noff = [&](int n) { return noff0 + (n % kCellSlots) * 24; };
  // 1 / M_D of a cell's interior nodes, after the last group's buffers: a node inside one cell
  // has the same mass in every cell of a launch (all of its systems share p and the edges)
  constexpr int NIN = NP - 2;
  float* wint = reinterpret_cast<float*>(sm_raw + blockDim.x / GT * cell_group_smem<NP, VB, FS>());
  {
    const MeshDev& m = sys[0].mesh;
    for (int i = threadIdx.x; i < NIN * NIN * NIN; i += blockDim.x) {
      const int x = i % NIN + m.periodic[0], y = (i / NIN) % NIN + m.periodic[1],
                z = i / (NIN * NIN) + m.periodic[2];
      wint[i] = __ldg(sys[0].invmd + ((long long)z * m.nfree[1] + y) * m.nfree[0] + x);
    }
    __syncthreads();
  }
  const int lane = tid & 31, warp = tid / 32;
  constexpr int NW = GT / 32;
  // PL: the x and y stages, the gather and the assembly of the planes z0 .. z0 + nz - 1 are
  // one warp's, ordered by warp barriers alone; otherwise all planes belong to the group
  constexpr bool PL = cell_planes<NP>();
  // the helper warp stages the fields and posts items before the x stage; at p = 7 it has a
  // full share of pencils, and all threads stage and it posts after the z stage
  constexpr bool EARLY = NP < 8;
  constexpr int PZW = PL ? (NP + NW - 1) / NW : NP;
  const int z0 = PL ? min(NP, warp * PZW) : 0, nz = PL ? min(NP - z0, PZW) : NP;
  constexpr int US = PL ? 32 : GT;           // threads that share a plane's units
  const int ut = PL ? lane : tid;
  auto psync = [&]() {
    if (PL) __syncwarp();
    else sync();
  };
  const bool helper = warp == NW - 1;

  // warp ``helper``: write the record and the offsets of item n, the counter's value ``it``
  auto post = [&](int n, long long it) {
    CellItem r{0, -1, 0, 0};
    if (lane == 0) {
      r = decode(it);
      rec[n % kCellSlots] = r;
    }
    r.q = __shfl_sync(0xffffffffu, r.q, 0);
    r.e = __shfl_sync(0xffffffffu, r.e, 0);
    if (r.e >= 0 && lane < 3 * NP) {
      const MeshDev& m = sys[r.q].mesh;
      const int dd = lane / NP, i = lane % NP;
      const int c = dd == 0 ? r.e % m.ncell[0]
                  : dd == 1 ? (r.e / m.ncell[0]) % m.ncell[1] : r.e / (m.ncell[0] * m.ncell[1]);
      const int gc = c * m.p + i;
      int f;
      if (m.periodic[dd]) f = gc >= m.period[dd] ? gc - m.period[dd] : gc;
      else f = (gc == 0 || gc == m.period[dd]) ? -1 : gc - 1;
      const int scale = dd == 0 ? 1 : dd == 1 ? m.nfree[0] : m.nfree[0] * m.nfree[1];
      noff(n)[dd * 8 + i] = f < 0 ? kNoNode : f * scale;
    }
  };
  // asynchronous gather of the thread's planes of item n into A: thread -> (vector, spin, x
  // pencil), vector fastest; absent nodes (Dirichlet faces) and vectors beyond nvec are
  // zero-filled
  auto gather = [&](int n) {
    const CellItem it = rec[n % kCellSlots];
    const CellSys& g = sys[it.q];
    const int* no = noff(n);
    const long long step = 2 * (long long)g.ldx;
    for (int i = ut; i < VB * 2 * NP * nz; i += US) {
      const int v = i % VB, s = (i / VB) & 1, pen = i / (2 * VB);
      const int y = pen % NP, z = z0 + pen / NP;
      const int Iyz = no[8 + y] + no[16 + z];
      const bool ok0 = Iyz >= 0 && it.v0 + v < g.nvec;
      float2* dst = reinterpret_cast<float2*>(&Ab(v)[pa(0, y, z)]) + s;
      const float2* src = g.X + (long long)s * g.ldx + it.v0 + v;
      // nodes x = 1 .. NP-2 are consecutive; the two on x faces may wrap or be absent
      const int I1 = Iyz + no[1];
      const float2* p = src + I1 * step;
#pragma unroll
      for (int x = 1; x < NP - 1; ++x, p += step) {
        const bool ok = ok0 && GBC_IN_RANGE(GBC_SITE_CELL_GATHER, I1 + x - 1, g.mesh.M);
        cp_async8(dst + 2 * x, ok ? p : g.X, ok ? 8 : 0);
      }
#pragma unroll
      for (int x = 0; x < NP; x += NP - 1) {
        const int I = Iyz + no[x];
        const bool ok = ok0 && I >= 0 && GBC_IN_RANGE(GBC_SITE_CELL_GATHER, I, g.mesh.M);
        cp_async8(dst + 2 * x, ok ? src + I * step : g.X, ok ? 8 : 0);
      }
    }
    cp_async_commit();
  };

  // fields of an item's cell into shared memory
  auto stage_fields = [&](const CellItem& it, int t, int nt) {
    if (!FS) return;
    const float4* src = reinterpret_cast<const float4*>(sys[it.q].fields) + (size_t)it.e * NQ3;
    for (int i = t; i < NQ3; i += nt) cp_async16(fsm + i, src + i);
    cp_async_commit();
  };

  // Items are taken two ahead by the helper warp.  A group's first item is its own: those of a
  // CTA are gridDim.x apart, so few items spread over the SMs.
  const long long ngroups = (long long)gridDim.x * (blockDim.x / GT);
  auto take = [&]() {
    long long it = 0;
    if (lane == 0) it = ngroups + (long long)atomicAdd(ctr, 1ULL);
    return it;
  };
  if (helper) {
    post(0, (long long)group * gridDim.x + blockIdx.x);
    post(1, take());
  }
  sync();
  if (rec[0].e >= 0) {
    gather(0);
    if (!EARLY) stage_fields(rec[0], tid, GT);
  }
#pragma unroll 1
  for (int n = 0;; ++n) {
    const CellItem item = rec[n % kCellSlots];
    if (item.e < 0) break;
    const CellSys& d = sys[item.q];
    const int e = item.e;
    const int vbase = item.v0;
    const int* no = noff(n);
    long long taken = 0;
    if (helper) taken = take();
    if (EARLY && helper) {
      stage_fields(item, lane, 32);
      post(n + 2, taken);
    }
    cp_async_wait_all();
    psync();

    // ---- x pencils: T1 = N'^T X, A = B_x X (in place), T2 = G_x X
    for (int u = ut; u < VB * NP * nz; u += US) {
      const int v = u % VB, pen = u / VB;
      const int y = pen % NP, z = z0 + pen / NP;
      float4 *A = Ab(v) + pa(0, y, z), *K = T2b(v) + pa(0, y, z), *Q = T1b(v) + pq(0, y, z);
      Parts<NP> s;
      load_parts<PACKED>(s, [&](int j) { return A[j]; });
#pragma unroll
      for (int i = 0; i < HQ; ++i) {
        Acc a;
        row_sym<true, NQ>(tb.Ni, i, s, a);
        put_rows<PACKED, NQ>(i, a, [&](int r, float4 val) { Q[r] = val; });
      }
#pragma unroll
      for (int i = 0; i < HP; ++i) {
        Acc a;
        row_sym<true, NP>(tb.B[0], i, s, a);
        put_rows<PACKED, NP>(i, a, [&](int r, float4 val) { A[r] = val; });
        row_sym<true, NP>(tb.Gr[0], i, s, a);
        if (KPT) row_anti<NP>(tb.Gi[0], i, s, a);
        put_rows<PACKED, NP>(i, a, [&](int r, float4 val) { K[r] = val; });
      }
    }
    psync();

    // ---- y pencils (in place): T1 = N'^T T1; T2 = G_y A + B_y T2
    for (int u = ut; u < VB * NQ * nz; u += US) {
      const int v = u % VB, pen = u / VB;
      float4* Q = T1b(v) + pq(pen % NQ, 0, z0 + pen / NQ);
      Parts<NP> s;
      load_parts<PACKED>(s, [&](int j) { return Q[j * L::QY]; });
#pragma unroll
      for (int i = 0; i < HQ; ++i) {
        Acc a;
        row_sym<true, NQ>(tb.Ni, i, s, a);
        put_rows<PACKED, NQ>(i, a, [&](int r, float4 val) { Q[r * L::QY] = val; });
      }
    }
    // (the threads left idle by the last round above take the first units here)
    for (int u = (ut + US - VB * NQ * nz % US) % US; u < VB * NP * nz; u += US) {
      const int v = u % VB, pen = u / VB;
      const int o = pa(pen % NP, 0, z0 + pen / NP);
      const float4* A = Ab(v) + o;
      float4* K = T2b(v) + o;
      Parts<NP> s1, s2;
      load_parts<PACKED>(s1, [&](int j) { return A[j * L::AY]; });
      load_parts<PACKED>(s2, [&](int j) { return K[j * L::AY]; });
#pragma unroll
      for (int i = 0; i < HP; ++i) {
        Acc a;
        row_sym<true, NP>(tb.Gr[1], i, s1, a);
        if (KPT) row_anti<NP>(tb.Gi[1], i, s1, a);
        row_sym<false, NP>(tb.B[1], i, s2, a);
        put_rows<PACKED, NP>(i, a, [&](int r, float4 val) { K[r * L::AY] = val; });
      }
    }
    psync();
    // the planes of A are free: start the next item's gather
    if (rec[(n + 1) % kCellSlots].e >= 0) gather(n + 1);
    if (PL) sync();

    // ---- z pencils (in place): T1 = N' F N'^T T1 + G'_z T1; T2 = B_z T2
    constexpr int UZ = VB * NQ * NQ;
    {
      const float4* __restrict__ fld = reinterpret_cast<const float4*>(d.fields) + (size_t)e * NQ3;
      for (int u = tid; u < UZ; u += GT) {
        const int v = u % VB, pen = u / VB;
        const int x = pen % NQ, y = pen / NQ;
        float4* Q = T1b(v) + pq(x, y, 0);
        Parts<NP> s;
        load_parts<PACKED>(s, [&](int j) { return Q[j * L::QZ]; });
        // up:   (V + bz) u + (bx - i by) d
        // down: (V - bz) d + (bx + i by) u
        auto spin_op = [&](int q, float4 o) {
          const float4 F = FS ? fsm[(q * NQ + y) * NQ + x] : __ldg(fld + (q * NQ + y) * NQ + x);
          const float vp = F.x + F.w, vm = F.x - F.w;
          return make_float4(fmaf(F.z, o.w, fmaf(F.y, o.z, vp * o.x)),
                             fmaf(-F.z, o.z, fmaf(F.y, o.w, vp * o.y)),
                             fmaf(-F.z, o.y, fmaf(F.y, o.x, vm * o.z)),
                             fmaf(F.z, o.x, fmaf(F.y, o.y, vm * o.w)));
        };
        Parts<NQ> w;
#pragma unroll
        for (int i = 0; i < HQ; ++i) {
          Acc a;
          float4 r0, r1;
          row_sym<true, NQ>(tb.Ni, i, s, a);
          put_rows<PACKED, NQ>(i, a, [&](int r, float4 val) {
            if (r == i) r0 = spin_op(r, val);
            else r1 = spin_op(r, val);
          });
          if (NQ - 1 - i == i) {
            w.m[0] = lo2(r0);
            w.m[1] = hi2(r0);
          } else {
            set_part<PACKED>(w, i, r0, r1);
          }
        }
#pragma unroll
        for (int i = 0; i < HP; ++i) {
          Acc a;
          row_sym<true, NP>(tb.Nt, i, w, a);
          row_sym<false, NP>(tb.Gr[2], i, s, a);
          if (KPT) row_anti<NP>(tb.Gi[2], i, s, a);
          put_rows<PACKED, NP>(i, a, [&](int r, float4 val) { Q[r * L::QZ] = val; });
        }
      }
    }
    for (int u = (tid + GT - UZ % GT) % GT; u < VB * NP * NP; u += GT) {
      const int v = u % VB, pen = u / VB;
      float4* K = T2b(v) + pa(pen % NP, pen / NP, 0);
      Parts<NP> s;
      load_parts<PACKED>(s, [&](int j) { return K[j * L::AZ]; });
#pragma unroll
      for (int i = 0; i < HP; ++i) {
        Acc a;
        row_sym<true, NP>(tb.B[2], i, s, a);
        put_rows<PACKED, NP>(i, a, [&](int r, float4 val) { K[r * L::AZ] = val; });
      }
    }
    sync();

    if (!EARLY) {
      if (helper) post(n + 2, taken);
      const CellItem next = rec[(n + 1) % kCellSlots];
      if (next.e >= 0) stage_fields(next, tid, GT);
    }
    // ---- y pencils of the planes (in place): T1 = N' T1
    for (int u = ut; u < VB * NQ * nz; u += US) {
      const int v = u % VB, pen = u / VB;
      float4* Q = T1b(v) + pq(pen % NQ, 0, z0 + pen / NQ);
      Parts<NQ> s;
      load_parts<PACKED>(s, [&](int j) { return Q[j * L::QY]; });
#pragma unroll
      for (int i = 0; i < HP; ++i) {
        Acc a;
        row_sym<true, NP>(tb.Nt, i, s, a);
        put_rows<PACKED, NP>(i, a, [&](int r, float4 val) { Q[r * L::QY] = val; });
      }
    }
    psync();

    // ---- x pencils: N' T1 + T2, assembled (vector fastest across threads; NS spins a thread)
    auto assemble = [&](auto ns) {
      constexpr int NS = decltype(ns)::value;
      for (int u = ut; u < VB * NP * nz * (3 - NS); u += US) {
        const int s0 = NS == 2 ? 0 : u / (VB * NP * NP);
        const int v = u % VB, pen = (u - s0 * VB * NP * NP) / VB;
        const int y = pen % NP, z = z0 + pen / NP;
        const int vec = vbase + v;
        if (vec >= d.nvec) continue;
        float2 out[NS][NP];
        {
          const float4* Q = T1b(v) + pq(0, y, z);
          const float4* K = T2b(v) + pa(0, y, z);
          // both spins of a point, or one of them twice (what the second half would do is not compiled)
          auto ld = [&](const float4* p) {
            if (NS == 2) return *p;
            const float2 a = reinterpret_cast<const float2*>(p)[s0];
            return cat2(a, a);
          };
          Parts<NQ> s;
          load_parts<PACKED>(s, [&](int j) { return ld(Q + j); });
#pragma unroll
          for (int i = 0; i < HP; ++i) {
            Acc a;
            row_sym<true, NP>(tb.Nt, i, s, a);
            put_rows<PACKED, NP>(i, a, [&](int r, float4 val) {
              const float4 k = ld(K + r);
              out[0][r] = c_add<PACKED>(lo2(val), lo2(k));
              if (NS == 2) out[NS - 1][r] = c_add<PACKED>(hi2(val), hi2(k));
            });
          }
        }
        const bool yz_in = y > 0 && y < NP - 1 && z > 0 && z < NP - 1;
        const int Iyz = no[8 + y] + no[16 + z];
#pragma unroll
        for (int si = 0; si < NS; ++si) {
          const int s = s0 + si;
          if (d.cheb && yz_in) {
            // nodes x = 1 .. NP-2 of this pencil are interior to the cell: every load is
            // issued before the first update (X_out may alias X_prev), so their latencies
            // overlap
            float2 yv[NIN], xv[NIN], pv[NIN];
            const long long step = 2 * (long long)d.ldx;
            const int I1 = Iyz + no[1];   // consecutive from here
            const long long o1 = I1 * step + (long long)s * d.ldx + vec;
            const float* w = wint + ((z - 1) * NIN + y - 1) * NIN;
#pragma unroll
            for (int j = 0; j < NIN; ++j) {
              const long long o = o1 + j * step;
              if (GBC_IN_RANGE(GBC_SITE_CELL_STORE, I1 + j, d.mesh.M)) {
                yv[j] = d.Y[o];
                xv[j] = __ldg(&d.X[o]);
                pv[j] = d.Xprev ? d.Xprev[o] : make_float2(0.f, 0.f);
              } else {
                yv[j] = xv[j] = pv[j] = make_float2(0.f, 0.f);
              }
            }
#pragma unroll
            for (int j = 0; j < NIN; ++j) {
              const long long o = o1 + j * step;
              const float2 yt = p_add(yv[j], out[si][1 + j]);
              const float2 xn = p_fma(dup(-d.cb), pv[j],
                                      p_mul(dup(d.ca), p_fma(dup(-d.cc), xv[j], p_mul(dup(w[j]), yt))));
              if (GBC_IN_RANGE(GBC_SITE_CELL_STORE, I1 + j, d.mesh.M)) d.Xout[o] = xn;
            }
#pragma unroll
            for (int i = 0; i < NP; i += NP - 1) {   // the pencil's two face nodes
              const int I = Iyz + no[i];
              if (I >= 0 && GBC_IN_RANGE(GBC_SITE_CELL_STORE, I, d.mesh.M))
                atomicAdd(&d.Y[((long long)I * 2 + s) * d.ldx + vec], out[si][i]);
            }
          } else {
#pragma unroll
            for (int i = 0; i < NP; ++i) {
              const int I = Iyz + no[i];
              if (I >= 0 && GBC_IN_RANGE(GBC_SITE_CELL_STORE, I, d.mesh.M))
                atomicAdd(&d.Y[((long long)I * 2 + s) * d.ldx + vec], out[si][i]);
            }
          }
        }
      }
    };
    if (cell_split_spins<NP, VB>() && d.cheb) assemble(std::integral_constant<int, cell_split_spins<NP, VB>() ? 1 : 2>());
    else assemble(std::integral_constant<int, 2>());
  }
}

// One persistent launch over systems that share p, the cell edges and the k-point;
// the groups of the CTAs take their work items from the zeroed counter *ctr in ascending
// order.
template <int NP, int NQ, bool KPT, int VB, int NT, int MINB, bool PACKED>
__global__ void __launch_bounds__(NT, MINB)
hx_cell_kernel(const __grid_constant__ CellArgs a,
               const __grid_constant__ CellTables<NP, NQ, PACKED> tb,
               unsigned long long* __restrict__ ctr) {
  cell_body<NP, NQ, KPT, VB, cell_group_threads<NP, VB>(), PACKED, cell_stage_fields<NP, VB, NT, MINB>()>(
      a.sys, a.nsys, a.nitems, tb, ctr);
}

template <int NO, int NI>
inline void cvt_table(const EO<float, NO, NI>& src, EO<float, NO, NI>& dst) { dst = src; }
template <int NO, int NI>
inline void cvt_table(const EO<float, NO, NI>& src, EO2<NO, NI>& dst) {
  for (int i = 0; i < EO2<NO, NI>::HO; ++i) {
    for (int j = 0; j < EO2<NO, NI>::HI; ++j) {
      dst.E[i][j] = make_float2(src.E[i][j], src.E[i][j]);
      dst.O[i][j] = make_float2(src.O[i][j], src.O[i][j]);
    }
    dst.Mid[i] = make_float2(src.Mid[i], src.Mid[i]);
  }
}

template <int NP, int NQ, bool PACKED>
inline bool make_cell_tables(const gbc_ctx* c, CellTables<NP, NQ, PACKED>* t) {
  TablesEO<float, NP, NQ> f;
  if (!make_tables_eo<float, NP, NQ>(c, &f)) return false;
  for (int d = 0; d < 3; ++d) {
    cvt_table(f.B[d], t->B[d]);
    cvt_table(f.Gr[d], t->Gr[d]);
    cvt_table(f.Gi[d], t->Gi[d]);
  }
  cvt_table(f.Ni, t->Ni);
  cvt_table(f.Nt, t->Nt);
  return true;
}

// descriptor of one system (items numbered from item0)
inline void fill_sys(CellSys& d, const CellJob& j, int vb, long long item0) {
    const gbc_ctx* c = j.c;
    d.X = (const float2*)j.X;
    d.Y = (float2*)j.Y;
    d.fields = c->d_fields32;
    d.Xout = (float2*)j.Xout;
    d.Xprev = (const float2*)j.Xprev;
    d.invmd = c->d_invmd32;
    d.ca = (float)j.a;
    d.cc = (float)j.cshift;
    d.cb = (float)j.b;
    d.cheb = j.Xout != nullptr;
    d.ldx = j.ldx;
    d.nvec = j.nvec;
    d.vchunks = (j.nvec + vb - 1) / vb;
    d.item0 = item0;
    d.mesh = c->mesh;
}

// One launch over up to GBC_MAX_SYS systems sharing p, the cell edges and the
// k-point.
template <int NP, int VB, int NT, int MINB, bool PACKED>
cudaError_t launch_cell_group_p(const CellJob* jobs, int n, cudaStream_t s) {
  constexpr int NQ = NP + 1;   // nq = p + 2
  if (n < 1 || n > GBC_MAX_SYS) return cudaErrorInvalidValue;
  CellArgs a;
  long long item = 0;
  for (int i = 0; i < GBC_MAX_SYS; ++i) {
    CellSys& d = a.sys[i];
    if (i >= n) {
      d = a.sys[0];
      d.item0 = 0x7fffffffffffffffLL;
      continue;
    }
    fill_sys(d, jobs[i], VB, item);
    item += (long long)jobs[i].c->mesh.E * d.vchunks;
  }
  a.nsys = n;
  a.nitems = item;
  if (item <= 0) return cudaSuccess;
  const gbc_ctx* c0 = jobs[0].c;
  CellTables<NP, NQ, PACKED> tb;
  if (!make_cell_tables<NP, NQ, PACKED>(c0, &tb)) return cudaErrorInvalidValue;
  const bool kpt = (c0->k[0] != 0.0 || c0->k[1] != 0.0 || c0->k[2] != 0.0);
  constexpr size_t smem = cell_smem<NP, VB, NT, MINB>();
  int dev = 0, nsm = 0, per_sm = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err != cudaSuccess) return err;
  err = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (err != cudaSuccess) return err;
  unsigned long long* ctr = c0->d_cell_ctr;   // the first system's work counter
  if (!ctr) return cudaErrorInvalidValue;
  auto run = [&](auto kern) -> cudaError_t {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NT, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    const long long nblk = std::min<long long>(item, (long long)nsm * per_sm);
    e = cudaMemsetAsync(ctr, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)nblk, NT, smem, s>>>(a, tb, ctr);
    return cudaGetLastError();
  };
  if (smem > 227 * 1024) return cudaErrorInvalidConfiguration;
  if (kpt) return run(hx_cell_kernel<NP, NQ, true, VB, NT, MINB, PACKED>);
  return run(hx_cell_kernel<NP, NQ, false, VB, NT, MINB, PACKED>);
}

template <int VB, int NT, int MINB, bool PACKED>
cudaError_t launch_cell_group(const CellJob* jobs, int n, cudaStream_t s) {
  for (int i = 0; i < n; ++i)   // node offsets are 32-bit
    if (jobs[i].c->mesh.M >= (1LL << 29)) return cudaErrorInvalidValue;
  switch (jobs[0].c->mesh.p) {
    case 2: return launch_cell_group_p<3, VB, NT, MINB, PACKED>(jobs, n, s);
    case 3: return launch_cell_group_p<4, VB, NT, MINB, PACKED>(jobs, n, s);
    case 4: return launch_cell_group_p<5, VB, NT, MINB, PACKED>(jobs, n, s);
    case 5: return launch_cell_group_p<6, VB, NT, MINB, PACKED>(jobs, n, s);
    default: break;
  }
  if constexpr (MINB < 3) {   // see launch_cell_f32
    if (jobs[0].c->mesh.p == 6) return launch_cell_group_p<7, VB, NT, MINB, PACKED>(jobs, n, s);
    if (jobs[0].c->mesh.p == 7) return launch_cell_group_p<8, VB, NT, MINB, PACKED>(jobs, n, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace gbc
