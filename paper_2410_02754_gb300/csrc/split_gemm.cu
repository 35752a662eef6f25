// Gram matrices and block rotations of CholGS / Rayleigh-Ritz as exact split products on the
// tcgen05 tensor cores (BF16 digits, FP32 accumulation without rounding, integer recombination).
//
// Paper: Sec. III.B.2 (X^H M X, X^H H X, U = X Q).  Method: the error-free transformation of a
// matrix product by splitting both factors (Ozaki, Ogita, Oishi, Rump, Numer. Algorithms 59,
// 2012), with balanced base-256 digits: a value x with |x| < 2^E is
//   x = 2^(E-6) sum_k d_k 256^-k,  |d_0| <= 65, d_k in [-128, 127],
// so every digit is a BF16 number and a product of two digits an integer below 2^14; S digits
// carry 8 S - 2 bits below 2^E.  The partial products of order t = i + j < T,
// G_t = sum_{i+j=t} A_i B_j, are integers that FP32 holds exactly while S K 2^14 <= 2^24;
// the accumulators are read out (to 64-bit integers) every kFlush K chunks to keep that, and
// sum_t G_t 256^-t is rounded at the end (Gram matrices and projections: once per part
// of K, the parts added in FP64).  Exponents are per row of A and B: per block
// row and per column of Q for a rotation, per column of the block (over all rows) for a Gram
// matrix.  A row with an infinity or a NaN is marked and gives NaN, as in FP arithmetic.
//
// S = 7 digits: an entry is off by at most 2^-55 of its row's largest.  FP32 blocks are rounded to
// FP32 once.  The rotation of CholGS, whose terms can cancel, takes its columns at a common size, by
// powers of two; that of Rayleigh-Ritz rests on an M_D-orthonormal block, whose columns have one size.
// Orders t < T are summed.  What is left out of a sum over K terms is about sqrt(K) 2^-54 of the
// product of the largest entries at T = S, sqrt(K) 2^-62 at T = S + 1, which counts where a sum is
// small against that: the rotation of a nearly converged block (Q close to the identity), Gram
// entries of columns that peak in a few of many rows, projectors over most of their support.  FP64:
// T = S + 1.  FP64 columns with one of 746,000 rows 1000 times the others came out of CholGS
// orthonormal to 5e-14 with T = S, to 1.3e-15 now (direct FP64 2.2e-15; 10^5 times: 5e-13, direct
// 6e-13).  FP32 blocks: T = S, which is closer than the float-float sums of before (Ritz values of
// such FP32 columns 3.4e-15 of the largest, float-float 4.7e-14) and far below the rounding to
// FP32.  S = T = 4 was not: columns of a nearly converged FP32 block of 256 came out 6.2e-8 off,
// 2.5e-8 (their rounding) now.
//
// GB300's FP64 pipe gives 1.05 TFLOP/s and float-float arithmetic on the FP32 pipes about 6;
// 28 (34) BF16 products at T = S (S + 1) and 1.9 PFLOP/s are an FP64-accurate 68 (56) TFLOP/s.  Measured, 884,736 nodes x 256
// FP32 columns: Gram 122 -> 22.6 ms, rotation 163 -> 26.6 ms; 373,248 nodes x 256 in FP64: 333 ->
// 11.5 and 527 -> 13.0 ms.  Per tile (128 x 64) every order has its own accumulator in tensor memory and all S
// digit slices of a 64-wide K chunk are in shared memory at once (one TMA box each), so a
// slice is loaded once per tile and used in up to S products.  Step i multiplies A_i with all
// of B_0 .. B_{T-1-i} in instructions of up to 256 columns (one product per instruction, 64
// columns, ran at a quarter of this rate); A_i's next chunk then loads behind the other steps,
// B is double-buffered.
#include <algorithm>
#include <cmath>
#include <cuda.h>

#include "gbc_internal.h"
#include "tc.cuh"

namespace {

constexpr int kTM = 128;              // tile rows
constexpr int kKC = 64;               // K chunk: one 128-byte swizzled row
constexpr int kBad = 0x7fffffff;      // exponent of a row with an infinity or a NaN
constexpr int kEpi = 16;              // read-out warps
constexpr int kSplitThreads = 64 + 32 * kEpi;
constexpr int S = 7;                  // digits
constexpr int kTN = 64;               // tile columns
constexpr int kFlush = 2;             // K chunks between read-outs
constexpr int kABytes = kTM * 128, kBBytes = kTN * 128;
constexpr size_t kSplitSmem = 1024 + (size_t)S * (kABytes + 2 * kBBytes) + 256;
static_assert((long long)S * kFlush * kKC << 14 <= 1LL << 24, "exact accumulation");
static_assert(kSplitSmem <= 227 * 1024, "shared memory");

// PROJ, EXPD: the FP64 projector contractions C += P^H X and Y += P C' (see nl_split_project)
enum { ROT32, ROT64, GRAM32, GRAM64, PROJ, EXPD };
// orders summed (order S: digits 1 .. S-1 only)
template <int MODE> __host__ __device__ constexpr int split_orders() {
  return MODE == ROT32 || MODE == GRAM32 ? S : S + 1;
}
constexpr int kNlRows = 1024;         // rows of a support chunk's place in the digit buffers
struct SplitArgs {
  int rows_a, rows_b;      // rows of a slice of A and B
  int nchunk, kper;        // K chunks; chunks per work item (GRAM: a part of them)
  int ntn;                 // column tiles
  int ntiles, nwork;       // tiles; work items (tiles, GRAM: x K parts)
  const int *ea, *eb;      // unit exponents (E - 6) of the rows of A and B
  long long rows;          // rotation: valid rows of the chunk; EXPD: free nodes of the mesh
  int n;                   // complex columns
  int ldo;                 // rotation, EXPD: complex leading dimension of out
  void* out;
  int* err;                // the context's word for an expired wait
  // PROJ, EXPD: chunks (atom, first node, count, node offset of the atom), supports, projectors
  // and first row of C of an atom
  const int4* chunks;
  const long long* nodes;
  const int *npj, *c_off;
};

// Persistent: CTAs take work items blockIdx.x, + gridDim.x, ...; the roles run on across items.
template <int MODE>
__global__ void __launch_bounds__(kSplitThreads, 1)
k_split_gemm(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb,
             const SplitArgs a) {
  constexpr int N = kTN, T = split_orders<MODE>();
  constexpr bool GRAM = MODE == GRAM32 || MODE == GRAM64;
  static_assert(T * N <= 512 && T <= 8, "tensor memory columns");
  struct Item { int m0, n0, k0, nk, b; };   // b: chunk of the batch
  auto decode = [&](int w) {
    Item it{0, 0, 0, a.nchunk, 0};
    if (GRAM) {   // tiles that reach the diagonal or above it, row by row
      int I = 0, t = w % a.ntiles, first = 0;
      while (t >= a.ntn - first) {
        t -= a.ntn - first;
        ++I;
        first = I * (kTM / N);
      }
      it.m0 = I * kTM;
      it.n0 = (first + t) * N;
      it.k0 = (w / a.ntiles) * a.kper;
      it.nk = min(a.kper, a.nchunk - it.k0);
    } else if (MODE == PROJ) {   // X columns x projectors over the chunk's nodes
      it.b = w / a.ntn;
      it.m0 = w % a.ntn * kTM;
      it.k0 = it.b * (kNlRows / kKC);
      it.nk = (a.chunks[it.b].z + 127) / 128 * (128 / kKC);
    } else if (MODE == EXPD) {   // nodes x columns of C' over the atom's projectors (B per chunk)
      const int mt = w / a.ntn;
      it.b = mt / (kNlRows / kTM);
      const int4 ch = a.chunks[it.b];
      it.m0 = mt * kTM;
      it.n0 = (it.b * a.ntn + w % a.ntn) * N;
      it.nk = it.m0 - it.b * kNlRows < ch.z ? 1 : 0;
    } else {   // column tiles of a row tile next to each other (its digits stay in L2)
      it.m0 = w / a.ntn * kTM;
      it.n0 = w % a.ntn * N;
    }
    return it;
  };
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* st = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* fulla = reinterpret_cast<uint64_t*>(st + S * (kABytes + 2 * kBBytes));   // [S]
  uint64_t* emptya = fulla + S;                                                          // [S]
  uint64_t* fullb = emptya + S;                                                          // [2]
  uint64_t* emptyb = fullb + 2;                                                          // [2]
  uint64_t* accf = emptyb + 2;                                       // accumulators complete
  uint64_t* acce = accf + 1;                                         // accumulators read out
  uint64_t* drain = acce + 1;                                        // every MMA complete
  uint32_t* tslot = reinterpret_cast<uint32_t*>(drain + 1);
  int* fail = reinterpret_cast<int*>(tslot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // A: one buffer per digit slice; B: two buffers of all slices back to back
  auto A = [&](int s) { return tc::smem_u32(st + s * kABytes); };
  auto B = [&](int buf, int s) {
    return tc::smem_u32(st + S * kABytes + (buf * S + s) * kBBytes);
  };
  auto failed = [&]() { return *reinterpret_cast<volatile int*>(fail) != 0; };

  if (warp == 0) {
    tc::tmem_alloc(tc::smem_u32(tslot), 512);
    tc::tmem_relinquish();
  }
  if (threadIdx.x == 32) {
    for (int s = 0; s < S; ++s) {
      tc::mbar_init(tc::smem_u32(&fulla[s]), 1);
      tc::mbar_init(tc::smem_u32(&emptya[s]), 1);
    }
    for (int s = 0; s < 2; ++s) {
      tc::mbar_init(tc::smem_u32(&fullb[s]), 1);
      tc::mbar_init(tc::smem_u32(&emptyb[s]), 1);
    }
    tc::mbar_init(tc::smem_u32(accf), 1);
    tc::mbar_init(tc::smem_u32(acce), kEpi);
    tc::mbar_init(tc::smem_u32(drain), 1);
    *fail = 0;
    tc::fence_mbar_init();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *tslot;

  if (warp == 0 && lane == 0) {
    // producer: chunk q of the CTA; A slice s once step s of chunk q - 1 is done, B buffer
    // q & 1 once chunk q - 2 is done
    int q = 0, ib = 0, ia[S];
#pragma unroll
    for (int s = 0; s < S; ++s) ia[s] = 0;
    for (int w = blockIdx.x; w < a.nwork && !failed(); w += gridDim.x) {
      const Item it = decode(w);
      for (int c = 0; c < it.nk && !failed(); ++c, ++q) {
        const int x = (it.k0 + c) * kKC, buf = q & 1;
        if (q > 1 && !tc::mbar_wait_bounded(tc::smem_u32(&emptyb[buf]), (q / 2 - 1) & 1)) atomicExch(fail, 1);
        if (failed()) break;
        const uint32_t fb = tc::smem_u32(&fullb[buf]);
        tc::mbar_arrive_expect_tx(fb, S * kBBytes);
#pragma unroll
        for (int s = 0; s < S; ++s) tc::tma_load_2d(B(buf, s), &tb, x, s * a.rows_b + it.n0, fb);
        ib = q + 1;
#pragma unroll
        for (int s = 0; s < S; ++s) {
          if (q > 0 && !tc::mbar_wait_bounded(tc::smem_u32(&emptya[s]), (q - 1) & 1)) atomicExch(fail, 1);
          if (failed()) break;
          const uint32_t fa = tc::smem_u32(&fulla[s]);
          tc::mbar_arrive_expect_tx(fa, kABytes);
          tc::tma_load_2d(A(s), &ta, x, s * a.rows_a + it.m0, fa);
          ia[s] = q + 1;
        }
      }
    }
    if (failed()) {   // let the copies in flight land first
#pragma unroll
      for (int s = 0; s < S; ++s)
        if (ia[s]) tc::mbar_wait_bounded(tc::smem_u32(&fulla[s]), (ia[s] - 1) & 1);
      for (int j = max(0, ib - 2); j < ib; ++j)
        tc::mbar_wait_bounded(tc::smem_u32(&fullb[j & 1]), (j / 2) & 1);
    }
  } else if (warp == 1 && lane == 0) {
    int q = 0, win = 0;
    for (int w = blockIdx.x; w < a.nwork && !failed(); w += gridDim.x) {
      const Item it = decode(w);
      for (int c = 0; c < it.nk && !failed(); ++c, ++q) {
        const bool first = c % kFlush == 0;
        if (first && win > 0 && !tc::mbar_wait_bounded(tc::smem_u32(acce), (win - 1) & 1)) atomicExch(fail, 1);
        const int buf = q & 1;
        if (!tc::mbar_wait_bounded(tc::smem_u32(&fullb[buf]), (q / 2) & 1)) atomicExch(fail, 1);
#pragma unroll
        for (int i = 0; i < S; ++i) {
          if (!tc::mbar_wait_bounded(tc::smem_u32(&fulla[i]), q & 1)) atomicExch(fail, 1);
          tc::fence_after_sync();
          // A_i against B_0 .. B_{T-1-i} at once: the slices are consecutive rows of one operand
          // and their orders i .. T-1 consecutive accumulators, so an instruction is up to 256
          // columns wide (64 columns take as long as 256)
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
#pragma unroll
            for (int j = 0; j < (T - i < S ? T - i : S); j += 256 / N) {
              constexpr int W = 256 / N;
              const int nb = T - i < S ? T - i : S, cnt = nb - j < W ? nb - j : W;
              auto mma = [&](int j, int cnt, unsigned acc) {
                tc::mma_bf16(tmem + (i + j) * N, tc::sdesc_sw128(A(i) + kk * 32),
                             tc::sdesc_sw128(B(buf, j) + kk * 32), tc::idesc_bf16(kTM, cnt * N), acc);
              };
              if (T > S && i == 1 && kk == 0 && j + cnt == S && first) {   // order S starts here
                if (cnt > 1) mma(j, cnt - 1, 1u);
                mma(S - 1, 1, 0u);
              } else {
                mma(j, cnt, (first && i == 0 && kk == 0) ? 0u : 1u);
              }
            }
          tc::mma_commit(tc::smem_u32(&emptya[i]));
        }
        tc::mma_commit(tc::smem_u32(&emptyb[buf]));
        if ((c + 1) % kFlush == 0 || c + 1 == it.nk) {
          tc::mma_commit(tc::smem_u32(accf));
          ++win;
        }
      }
    }
    // tensor memory is given back only after the issued MMAs (also after a failure)
    tc::mma_commit(tc::smem_u32(drain));
    if (!tc::mbar_wait_bounded(tc::smem_u32(drain), 0)) atomicExch(fail, 1);
  } else if (warp >= 2) {
    const int g = warp & 3, part = (warp - 2) >> 2;
    constexpr int NC = N / (kEpi / 4);               // columns of a thread
    const uint32_t tl = tmem + ((uint32_t)(g * 32) << 16) + (uint32_t)(part * NC);
    int win = 0;
    bool ok = true;
    for (int w = blockIdx.x; w < a.nwork && ok; w += gridDim.x) {
      const Item it = decode(w);
      // orders 0..3 and 4..T-1 as 64-bit integers, in units of 256^-3 and 256^-(T-1)
      long long hi[NC], lo[NC];
#pragma unroll
      for (int i = 0; i < NC; ++i) {
        hi[i] = 0;
        lo[i] = 0;
      }
      const int nwin = (it.nk + kFlush - 1) / kFlush;
      for (int v = 0; v < nwin && ok; ++v, ++win) {
        ok = tc::mbar_wait_bounded(tc::smem_u32(accf), win & 1);
        if (!ok) atomicExch(fail, 1);
        ok = ok && !failed();
        tc::fence_after_sync();
        if (ok) {
#pragma unroll
          for (int c0 = 0; c0 < NC; c0 += 8) {
            // orders 0..3, then the others: half of the registers at a time
            uint32_t r[4][8];
#pragma unroll
            for (int t = 0; t < 4; ++t) tc::tmem_ld8_nowait(tl + t * N + c0, r[t]);
            tc::tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
              for (int t = 0; t < 4; ++t)
                hi[c0 + i] += (long long)__float2int_rn(__uint_as_float(r[t][i])) * (1 << (8 * (3 - t)));
#pragma unroll
            for (int t = 4; t < T; ++t) tc::tmem_ld8_nowait(tl + t * N + c0, r[t - 4]);
            tc::tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
              for (int t = 4; t < T; ++t)
                lo[c0 + i] += (long long)__float2int_rn(__uint_as_float(r[t - 4][i])) * (1 << (8 * (T - 1 - t)));
          }
        }
        tc::fence_before_sync();
        if (lane == 0) tc::mbar_arrive(tc::smem_u32(acce));
      }
      if (T > S) {   // back to units of 256^-(S-1)
#pragma unroll
        for (int i = 0; i < NC; ++i) lo[i] = (lo[i] + 128) >> 8;
      }
      if (ok && it.nk > 0) {
        const int mr = it.m0 + g * 32 + lane;
        const int ea = a.ea[mr + (MODE == PROJ ? it.b * a.rows_a : 0)];
        const int cb = it.n0 + part * NC;
        const int* eb = a.eb + cb + (MODE == PROJ ? it.b * a.rows_b : 0);
        // a rotation's sum (|hi| < 2^47) as one integer in units of 2^(ea + eb - 24 - sh): exact
        // where |hi| < 2^38, else cut 2^-53 below its leading bit; rounded once
        auto value = [&](int i, int& sh) {
          const bool small = llabs(hi[i]) < (1LL << 38);
          sh = small ? 24 : 15;
          return small ? (hi[i] << 24) + lo[i] : (hi[i] << 15) + (lo[i] >> 9);
        };
        if (MODE == ROT32) {
          if (mr < a.rows) {
            float2* o = reinterpret_cast<float2*>(a.out) + (size_t)mr * a.ldo + cb / 2;
#pragma unroll
            for (int i = 0; i < NC; i += 2) {
              if (cb + i >= 2 * a.n) break;
              float v[2];
#pragma unroll
              for (int q = 0; q < 2; ++q) {
                int sh;
                const float f = __ll2float_rn(value(i + q, sh));
                const int e = eb[i + q];
                v[q] = (ea == kBad || e == kBad) ? NAN : scalbnf(f, ea + e - 24 - sh);
              }
              o[i / 2] = make_float2(v[0], v[1]);
            }
          }
        } else {
          int4 ch{};
          int cols = 2 * a.n, c0 = cb;   // valid real columns, the thread's first
          if (MODE == PROJ) {
            ch = a.chunks[it.b];
            cols = mr < 4 * a.n ? 2 * a.npj[ch.x] : 0;
          }
          if (MODE == EXPD) {
            ch = a.chunks[it.b];
            c0 = cb - it.b * a.ntn * N;
            cols = mr - it.b * kNlRows < ch.z ? 4 * a.n : 0;
          }
#pragma unroll
          for (int i = 0; i < NC; i += 2) {
            if (c0 + i >= cols) break;
            double v[2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
              int sh = 0;
              if (GRAM)   // hi may use all of its 53 bits here: hi + 2^-24 lo, rounded once
                v[q] = fma(__ll2double_rn(lo[i + q]), 0x1p-24, __ll2double_rn(hi[i + q]));
              else
                v[q] = __ll2double_rn(value(i + q, sh));
              const int e = eb[i + q];
              const bool bad = ea == kBad || e == kBad;
              const int x = bad ? 0 : ea + e - 24 - sh;
              if (bad) v[q] = NAN;
              else if (abs(x) > 900) v[q] = scalbn(v[q], x);
              else if (v[q] != 0.0)   // a multiplication by 2^x on the integer pipe (2^-24 <= |v| < 2^63)
                v[q] = __hiloint2double(__double2hiint(v[q]) + (x << 20), __double2loint(v[q]));
            }
            if (MODE == ROT64) {
              if (mr < a.rows)
                reinterpret_cast<double2*>(a.out)[(size_t)mr * a.ldo + (cb + i) / 2] = make_double2(v[0], v[1]);
            } else if (MODE == PROJ) {
              // conj(p) x: re = pr xr + pi xi, im = pr xi - pi xr; the row is one part of x
              const int xc = mr >> 1, sp = xc >= a.n, vec = xc - sp * a.n;
              double2* o = reinterpret_cast<double2*>(a.out) +
                           (size_t)(a.c_off[ch.x] + 2 * ((c0 + i) >> 1) + sp) * a.n + vec;
              atomicAdd(&o->x, (mr & 1) ? v[1] : v[0]);
              atomicAdd(&o->y, (mr & 1) ? v[0] : -v[1]);
            } else if (MODE == EXPD) {
              const int yc = (c0 + i) >> 1, sp = yc >= a.n, vec = yc - sp * a.n;
              const long long node = a.nodes[ch.w + ch.y + mr - it.b * kNlRows];
              if (!GBC_IN_RANGE(GBC_SITE_NL_NODE, node, a.rows)) break;
              double2* o = reinterpret_cast<double2*>(a.out) + (node * 2 + sp) * a.ldo + vec;
              atomicAdd(&o->x, v[0]);
              atomicAdd(&o->y, v[1]);
            } else {
              // conj(x) y of complex columns (mr / 2, (cb + i) / 2): re = rr + ii, im = ri - ir
              const int ci = mr >> 1, cj = (cb + i) >> 1;
              if (ci < a.n && ci <= cj) {
                double2* s = reinterpret_cast<double2*>(a.out) + (size_t)ci * a.n + cj;
                atomicAdd(&s->x, (mr & 1) ? v[1] : v[0]);
                atomicAdd(&s->y, (mr & 1) ? -v[0] : v[1]);
              }
            }
          }
        }
      }
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (failed() && threadIdx.x == 0) atomicExch(a.err, 1);
  if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

// ---------------------------------------------------------------------------
// splitting
// ---------------------------------------------------------------------------
// largest-magnitude key of a value (ordered as an unsigned integer) and its exponent E
// (|x| < 2^E), kBad for an infinity or a NaN
__device__ __forceinline__ unsigned mag_key(float x) { return __float_as_uint(x) & 0x7fffffffu; }
__device__ __forceinline__ unsigned mag_key(double x) {
  return (unsigned)__double2hiint(x) & 0x7fffffffu;
}
template <typename T> __device__ __forceinline__ int key_exponent(unsigned k) {
  if (sizeof(T) == 4) {
    if (k >= 0x7f800000u) return kBad;
    return k == 0 ? 0 : max((int)(k >> 23), 1) - 126;
  }
  if (k >= 0x7ff00000u) return kBad;
  return k == 0 ? 0 : max((int)(k >> 20), 1) - 1022;
}
// x as a fixed-point integer with unit 2^(E - 6 - 8 (S - 1)), rounded to nearest
template <typename T> __device__ __forceinline__ long long to_fixed(T x, int E) {
  long long m;
  int sh;
  bool neg;
  if (sizeof(T) == 4) {
    const unsigned b = __float_as_uint((float)x);
    const int ex = (b >> 23) & 0xff;
    m = (b & 0x7fffffu) | (ex ? 0x800000u : 0u);
    neg = b >> 31;
    sh = max(ex, 1) - 150;
  } else {
    const long long b = __double_as_longlong((double)x);
    const int ex = (int)((b >> 52) & 0x7ff);
    m = (b & 0xfffffffffffffLL) | (ex ? 0x10000000000000LL : 0LL);
    neg = b < 0;
    sh = max(ex, 1) - 1075;
  }
  sh += 6 + 8 * (S - 1) - E;
  if (sh >= 0) m = sh > 30 ? 0 : m << sh;   // more only for a subnormal that the exponent left out
  else m = sh < -60 ? 0 : (m + (1LL << (-sh - 1))) >> -sh;
  return neg ? -m : m;
}
// the biased digits of q (byte k of the result is digit S-1-k plus 128)
__device__ __forceinline__ unsigned long long digits(long long q) {
  return (unsigned long long)q + (0x8080808080808080ULL >> (64 - 8 * S));
}
// digit s (0 = leading) of two values, as two BF16 (a low, b high)
__device__ __forceinline__ unsigned pack2(unsigned long long a, unsigned long long b, int s) {
  const int sh = 8 * (S - 1 - s);
  const float fa = __uint_as_float(0x4B000000u | ((unsigned)(a >> sh) & 255u)) - 8388736.f;
  const float fb = __uint_as_float(0x4B000000u | ((unsigned)(b >> sh) & 255u)) - 8388736.f;
  return __byte_perm(__float_as_uint(fa), __float_as_uint(fb), 0x7632);
}

// exponent of the larger part of a complex value that counts 2^c: kNone for zero, kBad for an
// infinity or a NaN
constexpr int kNone = -(1 << 30);
template <typename T, typename V> __device__ __forceinline__ int scaled_exponent(V x, int c) {
  const unsigned k = max(mag_key(x.x), mag_key(x.y));
  const int e = key_exponent<T>(k);
  return k == 0 ? kNone : e == kBad ? kBad : e + c;
}

// rows of a block (2n reals each) -> digits [S][rows_pad][kp] and unit exponents, one warp per
// row; rows >= rows are written as zeros.  cs: exponents that multiply the columns (or null).  They
// are added to the exponents and never multiplied in: they may be larger than the type's range.
template <typename T>
__global__ void __launch_bounds__(256)
k_split_rows(const cplx<T>* __restrict__ X, int ldx, int n, long long rows, int rows_pad, int kp,
             const int* __restrict__ cs, uint16_t* __restrict__ D, int* __restrict__ eu) {
  const int lane = threadIdx.x & 31;
  const long long r = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  if (r >= rows_pad) return;
  constexpr int IT = 512 / 64;                 // n <= 512: 64 complex columns per iteration
  T v[IT][4];
  int E = kNone;
#pragma unroll
  for (int i = 0; i < IT; ++i) {
    if (i * 128 >= kp) break;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int c = i * 64 + 2 * lane + q;
      cplx<T> x = cmake<cplx<T>>(0, 0);
      if (r < rows && c < n) x = X[r * ldx + c];
      v[i][2 * q] = x.x;
      v[i][2 * q + 1] = x.y;
      E = max(E, scaled_exponent<T>(x, cs && c < n ? cs[c] : 0));
    }
  }
  E = __reduce_max_sync(0xffffffffu, E);
  if (E == kNone) E = 0;
  if (lane == 0) eu[r] = E == kBad ? kBad : E - 6;
#pragma unroll
  for (int i = 0; i < IT; ++i) {
    if (i * 128 >= kp) break;
    const int k = i * 128 + 4 * lane;
    if (k >= kp) continue;
    unsigned long long d[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int c = i * 64 + 2 * lane + q / 2;
      d[q] = digits(E == kBad ? 0 : to_fixed(v[i][q], E - (cs && c < n ? cs[c] : 0)));
    }
#pragma unroll
    for (int s = 0; s < S; ++s)
      *reinterpret_cast<uint2*>(&D[((size_t)s * rows_pad + r) * kp + k]) =
          make_uint2(pack2(d[0], d[1], s), pack2(d[2], d[3], s));
  }
}

// Q (n x n, rows scaled by 2^-cs) -> the real right factor of the rotation: row 2j + part of
// output column j's part, over the reals k of a block row; one warp per output row
__global__ void __launch_bounds__(256)
k_split_q(const double2* __restrict__ Q, int n, int rows_pad, int kp, const int* __restrict__ cs,
          uint16_t* __restrict__ D, int* __restrict__ eu) {
  const int lane = threadIdx.x & 31;
  const int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (r >= rows_pad) return;
  const int j = r >> 1, part = r & 1;
  auto at = [&](int i) {   // (factor of x_i.re, factor of x_i.im) in output part ``part``
    if (j >= n || i >= n) return make_double2(0, 0);
    const double2 q = Q[(size_t)i * n + j];
    return part ? make_double2(q.y, q.x) : make_double2(q.x, -q.y);
  };
  int E = kNone;
  for (int i = lane; i < n; i += 32) E = max(E, scaled_exponent<double>(at(i), cs ? -cs[i] : 0));
  E = __reduce_max_sync(0xffffffffu, E);
  if (E == kNone) E = 0;
  if (lane == 0) eu[r] = E == kBad ? kBad : E - 6;
  for (int i = lane; 2 * i < kp; i += 32) {
    const double2 q = at(i);
    const int Ei = cs && i < n && E != kBad ? E + cs[i] : E;
    const unsigned long long a = digits(E == kBad ? 0 : to_fixed(q.x, Ei)),
                             b = digits(E == kBad ? 0 : to_fixed(q.y, Ei));
#pragma unroll
    for (int s = 0; s < S; ++s)
      *reinterpret_cast<unsigned*>(&D[((size_t)s * rows_pad + r) * kp + 2 * i]) = pack2(a, b, s);
  }
}

// exponents that bring the columns to a common size: 2^cs[i] ~ max_j sqrt(S_jj) / sqrt(S_ii), over
// the whole exponent range (a column that fell behind the common size would keep fewer digits)
__global__ void k_col_scale(const double2* __restrict__ diag, int n, int* __restrict__ cs) {
  __shared__ int big;
  if (threadIdx.x == 0) big = kNone;
  __syncthreads();
  auto half_exp = [&](int i) {   // exponent of the norm; a column that is zero or not finite: none
    const double d = diag[i].x;
    return d > 0.0 && isfinite(d) ? ilogb(d) >> 1 : kNone;
  };
  for (int i = threadIdx.x; i < n; i += blockDim.x) atomicMax(&big, half_exp(i));
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const int e = half_exp(i);
    cs[i] = e == kNone ? 0 : big - e;
  }
}

// largest magnitude key of every real column over all rows (WEIGHT: of |x| sqrt(w) rounded up
// by a factor of two)
template <typename T, bool WEIGHT>
__global__ void __launch_bounds__(256)
k_col_max(const cplx<T>* __restrict__ X, int ldx, int n, long long rows,
          const double* __restrict__ md, unsigned* __restrict__ key) {
  const int c = blockIdx.y * 32 + (threadIdx.x & 31);
  const long long step = (long long)gridDim.x * 8;
  unsigned kx = 0, ky = 0;
  if (c < n)
    for (long long r = blockIdx.x * 8LL + (threadIdx.x >> 5); r < rows; r += step) {
      cplx<T> x = X[r * ldx + c];
      if (WEIGHT) {
        const T w = 2 * (T)sqrtf((float)md[r >> 1]);
        x.x *= w;
        x.y *= w;
      }
      kx = max(kx, mag_key(x.x));
      ky = max(ky, mag_key(x.y));
    }
  __shared__ unsigned sk[2][8][32];
  sk[0][threadIdx.x >> 5][threadIdx.x & 31] = kx;
  sk[1][threadIdx.x >> 5][threadIdx.x & 31] = ky;
  __syncthreads();
  if (threadIdx.x < 64) {
    const int p = threadIdx.x >> 5, l = threadIdx.x & 31;
    unsigned k = 0;
    for (int w = 0; w < 8; ++w) k = max(k, sk[p][w][l]);
    const int cc = blockIdx.y * 32 + l;
    if (cc < n && k) atomicMax(&key[2 * cc + p], k);
  }
}

// columns of a block over the rows [r0, r0 + rows_pad) -> digits [S][cols_pad][rows_pad] (rows
// contiguous), rows >= rows as zeros; blocks of 64 rows x 32 complex columns are transposed
// through shared memory.  WEIGHT: x sqrt(w), an FP64 product, so that one set of digits serves
// both factors of X^H diag(w) X; and diag[.][c] += the column's |x|^2 w in FP64: a digit's product
// with itself does not average out, so the orders left out of the products (d_4^2 first) would add
// up to rows 2^-62 of the largest entry squared on the diagonal.  kDiagParts partial sums per column:
// one would be the sum of 23,000 atomics at 746,000 rows and off by their roundings.
constexpr int kDiagParts = 64;
template <typename T, bool WEIGHT>
__global__ void __launch_bounds__(256)
k_split_cols(const cplx<T>* __restrict__ X, int ldx, int n, long long r0, long long rows,
             int rows_pad, int cols_pad, const double* __restrict__ md,
             const unsigned* __restrict__ key, uint16_t* __restrict__ D, int* __restrict__ eu,
             double* __restrict__ diag) {
  using V = typename std::conditional<WEIGHT, double, T>::type;
  __shared__ V xs[64][65];                      // [real column][row]
  __shared__ double ws[64], sqs[8][32];
  const int rb = blockIdx.x * 64, cb = blockIdx.y * 32;
  if (WEIGHT) {
    if (threadIdx.x < 64)
      ws[threadIdx.x] = rb + threadIdx.x < rows ? sqrt(md[(r0 + rb + threadIdx.x) >> 1]) : 0.0;
    __syncthreads();
  }
  double sq = 0.0;
  for (int i = threadIdx.x; i < 64 * 32; i += 256) {
    const int c = i & 31, rr = i >> 5;
    const long long r = rb + rr;
    V a = 0, b = 0;
    if (r < rows && cb + c < n) {
      const cplx<T> x = X[(r0 + r) * ldx + cb + c];
      const double w = WEIGHT ? ws[rr] : 1.0;
      a = WEIGHT ? (V)((double)x.x * w) : (V)x.x;
      b = WEIGHT ? (V)((double)x.y * w) : (V)x.y;
    }
    if (WEIGHT) sq = fma((double)a, (double)a, fma((double)b, (double)b, sq));
    xs[2 * c][rr] = a;
    xs[2 * c + 1][rr] = b;
  }
  if (WEIGHT) sqs[threadIdx.x >> 5][threadIdx.x & 31] = sq;
  __syncthreads();
  if (WEIGHT && threadIdx.x < 32 && cb + threadIdx.x < n) {
    for (int w = 1; w < 8; ++w) sq += sqs[w][threadIdx.x];
    atomicAdd(&diag[(size_t)(blockIdx.x % kDiagParts) * n + cb + threadIdx.x], sq);
  }
  const int c = threadIdx.x >> 2, q = threadIdx.x & 3;   // real column, group of 16 rows
  const int col = 2 * cb + c;
  const int E = col < 2 * n ? key_exponent<T>(key[col]) : 0;
  if (q == 0 && blockIdx.x == 0) eu[col] = E == kBad ? kBad : E - 6;
  unsigned long long d[16];
#pragma unroll
  for (int i = 0; i < 16; ++i)
    d[i] = digits(E == kBad ? 0 : to_fixed(xs[c][q * 16 + i], E));
#pragma unroll
  for (int s = 0; s < S; ++s) {
    uint4* o = reinterpret_cast<uint4*>(&D[((size_t)s * cols_pad + col) * rows_pad + rb + q * 16]);
    o[0] = make_uint4(pack2(d[0], d[1], s), pack2(d[2], d[3], s), pack2(d[4], d[5], s),
                      pack2(d[6], d[7], s));
    o[1] = make_uint4(pack2(d[8], d[9], s), pack2(d[10], d[11], s), pack2(d[12], d[13], s),
                      pack2(d[14], d[15], s));
  }
}

// S_ii = sum of the parts of diag (NaN where it is not finite)
__global__ void k_set_diag(const double* __restrict__ diag, int n, double2* __restrict__ Sm) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    double d = 0.0;
    for (int p = 0; p < kDiagParts; ++p) d += diag[(size_t)p * n + i];
    Sm[(size_t)i * n + i] = make_double2(isfinite(d) ? d : NAN, 0.0);
  }
}

// Columns of a chunk's rows -> digits [S][cols_pad][kp] (rows contiguous; the chunk's at b *
// kNlRows, zeros up to a multiple of 128) and exponents [b][cols_pad], the maximum taken over
// the chunk.  X: row j, column s nvec + v is X[(node_j 2 + s) ldx + v]; PTAB: rows of the atom's P
// table.  The second pass over the rows finds them in L2.
template <bool PTAB>
__global__ void __launch_bounds__(256)
k_split_nodes(const double2* __restrict__ src, int ldx, int nvec, const int4* __restrict__ chunks,
              const long long* __restrict__ nodes, const int* __restrict__ atom_npj,
              const int* __restrict__ atom_pv_off, long long M, int cols_pad, int kp,
              uint16_t* __restrict__ D, int* __restrict__ eu) {
  __shared__ double xs[64][65];
  __shared__ unsigned sk[2][8][32];
  __shared__ int se[64];
  const int b = blockIdx.x, cb = blockIdx.y * 32, l = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int4 ch = chunks[b];
  const int npj = atom_npj[ch.x], c = cb + l;
  const bool ok = c < (PTAB ? npj : 2 * nvec);
  const int sp = !PTAB && c >= nvec;
  const double2* base = PTAB ? src + atom_pv_off[ch.x] + (size_t)ch.y * npj + c
                             : src + (size_t)sp * ldx + (c - sp * nvec);
  const long long* nd = nodes + ch.w + ch.y;
  auto at = [&](int j) {
    if (!ok || j >= ch.z) return make_double2(0, 0);
    if (PTAB) return base[(size_t)j * npj];
    const long long node = nd[j];
    return GBC_IN_RANGE(GBC_SITE_NL_NODE, node, M) ? base[node * 2 * ldx] : make_double2(0, 0);
  };
  unsigned kx = 0, ky = 0;
#pragma unroll 4
  for (int j = w; j < ch.z; j += 8) {
    const double2 x = at(j);
    kx = max(kx, mag_key(x.x));
    ky = max(ky, mag_key(x.y));
  }
  sk[0][w][l] = kx;
  sk[1][w][l] = ky;
  __syncthreads();
  if (threadIdx.x < 64) {   // real column 2 l' + part
    unsigned k = 0;
    for (int i = 0; i < 8; ++i) k = max(k, sk[threadIdx.x & 1][i][threadIdx.x >> 1]);
    const int E = key_exponent<double>(k);
    se[threadIdx.x] = E;
    eu[(size_t)b * cols_pad + 2 * cb + threadIdx.x] = E == kBad ? kBad : E - 6;
  }
  const int cc = threadIdx.x >> 2, q = threadIdx.x & 3;   // real column, group of 16 rows
  for (int rb = 0; rb < ch.z; rb += 128) {
#pragma unroll 1
    for (int h = 0; h < 128; h += 64) {
      __syncthreads();
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const double2 x = at(rb + h + w + 8 * i);
        xs[2 * l][w + 8 * i] = x.x;
        xs[2 * l + 1][w + 8 * i] = x.y;
      }
      __syncthreads();
      const int E = se[cc];
      unsigned long long d[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) d[i] = digits(E == kBad ? 0 : to_fixed(xs[cc][q * 16 + i], E));
#pragma unroll
      for (int s = 0; s < S; ++s) {
        uint4* o = reinterpret_cast<uint4*>(
            &D[((size_t)s * cols_pad + 2 * cb + cc) * kp + (size_t)b * kNlRows + rb + h + q * 16]);
        o[0] = make_uint4(pack2(d[0], d[1], s), pack2(d[2], d[3], s), pack2(d[4], d[5], s),
                          pack2(d[6], d[7], s));
        o[1] = make_uint4(pack2(d[8], d[9], s), pack2(d[10], d[11], s), pack2(d[12], d[13], s),
                          pack2(d[14], d[15], s));
      }
    }
  }
}

// one warp per row of up to 32 complex values -> digits [S][rows][64] and exponents.  COEF: the
// right factor of the expansion, row (chunk, real column (s, v, part)) of its atom's C'; else
// rows of the chunks' P tables (zeros up to a multiple of 128 rows of a chunk)
template <bool COEF>
__global__ void __launch_bounds__(256)
k_split_proj(const double2* __restrict__ src, int nvec, int rows, int cols, const int4* __restrict__ chunks,
             const int* __restrict__ atom_npj, const int* __restrict__ atom_off,
             uint16_t* __restrict__ D, int* __restrict__ eu) {
  const int lane = threadIdx.x & 31;
  const int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (r >= rows) return;
  double2 x = make_double2(0, 0);
  if (COEF) {
    const int atom = chunks[r / cols].x, rc = r % cols;   // cols: padded real columns
    const int yc = rc >> 1, sp = yc >= nvec, v = yc - sp * nvec;
    if (lane < atom_npj[atom] && rc < 4 * nvec) {
      x = src[(size_t)(atom_off[atom] + 2 * lane + sp) * nvec + v];
      x = (rc & 1) ? make_double2(x.y, x.x) : make_double2(x.x, -x.y);
    }
  } else {
    const int4 ch = chunks[r / kNlRows];
    const int i = r % kNlRows, npj = atom_npj[ch.x];
    if (i >= (ch.z + 127) / 128 * 128) return;
    if (i < ch.z && lane < npj) x = src[atom_off[ch.x] + (size_t)(ch.y + i) * npj + lane];
  }
  const unsigned key = __reduce_max_sync(0xffffffffu, max(mag_key(x.x), mag_key(x.y)));
  const int E = key_exponent<double>(key);
  if (lane == 0) eu[r] = E == kBad ? kBad : E - 6;
  const unsigned long long a = digits(E == kBad ? 0 : to_fixed(x.x, E)),
                           b = digits(E == kBad ? 0 : to_fixed(x.y, E));
#pragma unroll
  for (int s = 0; s < S; ++s)
    *reinterpret_cast<unsigned*>(&D[((size_t)s * rows + r) * 64 + 2 * lane]) = pack2(a, b, s);
}

inline int up(int x, int m) { return (x + m - 1) / m * m; }

template <int MODE>
cudaError_t run_split_gemm(const uint16_t* A, const uint16_t* B, int kpad, const SplitArgs& a,
                           cudaStream_t s) {
  CUtensorMap ta, tb;
  if (!tc_make_map_bf16(&ta, A, (long long)S * a.rows_a, kpad, kTM) ||
      !tc_make_map_bf16(&tb, B, (long long)S * a.rows_b, kpad, kTN))
    return cudaErrorInvalidValue;
  auto k = k_split_gemm<MODE>;
  const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSplitSmem);
  if (e != cudaSuccess) return e;
  k<<<(unsigned)std::min(a.nwork, gbc_sm_count()), kSplitThreads, kSplitSmem, s>>>(ta, tb, a);
  return cudaGetLastError();
}

// digit buffer of a chunk of rows: 884,736 x 256 CholGS 72 / 66 ms at 80 / 256 MB (fewer, longer
// launches; that the digits stay in L2 at 80 MB does not make up for it)
constexpr size_t kChunkBytes = size_t(512) << 20;
constexpr size_t kNlBytes = size_t(256) << 20;   // the same of a batch of support chunks
static_assert(GBC_MAX_NPJ <= 32, "a row of projectors is one 64-wide K chunk");

}  // namespace

// one warp waits on an mbarrier that nothing arrives at and gives up as k_split_gemm does
__global__ void k_split_wait_selftest(uint32_t max_iter, int* err) {
  __shared__ uint64_t bar;
  if (threadIdx.x == 0) {
    tc::mbar_init(tc::smem_u32(&bar), 1);
    tc::fence_mbar_init();
  }
  __syncwarp();
  if (!tc::mbar_wait_bounded(tc::smem_u32(&bar), 0, max_iter) && threadIdx.x == 0) atomicExch(err, 1);
}

extern "C" gbc_status gbc_split_wait_selftest(gbc_ctx* c, int max_iter, void* stream) {
  if (!c) return GBC_EINVAL;
  if (max_iter < 1 || max_iter > (1 << 20)) return gbc_fail(c, GBC_EINVAL, "max_iter must be in [1, 2^20]");
  cudaStream_t s = (cudaStream_t)stream;
  GBC_CU(c, cudaSetDevice(c->dev));
  k_split_wait_selftest<<<1, 32, 0, s>>>((uint32_t)max_iter, c->d_flag + 1);
  GBC_CU(c, cudaGetLastError());
  GBC_CU(c, cudaStreamSynchronize(s));
  return GBC_OK;
}

// X <- X Q in place, chunk of rows by chunk.  diag: the diagonal of X's Gram matrix (the columns'
// sizes squared), or null for columns of one size
template <typename T>
gbc_status launch_rotate_split(gbc_ctx* c, cplx<T>* X, const double2* Q, long long M, int n, int ldx,
                               const double2* diag, cudaStream_t s) {
  constexpr int MODE = sizeof(T) == 4 ? ROT32 : ROT64;
  const long long rows = 2 * M;
  const int kp = up(2 * n, kKC), nb = up(2 * n, kTN);
  const long long per = std::max<long long>(kTM, (long long)(kChunkBytes / (2 * S * (size_t)kp)) / kTM * kTM);
  const int rc = (int)std::min<long long>(per, (rows + kTM - 1) / kTM * kTM);
  const size_t ab = (size_t)2 * S * rc * kp, bb = (size_t)2 * S * nb * kp;
  GBC_TRY(gbc_ensure_work(c, 13, ab + bb + sizeof(int) * ((size_t)rc + nb + n) + 1024));
  uint16_t* A = (uint16_t*)c->work[13];
  uint16_t* B = (uint16_t*)((char*)A + ab);
  int* ea = (int*)((char*)B + bb);
  int* eb = ea + rc;
  int* cs = diag ? eb + nb : nullptr;
  if (cs) k_col_scale<<<1, 256, 0, s>>>(diag, n, cs);
  k_split_q<<<(nb + 7) / 8, 256, 0, s>>>(Q, n, nb, kp, cs, B, eb);
  GBC_CU(c, cudaGetLastError());
  for (long long r0 = 0; r0 < rows; r0 += rc) {
    const long long nr = std::min<long long>(rc, rows - r0);
    const int rp = up((int)nr, kTM);
    k_split_rows<T><<<(rp + 7) / 8, 256, 0, s>>>(X + r0 * ldx, ldx, n, nr, rp, kp, cs, A, ea);
    GBC_CU(c, cudaGetLastError());
    const int ntn = nb / kTN, tiles = rp / kTM * ntn;
    SplitArgs a{rp, nb, kp / kKC, kp / kKC, ntn, tiles, tiles, ea, eb, nr, n, ldx, X + r0 * ldx,
                c->d_flag + 1};
    GBC_CU(c, run_split_gemm<MODE>(A, B, kp, a, s));
  }
  return GBC_OK;
}
template gbc_status launch_rotate_split<float>(gbc_ctx*, float2*, const double2*, long long, int, int,
                                               const double2*, cudaStream_t);
template gbc_status launch_rotate_split<double>(gbc_ctx*, double2*, const double2*, long long, int, int,
                                                const double2*, cudaStream_t);

// Sm (upper triangle) = X^H diag(md) X (Y null), or X^H Y (md null)
template <typename TX, typename TY>
gbc_status launch_gram_split(gbc_ctx* c, const cplx<TX>* X, int ldx, const cplx<TY>* Y, int ldy,
                             const double* md, long long M, int n, double2* Sm, cudaStream_t s) {
  const long long rows = 2 * M;
  const int ma = up(2 * n, kTM), nb = ma;    // both padded to a row tile
  const size_t rowb = (size_t)2 * S * (Y ? ma + nb : ma);
  const int win = kFlush * kKC;
  const long long per = std::max<long long>(win, (long long)(kChunkBytes / rowb) / win * win);
  const int rc = (int)std::min<long long>(per, (rows + win - 1) / win * win);
  const size_t ab = (size_t)2 * S * ma * rc, bb = Y ? (size_t)2 * S * nb * rc : 0;
  GBC_TRY(gbc_ensure_work(c, 13, ab + bb + sizeof(int) * 4 * (size_t)ma + sizeof(double) * kDiagParts * n + 1024));
  uint16_t* A = (uint16_t*)c->work[13];
  uint16_t* B = Y ? (uint16_t*)((char*)A + ab) : A;   // one set of digits for both factors
  int* ea = (int*)((char*)A + ab + bb);
  int* eb = Y ? ea + ma : ea;
  unsigned* ka = (unsigned*)(ea + 2 * (size_t)ma);
  unsigned* kb = ka + ma;
  double* diag = (double*)(kb + ma);
  GBC_CU(c, cudaMemsetAsync(Sm, 0, sizeof(double2) * (size_t)n * n, s));
  GBC_CU(c, cudaMemsetAsync(ka, 0, sizeof(unsigned) * 2 * (size_t)ma + sizeof(double) * kDiagParts * n, s));
  const unsigned ncb = (unsigned)((n + 31) / 32);
  const dim3 gm((unsigned)std::max<long long>(1, std::min<long long>((rows + 63) / 64, 16LL * gbc_sm_count() / ncb + 1)), ncb);
  if (md) k_col_max<TX, true><<<gm, 256, 0, s>>>(X, ldx, n, rows, md, ka);
  else k_col_max<TX, false><<<gm, 256, 0, s>>>(X, ldx, n, rows, md, ka);
  if (Y) k_col_max<TY, false><<<gm, 256, 0, s>>>(Y, ldy, n, rows, nullptr, kb);
  GBC_CU(c, cudaGetLastError());
  int tiles = 0;
  const int ntn = nb / kTN;
  for (int I = 0; I < ma / kTM; ++I) tiles += ntn - I * (kTM / kTN);
  for (long long r0 = 0; r0 < rows; r0 += rc) {
    const long long nr = std::min<long long>(rc, rows - r0);
    const int rp = up((int)nr, win);
    const dim3 gs((unsigned)(rp / 64), (unsigned)(ma / 64));
    if (md) k_split_cols<TX, true><<<gs, 256, 0, s>>>(X, ldx, n, r0, nr, rp, ma, md, ka, A, ea, diag);
    else k_split_cols<TX, false><<<gs, 256, 0, s>>>(X, ldx, n, r0, nr, rp, ma, md, ka, A, ea, nullptr);
    if (Y) k_split_cols<TY, false><<<gs, 256, 0, s>>>(Y, ldy, n, r0, nr, rp, nb, nullptr, kb, B, eb, nullptr);
    GBC_CU(c, cudaGetLastError());
    // K split so that the CTAs fill the SMs about once, in whole read-out windows
    const int nwin = rp / win;
    const int split = std::max(1, std::min(nwin, gbc_sm_count() / std::max(1, tiles)));
    const int kper = (nwin + split - 1) / split * kFlush;
    const int parts = (rp / kKC + kper - 1) / kper;
    SplitArgs a{ma, nb, rp / kKC, kper, ntn, tiles, tiles * parts, ea, eb, nr, n, 0, Sm, c->d_flag + 1};
    GBC_CU(c, (run_split_gemm<sizeof(TX) == 4 ? GRAM32 : GRAM64>(A, B, rp, a, s)));
  }
  if (md) k_set_diag<<<1, 256, 0, s>>>(diag, n, Sm);
  GBC_CU(c, cudaGetLastError());
  return GBC_OK;
}
template gbc_status launch_gram_split<float, float>(gbc_ctx*, const float2*, int, const float2*, int,
                                                    const double*, long long, int, double2*, cudaStream_t);
template gbc_status launch_gram_split<float, double>(gbc_ctx*, const float2*, int, const double2*, int,
                                                     const double*, long long, int, double2*, cudaStream_t);
template gbc_status launch_gram_split<double, double>(gbc_ctx*, const double2*, int, const double2*, int,
                                                      const double*, long long, int, double2*, cudaStream_t);

// FP64 projector contractions as split products, in batches of support chunks (at most kNlRows
// nodes of one atom each).  Projection: C1 += P^H X over the chunk's nodes, exponents per chunk
// and column; expansion: Y += P C2 over the atom's projectors, exponents per node and per column
// of C2.  C1 is zero on entry; both add with FP64 atomics, as the direct kernels do.  The digits
// live in work slot 14: nl_split_bytes, which does not shrink with nvec as long as it is used.
// Batches keep the workspace bounded; within one the chunks are independent tiles.  Measured per
// launch at 58 chunks x 64 vectors x 18 projectors: splitting X 0.17 ms and P 0.10 ms (latency of a
// CTA's walk over its chunk), projection products 0.086 ms (tensor pipe 43%); the direct kernels
// run both contractions at the FP64 rate.  Error against 80-bit and wider sums, relative to the
// result: 1.58e-15 (direct 1.63e-15) at 6,300-node supports and 33 vectors, 2.07e-15 (2.06e-15) at
// 17,000 nodes.  One order less (as in the Gram products) measured up to 1.17 times the direct
// kernels' error.
static size_t nl_split_chunk(int nvec, bool project) {
  const size_t cols = up(4 * nvec, project ? kTM : kTN);
  return project ? (2 * S * (size_t)kNlRows + sizeof(int)) * (cols + 64)
                 : (2 * S * 64 + sizeof(int)) * (kNlRows + cols);
}
static int nl_split_batch(const gbc_ctx* c, size_t per) {
  return (int)std::min<size_t>(c->proj.nchunks, std::max<size_t>(1, kNlBytes / per));
}
size_t nl_split_bytes(const gbc_ctx* c, int nvec) {
  const size_t per = std::max(nl_split_chunk(nvec, true), nl_split_chunk(nvec, false));
  return std::min(per * c->proj.nchunks, std::max(per, kNlBytes));
}

cudaError_t nl_split_project(gbc_ctx* c, const double2* X, int nvec, int ldx, double2* C1, cudaStream_t s) {
  const ProjDev& pj = c->proj;
  const int cols = up(4 * nvec, kTM), nb = nl_split_batch(c, nl_split_chunk(nvec, true));
  for (int b0 = 0; b0 < pj.nchunks; b0 += nb) {
    const int n = std::min(nb, pj.nchunks - b0), kp = n * kNlRows;
    uint16_t* A = (uint16_t*)c->work[14];
    uint16_t* B = A + (size_t)S * kp * cols;
    int* ea = (int*)(B + (size_t)S * kp * 64);
    int* eb = ea + (size_t)n * cols;
    const int4* ch = pj.d_chunks + b0;
    // (rows of A past the last 64 columns stay as they are: nothing of theirs is used)
    k_split_nodes<false><<<dim3(n, up(4 * nvec, 64) / 64), 256, 0, s>>>(
        X, ldx, nvec, ch, pj.d_nodes, pj.d_atom_npj, pj.d_atom_pv_off, c->mesh.M, cols, kp, A, ea);
    k_split_nodes<true><<<dim3(n, 1), 256, 0, s>>>(pj.d_P64, 0, 0, ch, pj.d_nodes, pj.d_atom_npj,
                                                      pj.d_atom_pv_off, c->mesh.M, 64, kp, B, eb);
    const int ntm = cols / kTM;
    SplitArgs a{cols, 64, 0, 0, ntm, n * ntm, n * ntm, ea, eb, 0, nvec, 0, C1, c->d_flag + 1, ch, pj.d_nodes,
                pj.d_atom_npj, pj.d_atom_c_off};
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = run_split_gemm<PROJ>(A, B, kp, a, s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t nl_split_expand(gbc_ctx* c, double2* Y, int nvec, int ldx, const double2* C2, cudaStream_t s) {
  const ProjDev& pj = c->proj;
  const int cols = up(4 * nvec, kTN), nb = nl_split_batch(c, nl_split_chunk(nvec, false));
  for (int b0 = 0; b0 < pj.nchunks; b0 += nb) {
    const int n = std::min(nb, pj.nchunks - b0), ra = n * kNlRows, rb = n * cols;
    uint16_t* A = (uint16_t*)c->work[14];
    uint16_t* B = A + (size_t)S * ra * 64;
    int* ea = (int*)(B + (size_t)S * rb * 64);
    int* eb = ea + ra;
    const int4* ch = pj.d_chunks + b0;
    k_split_proj<false><<<ra / 8, 256, 0, s>>>(pj.d_P64, nvec, ra, 0, ch, pj.d_atom_npj,
                                                  pj.d_atom_pv_off, A, ea);
    k_split_proj<true><<<rb / 8, 256, 0, s>>>(C2, nvec, rb, cols, ch, pj.d_atom_npj,
                                                 pj.d_atom_c_off, B, eb);
    const int ntn = cols / kTN, tiles = ra / kTM * ntn;
    SplitArgs a{ra, rb, 1, 1, ntn, tiles, tiles, ea, eb, c->mesh.M, nvec, ldx, Y, c->d_flag + 1, ch, pj.d_nodes,
                pj.d_atom_npj, pj.d_atom_c_off};
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = run_split_gemm<EXPD>(A, B, 64, a, s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}
