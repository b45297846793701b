// Solve phase of VBARMS on the GPU: Alg. 2 (VBARMS_Solve) over the levels,
// the sync-free block triangular solves of the last level, the VBCSR SpMV and
// the vector kernels of FGMRES.
//
// Vectors are FP64.  FP64 factors are applied in the oracle's operation
// order; FP32 factors are promoted to FP64 as they are read.
#include <type_traits>
#include "prec.cuh"
#include "vbsr_ops.cuh"

namespace vb {
namespace {

constexpr int TRI_R = 4;  // scalar rows per lane in the triangular solves (blocks up to 128)

template <typename T>
__device__ __forceinline__ double ld(const T* p) {
  return (double)*p;
}

// bh[q] = r[sp[q]] * b[sp[q]]
__global__ void k_gather_scale(int64_t n, const int32_t* __restrict__ sp, const double* __restrict__ r,
                               const double* __restrict__ b, double* __restrict__ bh) {
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
    const int32_t o = sp[q];
    bh[q] = __dmul_rn(r[o], b[o]);
  }
}

// x[sp[q]] = c[sp[q]] * xh[q]
__global__ void k_scatter_scale(int64_t n, const int32_t* __restrict__ sp, const double* __restrict__ c,
                                const double* __restrict__ xh, double* __restrict__ x) {
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
    const int32_t o = sp[q];
    x[o] = __dmul_rn(c[o], xh[q]);
  }
}

// (double)v by integer operations (normal values; the conversion instruction
// takes the FP64 unit).
__device__ __forceinline__ double tri_widen(float v) {
  const unsigned u = (unsigned)__float_as_int(v);
  if ((u & 0x7f800000u) - 0x00800000u < 0x7f000000u)
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(u << 29));
  return (double)v;
}
__device__ __forceinline__ double tri_widen(double v) { return v; }

// a / b correctly rounded from y = RN(1/b) and z, the rest of 1/b (tri_recip):
// q0 = a y + a z is within one ulp of a / b, a - b q0 is exact, and the
// correction by it rounds to RN(a / b) (Markstein's theorem; exact remainder
// and correctly rounded reciprocal).  Four operations instead of a division's
// 84 (FP32) or 560 (FP64) cycles.  Operands outside the range where no
// intermediate can underflow or overflow (y = 0 marks such a b) are divided.
__device__ __forceinline__ void tri_recip(float b, float& y, float& z) {
  y = 0.f, z = 0.f;
  if (fabsf(b) >= 0x1p-40f && fabsf(b) <= 0x1p40f) {
    y = __frcp_rn(b);
    z = __fmul_rn(__fmaf_rn(-b, y, 1.f), y);
  }
}
__device__ __forceinline__ void tri_recip(double b, double& y, double& z) {
  y = 0.0, z = 0.0;
  if (fabs(b) >= 0x1p-300 && fabs(b) <= 0x1p300) {
    y = __drcp_rn(b);
    z = __dmul_rn(__fma_rn(-b, y, 1.0), y);
  }
}
__device__ __forceinline__ double tri_div(double a, double b, double y, double z) {
  const unsigned e = ((unsigned)__double2hiint(a) >> 20) & 0x7ff;  // |a| in [2^-300, 2^300): integer compares
  if (__double2hiint(y) != 0 && e >= 1023 - 300 && e < 1023 + 300) {
    const double q = __fma_rn(a, y, __dmul_rn(a, z));
    return __fma_rn(__fma_rn(-b, q, a), y, q);
  }
  if (__double2hiint(y) != 0 && __double_as_longlong(a) << 1 == 0) return __dmul_rn(a, y);  // a zero
  return __ddiv_rn(a, b);
}

// The reduction levels' pivot blocks of at most PIV_R rows are solved in a
// thread's registers, every load before the chain of operations; larger ones by
// the warp together.  One thread's walk through the largest block, one global
// load after another, was what each launch waited for (720 000 unknowns, up to
// 20 rows, eight launches in an application: 60 us each, 19 forward and 45
// backward now, where an FP64 division still costs 256 cycles a row).  PivShape
// says where a thread to a block is still the better way.
constexpr int PIV_R = 8;

template <typename TL>
__device__ __forceinline__ void pivot_forward_reg(const TL* __restrict__ lu, const int32_t* __restrict__ pv, int m,
                                                  double* __restrict__ u) {
  double x[PIV_R];
  int p[PIV_R];
  TL l[PIV_R * PIV_R];
#pragma unroll
  for (int k = 0; k < PIV_R; ++k)
    if (k < m) x[k] = u[k], p[k] = pv[k];
#pragma unroll
  for (int i = 1; i < PIV_R; ++i)
#pragma unroll
    for (int k = 0; k < i; ++k)
      if (i < m) l[i * PIV_R + k] = lu[i * m + k];
#pragma unroll
  for (int k = 0; k < PIV_R; ++k)
    if (k < m) {
#pragma unroll
      for (int q = k + 1; q < PIV_R; ++q)
        if (q < m && q == p[k]) {
          const double t = x[k];
          x[k] = x[q];
          x[q] = t;
        }
    }
#pragma unroll
  for (int i = 1; i < PIV_R; ++i)
    if (i < m) {
#pragma unroll
      for (int k = 0; k < i; ++k) x[i] = __dsub_rn(x[i], __dmul_rn(tri_widen(l[i * PIV_R + k]), x[k]));
    }
#pragma unroll
  for (int k = 0; k < PIV_R; ++k)
    if (k < m) u[k] = x[k];
}

// x <- U^{-1} u
template <typename TL>
__device__ __forceinline__ void pivot_backward_reg(const TL* __restrict__ lu, int m, const double* __restrict__ u,
                                                   double* __restrict__ x) {
  double s[PIV_R];
  TL l[PIV_R * PIV_R];
#pragma unroll
  for (int k = 0; k < PIV_R; ++k)
    if (k < m) s[k] = u[k];
#pragma unroll
  for (int i = 0; i < PIV_R; ++i)
#pragma unroll
    for (int k = i; k < PIV_R; ++k)
      if (k < m) l[i * PIV_R + k] = lu[i * m + k];
#pragma unroll
  for (int i = PIV_R - 1; i >= 0; --i)
    if (i < m) {
#pragma unroll
      for (int k = i + 1; k < PIV_R; ++k)
        if (k < m) s[i] = __dsub_rn(s[i], __dmul_rn(tri_widen(l[i * PIV_R + k]), s[k]));
      s[i] = __ddiv_rn(s[i], tri_widen(l[i * PIV_R + i]));
    }
#pragma unroll
  for (int k = 0; k < PIV_R; ++k)
    if (k < m) x[k] = s[k];
}

// u <- L^{-1} P u per pivot block (one thread per block).
template <typename TL>
__device__ void pivot_forward(const TL* lu, const int32_t* pv, int m, double* u) {
  for (int k = 0; k < m; ++k)
    if (pv[k] != k) {
      const double t = u[k];
      u[k] = u[pv[k]];
      u[pv[k]] = t;
    }
  for (int i = 1; i < m; ++i)
    for (int k = 0; k < i; ++k) u[i] = __dsub_rn(u[i], __dmul_rn(ld(lu + i * m + k), u[k]));
}

template <typename TL>
__device__ void pivot_backward(const TL* lu, int m, double* u) {
  for (int i = m - 1; i >= 0; --i) {
    double s = u[i];
    for (int k = i + 1; k < m; ++k) s = __dsub_rn(s, __dmul_rn(ld(lu + i * m + k), u[k]));
    u[i] = __ddiv_rn(s, ld(lu + i * m + i));
  }
}

// Blocks of more than PIV_R and at most 32 rows: the whole warp, lane a with
// row a.  L column by column over all rows at once; in U the products with the
// newest unknown are formed for all rows at once (in S, the staged block, rows
// m | 1 apart), so that only the subtractions of one row stay serial.
template <typename TL>
__device__ __forceinline__ void pivot_forward_warp(const TL* __restrict__ lu, const int32_t* __restrict__ pv, int m,
                                                   double* __restrict__ u, int lane) {
  double y = lane < m ? u[lane] : 0.0;
  const int p = lane < m ? pv[lane] : lane;
#pragma unroll 1
  for (int k = 0; k < m; ++k) {
    const int q = __shfl_sync(0xffffffffu, p, k) & 31;
    const double a = __shfl_sync(0xffffffffu, y, k), b = __shfl_sync(0xffffffffu, y, q);
    if (lane == k) y = b;
    if (lane == q) y = a;
  }
  const TL* row = lu + (lane < m ? lane : 0) * m;
#pragma unroll 1
  for (int k0 = 0; k0 + 1 < m; k0 += 8) {
    TL l[8];
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (k0 + k < m) l[k] = row[k0 + k];
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (k0 + k + 1 < m) {
        const double yk = __shfl_sync(0xffffffffu, y, k0 + k);
        if (lane > k0 + k && lane < m) y = __dsub_rn(y, __dmul_rn(tri_widen(l[k]), yk));
      }
  }
  if (lane < m) u[lane] = y;
}

template <typename TL>
__device__ __forceinline__ void pivot_backward_warp(const TL* __restrict__ lu, int m, const double* __restrict__ u,
                                                    double* __restrict__ x, double* S, int lane) {
  double y = lane < m ? u[lane] : 0.0;
  const int d = m | 1;
#pragma unroll 4
  for (int e = lane; e < m * m; e += 32) {
    const int a = e / m;
    S[a * d + e - a * m] = tri_widen(lu[e]);
  }
  __syncwarp();
  double dg = 1.0, ry, rz;
  if (lane < m) dg = S[lane * (d + 1)];
  tri_recip(dg, ry, rz);
#pragma unroll 1
  for (int i = m - 1; i >= 0; --i) {
    if (lane == i) {
#pragma unroll 4
      for (int k = i + 1; k < m; ++k) y = __dsub_rn(y, S[i * d + k]);
      y = tri_div(y, dg, ry, rz);
    }
    const double v = __shfl_sync(0xffffffffu, y, i);
    if (lane < i) S[lane * d + i] = __dmul_rn(S[lane * d + i], v);
    __syncwarp();
  }
  if (lane < m) x[lane] = y;
  __syncwarp();
}

constexpr int PIV_T = 128;  // threads per block of the two kernels below

// How a launch deals out nD pivot blocks: per of them to a warp (fewer than 8
// while the quarters of the SMs, 608, have no more than two warps each, so that a
// warp meets few large blocks one after the other; an FP64 operation costs the same
// for 8 lanes as for 32), and whether the large ones are solved by a thread each all
// the same.  That is the cheaper way from three blocks a warp on, if most are large
// (nval values: more than PIV_R rows on average): 32 chains share their operations'
// time.  One application, two levels, FP32, blocks of one size on a grid; with a
// thread, with a warp for every block (8 or 32 a warp) and with this rule: 16 rows,
// 30 000 unknowns 0.27, 0.34 and 0.16 ms; 20 rows, 160 000 unknowns (about 3 000
// blocks a launch) 0.29, 0.34 (four a warp) and 0.27, 1.0 million 0.52, 1.22 and
// 0.44.  160 000 nodes of 6 (20 600 blocks, most of them small), 8 and 32 a warp:
// 3.36 and 3.47 ms; 320 000 nodes (41 500 blocks) 4.35 and 4.32.
struct PivShape {
  int per;
  bool threads;
  PivShape(int64_t nD, int64_t nval) {
    per = nD <= 1216 ? 1 : nD <= 2432 ? 2 : nD <= 4864 ? 4 : nD <= 32768 ? 8 : 32;
    threads = nD > 2432 && nval > nD * PIV_R * PIV_R;
    if (threads) per = 32;
  }
};
inline unsigned piv_grid(int64_t nD, const PivShape& p) { return grid_for(nD, PIV_T / 32 * p.per); }

__global__ void __launch_bounds__(PIV_T)
    k_pivot_fwd(int64_t nD, int per, bool threads, const int32_t* __restrict__ sz, const int64_t* __restrict__ roff,
                const int64_t* __restrict__ voff, const double* __restrict__ lu64, const float* __restrict__ lu32,
                const int32_t* __restrict__ ptag, const int32_t* __restrict__ piv, double* __restrict__ u) {
  const int lane = threadIdx.x & 31;
  const int64_t wpg = (int64_t)gridDim.x * (PIV_T / 32);
  for (int64_t y0 = (blockIdx.x * (int64_t)(PIV_T / 32) + (threadIdx.x >> 5)) * per; y0 < nD; y0 += wpg * per) {
    const int64_t y = y0 + lane;
    const bool has = lane < per && y < nD;
    const int m = has ? sz[y] : 0;
    const bool f32 = has && lu32 && !ptag[y];
    if (m > 0 && m <= PIV_R) {
      if (f32)
        pivot_forward_reg<float>(lu32 + voff[y], piv + roff[y], m, u + roff[y]);
      else
        pivot_forward_reg<double>(lu64 + voff[y], piv + roff[y], m, u + roff[y]);
    } else if (m > 32 || (m > PIV_R && threads)) {
      if (f32)
        pivot_forward<float>(lu32 + voff[y], piv + roff[y], m, u + roff[y]);
      else
        pivot_forward<double>(lu64 + voff[y], piv + roff[y], m, u + roff[y]);
    }
    __syncwarp();
    const unsigned f = __ballot_sync(0xffffffffu, f32);
    for (unsigned w = __ballot_sync(0xffffffffu, !threads && m > PIV_R && m <= 32); w; w &= w - 1) {
      const int o = __ffs(w) - 1, mo = __shfl_sync(0xffffffffu, m, o);
      if (f >> o & 1)
        pivot_forward_warp<float>(lu32 + voff[y0 + o], piv + roff[y0 + o], mo, u + roff[y0 + o], lane);
      else
        pivot_forward_warp<double>(lu64 + voff[y0 + o], piv + roff[y0 + o], mo, u + roff[y0 + o], lane);
    }
  }
}

__global__ void __launch_bounds__(PIV_T)
    k_pivot_bwd(int64_t nD, int per, bool threads, const int32_t* __restrict__ sz, const int64_t* __restrict__ roff,
                const int64_t* __restrict__ voff, const double* __restrict__ lu64, const float* __restrict__ lu32,
                const int32_t* __restrict__ ptag, const double* __restrict__ u, double* __restrict__ x) {
  __shared__ double stage[PIV_T / 32][32 * 33];
  const int lane = threadIdx.x & 31;
  double* S = stage[threadIdx.x >> 5];
  const int64_t wpg = (int64_t)gridDim.x * (PIV_T / 32);
  for (int64_t y0 = (blockIdx.x * (int64_t)(PIV_T / 32) + (threadIdx.x >> 5)) * per; y0 < nD; y0 += wpg * per) {
    const int64_t y = y0 + lane;
    const bool has = lane < per && y < nD;
    const int m = has ? sz[y] : 0;
    const bool f32 = has && lu32 && !ptag[y];
    if (m > 0 && m <= PIV_R) {
      if (f32)
        pivot_backward_reg<float>(lu32 + voff[y], m, u + roff[y], x + roff[y]);
      else
        pivot_backward_reg<double>(lu64 + voff[y], m, u + roff[y], x + roff[y]);
    } else if (m > 32 || (m > PIV_R && threads)) {
      for (int a = 0; a < m; ++a) x[roff[y] + a] = u[roff[y] + a];
      if (f32)
        pivot_backward<float>(lu32 + voff[y], m, x + roff[y]);
      else
        pivot_backward<double>(lu64 + voff[y], m, x + roff[y]);
    }
    __syncwarp();
    const unsigned f = __ballot_sync(0xffffffffu, f32);
    for (unsigned w = __ballot_sync(0xffffffffu, !threads && m > PIV_R && m <= 32); w; w &= w - 1) {
      const int o = __ffs(w) - 1, mo = __shfl_sync(0xffffffffu, m, o);
      if (f >> o & 1)
        pivot_backward_warp<float>(lu32 + voff[y0 + o], mo, u + roff[y0 + o], x + roff[y0 + o], S, lane);
      else
        pivot_backward_warp<double>(lu64 + voff[y0 + o], mo, u + roff[y0 + o], x + roff[y0 + o], S, lane);
    }
  }
}

// One row of a block times its unknowns, op(value, unknown) column by column.
// K = 1: a plain loop.  K > 1: the loads of K columns first, then their
// operations; the loop over these is left at the block's end (an FP64 operation
// takes its 64 cycles whether or not a lane wants its result).
// Rows of a warp that meet blocks of different sizes wait for one another's loads
// in the plain loop.  Twenty cycles of FGMRES(1), 360 000 unknowns, 15 neighbours,
// approximate blocks, plain and K = 8: of 2 unknowns 9.4 and 7.6 ms, of 6 (tau 0.8)
// 15.7 and 13.0, of 6 (tau 0.9) 23.8 and 18.7, of 10 20.6 and 17.9.  Blocks that
// are all of one size, 600 000 unknowns on a grid: of 1 4.5 and 4.9, of 4 5.7 and
// 5.9, of 6 7.2 and 7.2, of 7 7.9 and 8.4, of 8 8.6 and 8.4, of 20 16.1 and 16.1: up
// to SPMV_PLAIN they take the plain loop.
constexpr int SPMV_K = 8;
constexpr int SPMV_PLAIN = 7;

template <int K, typename T, typename Op>
__device__ __forceinline__ void row_times(const T* v, const double* x, int nc, Op&& op) {
  if constexpr (K == 1) {
    for (int k = 0; k < nc; ++k) op(v[k], x[k]);
  } else {
    for (int k0 = 0; k0 < nc; k0 += K) {
      T vk[K];
      double xk[K];
#pragma unroll
      for (int k = 0; k < K; ++k)
        if (k0 + k < nc) vk[k] = v[k0 + k], xk[k] = x[k0 + k];
#pragma unroll
      for (int k = 0; k < K; ++k) {
        if (k0 + k >= nc) break;
        op(vk[k], xk[k]);
      }
    }
  }
}

// All blocks are s x s for one s <= SPMV_PLAIN, as far as their number and values
// tell.
template <typename T>
bool spmv_plain(const VBDev<T>& M) {
  for (int64_t s = 1; s <= SPMV_PLAIN; ++s)
    if (M.nval == s * s * M.nnzb) return true;
  return false;
}

// y_row -= M x  for every scalar row of a VBCSR M (one thread per scalar row,
// blocks in order, then the entries of the row).
template <typename T, int K>
__global__ void k_bsr_sub(VBView<T> M, const int64_t* __restrict__ rowblk, int64_t nrows,
                          const double* __restrict__ x, double* __restrict__ y) {
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nrows; q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t I = rowblk[q];
    const int a = (int)(q - M.roff[I]);
    if (sizeof(T) == sizeof(float)) {
      // FP32 factor blocks: products summed in FP32, the result in FP64
      float acc = 0.f;
      for (int64_t b = M.bptr[I]; b < M.bptr[I + 1]; ++b) {
        const int32_t J = M.bcol[b];
        const int nc = M.csz[J];
        row_times<K>(M.val + M.voff[b] + (int64_t)a * nc, x + M.coff[J], nc,
                     [&](T v, double xk) { acc = __fmaf_rn((float)v, (float)xk, acc); });
      }
      y[q] = y[q] - (double)acc;
      continue;
    }
    double s = y[q];
    for (int64_t b = M.bptr[I]; b < M.bptr[I + 1]; ++b) {
      const int32_t J = M.bcol[b];
      const int nc = M.csz[J];
      row_times<K>(M.val + M.voff[b] + (int64_t)a * nc, x + M.coff[J], nc,
                   [&](T v, double xk) { s = __dsub_rn(s, __dmul_rn((double)v, xk)); });
    }
    y[q] = s;
  }
}

// y = A x (FP64), one thread per scalar row.
template <int K>
__global__ void k_spmv(VBView<double> A, const int64_t* __restrict__ rowblk, int64_t nrows,
                       const double* __restrict__ x, double* __restrict__ y) {
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nrows; q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t I = rowblk[q];
    const int a = (int)(q - A.roff[I]);
    double s = 0.0;
    for (int64_t b = A.bptr[I]; b < A.bptr[I + 1]; ++b) {
      const int32_t J = A.bcol[b];
      const int nc = A.csz[J];
      row_times<K>(A.val + A.voff[b] + (int64_t)a * nc, x + A.coff[J], nc,
                   [&](double v, double xk) { s = __dadd_rn(s, __dmul_rn(v, xk)); });
    }
    y[q] = s;
  }
}

__global__ void k_rowblk(int64_t nbr, const int64_t* __restrict__ roff, int64_t* __restrict__ rowblk) {
  const int lane = threadIdx.x & 31;
  const int64_t wpb = blockDim.x >> 5;
  for (int64_t I = blockIdx.x * wpb + (threadIdx.x >> 5); I < nbr; I += (int64_t)gridDim.x * wpb)
    for (int64_t q = roff[I] + lane; q < roff[I + 1]; q += 32) rowblk[q] = I;
}

// ---------------------------------------------------------------------------
// The last level's triangular sweeps.
//
// Publication.  A row's unknowns are their own flags: the sweep's records
// start as kTriEmpty in every word, a row stores its finished values there
// with relaxed stores, and a dependant polls exactly the values that it needs
// until none is empty.  No other data hangs on them, so neither side takes a
// fence, and a link of the dependency chain costs one store and one load
// through L2 (0.53 us measured from warp to warp) instead of store, fence,
// flag, poll, fence and load.  The empty word is a NaN that no operation
// produces; a value that carries those bits all the same (an input's payload)
// is stored as the canonical NaN.
//
// Records are of type R.  The FP32 sweeps publish each unknown rounded to
// FP32, the form its dependants use (a conversion from FP64 costs a dependant
// 100 cycles a value on this part), beside the FP64 value (dbl), which block
// rows of more than TRI_MR scalars read.  With R = double the record serves
// both; that form needs less memory and is the one of the fixed-scratch solve.
// A record starts on a 16-byte boundary: with w = 16 / sizeof(R), row k's at
// coff[k] + (w - 1) k rounded down to a multiple of w.
template <typename R>
__device__ __forceinline__ int64_t tri_rec(int64_t off, int64_t k) {
  constexpr int64_t w = 16 / sizeof(R);
  return (off + (w - 1) * k) & ~(w - 1);
}
template <typename R>
int64_t rec_words(int64_t n_last, int64_t p) {  // a whole number of 16-byte groups
  constexpr int64_t w = 16 / sizeof(R);
  return (n_last + (w - 1) * p + w - 1) & ~(w - 1);
}

__device__ __forceinline__ bool tri_ready(double v) { return __double_as_longlong(v) != -1LL; }
__device__ __forceinline__ bool tri_ready(float v) { return __float_as_int(v) != -1; }
__device__ __forceinline__ void tri_publish(double* p, double v) {
  if (!tri_ready(v)) v = __longlong_as_double(0x7ff8000000000000LL);
  asm volatile("st.relaxed.gpu.global.f64 [%0], %1;" ::"l"(p), "d"(v) : "memory");
}
__device__ __forceinline__ void tri_publish(float* p, float v) {
  if (!tri_ready(v)) v = __int_as_float(0x7fc00000);
  asm volatile("st.relaxed.gpu.global.f32 [%0], %1;" ::"l"(p), "f"(v) : "memory");
}
__device__ __forceinline__ double tri_load(const double* p) {
  double v;
  asm volatile("ld.relaxed.gpu.global.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
  return v;
}

constexpr int TRI_W = 4;         // warps per block
constexpr int TRI_MR = 16;       // block rows up to this size use the lane-per-block path
constexpr int TRI_MP = 32;       // pivot blocks up to this size are solved from shared memory
constexpr int TRI_STAGE = 1024;  // values of a row staged in shared memory per warp
constexpr int TRI_XQ = 8;        // dependency values polled at once

// Blocks per SM.  The chain of rows bounds the sweeps, not the number of rows
// in flight: 8 warps an SM with all their registers measured 82.5 ms on the
// FGMRES of 720 000 unknowns, 12 warps 85.3 and 16 (128 registers) 95.9.
constexpr int TRI_B = 2;

// Shared memory of one warp.
template <typename T>
struct alignas(16) TriSmem {
  // the row's block values: TRI_STAGE of them, all of val when the row has more
  // than TRI_MR scalars; behind TRI_STAGE, per block of the row (modulo 32), its
  // product, or a large pivot block's unknowns and products
  T val[TRI_STAGE + 32 * TRI_MR];
  // the factored pivot block and the reciprocals of its diagonal (tri_recip):
  // up to TRI_MP rows of T, or up to TRI_MP / 2 rows of a tagged FP64 block
  T lu[TRI_MP * (TRI_MP + 1)];
  T ry[TRI_MP], rz[TRI_MP];
  __device__ __forceinline__ T* part() { return val + TRI_STAGE; }
  static_assert(2 * 32 * TRI_R * sizeof(double) <= 32 * TRI_MR * sizeof(T), "part: a large block's unknowns and products");
};

// The wait of one warp between two polls: a short sleep, the abort word and
// the time budget every 16th poll.  it = 0 starts it anew: the budget is that of
// one wait, from arrival to arrival, not of all the waits of a row.  False when
// the wait gave up.
struct TriWait {
  unsigned it = 0;
  unsigned long long t0 = 0;
  __device__ __forceinline__ bool pause(int* abort, unsigned long long limit, int* st) {
    if (it == 0) t0 = global_ns();
    ++it;
    __nanosleep(32);
    if ((it & 15) == 0) {
      if (*((volatile int*)abort) != 0) return false;
      if (global_ns() - t0 > limit) {
        dev_fail(st, DEV_ETIMEOUT);
        atomicExch(abort, 1);
        return false;
      }
    }
    return true;
  }
};

// The first cnt (1 to TRI_XQ) values of a record into x; false while one of
// them is still empty.
template <typename TA>
__device__ __forceinline__ bool tri_take(const double* p, int cnt, TA* x) {
  bool ok = true;
#pragma unroll
  for (int q = 0; q < TRI_XQ; q += 2)
    if (q < cnt) {
      double a, b;
      asm volatile("ld.relaxed.gpu.global.v2.f64 {%0, %1}, [%2];" : "=d"(a), "=d"(b) : "l"(p + q) : "memory");
      ok = ok && tri_ready(a) && (q + 1 >= cnt || tri_ready(b));
      x[q] = (TA)a;
      x[q + 1] = (TA)b;
    }
  return ok;
}
__device__ __forceinline__ bool tri_take(const float* p, int cnt, float* x) {
  bool ok = true;
#pragma unroll
  for (int q = 0; q < TRI_XQ; q += 4)
    if (q < cnt) {
      asm volatile("ld.relaxed.gpu.global.v4.f32 {%0, %1, %2, %3}, [%4];"
                   : "=f"(x[q]), "=f"(x[q + 1]), "=f"(x[q + 2]), "=f"(x[q + 3])
                   : "l"(p + q)
                   : "memory");
#pragma unroll
      for (int u = 0; u < 4; ++u) ok = ok && (q + u >= cnt || tri_ready(x[q + u]));
    }
  return ok;
}

// RN32(RN64(R - s)) for an FP64 R and an FP32 s by FP32 operations: R is held
// as the exact sum h + m + l of three floats; t + e = h - s and f + e2 = t + w
// exactly (Knuth's two-sum), w = e + m.  f is the answer when e2 and all that
// was rounded or left out (2^-24 |w| + |l| + 2^-53 |f|, less than 2^-8 of half
// an ulp of f under the two range conditions) stay within half an ulp, which
// is not asked of a power of two.  Otherwise (one row in some hundred) the
// FP64 unit is used: a subtraction between two conversions, 290 cycles on the
// chain against 100.
struct TriSplit {
  float h, m, l;
  bool ok;
};
__device__ __forceinline__ TriSplit tri_split(double R) {
  TriSplit p;
  p.h = (float)R;
  const double d = R - (double)p.h;
  p.m = (float)d;
  p.l = (float)(d - (double)p.m);
  p.ok = fabsf(p.h) >= 0x1p-40f && fabsf(p.h) <= 0x1p40f;
  return p;
}
__device__ __forceinline__ float tri_sub32(double R, const TriSplit& p, float s, bool wanted) {
  const float t = __fsub_rn(p.h, s);
  const float tb = __fsub_rn(t, p.h);
  const float e = __fadd_rn(__fsub_rn(p.h, __fsub_rn(t, tb)), __fsub_rn(-s, tb));
  const float w = __fadd_rn(e, p.m);
  const float f = __fadd_rn(t, w);
  const float fb = __fsub_rn(f, t);
  const float e2 = __fadd_rn(__fsub_rn(t, __fsub_rn(f, fb)), __fsub_rn(w, fb));
  const unsigned u = (unsigned)__float_as_int(f);
  const float lead = __int_as_float((int)(u & 0x7f800000u));  // 2^ef
  const bool ok = p.ok && (u & 0x7fffffu) != 0 && fabsf(f) >= 0x1p-60f && fabsf(w) <= lead * 0x1p-10f &&
                  fabsf(p.h) <= lead * 0x1p10f && fabsf(e2) <= lead * (0x1p-24f - 0x1p-32f);
  return ok || !wanted ? f : (float)(R - (double)s);
}

// The block row that a warp works on.
template <typename T>
struct TriRow {
  const int32_t* bcol;  // its blocks' columns and value offsets
  const int64_t* voff;
  const int32_t* csz;   // the matrix's column partition
  const int64_t* coff;
  int64_t v0;           // its first value
  int nb, ni;           // blocks, scalar rows
};

// sum_b B_ib x_b of the calling warp's block row (ni <= G rows, G = 8 or 16),
// row a's sum on lane a.  Lane l owns the blocks l, l + 32, ... of the row, in
// units of up to TRI_XQ columns, and polls for its next two units; as soon as
// some lanes' units have arrived, all lanes multiply those (G lanes to a
// unit, one per row), so that when the last dependency arrives only its own
// product is left.  The products are kept per owner lane, each element's
// additions in the order of its blocks and columns, and then summed over the
// owners as a butterfly over lane ^ 16, 8, 4, 2, 1 would.  An FP64 operation
// occupies the unit of a warp's quarter of the SM for 64 cycles whatever the
// number of lanes, so the additions of owners that do not exist (+0.0) are
// left out there; the one effect they have, -0.0 becoming +0.0, is applied.
template <int G, typename T, typename R>
__device__ __forceinline__ bool tri_row(const TriRow<T>& row, const T* sval, const R* rec, T* part, int* abort,
                                        unsigned long long limit, int* st, int lane, T* sum) {
  const int nb = row.nb, ni = row.ni;
  constexpr int NG = 32 / G;
  const int g = lane / G, a = lane % G;
  // the lane's units: the generator's block and column, then unit A and unit B
  int gb = lane - 32, gq = 0, gnk = 0, gvo = 0;
  const R* gx = rec;
  auto next = [&](int& meta, int& vo, const R*& x) {
    if (gq + TRI_XQ < gnk) {
      gq += TRI_XQ;
    } else {
      gb += 32;
      gq = 0;
      gnk = 0;
      if (gb < nb) {
        const int32_t k = row.bcol[gb];
        gnk = row.csz[k];
        gvo = (int)(row.voff[gb] - row.v0);
        gx = rec + tri_rec<R>(row.coff[k], k);
      }
    }
    meta = gnk ? min(TRI_XQ, gnk - gq) | (gb < 32 && gq == 0 ? 16 : 0) | gnk << 8 : 0;
    vo = gvo + gq;
    x = gx + gq;
  };
  // a unit: its columns cnt, the block's columns nk, whether it opens its
  // owner's sum, and its first value's place
  int metaA, voA, metaB, voB;
  bool okA = false, okB = false;
  const R *pA, *pB;
  T xA[TRI_XQ], xB[TRI_XQ];
  next(metaA, voA, pA);
  next(metaB, voB, pB);
  int units = 0;  // of all lanes, still to come
  for (int b = lane; b < nb; b += 32) units += (row.csz[row.bcol[b]] + TRI_XQ - 1) / TRI_XQ;
  units = __reduce_add_sync(0xffffffffu, units);
  TriWait w;
  while (units > 0) {
    if (metaA && !okA) okA = tri_take(pA, metaA & 15, xA);
    if (metaB && !okB) okB = tri_take(pB, metaB & 15, xB);
    const unsigned arrived = __ballot_sync(0xffffffffu, okA);
    if (!arrived) {
      const bool go = w.pause(abort, limit, st);
      if (!__all_sync(0xffffffffu, go)) return false;
      continue;
    }
    w.it = 0;
    for (unsigned left = arrived; left;) {
      unsigned mine = left;  // the group's owner: the g-th lowest lane left
#pragma unroll
      for (int j = 0; j < NG; ++j) {
        if (j < g) mine &= mine - 1;
        left &= left - 1;
      }
      const int o = mine ? __ffs(mine) - 1 : 0;
      const int meta = __shfl_sync(0xffffffffu, metaA, o);
      const int vo = __shfl_sync(0xffffffffu, voA, o);
      const int cnt = mine != 0 && a < ni ? meta & 15 : 0;
      const int nk = meta >> 8;
      T acc = cnt && !(meta & 16) ? part[o * G + a] : (T)0;
      const T* v = sval + vo + a * nk;
      if constexpr (sizeof(T) == sizeof(double)) {
        const int most = __reduce_max_sync(0xffffffffu, cnt);
#pragma unroll
        for (int q = 0; q < TRI_XQ; ++q) {
          if (q >= most) break;
          const T x = __shfl_sync(0xffffffffu, xA[q], o);
          if (q < cnt) acc = fma(v[q], x, acc);
        }
      } else {
#pragma unroll
        for (int q = 0; q < TRI_XQ; ++q) {
          const T x = __shfl_sync(0xffffffffu, xA[q], o);
          if (q < cnt) acc = fma(v[q], x, acc);
        }
      }
      if (cnt) part[o * G + a] = acc;
      __syncwarp();
    }
    units -= __popc(arrived);
    if (units == 0) break;
    if (okA) {
#pragma unroll
      for (int q = 0; q < TRI_XQ; ++q) xA[q] = xB[q];
      metaA = metaB, voA = voB, pA = pB, okA = okB;
      okB = false;
      next(metaB, voB, pB);
    }
  }
  // owners l = g + NG j in lane group g: j ^ (16 / NG) ... j ^ 1 within the
  // lane, then g ^ (NG / 2) ... g ^ 1 by shuffles
  constexpr int J = 32 / NG;
  const int own = min(nb, 32);
  T p[J];
#pragma unroll
  for (int j = 0; j < J; ++j) p[j] = a < ni && g + NG * j < own ? part[(g + NG * j) * G + a] : (T)0;
  if constexpr (sizeof(T) == sizeof(double)) {
    if (own <= 16) {
#pragma unroll
      for (int j = 0; j < J; ++j)
        if (__double_as_longlong(p[j]) == (long long)0x8000000000000000ULL) p[j] = 0.0;
    }
#pragma unroll
    for (int h = J / 2; h >= 1; h >>= 1)
      if (own > h * NG) {
#pragma unroll
        for (int j = 0; j < h; ++j) p[j] = p[j] + p[j + h];
      }
#pragma unroll
    for (int h = NG / 2; h >= 1; h >>= 1)
      if (own > h) p[0] += __shfl_xor_sync(0xffffffffu, p[0], h * G);
  } else {
#pragma unroll
    for (int h = J / 2; h >= 1; h >>= 1)
#pragma unroll
      for (int j = 0; j < h; ++j) p[j] = p[j] + p[j + h];
#pragma unroll
    for (int h = NG / 2; h >= 1; h >>= 1) p[0] += __shfl_xor_sync(0xffffffffu, p[0], h * G);
  }
  *sum = p[0];
  return true;
}

// The row of up to TRI_MR scalars that is not the common one (9 rows or more,
// or values that did not fit on chip): kept out of line, as are the large rows
// and the larger pivot blocks below, so that the common row's code stays
// small (inlined, they made it 1.5 times slower).
template <typename T, typename R>
__device__ __noinline__ bool tri_row16(TriRow<T> row, const T* sval, const R* rec, T* part, int* abort,
                                       unsigned long long limit, int* st, int lane, T* sum) {
  return tri_row<16>(row, sval, rec, part, abort, limit, st, lane, sum);
}

// s[t] -= sum_b B_ib x_b for the rows lane + 32 t of a block row of more than
// TRI_MR scalars: FP64 sums in the order of the blocks and columns.  Every lane
// polls its own block's first unknowns; the blocks are taken in their order,
// each as soon as it has arrived.  xw: the FP64 unknowns, record k at
// coff[k] (dense) or at tri_rec.
template <typename T>
__device__ __noinline__ bool tri_large(TriRow<T> row, const T* sval, const double* xw, bool dense, double* s,
                                       int* abort, unsigned long long limit, int* st, int lane) {
  const int nb = row.nb, ni = row.ni;
  for (int base = 0; base < nb; base += 32) {
    // lane l: block base + l, its first unknown and its values
    int nk = 0, vo = 0;
    const double* xk = nullptr;
    if (base + lane < nb) {
      const int32_t k = row.bcol[base + lane];
      nk = row.csz[k];
      vo = (int)(row.voff[base + lane] - row.v0);
      xk = xw + (dense ? row.coff[k] : tri_rec<double>(row.coff[k], k));
    }
    // every lane polls its own block's first unknowns; the blocks are
    // taken in their order, each as soon as it has arrived
    double x[TRI_XQ];
    bool ok = nk == 0;
    TriWait w;
    const int cnt = min(32, nb - base);
    for (int b = 0; b < cnt;) {
      if (!ok) {
        ok = true;
#pragma unroll
        for (int q = 0; q < TRI_XQ; ++q)
          if (q < nk) {
            x[q] = tri_load(xk + q);
            ok = ok && tri_ready(x[q]);
          }
        for (int q = TRI_XQ; q < nk; ++q) ok = ok && tri_ready(tri_load(xk + q));
      }
      const unsigned arrived = __ballot_sync(0xffffffffu, ok);
      if (!(arrived >> b & 1)) {
        const bool go = w.pause(abort, limit, st);
        if (!__all_sync(0xffffffffu, go)) return false;
        continue;
      }
      w.it = 0;
      __syncwarp();  // the loads below come after the polls that saw the values (a ballot orders no memory)
      for (; b < cnt && (arrived >> b & 1); ++b) {
        const int bk = __shfl_sync(0xffffffffu, nk, b), bv = __shfl_sync(0xffffffffu, vo, b);
        const double* bx = (const double*)__shfl_sync(0xffffffffu, (unsigned long long)xk, b);
        for (int q0 = 0; q0 < bk; q0 += TRI_XQ) {
          T v[TRI_XQ];
          double xq[TRI_XQ];
#pragma unroll
          for (int q = 0; q < TRI_XQ; ++q)
            if (q0 + q < bk) xq[q] = q0 == 0 ? __shfl_sync(0xffffffffu, x[q], b) : tri_load(bx + q0 + q);
#pragma unroll
          for (int t = 0; t < TRI_R; ++t) {
            if (32 * t >= ni) break;
            const int a = lane + 32 * t;
#pragma unroll
            for (int q = 0; q < TRI_XQ; ++q)
              if (a < ni && q0 + q < bk) v[q] = sval[bv + a * bk + q0 + q];
#pragma unroll
            for (int q = 0; q < TRI_XQ; ++q) {
              if (q0 + q >= bk) break;
              if (a < ni) s[t] = fma(-tri_widen(v[q]), xq[q], s[t]);
            }
          }
        }
      }
    }
  }
  return true;
}

// Row stride of a staged pivot block of m rows.
__device__ __forceinline__ int tri_stride(int m, bool f32) {
  if (!f32) return m | 1;
  return m <= 8 ? 8 : m <= 12 ? 12 : m <= 16 ? 16 : m <= 20 ? 20 : 32;
}

// U^{-1} L^{-1} P u of a staged FP32 pivot block of m <= M rows (row stride S,
// a multiple of 4; the block is padded to M rows with those of the identity),
// the operations of the sequential solve in their order: lane a holds u_a and
// gets x_a, src is the lane's interchanged source row.  Every lane solves the
// whole block in registers: its operations form one serial chain (each row of
// U starts with the unknown found last), which no split shortens; the block's
// entries come as broadcast 16-byte loads that do not depend on it.  The
// padding adds -0.0 to the rows of the block, which changes none of them.
// FAST divides as tri_div does; *ok tells whether all dividends were in its
// range.
template <int M, int S, bool FAST>
__device__ __forceinline__ float tri_pivot_f32(const float* lu, const float* ry, const float* rz, int m, int src,
                                               float u, int lane, bool* ok) {
  const float up = __shfl_sync(0xffffffffu, u, src);
  float x[M];
#pragma unroll
  for (int k = 0; k < M; ++k) x[k] = __shfl_sync(0xffffffffu, up, k);
#pragma unroll
  for (int i = 1; i < M; ++i) {
#pragma unroll
    for (int k4 = 0; k4 < i; k4 += 4) {
      const float4 l = *reinterpret_cast<const float4*>(lu + i * S + k4);
      const float lv[4] = {l.x, l.y, l.z, l.w};
#pragma unroll
      for (int k = k4; k < i && k < k4 + 4; ++k) x[i] = __fmaf_rn(-lv[k - k4], x[k], x[i]);
    }
    if (i >= m) x[i] = 0.f;  // also where the block's unknowns are infinite
  }
  float lo = 1.f, hi = 1.f;
#pragma unroll
  for (int i = M - 1; i >= 0; --i) {
#pragma unroll
    for (int k4 = (i + 1) & ~3; k4 < M; k4 += 4) {
      const float4 l = *reinterpret_cast<const float4*>(lu + i * S + k4);
      const float lv[4] = {l.x, l.y, l.z, l.w};
#pragma unroll
      for (int k = k4; k < M && k < k4 + 4; ++k)
        if (k > i) x[i] = __fmaf_rn(-lv[k - k4], x[k], x[i]);
    }
    if (FAST) {
      const float s = fabsf(x[i]), q = __fmaf_rn(x[i], ry[i], __fmul_rn(x[i], rz[i]));
      if (i < m) lo = fminf(lo, s == s ? s : 0.f), hi = fmaxf(hi, s);
      x[i] = __fmaf_rn(__fmaf_rn(-lu[i * S + i], q, x[i]), ry[i], q);
      if (i >= m) x[i] = 0.f;
    } else {
      x[i] = i < m ? __fdiv_rn(x[i], lu[i * S + i]) : 0.f;
    }
  }
  *ok = lo >= 0x1p-40f && hi <= 0x1p40f;
  float r = x[0];
#pragma unroll
  for (int k = 1; k < M; ++k)
    if (lane == k) r = x[k];
  return r;
}

// The same in FP64, lane a with row a: L column by column over all rows at
// once; in U the products with the newest unknown are formed for all rows at
// once, so that only the subtractions of one row stay serial.  (An FP64
// operation takes 64 cycles for one lane as for 32.)
template <int M>
__device__ __forceinline__ double tri_pivot_f64(const double* lu, const double* ry, const double* rz, int m, int S,
                                                int src, double u, int lane) {
  double y = __shfl_sync(0xffffffffu, u, src);
  const double* row = lu + (lane < m ? lane : 0) * S;
  double prod[M];  // k < a: l_ak, k >= a: u_ak, then its product with x_k
#pragma unroll
  for (int k = 0; k < M; ++k) prod[k] = k < m ? row[k] : 0.0;
  const double d = lu[(lane < m ? lane : 0) * (S + 1)], dy = ry[lane < m ? lane : 0], dz = rz[lane < m ? lane : 0];
#pragma unroll
  for (int k = 0; k + 1 < M; ++k)
    if (k + 1 < m) {
      const double yk = __shfl_sync(0xffffffffu, y, k);
      if (lane > k && lane < m) y = __dsub_rn(y, __dmul_rn(prod[k], yk));
    }
#pragma unroll
  for (int i = M - 1; i >= 0; --i)
    if (i < m) {
      if (lane == i) {
#pragma unroll
        for (int k = i + 1; k < M; ++k)
          if (k < m) y = __dsub_rn(y, prod[k]);
        y = tri_div(y, d, dy, dz);
      }
      const double x = __shfl_sync(0xffffffffu, y, i);
      if (lane < i) prod[i] = __dmul_rn(prod[i], x);
    }
  return y;
}

// The FP64 solve for m <= TRI_MP rows, in loops; the products take the place
// of the entries above the diagonal in shared memory.
__device__ __noinline__ double tri_pivot_f64_wide(double* lu, const double* ry, const double* rz, int m, int S,
                                                     int src, double u, int lane) {
  double y = __shfl_sync(0xffffffffu, u, src);
  for (int k = 0; k + 1 < m; ++k) {
    const double yk = __shfl_sync(0xffffffffu, y, k);
    if (lane > k && lane < m) y = __dsub_rn(y, __dmul_rn(lu[lane * S + k], yk));
  }
  for (int i = m - 1; i >= 0; --i) {
    if (lane == i) {
#pragma unroll 4
      for (int k = i + 1; k < m; ++k) y = __dsub_rn(y, lu[i * S + k]);
      y = tri_div(y, lu[i * S + i], ry[i], rz[i]);
    }
    const double x = __shfl_sync(0xffffffffu, y, i);
    if (lane < i) lu[lane * S + i] = __dmul_rn(lu[lane * S + i], x);
    __syncwarp();
  }
  return y;
}

// The FP32 solve for m <= TRI_MP rows; fast: every diagonal entry has its
// reciprocal (tri_recip).
template <int M, int S>
__device__ __forceinline__ float tri_pivot_any(const float* lu, const float* ry, const float* rz, int m, int src,
                                               bool fast, float u, int lane) {
  bool ok;
  if (fast) {
    const float x = tri_pivot_f32<M, S, true>(lu, ry, rz, m, src, u, lane, &ok);
    if (ok) return x;
  }
  return tri_pivot_f32<M, S, false>(lu, ry, rz, m, src, u, lane, &ok);
}
__device__ __noinline__ float tri_pivot_f32_wide(const float* lu, const float* ry, const float* rz, int m, int src,
                                                 bool fast, float u, int lane) {
  return m <= 8    ? tri_pivot_any<8, 8>(lu, ry, rz, m, src, fast, u, lane)
         : m <= 12 ? tri_pivot_any<12, 12>(lu, ry, rz, m, src, fast, u, lane)
         : m <= 16 ? tri_pivot_any<16, 16>(lu, ry, rz, m, src, fast, u, lane)
         : m <= 20 ? tri_pivot_any<20, 20>(lu, ry, rz, m, src, fast, u, lane)
                   : tri_pivot_any<32, 32>(lu, ry, rz, m, src, fast, u, lane);
}

// x <- U^{-1} L^{-1} P x with a pivot block of up to 32 TRI_R rows that is read in
// place; x and pr (32 TRI_R values each) in shared memory, lane a with the rows a,
// a + 32, ...  L column by column over all rows at once; in U a row's products at
// once, the next row's entries loaded meanwhile, and their subtractions one after
// the other, on every lane.  The operations of the sequential solve in their order,
// which one lane did before: an application on 300 block rows of 33 to 40 scalars
// FP64 50.7 and 26.1 ms, of 17 to 32 in FP32 with tagged pivots 35.7 and 20.2.
template <typename TL>
__device__ __noinline__ void tri_pivot_large(const TL* __restrict__ lu, const int32_t* __restrict__ pv, int m,
                                             double* x, double* pr, int lane) {
#pragma unroll 1
  for (int k0 = 0; k0 < m; k0 += 32) {
    const int p = k0 + lane < m ? pv[k0 + lane] : 0;
#pragma unroll 1
    for (int k = k0; k < min(m, k0 + 32); ++k) {
      const int q = __shfl_sync(0xffffffffu, p, k - k0);
      if (lane == 0 && q != k) {
        const double v = x[k];
        x[k] = x[q];
        x[q] = v;
      }
    }
  }
  __syncwarp();
  TL l[TRI_R];  // the next column of L, then the next row of U
  auto fetch = [&](int from, int stride, int at) {
#pragma unroll
    for (int t = 0; t < TRI_R; ++t) {
      const int i = lane + 32 * t;
      if (i < m && i >= from) l[t] = lu[i * stride + at];
    }
  };
  fetch(1, m, 0);
#pragma unroll 1
  for (int k = 0; k + 1 < m; ++k) {
    const double xk = x[k];
    TL c[TRI_R];
#pragma unroll
    for (int t = 0; t < TRI_R; ++t) c[t] = l[t];
    fetch(k + 2, m, k + 1);
#pragma unroll
    for (int t = 0; t < TRI_R; ++t) {
      if (32 * t >= m) break;
      const int i = lane + 32 * t;
      if (i < m && i > k) x[i] = __dsub_rn(x[i], __dmul_rn(tri_widen(c[t]), xk));
    }
    __syncwarp();
  }
  fetch(m - 1, 1, (m - 1) * m);
#pragma unroll 1
  for (int i = m - 1; i >= 0; --i) {
    const double d = tri_widen(lu[i * (m + 1)]);
#pragma unroll
    for (int t = 0; t < TRI_R; ++t) {
      if (32 * t >= m) break;
      const int k = lane + 32 * t;
      if (k < m && k > i) pr[k] = __dmul_rn(tri_widen(l[t]), x[k]);
    }
    if (i > 0) fetch(i, 1, (i - 1) * m);
    __syncwarp();
    double v = x[i];
#pragma unroll 4
    for (int k = i + 1; k < m; ++k) v = __dsub_rn(v, pr[k]);
    v = __ddiv_rn(v, d);
    __syncwarp();
    if (lane == 0) x[i] = v;
    __syncwarp();
  }
}

// Sync-free block triangular sweep over the last-level factors, one warp per
// block row, rows handed out in level order (order[ticket]): every dependency
// of a row sits in an earlier level and so holds an earlier ticket.
//   forward  (BWD = false): y_i <- r_i g_i - sum_{k<i} L_ik y_k
//                           (rhs g, scl r; y to out and the records)
//   backward (BWD = true):  x_i <- D_i^{-1} (y_i - sum_{j>i} U_ij x_j)
//                           (rhs y; x to the records, c_i x_i to out, scl c;
//                           rows flagged in fixed take x_i = fixv_i / c_i)
// rec: the records; dbl: the FP64 unknowns (R = float; forward: out).  Both
// start as 0xff bytes.  Rows of up to TRI_MR scalars: everything static (the
// row's values, the pivot LU, its interchanges and its diagonal's
// reciprocals) is on chip before the first poll; then tri_row.  Larger rows
// (FP64 sums, block by block) use a lane per scalar row.
//
// Bound: the levels of the dependency DAG times the latency of a link.  A
// publication reaches a poller in 0.53 us; a link's own work is then about
// 0.35 us forward and 0.8 us backward in FP32 (products of the last arrival
// 330 cycles, sum over the owners 160, subtraction 100, pivot solve 700), and
// several times that in FP64, whose operations take 64 cycles each.  One
// application's two sweeps, with flags, fences and one-lane pivot solves before and
// now: 3.0 million unknowns FP32 (2 650 levels each way) 33.2 and 9.6 ms; 48 000
// unknowns at tau 0.9 FP32 (5 100 and 6 190 levels) 60.0 and 16.7 ms; 360 000
// unknowns FP64 (1 930 levels) 51 and 14.9 ms; 18 000 FP64 (the whole application)
// 10.2 and 3.2 ms.
template <typename T, bool BWD, typename R>
__global__ void __launch_bounds__(TRI_W * 32, TRI_B)
    k_tri(VBView<T> M, const int64_t* __restrict__ dgoff, const double* __restrict__ lu64,
          const float* __restrict__ lu32, const int32_t* __restrict__ ptag, const int32_t* __restrict__ piv,
          const double* __restrict__ rhs, const double* __restrict__ scl, R* rec, double* dbl, double* out,
          const int32_t* __restrict__ order, unsigned long long* ticket, int* abort, unsigned long long wait_limit,
          int* st, const int32_t* __restrict__ fixed, const double* __restrict__ fixv) {
  extern __shared__ __align__(16) unsigned char tri_sm[];
  const int lane = threadIdx.x & 31;
  TriSmem<T>& sm = reinterpret_cast<TriSmem<T>*>(tri_sm)[threadIdx.x >> 5];
  // the finished unknown a of row i, whose scalars start at r0
  auto publish = [&](int64_t i, int64_t r0, int a, double x, double sc) {
    R* ri = rec + tri_rec<R>(r0, i);
    if constexpr (std::is_same<R, float>::value) tri_publish(ri + a, (float)x);
    if constexpr (std::is_same<R, double>::value) tri_publish(ri + a, x);
    if (std::is_same<R, float>::value) tri_publish(dbl + r0 + a, x);
    if (BWD)
      out[r0 + a] = __dmul_rn(sc, x);
    else if (std::is_same<R, double>::value)
      out[r0 + a] = x;
  };
  for (;;) {
    long long t0 = 0;
    if (lane == 0) t0 = (long long)atomicAdd(ticket, 1ULL);
    t0 = __shfl_sync(0xffffffffu, t0, 0);
    if (t0 >= M.nbr) break;
    const int64_t i = order[t0];
    const int ni = M.rsz[i];
    const int64_t r0 = M.roff[i];
    if (BWD && fixed && fixed[i]) {  // the caller gave this row's unknowns
      for (int a = lane; a < ni; a += 32) publish(i, r0, a, __ddiv_rn(fixv[r0 + a], scl[r0 + a]), scl[r0 + a]);
      continue;
    }
    const int64_t b0 = M.bptr[i], b1 = M.bptr[i + 1];
    const int nb = (int)(b1 - b0);
    // the pivot block: applied in FP32 (f32p) or FP64, from shared memory (sp)
    const bool f32p = BWD && lu32 && !ptag[i];
    const int S = tri_stride(ni, f32p);
    const bool sp = BWD && ni <= (f32p || sizeof(T) == sizeof(double) ? TRI_MP : TRI_MP / 2);
    int src = lane;     // interchanged source row
    bool fast = false;  // every diagonal entry of the FP32 block has its reciprocal
    if (sp) {
      const int64_t lo = dgoff[i];
      if (f32p) {
        for (int e = lane; e < S * S; e += 32) {
          const int a = e / S, c = e - a * S;
          reinterpret_cast<float*>(sm.lu)[e] = a < ni && c < ni ? lu32[lo + a * ni + c] : a == c ? 1.f : 0.f;
        }
      } else {
        for (int e = lane; e < ni * ni; e += 32) {
          const int a = e / ni;
          reinterpret_cast<double*>(sm.lu)[a * S + (e - a * ni)] = lu64[lo + e];
        }
      }
      const int pv = lane < ni ? piv[r0 + lane] : lane;
      for (int k = 0; k < ni; ++k) {
        const int pk = __shfl_sync(0xffffffffu, pv, k);
        const int vk = __shfl_sync(0xffffffffu, src, k), vp = __shfl_sync(0xffffffffu, src, pk & 31);
        if (lane == k) src = vp;
        if (lane == pk) src = vk;
      }
      __syncwarp();
      if (f32p) {
        float y = 1.f, z = 0.f;
        if (lane < ni) tri_recip(reinterpret_cast<float*>(sm.lu)[lane * (S + 1)], y, z);
        reinterpret_cast<float*>(sm.ry)[lane] = y;
        reinterpret_cast<float*>(sm.rz)[lane] = z;
        fast = __all_sync(0xffffffffu, y != 0.f);
      } else if (lane < ni) {
        double y, z;
        tri_recip(reinterpret_cast<double*>(sm.lu)[lane * (S + 1)], y, z);
        reinterpret_cast<double*>(sm.ry)[lane] = y;
        reinterpret_cast<double*>(sm.rz)[lane] = z;
      }
    }
    const int64_t v0 = M.voff[b0];
    const int64_t nv = M.voff[b1] - v0;
    const bool staged = nv <= (ni > TRI_MR ? TRI_STAGE + 32 * TRI_MR : TRI_STAGE);
    if (staged) {
#pragma unroll 4
      for (int64_t e = lane; e < nv; e += 32) sm.val[e] = M.val[v0 + e];
    }
    const T* sval = staged ? sm.val : M.val + v0;
    const TriRow<T> row{M.bcol + b0, M.voff + b0, M.csz, M.coff, v0, nb, ni};
    double u = 0.0, sc = 0.0;  // lane a: row a's unknown, its scale
    if (lane < ni) {
      sc = scl[r0 + lane];
      u = BWD ? rhs[r0 + lane] : __dmul_rn(sc, rhs[r0 + lane]);
    }
    __syncwarp();
    TriSplit us{0.f, 0.f, 0.f, false};
    constexpr bool narrow = std::is_same<R, float>::value;
    if constexpr (narrow) us = tri_split(u);
    float uf = 0.f;   // u rounded to FP32 (FP32 records)
    double s[TRI_R];  // rows lane + 32 t of a large row
    if (ni <= TRI_MR) {
      // FP32 factors are applied in FP32 (the products and their sums), FP64
      // ones in FP64; the row's result is formed in FP64
      T sa;
      const bool ok = ni <= 8 && staged
                          ? tri_row<8>(row, sm.val, rec, sm.part(), abort, wait_limit, st, lane, &sa)
                          : tri_row16<T, R>(row, sval, rec, sm.part(), abort, wait_limit, st, lane, &sa);
      if (!ok) return;
      if constexpr (narrow) uf = tri_sub32(u, us, sa, lane < ni);
      if (!narrow || (BWD && !f32p)) u = lane < ni ? u - (double)sa : 0.0;
      if constexpr (narrow && !BWD) {  // the record first: the FP64 unknown is not on the chain
        if (lane < ni) {
          tri_publish(rec + tri_rec<R>(r0, i) + lane, uf);
          tri_publish(dbl + r0 + lane, u - (double)sa);
        }
        __syncwarp();  // the staged data is read no more
        continue;
      }
    } else {
      if (ni > 32 * TRI_R) {
        if (lane == 0) {
          dev_fail(st, DEV_INTERNAL);
          atomicExch(abort, 1);
        }
        return;
      }
      s[0] = u;
#pragma unroll
      for (int t = 1; t < TRI_R; ++t) {
        const int64_t q = r0 + lane + 32 * t;
        s[t] = lane + 32 * t < ni ? (BWD ? rhs[q] : __dmul_rn(scl[q], rhs[q])) : 0.0;
      }
      const bool dense = std::is_same<R, float>::value;
      if (!tri_large<T>(row, sval, dense ? dbl : (const double*)rec, dense, s, abort, wait_limit, st, lane)) return;
      u = s[0];
    }
    if (ni <= TRI_MP && (!BWD || sp)) {
      if (BWD) {
        if (f32p) {
          if (!narrow || ni > TRI_MR) uf = (float)u;
          if constexpr (sizeof(T) == sizeof(float)) {  // FP32 pivot blocks belong to FP32 factors only
            bool ok = false;
            float x = 0.f;
            // in line up to 6 rows only (applications of 200 000 unknowns in blocks of
            // 4, 6 and 8, two levels: up to 6 0.449, 0.466, 0.455 ms; up to 8 0.449,
            // 0.470, 0.436; none 0.477, 0.493, 0.455)
            if (ni <= 6 && fast) x = tri_pivot_f32<6, 8, true>(sm.lu, sm.ry, sm.rz, ni, src, uf, lane, &ok);
            if (!ok) x = tri_pivot_f32_wide(sm.lu, sm.ry, sm.rz, ni, src, fast, uf, lane);
            if constexpr (narrow)
              if (lane < ni) tri_publish(rec + tri_rec<R>(r0, i) + lane, x);
            u = (double)x;
          }
        } else {
          double* l = reinterpret_cast<double*>(sm.lu);
          const double* ry = reinterpret_cast<const double*>(sm.ry);
          const double* rz = reinterpret_cast<const double*>(sm.rz);
          u = sizeof(T) == sizeof(double) && ni <= 8 ? tri_pivot_f64<8>(l, ry, rz, ni, S, src, u, lane)
                                                     : tri_pivot_f64_wide(l, ry, rz, ni, S, src, u, lane);
        }
      }
      if (lane < ni) publish(i, r0, lane, u, sc);
    } else {  // pivot blocks of more than TRI_MP rows (tagged FP64 ones in FP32 factors: TRI_MP / 2)
      double* sv = reinterpret_cast<double*>(sm.part());
      __syncwarp();  // a large row's values may reach behind TRI_STAGE: every lane has read them
#pragma unroll
      for (int t = 0; t < TRI_R; ++t)
        if (lane + 32 * t < ni) sv[lane + 32 * t] = ni <= TRI_MR ? u : s[t];
      __syncwarp();
      if (BWD) {
        if (f32p)
          tri_pivot_large<float>(lu32 + dgoff[i], piv + r0, ni, sv, sv + 32 * TRI_R, lane);
        else
          tri_pivot_large<double>(lu64 + dgoff[i], piv + r0, ni, sv, sv + 32 * TRI_R, lane);
      }
      for (int a = lane; a < ni; a += 32) publish(i, r0, a, sv[a], scl[r0 + a]);
    }
    __syncwarp();  // the staged data is read no more
  }
}

// Deterministic two-stage dot product.
constexpr int RT = 256;
constexpr int RB = 512;

__global__ void __launch_bounds__(RT) k_dot_partial(const double* __restrict__ x, const double* __restrict__ y,
                                                    int64_t n, double* __restrict__ part) {
  __shared__ double red[RT / 32];
  double s = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)RT + threadIdx.x; i < n; i += (int64_t)gridDim.x * RT) s += x[i] * y[i];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    double v = threadIdx.x < RT / 32 ? red[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (threadIdx.x == 0) part[blockIdx.x] = v;
  }
}

__global__ void k_dot_final(const double* __restrict__ part, int nb, double* __restrict__ out) {
  __shared__ double red[RB];
  double s = 0.0;
  for (int i = threadIdx.x; i < nb; i += blockDim.x) s += part[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = red[0];
}

__global__ void k_axpy_dev(double* __restrict__ y, const double* __restrict__ x, const double* __restrict__ a,
                           double sign, int64_t n) {
  const double al = sign * *a;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] += al * x[i];
}
__global__ void k_axpy_host(double* __restrict__ y, const double* __restrict__ x, double a, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] += a * x[i];
}
__global__ void k_scale_dev(double* __restrict__ y, const double* __restrict__ x, const double* __restrict__ d,
                            int64_t n) {
  const double dv = *d;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = x[i] / dv;
}
__global__ void k_sub(double* __restrict__ r, const double* __restrict__ b, const double* __restrict__ ax, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    r[i] = b[i] - ax[i];
}
__global__ void k_gather(double* __restrict__ y, const double* __restrict__ x, const int32_t* __restrict__ idx,
                         int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = x[idx[i]];
}
__global__ void k_scatter(double* __restrict__ y, const double* __restrict__ x, const int32_t* __restrict__ idx,
                          int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[idx[i]] = x[i];
}

__global__ void k_sperm(int64_t p, const int32_t* __restrict__ pI, const int32_t* __restrict__ rsz,
                        const int64_t* __restrict__ roff, const int64_t* __restrict__ newoff,
                        int32_t* __restrict__ sperm) {
  const int lane = threadIdx.x & 31;
  const int64_t wpb = blockDim.x >> 5;
  for (int64_t k = blockIdx.x * wpb + (threadIdx.x >> 5); k < p; k += (int64_t)gridDim.x * wpb) {
    const int32_t Y = pI[k];
    for (int a = lane; a < rsz[Y]; a += 32) sperm[newoff[k] + a] = (int32_t)(roff[Y] + a);
  }
}

__global__ void k_perm_sizes2(int64_t p, const int32_t* __restrict__ pI, const int32_t* __restrict__ rsz,
                              int32_t* __restrict__ out) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < p; k += (int64_t)gridDim.x * blockDim.x)
    out[k] = rsz[pI[k]];
}

}  // namespace

// --------------------------------------------------------------------------
void dot_dev(const double* x, const double* y, int64_t n, double* out, double* scratch, cudaStream_t s) {
  const int nb = (int)std::min<int64_t>(RB, std::max<int64_t>(1, (n + RT - 1) / RT));
  launch(k_dot_partial, nb, RT, 0, s, x, y, n, scratch);
  launch(k_dot_final, 1, RB, 0, s, scratch, nb, out);
  VB_LAUNCH_CHECK();
}
void axpy_dev(double* y, const double* x, const double* a, double sign, int64_t n, cudaStream_t s) {
  if (n) launch(k_axpy_dev, grid_for(n, 256, 152LL * 16), 256, 0, s, y, x, a, sign, n);
  VB_LAUNCH_CHECK();
}
void axpy_host(double* y, const double* x, double a, int64_t n, cudaStream_t s) {
  if (n) launch(k_axpy_host, grid_for(n, 256, 152LL * 16), 256, 0, s, y, x, a, n);
  VB_LAUNCH_CHECK();
}
void scale_dev(double* y, const double* x, const double* d, int64_t n, cudaStream_t s) {
  if (n) launch(k_scale_dev, grid_for(n, 256, 152LL * 16), 256, 0, s, y, x, d, n);
  VB_LAUNCH_CHECK();
}
void sub_dev(double* r, const double* b, const double* ax, int64_t n, cudaStream_t s) {
  if (n) launch(k_sub, grid_for(n, 256, 152LL * 16), 256, 0, s, r, b, ax, n);
  VB_LAUNCH_CHECK();
}
void gather_dev(double* y, const double* x, const int32_t* idx, int64_t n, cudaStream_t s) {
  if (n) launch(k_gather, grid_for(n, 256, 152LL * 16), 256, 0, s, y, x, idx, n);
  VB_LAUNCH_CHECK();
}
void scatter_dev(double* y, const double* x, const int32_t* idx, int64_t n, cudaStream_t s) {
  if (n) launch(k_scatter, grid_for(n, 256, 152LL * 16), 256, 0, s, y, x, idx, n);
  VB_LAUNCH_CHECK();
}

// Row-block map of a VBCSR (scalar row -> block row), cached per matrix.
static void make_rowblk(int64_t nbr, const int64_t* roff, int64_t n, DBuf<int64_t>& rb, cudaStream_t s) {
  rb.alloc(n, s);
  if (nbr) launch(k_rowblk, grid_for(nbr, 8), 256, 0, s, nbr, roff, rb.p);
  VB_LAUNCH_CHECK();
}

void spmv_vb(const VBDev<double>& A, const int64_t* rowblk, int64_t n, const double* x, double* y,
             cudaStream_t s) {
  if (n) launch(spmv_plain(A) ? k_spmv<1> : k_spmv<SPMV_K>, grid_for(n, 128, 152LL * 32), 128, 0, s, A.view(), rowblk, n, x, y);
  VB_LAUNCH_CHECK();
}

void rowblk_map(const VBDev<double>& A, int64_t n, DBuf<int64_t>& rb, cudaStream_t s) {
  make_rowblk(A.nbr, A.roff.p, n, rb, s);
}

template <typename T>
void build_level_maps(const LevelDev<T>& L, const int32_t* rsz, const int64_t* roff, int64_t p, LevelMaps& M,
                      cudaStream_t s) {
  M.n = p ? d2h(roff + p, s) : 0;
  M.sperm.alloc(M.n, s);
  DBuf<int32_t> psz(p, s);
  DBuf<int64_t> newoff(p + 1, s);
  if (p) {
    launch(k_perm_sizes2, grid_for(p, 256), 256, 0, s, p, L.pI.p, rsz, psz.p);
    VB_LAUNCH_CHECK();
  }
  scan_i32_to_i64(psz.p, newoff.p, p, s);
  M.nf = p ? d2h(newoff.p + L.nD, s) : 0;
  if (p) {
    launch(k_sperm, grid_for(p, 8), 256, 0, s, p, L.pI.p, rsz, roff, newoff.p, M.sperm.p);
    VB_LAUNCH_CHECK();
  }
}
template void build_level_maps<double>(const LevelDev<double>&, const int32_t*, const int64_t*, int64_t,
                                       LevelMaps&, cudaStream_t);
template void build_level_maps<float>(const LevelDev<float>&, const int32_t*, const int64_t*, int64_t, LevelMaps&,
                                      cudaStream_t);

// --------------------------------------------------------------------------
// The sweeps use more than 48 KB of dynamic shared memory: opt in once per
// device for each instantiation.
template <typename T>
void tri_attributes() {
  static bool set_on[64] = {};
  int dev = 0;
  VB_CUDA(cudaGetDevice(&dev));
  if (dev >= 0 && dev < 64 && set_on[dev]) return;
  auto opt_in = [](auto kernel) {
    VB_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(TRI_W * sizeof(TriSmem<T>))));
  };
  opt_in(k_tri<T, false, double>);
  opt_in(k_tri<T, true, double>);
  if constexpr (sizeof(T) == sizeof(float)) {
    opt_in(k_tri<T, false, float>);
    opt_in(k_tri<T, true, float>);
  }
  if (dev >= 0 && dev < 64) set_on[dev] = true;
}

template <typename T>
void PrecDev<T>::prepare_apply() {
  tri_attributes<T>();
  if (prepared) return;
  const int nl = (int)lev.size();
  int64_t total = 0;
  for (int l = 0; l < nl; ++l) {
    total += 2 * maps[l].n;
    LevelMaps& M = maps[l];
    const LevelDev<T>& L = lev[l];
    if (M.n - M.nf > 0) make_rowblk(L.G.nbr, L.G.roff.p, M.n - M.nf, M.grow, s);
    if (M.nf > 0) make_rowblk(L.W.nbr, L.W.roff.p, M.nf, M.wrow, s);
  }
  nlast = last.A.nbr ? last.A.nrows_scalar(s) : 0;
  work.alloc(std::max<int64_t>(total, 1), s);
  // the sweeps' records and FP64 unknowns, cleared together: FP32 records
  // twice, y and x, or FP64 records twice and y
  const bool narrow = sizeof(T) == sizeof(float);
  rec_bytes = narrow ? rec_words<float>(nlast, last.A.nbr) * 4 : rec_words<double>(nlast, last.A.nbr) * 8;
  rec.alloc(2 * rec_bytes + (narrow ? 2 : 1) * nlast * 8 + 16, s);
  tick.alloc(2, s);
  abort_flag.alloc(1, s);
  int dev = 0;
  VB_CUDA(cudaGetDevice(&dev));
  VB_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  prepared = true;
}

namespace {
constexpr int kMaxLev = 64;  // fixed host arrays: the scratch path allocates nothing

// Device buffers of one application of Alg. 2.
struct SolveBufs {
  double* bh[kMaxLev];          // per level: P_I S_1 b, then y = U^{-1}(u - W z)
  double* xh[kMaxLev];          // per level: [y; z] before S_2 P_I^T
  const int64_t* grow[kMaxLev]; // scalar row -> block row of G
  const int64_t* wrow[kMaxLev]; // scalar row -> block row of W
  double* fv[kMaxLev + 1];      // fixed values per level (fv[0]: the caller's)
  double* yy;                   // last level: L^{-1} S_1 g
  void* recf;                   // records of the forward sweep
  void* recb;                   // records of the backward sweep (may be recf)
  double* xx;                   // FP32 records: the FP64 unknowns of the backward sweep (else NULL)
  void* clear;                  // what starts as 0xff bytes: recf, and all else but a recb that is recf
  size_t clear_bytes;
  unsigned long long* tick;     // 2 tickets
  int* abort;
  int nsm;
};

// fv_next[q] = fv[sp[nf + q]] / c[sp[nf + q]]: the fixed values of the C rows
// in the next level's variables (the backward sweep forms x = c * z there).
__global__ void k_fix_down(int64_t n, const int32_t* __restrict__ sp, const double* __restrict__ c,
                           const double* __restrict__ fv, double* __restrict__ fnext) {
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
    const int32_t o = sp[q];
    fnext[q] = __ddiv_rn(fv[o], c[o]);
  }
}

// The last level's two sweeps: z = S2 (L U)^{-1} S1 g, with records of type R.
template <typename T, typename R>
void sweep_last(const PrecDev<T>& P, const SolveBufs& B, const double* g, double* z, int64_t n, const int32_t* fixed,
                const double* fixv) {
  cudaStream_t s = P.s;
  const auto& last = P.last;
  const int64_t p = last.A.nbr;
  // the buffers keep the previous call's contents
  VB_CUDA(cudaMemsetAsync(B.clear, 0xff, B.clear_bytes, s));
  VB_CUDA(cudaMemsetAsync(B.tick, 0, 2 * sizeof(unsigned long long), s));
  VB_CUDA(cudaMemsetAsync(B.abort, 0, sizeof(int), s));
  const unsigned nb =
      (unsigned)std::max<int64_t>(1, std::min<int64_t>((int64_t)B.nsm * TRI_B, (p + TRI_W - 1) / TRI_W));
  const size_t smem = TRI_W * sizeof(TriSmem<T>);
  launch(k_tri<T, false, R>, nb, TRI_W * 32, smem, s, last.L.view(), nullptr, nullptr, nullptr, nullptr, nullptr, g,
         last.r.p, (R*)B.recf, B.yy, B.yy, last.lorder.p, B.tick, B.abort, (unsigned long long)P.wait_limit,
         P.status.p, nullptr, nullptr);
  if (B.recb == B.recf) VB_CUDA(cudaMemsetAsync(B.recb, 0xff, B.clear_bytes, s));
  launch(k_tri<T, true, R>, nb, TRI_W * 32, smem, s, last.U.view(), last.Dg.voff.p, last.Dg.val.p,
         sizeof(T) == sizeof(float) ? last.Dg32.val.p : nullptr, last.ptag.p, last.piv.p, B.yy, last.c.p, (R*)B.recb,
         B.xx, z, last.uorder.p, B.tick + 1, B.abort, (unsigned long long)P.wait_limit, P.status.p, fixed, fixv);
  VB_LAUNCH_CHECK();
}

template <typename T>
void bsr_sub(const VBDev<T>& M, const int64_t* rowblk, int64_t n, const double* x, double* y, cudaStream_t s) {
  launch(spmv_plain(M) ? k_bsr_sub<T, 1> : k_bsr_sub<T, SPMV_K>, grid_for(n, 128), 128, 0, s, M.view(), rowblk, n, x, y);
}

// Alg. 2 over all levels, in the factorization's own numbering; enqueues
// work only.  fixv (may be NULL; factorizations with fixed rows only): the
// values the last level's backward sweep takes for its fixed rows instead of
// solving for them (Section 5, the recovery u_i = B_i^{-1}(f_i - F_i y_i)).
template <typename T>
void solve_core(const PrecDev<T>& P, const double* in, double* out, const SolveBufs& B, const double* fixv) {
  cudaStream_t s = P.s;
  const int nl = (int)P.lev.size();
  const bool mixed = sizeof(T) != sizeof(double);
  const auto& last = P.last;
  // forward sweep down the levels: u = L^{-1} P f, g' = g - G u
  for (int l = 0; l < nl; ++l) {
    const LevelDev<T>& L = P.lev[l];
    const LevelMaps& M = P.maps[l];
    const double* b = l == 0 ? in : B.bh[l - 1] + P.maps[l - 1].nf;
    if (M.n) launch(k_gather_scale, grid_for(M.n, 256), 256, 0, s, M.n, M.sperm.p, L.r.p, b, B.bh[l]);
    if (L.grouped)
      grouped_forward<T>(L, B.bh[l], s);
    else if (L.nD) {
      const PivShape ps(L.nD, L.D.nval);
      launch(k_pivot_fwd, piv_grid(L.nD, ps), PIV_T, 0, s, L.nD, ps.per, ps.threads, L.D.rsz.p, L.D.roff.p, L.D.voff.p,
             L.D.val.p, mixed ? L.D32.val.p : nullptr, L.ptag.p, L.piv.p, B.bh[l]);
    }
    const int64_t ng = M.n - M.nf;
    if (ng && L.G.nnzb)
      bsr_sub(L.G, B.grow[l], ng, B.bh[l], B.bh[l] + M.nf, s);
    if (fixv && ng)
      launch(k_fix_down, grid_for(ng, 256), 256, 0, s, ng, M.sperm.p + M.nf, L.c.p, l == 0 ? fixv : B.fv[l],
             B.fv[l + 1]);
    VB_LAUNCH_CHECK();
  }
  // last level: z = S2 (L U)^{-1} S1 g
  {
    const int64_t nl_last = nl == 0 ? P.n : P.maps[nl - 1].n - P.maps[nl - 1].nf;
    const double* g = nl == 0 ? in : B.bh[nl - 1] + P.maps[nl - 1].nf;
    double* z = nl == 0 ? out : B.xh[nl - 1] + P.maps[nl - 1].nf;
    if (nl_last) {
      if constexpr (sizeof(T) == sizeof(float)) {
        if (B.xx)
          sweep_last<T, float>(P, B, g, z, nl_last, fixv ? last.fixed.p : nullptr, nl == 0 ? fixv : B.fv[nl]);
        else
          sweep_last<T, double>(P, B, g, z, nl_last, fixv ? last.fixed.p : nullptr, nl == 0 ? fixv : B.fv[nl]);
      } else {
        sweep_last<T, double>(P, B, g, z, nl_last, fixv ? last.fixed.p : nullptr, nl == 0 ? fixv : B.fv[nl]);
      }
      VB_LAUNCH_CHECK();
    }
  }
  // backward sweep up the levels: y = U^{-1} (u - W z), x = S2 P_I^T [y; z]
  for (int l = nl - 1; l >= 0; --l) {
    const LevelDev<T>& L = P.lev[l];
    const LevelMaps& M = P.maps[l];
    double* xo = l == 0 ? out : B.xh[l - 1] + P.maps[l - 1].nf;
    if (M.nf && L.W.nnzb)
      bsr_sub(L.W, B.wrow[l], M.nf, B.xh[l] + M.nf, B.bh[l], s);
    if (L.grouped)
      grouped_backward<T>(L, B.bh[l], B.xh[l], s);
    else if (L.nD) {
      const PivShape ps(L.nD, L.D.nval);
      launch(k_pivot_bwd, piv_grid(L.nD, ps), PIV_T, 0, s, L.nD, ps.per, ps.threads, L.D.rsz.p, L.D.roff.p, L.D.voff.p,
             L.D.val.p, mixed ? L.D32.val.p : nullptr, L.ptag.p, B.bh[l], B.xh[l]);
    }
    if (M.n) launch(k_scatter_scale, grid_for(M.n, 256), 256, 0, s, M.n, M.sperm.p, L.c.p, B.xh[l], xo);
    VB_LAUNCH_CHECK();
  }
}

// Doubles of fixed-value work: the C rows of every level.
template <typename T>
int64_t fixed_work(const PrecDev<T>& P) {
  if (!P.last.fixed.p) return 0;
  int64_t t = 0;
  for (const auto& M : P.maps) t += M.n - M.nf;
  return t;
}
}  // namespace

template <typename T>
void PrecDev<T>::apply_perm(const double* x, double* y) {
  apply_fixed(x, y, nullptr);
}

template <typename T>
void PrecDev<T>::apply_fixed(const double* x, double* y, const double* fixv) {
  prepare_apply();
  const int nl = (int)lev.size();
  if (nl > kMaxLev) fail(VB_EINVAL, "more than 64 levels");
  if (fixv && !last.fixed.p) fail(VB_EINVAL, "the factorization has no fixed rows");
  SolveBufs B{};
  double* wp = work.p;
  for (int l = 0; l < nl; ++l) {
    B.bh[l] = wp;
    wp += maps[l].n;
    B.xh[l] = wp;
    wp += maps[l].n;
    B.grow[l] = maps[l].grow.p;
    B.wrow[l] = maps[l].wrow.p;
  }
  const bool narrow = sizeof(T) == sizeof(float);
  B.recf = rec.p;
  B.recb = rec.p + rec_bytes;
  B.yy = (double*)(rec.p + 2 * rec_bytes);
  B.xx = narrow ? B.yy + nlast : nullptr;
  B.clear = rec.p;
  B.clear_bytes = 2 * rec_bytes + (narrow ? 2 : 0) * nlast * 8;
  if (fixv) {
    const int64_t nf = fixed_work(*this);
    if ((int64_t)fwork.n < nf) fwork.alloc(std::max<int64_t>(nf, 1), s);
    double* fp = fwork.p;
    for (int l = 0; l < nl; ++l) {
      B.fv[l + 1] = fp;
      fp += maps[l].n - maps[l].nf;
    }
  }
  B.tick = tick.p;
  B.abort = abort_flag.p;
  B.nsm = nsm;
  solve_core(*this, x, y, B, fixv);
}

// ---- the same solve with caller-provided scratch (no allocation) ----------
// Layout of the scratch, each piece 256-byte aligned: the permuted x and y
// (n doubles each), the records of the sweeps (both use the same n_last +
// p_last doubles, in turn: p_last doubles, then the first n_last doubles of
// the next piece), the work vectors (n_last doubles of records, then the
// last level's y, then 2 n_l doubles per level), the row->block maps of G and
// W (n_l int64 per level), two tickets, the abort word, and (factorizations
// with fixed rows) the fixed-value work.
namespace {
struct ScratchPlan {
  size_t xp, yp, rec, work, maps, tick, abort, fwork, total;
};

inline size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }

template <typename T>
ScratchPlan plan_scratch(const PrecDev<T>& P) {
  ScratchPlan sp{};
  size_t o = 0;
  int64_t nwork = 0, nmap = 0;
  for (const auto& M : P.maps) {
    nwork += 2 * M.n;
    nmap += M.n;
  }
  const int64_t nlast = P.maps.empty() ? P.n : P.maps.back().n - P.maps.back().nf;
  nwork += 2 * nlast;
  sp.xp = o;
  o = align256(o + (size_t)P.n * 8);
  sp.yp = o;
  o = align256(o + (size_t)P.n * 8);
  sp.rec = o;
  o = align256(o + (size_t)P.last.A.nbr * 8);
  sp.work = o;
  o = align256(o + (size_t)nwork * 8);
  sp.maps = o;
  o = align256(o + (size_t)nmap * 8);
  sp.tick = o;
  o = align256(o + 2 * 8);
  sp.abort = o;
  o = align256(o + 4);
  sp.fwork = o;
  o = align256(o + (size_t)fixed_work(P) * 8);
  sp.total = o;
  return sp;
}
}  // namespace

template <typename T>
size_t PrecDev<T>::scratch_bytes() const {
  return plan_scratch(*this).total;
}

template <typename T>
void PrecDev<T>::apply_with_scratch(const double* x, double* y, unsigned char* scratch, int nsm_dev) {
  const ScratchPlan sp = plan_scratch(*this);
  double* xp = (double*)(scratch + sp.xp);
  double* yp = (double*)(scratch + sp.yp);
  gather_dev(xp, x, perm.p, n, s);
  solve_scratch(xp, yp, scratch, nsm_dev, nullptr);
  scatter_dev(y, yp, perm.p, n, s);
}

template <typename T>
void PrecDev<T>::solve_scratch(const double* x, double* y, unsigned char* scratch, int nsm_dev, const double* fixv) {
  tri_attributes<T>();
  const ScratchPlan sp = plan_scratch(*this);
  const int nl = (int)lev.size();
  if (nl > kMaxLev) fail(VB_EINVAL, "more than 64 levels");
  if (fixv && !last.fixed.p) fail(VB_EINVAL, "the factorization has no fixed rows");
  const int64_t nl_last = maps.empty() ? n : maps.back().n - maps.back().nf;
  double* wp = (double*)(scratch + sp.work) + nl_last;  // its first n_last doubles belong to the records
  int64_t* mp = (int64_t*)(scratch + sp.maps);
  double* fp = (double*)(scratch + sp.fwork);
  SolveBufs B{};
  // FP64 records, shared by the two sweeps: no more scratch than their flags took
  B.recf = B.recb = B.clear = scratch + sp.rec;
  B.clear_bytes = (size_t)(nl_last + last.A.nbr) * 8;  // exactly: y follows
  B.yy = wp;
  wp += nl_last;
  for (int l = 0; l < nl; ++l) {
    B.bh[l] = wp;
    wp += maps[l].n;
    B.xh[l] = wp;
    wp += maps[l].n;
    int64_t* gm = mp;
    int64_t* wm = mp + (maps[l].n - maps[l].nf);
    mp += maps[l].n;
    const LevelDev<T>& L = lev[l];
    if (maps[l].n - maps[l].nf > 0 && L.G.nbr)
      launch(k_rowblk, grid_for(L.G.nbr, 8), 256, 0, s, L.G.nbr, L.G.roff.p, gm);
    if (maps[l].nf > 0 && L.W.nbr) launch(k_rowblk, grid_for(L.W.nbr, 8), 256, 0, s, L.W.nbr, L.W.roff.p, wm);
    VB_LAUNCH_CHECK();
    B.grow[l] = gm;
    B.wrow[l] = wm;
    if (fixv) {
      B.fv[l + 1] = fp;
      fp += maps[l].n - maps[l].nf;
    }
  }
  B.tick = (unsigned long long*)(scratch + sp.tick);
  B.abort = (int*)(scratch + sp.abort);
  B.nsm = nsm_dev;
  solve_core(*this, x, y, B, fixv);
}

template <typename T>
void PrecDev<T>::export_mat(int l, int which, int64_t* nbr, int64_t* nbc, int64_t* nnzb, int64_t* nval,
                            int32_t* rsz, int32_t* csz, int64_t* bptr, int32_t* bcol, int64_t* voff, double* val) {
  const int nl = (int)lev.size();
  if (l < 0 || l > nl) fail(VB_EINVAL, "level out of range");
  if (l == nl) {
    switch (which) {
      case 0: return export_vb(last.A, s, nbr, nbc, nnzb, nval, rsz, csz, bptr, bcol, voff, val);
      case 1: return export_vb(last.Dg, s, nbr, nbc, nnzb, nval, rsz, csz, bptr, bcol, voff, val);
      case 8: return export_vb(last.L, s, nbr, nbc, nnzb, nval, rsz, csz, bptr, bcol, voff, val);
      case 9: return export_vb(last.U, s, nbr, nbc, nnzb, nval, rsz, csz, bptr, bcol, voff, val);
    }
    fail(VB_EINVAL, "matrix selector out of range");
  }
  const LevelDev<T>& L = lev[l];
  switch (which) {
    case 0:
      if (L.A64.nbr || !L.AT.nbr) return export_vb(L.A64, s, nbr, nbc, nnzb, nval, rsz, csz, bptr, bcol, voff, val);
      return export_vb(L.AT, s, nbr, nbc, nnzb, nval, rsz, csz, bptr, bcol, voff, val);
    case 1: return export_vb(L.D, s, nbr, nbc, nnzb, nval, rsz, csz, bptr, bcol, voff, val);
    case 2: return export_vb(L.F, s, nbr, nbc, nnzb, nval, rsz, csz, bptr, bcol, voff, val);
    case 3: return export_vb(L.E, s, nbr, nbc, nnzb, nval, rsz, csz, bptr, bcol, voff, val);
    case 4: return export_vb(L.C, s, nbr, nbc, nnzb, nval, rsz, csz, bptr, bcol, voff, val);
    case 5: return export_vb(L.W, s, nbr, nbc, nnzb, nval, rsz, csz, bptr, bcol, voff, val);
    case 6: return export_vb(L.G, s, nbr, nbc, nnzb, nval, rsz, csz, bptr, bcol, voff, val);
    case 7: return export_vb(L.S, s, nbr, nbc, nnzb, nval, rsz, csz, bptr, bcol, voff, val);
    case 10:
      if (!L.grouped) fail(VB_EINVAL, "not a grouped level");
      return export_vb(L.Lg, s, nbr, nbc, nnzb, nval, rsz, csz, bptr, bcol, voff, val);
    case 11:
      if (!L.grouped) fail(VB_EINVAL, "not a grouped level");
      return export_vb(L.Ug, s, nbr, nbc, nnzb, nval, rsz, csz, bptr, bcol, voff, val);
  }
  fail(VB_EINVAL, "matrix selector out of range");
}

template <typename T>
void PrecDev<T>::export_vec(int l, int which, double* d, int32_t* iv, int64_t* len) {
  const int nl = (int)lev.size();
  if (l < 0 || l > nl) fail(VB_EINVAL, "level out of range");
  const DBuf<double>* dv = nullptr;
  const DBuf<int32_t>* ivb = nullptr;
  if (l == nl) {
    if (which == 0) dv = &last.r;
    if (which == 1) dv = &last.c;
    if (which == 4) ivb = &last.piv;
    if (which == 5) ivb = &last.ptag;
  } else {
    const LevelDev<T>& L = lev[l];
    if (which == 0) dv = &L.r;
    if (which == 1) dv = &L.c;
    if (which == 2) dv = &L.w;
    if (which == 3) ivb = &L.pI;
    if (which == 4) ivb = &L.piv;
    if (which == 5) ivb = &L.ptag;
    if (which == 6) {  // group boundaries of a grouped level (ngroups + 1)
      if (!L.grouped) fail(VB_EINVAL, "not a grouped level");
      const std::vector<int64_t> g = d2h_vec(L.gptr.p, L.ngroups + 1, s);
      if (len) *len = (int64_t)g.size();
      if (iv)
        for (size_t k = 0; k < g.size(); ++k) iv[k] = (int32_t)g[k];
      return;
    }
  }
  if (!dv && !ivb) fail(VB_EINVAL, "vector selector out of range");
  const int64_t n = dv ? (int64_t)dv->n : (int64_t)ivb->n;
  if (len) *len = n;
  if (dv && d && n) VB_CUDA(cudaMemcpyAsync(d, dv->p, n * 8, cudaMemcpyDeviceToHost, s));
  if (ivb && iv && n) VB_CUDA(cudaMemcpyAsync(iv, ivb->p, n * 4, cudaMemcpyDeviceToHost, s));
  VB_CUDA(cudaStreamSynchronize(s));
}

template struct PrecDev<double>;
template struct PrecDev<float>;

}  // namespace vb
