// Last-level block ILUT of VBARMS on the GPU (Section 3 dropping rule, the
// block IKJ form of Alg. 3), on the scaled last Schur complement in natural
// order.
//
// Row i is processed by one warp that took ticket i (tickets are handed out
// in row order, so every row a warp waits for is already owned by a running
// warp).  A matrix made of independent diagonal blocks (a batch, or the
// subdomains of a domain decomposition) may instead hand out its rows
// interleaved across the blocks, each block's rows in ascending order: the
// blocks' dependency chains then advance side by side.
//
// The warp keeps its working row in a private workspace (hash table column ->
// slot, dense values): in shared memory when the row fits, else in global
// memory (a shared row whose fill would outgrow the buffer moves, slots and
// values as they are, to the global one before the blocks that overflow it are
// created).  The size of the shared workspace is chosen by timing from the
// last-level matrix (rows of a few large blocks, or rows of many small ones).
// The warp eliminates its L part in ascending column order including fill.
// For each column k it needs row k's factored pivot block and its U row:
// row k publishes them as one record (below) and a 64-bit word in done[k]
// telling where the record lies, so the dependant waits for one word and
// brings the record on chip with its own asynchronous copies; the record of
// the next pending column is fetched ahead while the current step computes.
// After the last column the warp thresholds its U part, applies lfil to it,
// sorts the kept blocks by column, factors its diagonal block (GEPP) and
// publishes; the L part, which no other row reads, is written after that.  Per
// element, the operation order is the oracle's, so FP64 results match it bit
// for bit; the mixed factor keeps its drop sums, drop tests and diagonal GEPP
// in FP32 (a block whose condition estimate exceeds the threshold is factored
// again in FP64).
//
// Bound: the chain of dependent rows times a link's latency (a dependant's step
// for the column it waited on, then its finish).  With 16 warps an SM, stages
// of 2 KB and 128 registers, the records of more than about ten U blocks (FP64:
// four) were read in place from L2, one dependent load after another, and half
// of the rows worked in global memory: 32 us a link (FP64 42 to 66).  Now 7
// warps an SM (FP64 5, wide rows 3) have up to 255 registers a thread (FP32: 64
// bytes spilled, FP64 none) and keep records and rows on chip; a step's update takes a column per lane, divisions by pivot
// entries are corrected products with their reciprocals, the pivot search and
// the reciprocals overlap, and FP64 drop tests are decided in FP32 where that
// is certain.  The kernel's time before and now: 3.0 million unknowns FP32 710
// and 385 ms, 360 000 FP64 498 and 261 ms, 48 000 at tau 0.9 786 and 254 ms.
//
// A wait that runs out sets VB_ETIMEOUT and raises an abort flag; a row that
// failed publishes kRowFailed so that its dependants stop too.  Overflowing a
// pool or the global workspace sets an overflow code and the host repeats the
// kernel with larger buffers.
#include <algorithm>
#include <chrono>
#include <climits>
#include <map>
#include <mutex>
#include <type_traits>

#include "internal.h"
#include "level.cuh"
#include "vbsr_ops.cuh"

namespace vb {
namespace {

enum : int { SL_LIVE = 0, SL_LKEPT = 1, SL_DEAD = 2 };

// ---------------------------------------------------------------------------
// Published rows.  Row k's record, in the U pool, 16-byte aligned:
//   int32 head[4]         ucnt (U blocks), nk, 2 depth + lu64 (lu64 = 1: the
//                         pivot LU is stored in FP64, else in the factor's
//                         type TL; depth: rows on the longest chain of waits
//                         that ends at the row), ncol (U columns)
//   int32 perm[nk]        row of the pivot block that GEPP brought to each place
//   TL lu[nk * S]         the factored pivot block, rows S = lu_stride apart
//   TL ry[nk], rz[nk]     reciprocals of its diagonal (recip_rn)
//   int32 ucol[ucnt]      U block columns, ascending
//   int32 ucst[ucnt]      each U block's first column within the row's U part
//   int32 unj[ucnt]       each U block's column count
//   T val[ncol * nk]      the U blocks, row-major, in column order (block q's
//                         values start at nk ucst[q])
// every part starting on a 16-byte boundary.  done[k] = (offset << 24) |
// length, both in 16-byte units, once the record is complete; kRowFailed when
// the row failed; 0 before.
constexpr unsigned long long kRowFailed = ~0ull;
constexpr int64_t kRecMaxUnits = (1LL << 24) - 1;

// Row stride of a record's pivot LU: FP32 blocks of at most 8 rows are read by
// unrolled code with fixed offsets.
__host__ __device__ __forceinline__ int lu_stride(int nk, int lu64, int tsize) {
  return !lu64 && tsize == 4 && nk <= 8 ? 8 : nk;
}

template <typename I>
struct RecLayout {
  I perm, lu, rcp, ucol, ucst, unj, val, bytes;
};
// I = int for a published record (at most 2^28 bytes), int64_t to size a new one.
template <typename I>
__host__ __device__ __forceinline__ RecLayout<I> rec_layout(int ucnt, int nk, int lu64, int ncol, int tsize) {
  RecLayout<I> L;
  const I tl = lu64 ? 8 : tsize, uc = ((I)ucnt * 4 + 15) & ~(I)15;
  L.perm = 16;
  L.lu = L.perm + (((I)nk * 4 + 15) & ~(I)15);
  L.rcp = L.lu + (((I)nk * lu_stride(nk, lu64, tsize) * tl + 15) & ~(I)15);
  L.ucol = L.rcp + ((2 * (I)nk * tl + 15) & ~(I)15);
  L.ucst = L.ucol + uc;
  L.unj = L.ucst + uc;
  L.val = L.unj + uc;
  L.bytes = L.val + (((I)ncol * nk * tsize + 15) & ~(I)15);
  return L;
}

struct Pools {
  // L rows: blocks in pool order; per row the first block and count
  int32_t* lcol;
  int64_t* lvo;  // value offset of each pool block
  int64_t* lstart;
  int32_t* lcnt;
  unsigned long long* done;  // per row: the published record word
  unsigned long long* ctr;   // [0] L blocks, [1] L values, [2] U record units, [4] ticket,
                             // [5] largest row values asked, [6] largest row slots asked
  int64_t lbcap, lvcap, ucap16;
  int* abort;
  // ticket -> row (nullptr: ticket t is row t); every row's dependencies
  // must come earlier in it
  const int32_t* order;
  // tickets handed out (the rows of the first nticket tickets: every prefix
  // of the ticket order holds its rows' dependencies, so it is factored
  // exactly on its own)
  int64_t nticket;
  // per row (may be NULL): 1 + the largest depth among the rows it waited
  // on (every pending L column, the dropped multipliers' included), i.e. the
  // length of the longest chain of waits ending at the row
  int32_t* depth;
};

// Global fallback workspace, per warp.
struct Workspace {
  int* keys;       // [ht]
  int* hpos;       // [smax]
  int* scol;       // [smax]
  int* soff;       // [smax]
  int* sstate;     // [smax]
  long long* sf2;  // [smax] norm key of each slot
  int* sncl;       // [smax] column count of each slot's block
  int* fin;        // [2 smax] candidate lists of the finish
  unsigned long long* srt;  // [4 smax] kept lists being sorted
  int ht, smax;
  int64_t vmax;
};

// Shared workspace of one warp, sized at launch (byte offsets in the warp's
// region; every part 16-byte aligned).
struct IlutGeom {
  int slots, hash, vbytes, stage, lcap;
  int o_misc, o_stage, o_vals, o_keys, o_hpos, o_scol, o_soff, o_sst, o_sf2, o_sncl, o_lc, o_ls;
  int bytes;
};

// Geometries chosen by timing, per device, precision and class of row sizes
// (the process keeps them), and the smallest matrix that is timed.
std::mutex g_geom_mu;
std::map<long long, struct IlutGeom> g_geom;
constexpr int64_t kTuneMinRows = 65536;

constexpr int PVMAX = 64;
constexpr int NSMALL = 8;   // FP32 pivot blocks up to this size are factored and applied in registers
constexpr int NPIV = 32;    // and up to this factored in registers
constexpr int MCOLS = 512;  // columns of a chunk of U blocks that the column update maps

// Per-warp scratch.  buf serves, one after the other: the lfil cut's histogram
// (256 int), a multiplier being formed, a chunk's column map (MCOLS bytes) and
// block descriptors (32 int4), the general update's tables.
template <typename T>
struct alignas(16) IlutMisc {
  int buf[256];
  T mt[1024 / sizeof(T)];  // rows of a step's multiplier, transposed: row a of column r at r * np + a
  T lu[NSMALL * NSMALL];   // the row's own small pivot LU (FP32)
  T ry[NPIV], rz[NPIV];    // reciprocals of its diagonal (FP32)
  int pv[PVMAX];           // GEPP interchanges of the row's own diagonal block
  int perm[PVMAX];         // and the rows they brought to each place
};
struct CopyTab {  // tables of the general update, in IlutMisc::buf
  int qpre[33];   // element prefix of a chunk's blocks
  int qoff[32];   // workspace value offset of each U block's target
  int quo[32];    // value offset of the U block within the record's values
  int qnj[32];
};
static_assert(sizeof(CopyTab) <= 1024, "tables exceed the scratch");

template <typename T>
__device__ __forceinline__ T msub(T acc, T a, T b);
template <>
__device__ __forceinline__ double msub<double>(double acc, double a, double b) {
  return __dsub_rn(acc, __dmul_rn(a, b));
}
template <>
__device__ __forceinline__ float msub<float>(float acc, float a, float b) {
  return __fmaf_rn(-a, b, acc);
}

__device__ __forceinline__ bool drop_rule(double f2, int m, int n, double t) {
  const double thr = __dmul_rn(__dmul_rn(t, (double)m), (double)n);
  return f2 < __dmul_rn(thr, thr);
}

// The same rule in FP32 for the mixed factor (FP64 operations are slow on
// this part and would sit on the critical path of every elimination step).
__device__ __forceinline__ bool drop_rule_f(float f2, int m, int n, float t) {
  const float thr = t * (float)m * (float)n;
  return f2 < thr * thr;
}

// Squared Frobenius norms are ranked (lfil) by their bit patterns: for
// non-negative IEEE values the integer order is the value order, so the
// comparisons stay on the integer pipes.  FP64 factor: the double's bits;
// mixed factor: the float's bits.
__device__ __forceinline__ long long norm_key(double f2) { return __double_as_longlong(f2); }
__device__ __forceinline__ long long norm_key(float f2) { return (long long)__float_as_int(f2); }

// x[perm[j]] <- x[j] for one row of length m, in place: every cycle of the
// permutation is turned from its smallest place (seen: the places below 128 that
// were turned; beyond, a walk along the cycle tells).
template <typename T, typename F>
__device__ __forceinline__ void row_permute(T* x, int m, F&& perm) {
  unsigned long long seen0 = 0, seen1 = 0;
#pragma unroll 1
  for (int j = 0; j < m; ++j) {
    int q = perm(j);
    if (q == j) continue;
    if (j < 64 ? seen0 >> j & 1 : j < 128 && (seen1 >> (j - 64) & 1)) continue;
    if (j >= 128) {
      while (q > j && q < m) q = perm(q);
      if (q != j) continue;  // j is not the smallest place of its cycle
    }
    T v = x[j];
#pragma unroll 1
    for (q = perm(j); q != j && q >= 0 && q < m; q = perm(q)) {
      const T t = x[q];
      x[q] = v;
      v = t;
      if (q < 64)
        seen0 |= 1ull << q;
      else if (q < 128)
        seen1 |= 1ull << (q - 64);
    }
    x[j] = v;
  }
}

// x (one row of length m) <- x (P^T L U)^{-1} = x U^{-1} L^{-1} P, arithmetic in
// TL, lu(q, j) the factored pivot block and perm(j) its permutation, UN loads in
// flight.
template <int UN, typename TL, typename T, typename L, typename F>
__device__ __forceinline__ void ainv_row(T* x, int m, L&& lu, F&& perm) {
#pragma unroll 1
  for (int j = 0; j < m; ++j) {
    TL s = (TL)x[j];
#pragma unroll UN
    for (int q = 0; q < j; ++q) s = msub<TL>(s, (TL)x[q], lu(q, j));
    x[j] = (T)(s / lu(j, j));
  }
#pragma unroll 1
  for (int j = m - 1; j >= 0; --j) {
    TL s = (TL)x[j];
#pragma unroll UN
    for (int q = j + 1; q < m; ++q) s = msub<TL>(s, (TL)x[q], lu(q, j));
    x[j] = (T)s;
  }
  row_permute(x, m, perm);
}

// The pivot block read through L2 (written by another warp); pm: the permutation
// on chip, or NULL and in place at pg.  One load after another took most of a link
// where blocks are large: 300 block rows of 28 to 32 scalars FP32 196 ms, 76 with
// eight in flight (and those of update_general); small blocks are quicker without.
template <typename T, typename TL>
__device__ __noinline__ void ainv_right_row(const TL* lu, int S, const int* pm, const int32_t* pg, int m, T* x) {
  auto at = [&](int q, int j) { return __ldcg(lu + q * S + j); };
  auto perm = [&](int j) { return pm ? pm[j] : __ldcg(pg + j); };
  if (m <= 8)
    ainv_row<1, TL>(x, m, at, perm);
  else
    ainv_row<8, TL>(x, m, at, perm);
}

// Workspace hash: keys[h] = -2 - slot, -1 = empty; the column of a slot is
// scol[slot].  Placement and lookup never run concurrently (separated by
// __syncwarp), and the columns inserted in one phase are distinct.
__device__ __forceinline__ int ws_place(int* keys, uint32_t mask, int slot, int col) {
  uint32_t h = hmix((uint32_t)col) & mask;
#pragma unroll 1
  for (uint32_t probe = 0; probe <= mask; ++probe) {
    if (atomicCAS(&keys[h], -1, -2 - slot) == -1) return (int)h;
    h = (h + 1) & mask;
  }
  return -1;
}

__device__ __forceinline__ int ws_lookup(const int* keys, const int* scol, uint32_t mask, int col) {
  uint32_t h = hmix((uint32_t)col) & mask;
#pragma unroll 1
  for (uint32_t probe = 0; probe <= mask; ++probe) {
    const int kv = keys[h];
    if (kv == -1) return -1;
    const int s = -2 - kv;
    if (scol[s] == col) return s;
    h = (h + 1) & mask;
  }
  return -1;
}

constexpr int MAX_SLOTS = 4096;  // largest workspace (blocks of one working row)

// Warp-cooperative copy with eight independent loads in flight per lane.
template <typename TD, typename T>
__device__ __noinline__ void warp_copy(TD* __restrict__ dst, const T* __restrict__ src, int64_t n, int lane) {
#pragma unroll 1
  for (int64_t e0 = lane; e0 < n; e0 += 32 * 8) {
    T v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int64_t e = e0 + 32 * u;
      if (e < n) v[u] = src[e];
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int64_t e = e0 + 32 * u;
      if (e < n) dst[e] = (TD)v[u];
    }
  }
}

// Squared Frobenius norm in row-major order (the oracle's summation order),
// with the loads issued eight at a time.
template <typename T>
__device__ __noinline__ double fro2_batched(const T* __restrict__ v, int n) {
  double s = 0.0;
#pragma unroll 1
  for (int e0 = 0; e0 < n; e0 += 8) {
    T x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) x[u] = e0 + u < n ? v[e0 + u] : (T)0;
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (e0 + u < n) {
        const double d = (double)x[u];
        s = __dadd_rn(s, __dmul_rn(d, d));
      }
  }
  return s;
}

// Squared Frobenius norm accumulated in FP32 (mixed factor).
template <typename T>
__device__ __forceinline__ float fro2_f32(const T* __restrict__ v, int n) {
  float s = 0.f;
  if (n <= 4) {
    float x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) x[u] = u < n ? (float)v[u] : 0.f;
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (u < n) s = __fmaf_rn(x[u], x[u], s);
    return s;
  }
#pragma unroll 1
  for (int e0 = 0; e0 < n; e0 += 16) {  // sixteen loads in flight, summed in element order
    float x[16];
#pragma unroll
    for (int u = 0; u < 16; ++u) x[u] = e0 + u < n ? (float)v[e0 + u] : 0.f;
#pragma unroll
    for (int u = 0; u < 16; ++u)
      if (e0 + u < n) s = __fmaf_rn(x[u], x[u], s);
  }
  return s;
}

// The same from a staged pivot block (values of type TS); x may live in shared
// memory.
template <typename T, typename TL, typename TS>
__device__ __noinline__ void ainv_right_row_sh(const TS* lu, int S, const int* pv, int m, T* x) {
  auto at = [&](int q, int j) { return (TL)lu[q * S + j]; };
  auto perm = [&](int j) { return pv[j]; };
  if (m <= 8)
    ainv_row<1, TL>(x, m, at, perm);
  else
    ainv_row<8, TL>(x, m, at, perm);
}

// |x| as an integer key: non-negative IEEE values order like their bit
// patterns, so pivot searches compare integers.
__device__ __forceinline__ long long abs_key(double x) { return __double_as_longlong(x) & 0x7fffffffffffffffLL; }
__device__ __forceinline__ long long abs_key(float x) { return (long long)(__float_as_int(x) & 0x7fffffff); }

// The largest of the lanes' non-negative values, NaN counting as 0 (as a chain
// of fmaxf from 0 has it).
__device__ __forceinline__ float warp_max_f(float v) {
  return __int_as_float((int)__reduce_max_sync(0xffffffffu, v == v ? (unsigned)__float_as_int(v) : 0u));
}

template <typename TL>
__device__ __forceinline__ TL div_rn(TL a, TL b);
template <>
__device__ __forceinline__ double div_rn<double>(double a, double b) {
  return __ddiv_rn(a, b);
}
template <>
__device__ __forceinline__ float div_rn<float>(float a, float b) {
  return __fdiv_rn(a, b);
}

// GEPP of the n x n row-major block a (max-abs pivot, ties to the lowest
// row), one warp: each elimination step finds its pivot by a warp reduction,
// then the lanes form the multipliers and update the trailing block, so every
// element receives the operations of the sequential algorithm in its order.
// Pivot rows go to gpiv (and pvs when not null).  Returns false when a pivot
// column is exactly zero.  FAR: a lies in global memory, where one element after
// another cost a trip to L2 each (30 block rows of 100 to 128 scalars FP64 642 ms,
// 577 with four rows in flight and the copies of the block too).
template <typename TL, bool FAR = false>
__device__ __noinline__ bool gepp_warp(TL* a, int n, int* pvs, int32_t* gpiv, int lane) {
#pragma unroll 1
  for (int kk = 0; kk < n; ++kk) {
    // the largest |a_ik|, its upper word first, the lowest row on ties
    unsigned long long key = 0;  // |a| + 1, 0: no row
    int idx = 0x7fffffff;
#pragma unroll(FAR ? 4 : 1)
    for (int ii = kk + lane; ii < n; ii += 32) {
      const unsigned long long v = (unsigned long long)abs_key(a[ii * n + kk]) + 1ull;
      if (v > key) {
        key = v;
        idx = ii;
      }
    }
    const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(key >> 32));
    const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(key >> 32) == hi ? (unsigned)key : 0u);
    const unsigned long long most = ((unsigned long long)hi << 32) | lo;
    idx = __reduce_min_sync(0xffffffffu, key == most ? idx : 0x7fffffff);
    key = most - 1;
    if (key == 0) return false;
    const int pr = idx;
    if (lane == 0) {
      gpiv[kk] = pr;
      if (pvs) pvs[kk] = pr;
    }
    if (pr != kk)
#pragma unroll 1
      for (int jj = lane; jj < n; jj += 32) {
        const TL t = a[kk * n + jj];
        a[kk * n + jj] = a[pr * n + jj];
        a[pr * n + jj] = t;
      }
    __syncwarp();
    const TL d = a[kk * n + kk];
    const int w = n - kk - 1;
    const float rw = __fdividef(1.f, (float)max(w, 1));
#pragma unroll 1
    for (int r = lane; r < w; r += 32) {
      TL* l = a + (kk + 1 + r) * n + kk;
      *l = div_rn<TL>(*l, d);
    }
    __syncwarp();
    if (FAR) {  // lanes over columns, four rows in flight
#pragma unroll 1
      for (int jj = kk + 1 + lane; jj < n; jj += 32) {
        const TL u = a[kk * n + jj];
        int ii = kk + 1;
#pragma unroll 1
        for (; ii + 4 <= n; ii += 4) {
          TL acc[4], l[4];
#pragma unroll
          for (int t = 0; t < 4; ++t) acc[t] = a[(ii + t) * n + jj], l[t] = a[(ii + t) * n + kk];
#pragma unroll
          for (int t = 0; t < 4; ++t) a[(ii + t) * n + jj] = msub<TL>(acc[t], l[t], u);
        }
#pragma unroll 1
        for (; ii < n; ++ii) a[ii * n + jj] = msub<TL>(a[ii * n + jj], a[ii * n + kk], u);
      }
    } else {
#pragma unroll 1
      for (int e = lane; e < w * w; e += 32) {
        int r = (int)((float)e * rw), c = e - r * w;  // e / w, corrected
        if (c < 0) --r, c += w;
        if (c >= w) ++r, c -= w;
        const int ii = kk + 1 + r, jj = kk + 1 + c;
        a[ii * n + jj] = msub<TL>(a[ii * n + jj], a[ii * n + kk], a[kk * n + jj]);
      }
    }
    __syncwarp();
  }
  return true;
}

// ||B^{-1}||_1 of a GEPP-factored FP32 block (n <= 32): lane c solves
// B x = e_c through the interchanges, L and U; the result is the largest
// column sum, on every lane.
__device__ __noinline__ float inv_norm1_f32(const float* a, int n, const int* pv, int lane) {
  float cs = 0.f;
  if (lane < n) {
    float x[32];
#pragma unroll 1
    for (int ii = 0; ii < n; ++ii) x[ii] = ii == lane ? 1.f : 0.f;
#pragma unroll 1
    for (int kk = 0; kk < n; ++kk) {
      const int pk = pv[kk];
      if (pk != kk) {
        const float t = x[kk];
        x[kk] = x[pk];
        x[pk] = t;
      }
    }
#pragma unroll 1
    for (int ii = 1; ii < n; ++ii) {
      float sum = x[ii];
#pragma unroll 1
      for (int kk = 0; kk < ii; ++kk) sum = __fmaf_rn(-a[ii * n + kk], x[kk], sum);
      x[ii] = sum;
    }
#pragma unroll 1
    for (int ii = n - 1; ii >= 0; --ii) {
      float sum = x[ii];
#pragma unroll 1
      for (int kk = ii + 1; kk < n; ++kk) sum = __fmaf_rn(-a[ii * n + kk], x[kk], sum);
      x[ii] = __fdiv_rn(sum, a[ii * n + ii]);
    }
#pragma unroll 1
    for (int ii = 0; ii < n; ++ii) cs += fabsf(x[ii]);
  }
  for (int o = 16; o > 0; o >>= 1) cs = fmaxf(cs, __shfl_xor_sync(0xffffffffu, cs, o));
  return cs;
}

// ---- division by a pivot entry -------------------------------------------
// a / b correctly rounded from y = RN(1/b) and z, the rest of 1/b: q = a y +
// a z is within one ulp of a / b, a - b q is exact, and the correction by it
// rounds to RN(a / b) (Markstein's theorem: exact remainder, correctly rounded
// reciprocal).  Valid while no intermediate can underflow or overflow, which
// the exponent ranges below ensure; y = 0 marks a b outside of its range.
__device__ __forceinline__ void recip_rn(float b, float& y, float& z) {
  y = 0.f, z = 0.f;
  if (fabsf(b) >= 0x1p-40f && fabsf(b) <= 0x1p40f) {
    y = __frcp_rn(b);
    z = __fmul_rn(__fmaf_rn(-b, y, 1.f), y);
  }
}
__device__ __forceinline__ void recip_rn(double b, double& y, double& z) {
  y = 0.0, z = 0.0;
  if (fabs(b) >= 0x1p-300 && fabs(b) <= 0x1p300) {
    y = __drcp_rn(b);
    z = __dmul_rn(__fma_rn(-b, y, 1.0), y);
  }
}
__device__ __forceinline__ float div_recip(float a, float b, float y, float z) {
  const float q = __fmaf_rn(a, y, __fmul_rn(a, z));
  return __fmaf_rn(__fmaf_rn(-b, q, a), y, q);
}
__device__ __forceinline__ double div_recip(double a, double b, double y, double z) {
  const double q = __fma_rn(a, y, __dmul_rn(a, z));
  return __fma_rn(__fma_rn(-b, q, a), y, q);
}
__device__ __forceinline__ bool div_range(float a, float y) {
  return y != 0.f && fabsf(a) >= 0x1p-40f && fabsf(a) <= 0x1p40f;
}
__device__ __forceinline__ bool div_range(double a, double y) {
  const unsigned e = ((unsigned)__double2hiint(a) >> 20) & 0x7ff;
  return __double2hiint(y) != 0 && e >= 1023 - 300 && e < 1023 + 300;
}

// ---- FP32 pivot blocks held in registers -----------------------------------
// The block's entries are read up front by broadcast 16-byte loads (rows 8
// floats apart for N <= 8, else N), so that only the chain of operations itself
// is left; a size n below N costs a uniform branch per row.  Small blocks are
// taken by the class 2, 4, 6 or 8 that holds them, since a class for 8 alone
// spends a row's and a column's instructions on every size below (that and the
// cheaper reductions and copies of a finish: 392 to 376 ms at 3.0 million unknowns,
// 267 to 253 at tau 0.9).  Each routine gives every element the
// operations of its generic counterpart (ainv_right_row_sh, gepp_warp,
// inv_norm1_f32) in the same order, so the results are identical bit for bit.
// A 6 x 6 block, one warp alone: multiplier 1 900 cycles with the entries read
// where they are used, factorization with condition estimate 6 200.

template <int N>
__device__ __forceinline__ constexpr int lu_rows() {  // distance of the rows
  return N <= 8 ? 8 : N;
}
template <int N>
__device__ __forceinline__ void load_lu(const float* lu, float* L) {
#pragma unroll
  for (int a = 0; a < N; ++a)
#pragma unroll
    for (int c = 0; c < N; c += 4) {
      const float4 v = *reinterpret_cast<const float4*>(lu + a * lu_rows<N>() + c);
      L[a * N + c] = v.x;
      if (c + 1 < N) L[a * N + c + 1] = v.y;
      if (c + 2 < N) L[a * N + c + 2] = v.z;
      if (c + 3 < N) L[a * N + c + 3] = v.w;
    }
}

// r <- r (P^T L U)^{-1} for one row x[0, n), n <= N <= 8; the result goes,
// permuted, to the row m and (unless NULL) to mt with stride np.
template <int N>
__device__ __forceinline__ void mult_row_n(const float* lu, const float* ry, const float* rz, const int* perm, int n,
                                           const float* x, float* m, float* mt, int np) {
  float L[N * N], r[N], y[N], z[N];
  int c[N];
#pragma unroll
  for (int j = 0; j < N; ++j) r[j] = j < n ? x[j] : 0.f;
  load_lu<N>(lu, L);
#pragma unroll
  for (int j = 0; j < N; ++j) {
    y[j] = j < n ? ry[j] : 1.f;
    z[j] = j < n ? rz[j] : 0.f;
    c[j] = j < n ? perm[j] : 0;
  }
  bool ok = true;
#pragma unroll
  for (int q = 0; q < N; ++q)
    if (q < n) {  // x_q is complete: divide, then take it out of the columns to its right
      ok = ok && div_range(r[q], y[q]);
      r[q] = div_recip(r[q], L[q * N + q], y[q], z[q]);
#pragma unroll
      for (int j = q + 1; j < N; ++j) r[j] = msub<float>(r[j], r[q], L[q * N + j]);
    }
  if (!ok) {  // a dividend or a divisor outside of the range: divide
#pragma unroll
    for (int j = 0; j < N; ++j) r[j] = j < n ? x[j] : 0.f;
#pragma unroll
    for (int q = 0; q < N; ++q)
      if (q < n) {
        r[q] = __fdiv_rn(r[q], L[q * N + q]);
#pragma unroll
        for (int j = q + 1; j < N; ++j) r[j] = msub<float>(r[j], r[q], L[q * N + j]);
      }
  }
#pragma unroll
  for (int j = N - 2; j >= 0; --j) {
#pragma unroll
    for (int q = j + 1; q < N; ++q)
      if (q < n) r[j] = msub<float>(r[j], r[q], L[q * N + j]);
  }
#pragma unroll
  for (int j = 0; j < N; ++j)
    if (j < n) {
      m[c[j]] = r[j];
      if (mt) mt[c[j] * np] = r[j];
    }
}

__device__ __forceinline__ void mult_row_small(const float* lu, const float* ry, const float* rz, const int* perm,
                                               int n, const float* x, float* m, float* mt, int np) {
  if (n <= 2)
    mult_row_n<2>(lu, ry, rz, perm, n, x, m, mt, np);
  else if (n <= 4)
    mult_row_n<4>(lu, ry, rz, perm, n, x, m, mt, np);
  else if (n <= 6)
    mult_row_n<6>(lu, ry, rz, perm, n, x, m, mt, np);
  else
    mult_row_n<8>(lu, ry, rz, perm, n, x, m, mt, np);
}

// GEPP of the n x n row-major FP32 block at src (n <= N), row i in lane i's
// registers: the pivot is the largest |a_ik| (the lowest position on ties)
// found by a warp max-reduction of the keys and a ballot, while every lane
// forms the reciprocal of its own candidate, so that the multipliers need no
// division.  Rows are not exchanged: pos is the position that a lane's row has
// come to.  The factored block goes to lu (rows N apart), its diagonal's
// reciprocals to ry and rz, the interchanges to pvs and gpiv, the rows' order
// to perm.  Then, on every lane, ||B^{-1}||_1 by solving B x = e_c on lane c.
// False when a pivot column is exactly zero.
template <int N>
__device__ __noinline__ bool gepp_cond(const float* src, int n, float* lu, float* ry, float* rz, int* pvs, int* perm,
                                       int32_t* gpiv, int lane, float* inv1) {
  constexpr int S = lu_rows<N>();
  float r[N];
#pragma unroll
  for (int j = 0; j < N; ++j) r[j] = lane < n && j < n ? src[lane * n + j] : 0.f;
  int pos = lane < n ? lane : 64;
  float yd = 0.f, zd = 0.f;  // the reciprocal of the pivot that a lane's row supplied
  bool done = lane >= n;
#pragma unroll
  for (int k = 0; k < N; ++k)
    if (k < n) {
      const unsigned key = done ? 0u : (unsigned)abs_key(r[k]) + 1u;
      float yc, zc;
      recip_rn(r[k], yc, zc);
      const unsigned mk = __reduce_max_sync(0xffffffffu, key);
      if (mk <= 1u) return false;  // the pivot column is exactly zero
      unsigned who = __ballot_sync(0xffffffffu, key == mk);
      if (who & (who - 1)) {
        const int pm = (int)__reduce_min_sync(0xffffffffu, key == mk ? (unsigned)pos : 64u);
        who = __ballot_sync(0xffffffffu, key == mk && pos == pm);
      }
      const int from = __ffs(who) - 1;
      float u[N];
#pragma unroll
      for (int j = k; j < N; ++j) u[j] = __shfl_sync(0xffffffffu, r[j], from);
      const float yp = __shfl_sync(0xffffffffu, yc, from), zp = __shfl_sync(0xffffffffu, zc, from);
      const int p = __shfl_sync(0xffffffffu, pos, from);
      if (lane == from) {
        pos = k;
        yd = yp, zd = zp;
        done = true;
      } else if (pos == k) {
        pos = p;
      }
      if (lane == 0) {
        gpiv[k] = p;
        pvs[k] = p;
      }
      if (!done) {
        const float l = div_range(r[k], yp) ? div_recip(r[k], u[k], yp, zp) : __fdiv_rn(r[k], u[k]);
        r[k] = l;
#pragma unroll
        for (int j = k + 1; j < N; ++j) r[j] = msub<float>(r[j], l, u[j]);
      }
    }
  if (lane < n) {
    perm[pos] = lane;
    ry[pos] = yd;
    rz[pos] = zd;
#pragma unroll
    for (int j = 0; j < N; ++j) lu[pos * S + j] = r[j];
  }
  __syncwarp();
  // x = P e_c: one at the place that row c was brought to (lanes without a
  // column follow lane 0's kind, so that they stay on the common path)
  float cs = 0.f;
  float x[N];
  const int pc = lane < n ? pos : 0;
#pragma unroll
  for (int i = 0; i < N; ++i) x[i] = i == pc ? 1.f : 0.f;
  if (N <= 8) {
    float L[N * N], y[N], z[N];
    load_lu<N>(lu, L);
#pragma unroll
    for (int i = 0; i < N; ++i) y[i] = i < n ? ry[i] : 1.f, z[i] = i < n ? rz[i] : 0.f;
#pragma unroll
    for (int i = 1; i < N; ++i) {
#pragma unroll
      for (int k = 0; k < i; ++k)
        if (i < n) x[i] = __fmaf_rn(-L[i * N + k], x[k], x[i]);
    }
#pragma unroll
    for (int i = N - 1; i >= 0; --i)
      if (i < n) {
#pragma unroll
        for (int k = i + 1; k < N; ++k)
          if (k < n) x[i] = __fmaf_rn(-L[i * N + k], x[k], x[i]);
        x[i] = div_range(x[i], y[i]) ? div_recip(x[i], L[i * (N + 1)], y[i], z[i])
                                     : __fdiv_rn(x[i], L[i * (N + 1)]);
      }
  } else {
#pragma unroll
    for (int i = 1; i < N; ++i)
      if (i < n) {
#pragma unroll
        for (int k4 = 0; k4 < i; k4 += 4) {
          const float4 v = *reinterpret_cast<const float4*>(lu + i * S + k4);
          const float l[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int k = k4; k < i && k < k4 + 4; ++k) x[i] = __fmaf_rn(-l[k - k4], x[k], x[i]);
        }
      }
#pragma unroll
    for (int i = N - 1; i >= 0; --i)
      if (i < n) {
#pragma unroll
        for (int k4 = (i + 1) & ~3; k4 < N; k4 += 4) {
          const float4 v = *reinterpret_cast<const float4*>(lu + i * S + k4);
          const float l[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int k = k4; k < N && k < k4 + 4; ++k)
            if (k > i && k < n) x[i] = __fmaf_rn(-l[k - k4], x[k], x[i]);
        }
        x[i] = div_range(x[i], ry[i]) ? div_recip(x[i], lu[i * (S + 1)], ry[i], rz[i])
                                      : __fdiv_rn(x[i], lu[i * (S + 1)]);
      }
  }
#pragma unroll
  for (int i = 0; i < N; ++i)
    if (i < n) cs += fabsf(x[i]);
  if (lane >= n) cs = 0.f;
  // (NaN in every lane, which takes 32 columns, stays NaN)
  *inv1 = N == 32 && __all_sync(0xffffffffu, cs != cs) ? cs : warp_max_f(cs);
  return true;
}

__device__ __forceinline__ bool gepp_cond_small(const float* src, int n, float* lu, float* ry, float* rz, int* pvs,
                                                int* perm, int32_t* gpiv, int lane, float* inv1) {
  return n <= 2   ? gepp_cond<2>(src, n, lu, ry, rz, pvs, perm, gpiv, lane, inv1)
         : n <= 4 ? gepp_cond<4>(src, n, lu, ry, rz, pvs, perm, gpiv, lane, inv1)
         : n <= 6 ? gepp_cond<6>(src, n, lu, ry, rz, pvs, perm, gpiv, lane, inv1)
                  : gepp_cond<8>(src, n, lu, ry, rz, pvs, perm, gpiv, lane, inv1);
}

// The same for any n and either type, in loops, the row held in shared memory
// at w[j * nw].
template <typename T>
__device__ __noinline__ void mult_row_loop(const T* lu, const T* ry, const T* rz, const int* perm, int n, T* w, int nw,
                                           T* m, T* mt, int np) {
#pragma unroll 1
  for (int j = 0; j < n; ++j) w[j * nw] = m[j];
#pragma unroll 1
  for (int j = 0; j < n; ++j) {
    T s = w[j * nw];
#pragma unroll 4
    for (int q = 0; q < j; ++q) s = msub<T>(s, w[q * nw], lu[q * n + j]);
    w[j * nw] = div_range(s, ry[j]) ? div_recip(s, lu[j * n + j], ry[j], rz[j]) : div_rn<T>(s, lu[j * n + j]);
  }
#pragma unroll 1
  for (int j = n - 2; j >= 0; --j) {
    T s = w[j * nw];
#pragma unroll 4
    for (int q = j + 1; q < n; ++q) s = msub<T>(s, w[q * nw], lu[q * n + j]);
    w[j * nw] = s;
  }
#pragma unroll 1
  for (int j = 0; j < n; ++j) {
    const int c = perm[j];
    m[c] = w[j * nw];
    if (mt) mt[c * np] = w[j * nw];
  }
}

// perm from the interchanges pvs of a block of n <= PVMAX rows (pvs and perm in
// shared memory).
__device__ __noinline__ void perm_of(const int* pvs, int n, int* perm, int lane) {
  if (lane == 0) {
#pragma unroll 1
    for (int k = 0; k < n; ++k) perm[k] = k;
#pragma unroll 1
    for (int k = 0; k < n; ++k) {
      const int p = pvs[k], t = perm[k];
      perm[k] = perm[p];
      perm[p] = t;
    }
  }
  __syncwarp();
}

// ---- the drop rule of an FP64 block, decided in FP32 where that is certain --
// |v| as an FP32 value from the upper bits of the FP64 one (an FP64 operation
// or conversion takes 64 to 100 cycles on this part); false outside 2^+-55.
__device__ __forceinline__ bool abs_f32(double v, float& f) {
  const unsigned h = (unsigned)__double2hiint(v) & 0x7fffffffu;
  f = __int_as_float((int)(((h - (896u << 20)) << 3) | ((unsigned)__double2loint(v) >> 29)));
  if (h - ((1023u - 55u) << 20) < (110u << 20)) return true;
  f = 0.f;
  return h == 0 && __double2loint(v) == 0;
}
// s: the FP32 sum of squares of n <= 4096 entries, ok: all were in range; none:
// the FP64 tolerance is zero (its FP32 value t also is when it is below 2^-150).
// 1: dropped, 0: kept, -1: too near the threshold.  Truncation, the sum and the
// threshold are off by less than (n + 8) 2^-23 together, the margin by 2^-10.
__device__ __forceinline__ int drop_f32(float s, bool ok, int m, int n, float t, bool none) {
  const float thr = t * (float)m * (float)n, thr2 = thr * thr;
  if (!ok || !(thr2 == 0.f ? none : thr2 >= 1e-30f) || !(thr2 <= 1e30f)) return -1;
  if (s * (1.f + 0x1p-10f) < thr2) return 1;
  if (s * (1.f - 0x1p-10f) >= thr2) return 0;
  return -1;
}

// ---------------------------------------------------------------------------
// A published record is brought on chip by the warp's own asynchronous copies
// (16 bytes a lane through L2, so that no line of L1 can be stale), which need
// no fence between proxies: from a publication to the record in the
// dependant's shared memory 1.2 us, against 2.3 us with a bulk copy completing
// on an mbarrier (1.5 KB records, one warp handing on to the next).
__device__ __forceinline__ void record_fetch(void* dst, const unsigned char* src, int bytes, int lane) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
#pragma unroll 1
  for (int e = lane * 16; e < bytes; e += 512)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + e), "l"(src + e) : "memory");
  asm volatile("cp.async.commit_group;" ::: "memory");
}
// All copies but the youngest `keep` groups have arrived, for the whole warp.
template <int KEEP>
__device__ __forceinline__ void record_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(KEEP) : "memory");
  __syncwarp();
}

__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

// The published word of a row: acquiring polls with a short backoff, the abort
// word and the time budget looked at only every 16th poll.  0 when the wait
// gave up.
__device__ __forceinline__ unsigned long long wait_word(const unsigned long long* w, int* abort,
                                                        unsigned long long limit, int* st) {
  unsigned long long v = ld_acquire_u64(w);
  if (v == 0) {
    const unsigned long long t0 = global_ns();
    unsigned nsl = 16;
#pragma unroll 1
    for (unsigned it = 1;; ++it) {
      __nanosleep(nsl);
      if (nsl < 128) nsl <<= 1;
      v = ld_acquire_u64(w);
      if (v != 0) break;
      if ((it & 15) == 0) {
        if (*((volatile int*)abort) != 0) return 0;
        if (global_ns() - t0 > limit) {
          dev_fail(st, DEV_ETIMEOUT);
          atomicExch(abort, 1);
          return 0;
        }
      }
    }
  }
  return v;
}

// Ascending bitonic sort of a[0, n2) (n2 a power of two) by one warp.
__device__ void warp_bitonic_sort(unsigned long long* a, int n2, int lane) {
#pragma unroll 1
  for (int k = 2; k <= n2; k <<= 1)
#pragma unroll 1
    for (int j = k >> 1; j > 0; j >>= 1) {
#pragma unroll 1
      for (int x = lane; x < n2; x += 32) {
        const int y = x ^ j;
        if (y > x) {
          const unsigned long long u = a[x], v = a[y];
          if ((u > v) == ((x & k) == 0)) {
            a[x] = v;
            a[y] = u;
          }
        }
      }
      __syncwarp();
    }
}

// lfil (Section 3 dropping rule with the lfil bound of the paper's ARMS
// parameters): of the n candidate slots cand[], keep the lfil with the
// largest norm keys, lower column first on equal keys; the others become
// SL_DEAD and cand[] is compacted to the kept ones.  The lfil-th largest key
// is found in registers when the keys are FP32 norms and n <= 256, else by
// radix selection, 8 bits a pass from the top (keybytes passes: the keys are
// the bit patterns of non-negative FP64 or FP32 norms, so their integer order
// is their value order).  Returns the number kept.
__device__ __noinline__ int lfil_cut(int* cand, int n, int lfil, const long long* sf2, const int* scol, int* sstate, int* hist,
                        int keybytes, int lane) {
  if (lfil < 0 || n <= lfil) return n;
  if (lfil == 0) {
#pragma unroll 1
    for (int c = lane; c < n; c += 32) sstate[cand[c]] = SL_DEAD;
    __syncwarp();
    return 0;
  }
  if (keybytes == 4 && n <= 256) {
    // keys of 31 bits, up to 8 a lane in registers: the lfil-th largest is
    // built from the top, bits kept if lfil keys reach the value with them
    unsigned kq[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) kq[u] = lane + 32 * u < n ? (unsigned)sf2[cand[lane + 32 * u]] + 1u : 0u;
    unsigned thr = 0;
#pragma unroll 1
    for (int bit = 30; bit >= 0; bit -= 2) {  // two bits at a time, three counts of at most 256 in one sum
      const unsigned t1 = thr | (1u << bit), t2 = thr | (2u << bit), t3 = thr | (3u << bit);
      unsigned c = 0;
#pragma unroll
      for (int u = 0; u < 8; ++u)
        c += (kq[u] >= t1 ? 1u : 0u) + (kq[u] >= t2 ? 1u << 10 : 0u) + (kq[u] >= t3 ? 1u << 20 : 0u);
      c = __reduce_add_sync(0xffffffffu, c);
      if ((int)(c >> 20) >= lfil)
        thr = t3;
      else if ((int)(c >> 10 & 1023) >= lfil)
        thr = t2;
      else if ((int)(c & 1023) >= lfil)
        thr = t1;
    }
    int above = 0, equal = 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) above += kq[u] > thr, equal += kq[u] == thr;
    above = __reduce_add_sync(0xffffffffu, above);
    equal = __reduce_add_sync(0xffffffffu, equal);
    const int want = lfil - above;  // of the keys equal to thr, those with the lowest columns
    unsigned keep = 0;
    int q[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int c = lane + 32 * u;
      q[u] = c < n ? cand[c] : -1;
      bool k = kq[u] > thr;
      if (kq[u] == thr && c < n) {
        int rank = 0;
        if (equal > want) {
          const int col = scol[q[u]];
#pragma unroll 1
          for (int c2 = 0; c2 < n; ++c2) {
            const int q2 = cand[c2];
            if ((unsigned)sf2[q2] + 1u == thr && scol[q2] < col) ++rank;
          }
        }
        k = rank < want;
      }
      if (c < n && !k) sstate[q[u]] = SL_DEAD;
      keep |= (unsigned)k << u;
    }
    __syncwarp();
    int kept = 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const unsigned bk = __ballot_sync(0xffffffffu, keep >> u & 1);
      if (keep >> u & 1) cand[kept + __popc(bk & ((1u << lane) - 1u))] = q[u];
      kept += __popc(bk);
    }
    __syncwarp();
    return kept;
  }
  unsigned long long prefix = 0, pmask = 0;
  int want = lfil;  // keys still to take at or below the current prefix
#pragma unroll 1
  for (int d = keybytes - 1; d >= 0; --d) {
    const int shift = 8 * d;
#pragma unroll 1
    for (int b = lane; b < 256; b += 32) hist[b] = 0;
    __syncwarp();
#pragma unroll 1
    for (int base = 0; base < n; base += 32) {
      const int c = base + lane;
      int bin = -1;
      if (c < n) {
        const unsigned long long key = (unsigned long long)sf2[cand[c]];
        if ((key & pmask) == prefix) bin = (int)((key >> shift) & 255);
      }
      // lanes with the same bin add once (keys of one row crowd a few bins)
      const unsigned peers = __match_any_sync(0xffffffffu, bin);
      if (bin >= 0 && (__ffs(peers) - 1) == lane) atomicAdd(&hist[bin], __popc(peers));
    }
    __syncwarp();
    // lane l holds bins 255 - 8 l - u, u = 0..7 (the highest bins first)
    int cnt[8];
    int s = 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      cnt[u] = hist[255 - 8 * lane - u];
      s += cnt[u];
    }
    int incl = s;
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    const int excl = incl - s;
    int bin = -1, above = 0;
    if (excl < want && want <= incl) {
      int run = excl;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        if (bin < 0 && run + cnt[u] >= want) {
          bin = 255 - 8 * lane - u;
          above = run;
        }
        run += cnt[u];
      }
    }
    const unsigned who = __ballot_sync(0xffffffffu, bin >= 0);
    const int src = __ffs(who) - 1;
    bin = __shfl_sync(0xffffffffu, bin, src);
    above = __shfl_sync(0xffffffffu, above, src);
    want -= above;
    prefix |= (unsigned long long)bin << shift;
    pmask |= 255ull << shift;
    __syncwarp();
  }
  // keys above prefix are kept; of the keys equal to it, the `want` with the
  // lowest columns.  Every cut slot is marked first (the tie ranks read the
  // whole list), then the list is compacted.
#pragma unroll 1
  for (int c = lane; c < n; c += 32) {
    const int q = cand[c];
    const unsigned long long key = (unsigned long long)sf2[q];
    bool keep = key > prefix;
    if (key == prefix) {
      const int col = scol[q];
      int rank = 0;
#pragma unroll 1
      for (int c2 = 0; c2 < n; ++c2) {
        const int q2 = cand[c2];
        if ((unsigned long long)sf2[q2] == prefix && scol[q2] < col) ++rank;
      }
      keep = rank < want;
    }
    if (!keep) sstate[q] = SL_DEAD;
  }
  __syncwarp();
  int kept = 0;
#pragma unroll 1
  for (int base = 0; base < n; base += 32) {
    const int c = base + lane;
    const int q = c < n ? cand[c] : -1;
    const bool keep = q >= 0 && sstate[q] != SL_DEAD;
    __syncwarp();
    const unsigned bk = __ballot_sync(0xffffffffu, keep);
    if (keep) cand[kept + __popc(bk & ((1u << lane) - 1u))] = q;
    kept += __popc(bk);
    __syncwarp();
  }
  return kept;
}

// The kept blocks of one part in column order: srt[p] = col << 32 | slot for
// p < k (space for the next power of two).
__device__ __noinline__ void sort_by_column(const int* cand, int k, const int* scol, unsigned long long* srt, int lane) {
  int n2 = 1;
  while (n2 < k) n2 <<= 1;
  if (k <= 64) {  // the keys are distinct: each goes to its rank
    const int qa = lane < k ? cand[lane] : 0, qb = 32 + lane < k ? cand[32 + lane] : 0;
    const unsigned ca = lane < k ? (unsigned)scol[qa] : ~0u, cb = 32 + lane < k ? (unsigned)scol[qb] : ~0u;
    int ra = 0, rb = 0;
#pragma unroll 4
    for (int j = 0; j < 32; ++j) {
      if (j >= k) break;
      const unsigned c = __shfl_sync(0xffffffffu, ca, j);
      ra += c < ca, rb += c < cb;
    }
#pragma unroll 4
    for (int j = 32; j < 64; ++j) {
      if (j >= k) break;
      const unsigned c = __shfl_sync(0xffffffffu, cb, j - 32);
      ra += c < ca, rb += c < cb;
    }
    if (lane < k) srt[ra] = ((unsigned long long)ca << 32) | (unsigned)qa;
    if (32 + lane < k) srt[rb] = ((unsigned long long)cb << 32) | (unsigned)qb;
    __syncwarp();
    return;
  }
  for (int p = lane; p < n2; p += 32)
    srt[p] = p < k ? ((unsigned long long)(unsigned)scol[cand[p]] << 32) | (unsigned)cand[p] : ~0ull;
  __syncwarp();
  warp_bitonic_sort(srt, n2, lane);
}

// Copy up to 32 blocks (lane p: sz values at src + so to dst + dof), eight
// lanes to a block and eight loads in flight a lane.
template <typename T>
__device__ __noinline__ void copy_blocks(int n, int sz, int so, long long dof, const T* __restrict__ src,
                                            T* __restrict__ dst, int lane) {
  if (__reduce_max_sync(0xffffffffu, lane < n ? sz : 0) <= 4) {  // a lane a block
    T v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (lane < n && u < sz) v[u] = src[so + u];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (lane < n && u < sz) dst[dof + u] = v[u];
    return;
  }
  const int g = lane >> 3, a = lane & 7;
#pragma unroll 1
  for (int p0 = 0; p0 < n; p0 += 4) {
    const int p = min(p0 + g, 31);
    const int s = __shfl_sync(0xffffffffu, sz, p), o = __shfl_sync(0xffffffffu, so, p);
    const long long d = __shfl_sync(0xffffffffu, dof, p);
    const int m = p0 + g < n ? s : 0;
#pragma unroll 1
    for (int e0 = a; e0 < m; e0 += 64) {
      T v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (e0 + 8 * u < m) v[u] = src[o + e0 + 8 * u];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (e0 + 8 * u < m) dst[d + e0 + 8 * u] = v[u];
    }
  }
}

// A factored pivot block (rows S apart) and the reciprocals of its diagonal into
// a record.
template <typename TL>
__device__ __noinline__ void put_pivot(const TL* __restrict__ lu, int S, int n, TL* __restrict__ o,
                                       TL* __restrict__ rcp, int lane) {
  if (S == n) {
#pragma unroll 4
    for (int e = lane; e < n * n; e += 32) o[e] = lu[e];
  } else {
#pragma unroll 1
    for (int e = lane; e < n * n; e += 32) {
      const int a = e / n;
      o[e] = lu[a * S + e - a * n];
    }
  }
#pragma unroll 1
  for (int a = lane; a < n; a += 32) {
    TL y, z;
    recip_rn(lu[a * (S + 1)], y, z);
    rcp[a] = y;
    rcp[n + a] = z;
  }
}

// One chunk of U blocks of a step: w(:, j) -= m U_kj for the chunk's columns and
// the rows [row0, row0 + ni) of the working row, whose multiplier is in mt.
// qinfo[q] = {workspace offset of the target, first column, columns, 1 if the
// target is new (its old values are zeros)}, cmap[c] = the block of column c.
// FP32: a lane takes a column, so that a value of U and the target's address
// serve ni rows, and the multiplier comes as broadcast 16-byte loads.
__device__ __forceinline__ void update_columns(const int4* qinfo, const unsigned char* cmap, int cols,
                                               const float* mt, int row0, int ni, int nk, int np, const float* U,
                                               float* wv, int lane) {
#pragma unroll 1
  for (int c = lane; c < cols; c += 32) {
    const int4 I = qinfo[cmap[c]];
    const int jj = c - I.y, nj = I.z;
    const float* u = U + nk * I.y + jj;
    float* z = wv + I.x + row0 * nj + jj;
#pragma unroll 1
    for (int a0 = 0; a0 < ni; a0 += 8) {
      float acc[8];
      if (I.w) {
#pragma unroll
        for (int a = 0; a < 8; ++a) acc[a] = 0.f;
      } else {
#pragma unroll
        for (int a = 0; a < 8; ++a)
          if (a0 + a < ni) acc[a] = z[(a0 + a) * nj];
      }
      const float* m = mt + a0;
#pragma unroll 2
      for (int r = 0; r < nk; ++r) {
        const float ur = u[r * nj];
        const float4 m0 = *reinterpret_cast<const float4*>(m + r * np);
        acc[0] = __fmaf_rn(-m0.x, ur, acc[0]);
        acc[1] = __fmaf_rn(-m0.y, ur, acc[1]);
        acc[2] = __fmaf_rn(-m0.z, ur, acc[2]);
        acc[3] = __fmaf_rn(-m0.w, ur, acc[3]);
        if (a0 + 4 < ni) {
          const float4 m1 = *reinterpret_cast<const float4*>(m + r * np + 4);
          acc[4] = __fmaf_rn(-m1.x, ur, acc[4]);
          acc[5] = __fmaf_rn(-m1.y, ur, acc[5]);
          acc[6] = __fmaf_rn(-m1.z, ur, acc[6]);
          acc[7] = __fmaf_rn(-m1.w, ur, acc[7]);
        }
      }
#pragma unroll
      for (int a = 0; a < 8; ++a)
        if (a0 + a < ni) z[(a0 + a) * nj] = acc[a];
    }
  }
}
// FP64: the operations themselves are the cost (64 cycles each for any number
// of lanes), so the elements are dealt out evenly, two a lane in flight.
__device__ __forceinline__ void update_columns(const int4* qinfo, const unsigned char* cmap, int cols,
                                               const double* mt, int row0, int ni, int nk, int np, const double* U,
                                               double* wv, int lane) {
  const int total = ni * cols;
  const float rc = 1.f / (float)cols;
#pragma unroll 1
  for (int e = lane; e < total; e += 32) {
    int a = (int)((float)e * rc);  // e / cols, corrected
    int c = e - a * cols;
    if (c < 0) --a, c += cols;
    if (c >= cols) ++a, c -= cols;
    const int4 I = qinfo[cmap[c]];
    const int jj = c - I.y, nj = I.z;
    const double* u = U + nk * I.y + jj;
    double* z = wv + I.x + (row0 + a) * nj + jj;
    double acc = I.w ? 0.0 : *z;
    const double* m = mt + a;
#pragma unroll 1
    for (int r = 0; r < nk; ++r) acc = msub<double>(acc, m[r * np], u[r * nj]);
    *z = acc;
  }
}

// One chunk of U blocks of any sizes (lane q: block q's target offset, first
// column and columns; missing: the target is new), the multiplier m row-major:
// lanes over the flattened elements, four per lane in flight.  A record that
// is not staged is read through L2.
template <typename T>
__device__ __noinline__ void update_general(CopyTab& tab, int nq, int off, int cst, int nj, bool missing, int ni,
                                            int nk, const T* m, const T* rval, bool staged, T* wv, int lane) {
  const int sz = ni * nj;
  if (missing) {
    T* z = wv + off;
#pragma unroll 4
    for (int e = 0; e < sz; ++e) z[e] = (T)0;
  }
  int incl = sz;
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  const int total = __shfl_sync(0xffffffffu, incl, 31);
  tab.qpre[lane] = incl - sz;
  if (lane == 31) tab.qpre[32] = total;
  tab.qoff[lane] = off;
  tab.quo[lane] = nk * cst;
  tab.qnj[lane] = nj;
  __syncwarp();
#pragma unroll 1
  for (int e0 = lane; e0 < total; e0 += 128) {
    T acc[4];
    T* dst[4];
    int a4[4], jj4[4], nj4[4], uo4[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = e0 + 32 * u;
      dst[u] = nullptr;
      if (e < total) {
        int lo = 0, hi = nq - 1;  // block tq with qpre[tq] <= e < qpre[tq + 1]
        while (lo < hi) {
          const int mid = (lo + hi + 1) >> 1;
          if (tab.qpre[mid] <= e)
            lo = mid;
          else
            hi = mid - 1;
        }
        const int njt = tab.qnj[lo];
        const int local = e - tab.qpre[lo];
        a4[u] = local / njt;
        jj4[u] = local - a4[u] * njt;
        nj4[u] = njt;
        uo4[u] = tab.quo[lo];
        dst[u] = wv + tab.qoff[lo] + local;
        acc[u] = *dst[u];
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (!dst[u]) continue;
      const T* U = rval + uo4[u];
      T av = acc[u];
      if (staged) {
#pragma unroll 1
        for (int r = 0; r < nk; ++r) av = msub<T>(av, m[a4[u] * nk + r], U[r * nj4[u] + jj4[u]]);
      } else {
#pragma unroll 8
        for (int r = 0; r < nk; ++r) av = msub<T>(av, m[a4[u] * nk + r], __ldcg(U + r * nj4[u] + jj4[u]));
      }
      *dst[u] = av;
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(256, 1)
    k_ilut(VBView<T> A, IlutGeom g, Workspace ws, T* __restrict__ wvals_all, Pools P, T* __restrict__ lval,
           unsigned char* __restrict__ upool, const int64_t* __restrict__ dgoff, double* __restrict__ dg,
           float* __restrict__ dg32, int32_t* __restrict__ piv, int32_t* __restrict__ ptag, int mixed,
           double cond_thr, double t, int lfil, unsigned long long wait_limit, int* st) {
  extern __shared__ __align__(128) unsigned char ilut_sm[];
  constexpr bool F32 = std::is_same<T, float>::value;
  constexpr int TS = (int)sizeof(T);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  unsigned char* const wb = ilut_sm + (size_t)warp * g.bytes;
  IlutMisc<T>& M = *reinterpret_cast<IlutMisc<T>*>(wb + g.o_misc);
  CopyTab& tab = *reinterpret_cast<CopyTab*>(M.buf);
  unsigned char* const cmap = reinterpret_cast<unsigned char*>(M.buf);
  int4* const qinfo = reinterpret_cast<int4*>(M.buf + MCOLS / 4);
  unsigned char* const stage0 = wb + g.o_stage;
  unsigned char* const stage1 = stage0 + g.stage;
  T* const sh_vals = reinterpret_cast<T*>(wb + g.o_vals);
  int* const sh_keys = reinterpret_cast<int*>(wb + g.o_keys);
  int* const sh_hpos = reinterpret_cast<int*>(wb + g.o_hpos);
  int* const sh_scol = reinterpret_cast<int*>(wb + g.o_scol);
  int* const sh_soff = reinterpret_cast<int*>(wb + g.o_soff);
  int* const sh_sst = reinterpret_cast<int*>(wb + g.o_sst);
  long long* const sh_sf2 = reinterpret_cast<long long*>(wb + g.o_sf2);
  int* const sh_sncl = reinterpret_cast<int*>(wb + g.o_sncl);
  int* const lc = reinterpret_cast<int*>(wb + g.o_lc);  // pending L columns (INT_MAX when processed)
  int* const ls = reinterpret_cast<int*>(wb + g.o_ls);  // their slots
  const int64_t wid = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;
  const int VSH = g.vbytes / TS;
  const float tf = (float)t, condf = (float)cond_thr;
  int* const gkeys = ws.keys + wid * ws.ht;
#pragma unroll 1
  for (int k = lane; k < ws.ht; k += 32) gkeys[k] = -1;
#pragma unroll 1
  for (int k = lane; k < g.hash; k += 32) sh_keys[k] = -1;
  __syncwarp();

  for (;;) {
    long long row = 0;
    if (lane == 0) {
      row = (long long)atomicAdd(P.ctr + 4, 1ULL);
      if (row >= P.nticket)
        row = A.nbr;
      else if (P.order)
        row = P.order[row];
    }
    row = __shfl_sync(0xffffffffu, row, 0);
    if (row >= A.nbr) break;
    const int64_t i = row;
    int maxdep = 0;  // the deepest row waited on
    const int ni = A.rsz[i];
    const int64_t b0 = A.bptr[i], b1 = A.bptr[i + 1];
    const int64_t v0 = A.voff[b0], nv = A.voff[b1] - v0;
    const int nb = (int)(b1 - b0);
    // The working row lives in shared memory when it leaves room for fill; a
    // row whose fill outgrows that moves to the warp's global workspace.
    bool in_sh = nb <= g.slots / 2 && nv <= VSH * 3 / 4;
    int status_local = 0;
    int* keys;
    int* hpos;
    int* scol;
    int* soff;
    int* sstate;
    long long* sf2;
    int* sncl;
    T* wv;
    int smax_c;
    int64_t vmax_c;
    uint32_t hmask;
    if (in_sh) {
      keys = sh_keys, hpos = sh_hpos, scol = sh_scol, soff = sh_soff, sstate = sh_sst, sf2 = sh_sf2;
      sncl = sh_sncl;
      wv = sh_vals;
      smax_c = g.slots, vmax_c = VSH, hmask = (uint32_t)g.hash - 1;
    } else {
      keys = gkeys, hpos = ws.hpos + wid * ws.smax, scol = ws.scol + wid * ws.smax;
      soff = ws.soff + wid * ws.smax, sstate = ws.sstate + wid * ws.smax, sf2 = ws.sf2 + wid * ws.smax;
      sncl = ws.sncl + wid * ws.smax;
      wv = wvals_all + wid * ws.vmax;
      smax_c = ws.smax, vmax_c = ws.vmax, hmask = (uint32_t)ws.ht - 1;
    }
    // the row's slots, values and pending L columns so far, and the slot of
    // its diagonal block: the same in every lane
    int ns = 0, nl = 0, dslot = -1;
    long long nval = 0;
    int ask_s = 0;  // what an overflowing row asked for
    long long ask_v = 0;
    // ---- load row i of A into the workspace: slot q is the row's block q
    // and the values arrive as one contiguous copy; columns left of the
    // diagonal enter the list of pending L columns
    if (nb > smax_c || nv > vmax_c) {
      status_local = DEV_OVERFLOW;
      ask_s = nb;
      ask_v = nv;
    } else {
#pragma unroll 1
      for (int base = 0; base < nb; base += 32) {
        const int slot = base + lane;
        int32_t J = INT_MAX;
        if (slot < nb) {
          const int64_t b = b0 + slot;
          J = A.bcol[b];
          scol[slot] = J;
          soff[slot] = (int)(A.voff[b] - v0);
          sstate[slot] = SL_LIVE;
          sncl[slot] = A.rsz[J];
          hpos[slot] = ws_place(keys, hmask, slot, J);  // the table holds 2 smax positions
        }
        const unsigned low = __ballot_sync(0xffffffffu, J < i), dia = __ballot_sync(0xffffffffu, J == i);
        if (J < i) {
          const int q = nl + __popc(low & lt);
          if (q < g.lcap) {
            lc[q] = J;
            ls[q] = slot;
          }
        }
        nl += __popc(low);
        if (dia) dslot = base + __ffs(dia) - 1;
      }
      warp_copy(wv, A.val + v0, nv, lane);
      ns = nb;
      nval = nv;
    }
    __syncwarp();
    // stage buffer bookkeeping, the same in every lane: the column whose
    // record a buffer holds or is being copied into (-1: free, and no copy into
    // it in flight: a step frees only the buffers of its own record, so that
    // one fetched ahead stays known across a step that reads its record in place)
    int btag0 = -1, btag1 = -1;
    int64_t last = -1;
    // ---- eliminate the L part in ascending column order (including fill)
    while (status_local == 0) {
      // the next pending L column and the one after it: from the list while
      // it has not overflowed, else by a scan of the workspace slots
      int c1 = INT_MAX, s1 = -1, p1 = -1, c2 = INT_MAX;
      if (nl <= g.lcap) {
#pragma unroll 1
        for (int q = lane; q < nl; q += 32) {
          const int c = lc[q];
          if (c < c1) {
            c2 = c1;
            c1 = c;
            p1 = q;
          } else if (c < c2) {
            c2 = c;
          }
        }
        if (p1 >= 0) s1 = ls[p1];
      } else {
#pragma unroll 1
        for (int sidx = lane; sidx < ns; sidx += 32) {
          const int c = scol[sidx];
          if (sstate[sidx] == SL_LIVE && c > last && c < i) {
            if (c < c1) {
              c2 = c1;
              c1 = c;
              s1 = sidx;
            } else if (c < c2) {
              c2 = c;
            }
          }
        }
      }
      const int kmin = __reduce_min_sync(0xffffffffu, c1);
      if (kmin == INT_MAX) break;
      const int owner = __ffs(__ballot_sync(0xffffffffu, c1 == kmin)) - 1;
      const int sk = __shfl_sync(0xffffffffu, s1, owner);
      const int knext = __reduce_min_sync(0xffffffffu, lane == owner ? c2 : c1);
      if (lane == owner && p1 >= 0) lc[p1] = INT_MAX;
      const int64_t k = kmin;
      last = k;
      const int nk = A.rsz[k];
      // ---- row k's record: already fetched ahead into a stage buffer, or
      // fetched now (a bounded wait for its word, then the copies); a record
      // too large for a buffer is read in place.  The word of the next pending
      // column is looked at meanwhile, and its record fetched into the other
      // buffer when its row is already published: beside the copies of this
      // one, or, when this one was fetched ahead, after the multiplier.
      // (bi: the buffer, 2: both as one, for a record larger than one.)
      int bi = btag0 == (int)k ? 0 : (btag1 == (int)k ? 1 : -1);
      const unsigned char* rec = nullptr;
      int64_t rlen = 0;
      const bool want_pf = knext != INT_MAX && btag0 != knext && btag1 != knext;
      unsigned long long w2 = 0;
      bool fetched = false;  // the next record is being fetched
      if (bi < 0) {
        unsigned long long word = 0;
        if (lane == 0) word = wait_word(P.done + k, P.abort, wait_limit, st);
        word = __shfl_sync(0xffffffffu, word, 0);
        __syncwarp();  // every lane's reads of the record come after lane 0's acquire (a shuffle orders no memory)
        if (word == 0 || word == kRowFailed) {
          status_local = DEV_ETIMEOUT;
          break;
        }
        rlen = (int64_t)(word & 0xFFFFFFull) * 16;
        const unsigned char* src = upool + (int64_t)(word >> 24) * 16;
        if (rlen <= g.stage) {
          // a free buffer, else one holding a record fetched ahead for a
          // later column, whose copies have to arrive before it is reused
          bi = btag0 < 0 ? 0 : (btag1 < 0 ? 1 : 0);
          if (btag0 >= 0 && btag1 >= 0) record_wait<0>();
          record_fetch(bi ? stage1 : stage0, src, (int)rlen, lane);
          (bi ? btag1 : btag0) = (int)k;
          if (want_pf && (bi ? btag0 : btag1) < 0) {
            if (lane == 0) w2 = ld_acquire_u64(P.done + knext);
            w2 = __shfl_sync(0xffffffffu, w2, 0);
            __syncwarp();
            if (w2 != 0 && w2 != kRowFailed && (int64_t)(w2 & 0xFFFFFFull) * 16 <= g.stage) {
              record_fetch(bi ? stage0 : stage1, upool + (int64_t)(w2 >> 24) * 16, (int)((w2 & 0xFFFFFFull) * 16),
                           lane);
              (bi ? btag0 : btag1) = knext;
              fetched = true;
            }
          }
          if (fetched)
            record_wait<1>();
          else
            record_wait<0>();
        } else if (rlen <= 2LL * g.stage) {
          record_wait<0>();
          record_fetch(stage0, src, (int)rlen, lane);
          bi = 2;
          btag0 = btag1 = (int)k;
          record_wait<0>();
        } else {
          rec = src;
        }
      } else {
        if (want_pf && lane == 0) w2 = ld_relaxed_u64(P.done + knext);
        record_wait<0>();
      }
      const bool staged = bi >= 0;
      if (staged) rec = bi == 1 ? stage1 : stage0;
      // header: U blocks, pivot size, pivot precision and depth, U columns
      const int4 hd = staged ? *reinterpret_cast<const int4*>(rec) : __ldcg(reinterpret_cast<const int4*>(rec));
      const int ucnt = hd.x, lu64 = hd.z & 1, ncol = hd.w;
      maxdep = max(maxdep, hd.z >> 1);
      const RecLayout<int> RL = rec_layout<int>(ucnt, nk, lu64, ncol, TS);
      if (hd.y != nk || ucnt < 0 || ncol < 0 || (!staged && RL.bytes > rlen) ||
          (staged && RL.bytes > (bi == 2 ? 2 : 1) * g.stage)) {
        status_local = DEV_INTERNAL;  // never true for a published row: record and skip
        break;
      }
      const int* rperm = reinterpret_cast<const int*>(rec + RL.perm);
      const int* rcol = reinterpret_cast<const int*>(rec + RL.ucol);
      const int* rcst = reinterpret_cast<const int*>(rec + RL.ucst);
      const int* rnj = reinterpret_cast<const int*>(rec + RL.unj);
      const T* rval = reinterpret_cast<const T*>(rec + RL.val);
      const unsigned char* const rs = bi == 1 ? stage1 : stage0;  // a staged record
      T* m = wv + soff[sk];
      // the multiplier m = a_ik (P^T L U)_k^{-1}, in place, one lane per row.
      // With a staged record whose pivot block is not too large (mb), np rows at
      // a time are also held transposed in M.mt, where the column update reads
      // them; when that is the whole multiplier (mall) the drop test does too.
      constexpr int CAP = 1024 / TS;
      const int np = ni > 8 && nk * 16 <= CAP ? 16 : 8;
      const bool mb = staged && nk * 8 <= CAP && !(F32 && lu64);
      const bool mall = mb && ni <= np;
      const int S = lu_stride(nk, lu64, TS);
      if (mb) {
        const T* lu = reinterpret_cast<const T*>(rs + RL.lu);
        const T* ry = reinterpret_cast<const T*>(rs + RL.rcp);
        const int* pm = reinterpret_cast<const int*>(rs + RL.perm);
        bool small = false;
        if constexpr (F32) {
          small = nk <= NSMALL;
          if (small) {
#pragma unroll 1
            for (int a = lane; a < ni; a += 32)
              mult_row_small(lu, ry, ry + nk, pm, nk, m + a * nk, m + a * nk, mall ? M.mt + a : nullptr, np);
          }
        }
        if (!small) {
#pragma unroll 1
          for (int a = lane; a < ni && lane < np; a += np)
            mult_row_loop<T>(lu, ry, ry + nk, pm, nk, reinterpret_cast<T*>(M.buf) + lane, np, m + a * nk,
                             mall ? M.mt + a : nullptr, np);
        }
        if (mall && lane >= ni && lane < np) {  // the padding rows of the transposed multiplier
#pragma unroll 1
          for (int r = 0; r < nk; ++r) M.mt[r * np + lane] = (T)0;
        }
      } else {
        const int* pm = nullptr;  // a record read in place: its permutation, on chip
        if (!staged && nk <= PVMAX) {
#pragma unroll 1
          for (int a = lane; a < nk; a += 32) M.perm[a] = __ldcg(rperm + a);
          __syncwarp();
          pm = M.perm;
        }
#pragma unroll 1
        for (int a = lane; a < ni; a += 32) {
          if (staged) {
            if (lu64)
              ainv_right_row_sh<T, double, double>(reinterpret_cast<const double*>(rec + RL.lu), S, rperm, nk,
                                                   m + a * nk);
            else
              ainv_right_row_sh<T, float, T>(reinterpret_cast<const T*>(rec + RL.lu), S, rperm, nk, m + a * nk);
          } else {
            if (lu64)
              ainv_right_row<T, double>(reinterpret_cast<const double*>(rec + RL.lu), S, pm, rperm, nk, m + a * nk);
            else
              ainv_right_row<T, T>(reinterpret_cast<const T*>(rec + RL.lu), S, pm, rperm, nk, m + a * nk);
          }
        }
      }
      __syncwarp();
      // the drop rule.  The norm of a kept FP32 multiplier is its lfil key; an
      // FP64 one's is formed after the row is published, if lfil asks for it.
      const int sz_m = ni * nk;
      const unsigned kinv = (65536u + (unsigned)nk - 1u) / (unsigned)nk;  // e / nk for e < 256, nk <= 32
      bool dropped;
      long long key = 0;
      if constexpr (F32) {  // FP32 squares, summed by a warp reduction
        float sf = 0.f;
#pragma unroll 1
        for (int e = lane; e < sz_m; e += 32) {
          float x;
          if (mall) {
            const int a = (int)((unsigned)e * kinv >> 16);
            x = (float)M.mt[(e - a * nk) * np + a];
          } else {
            x = (float)m[e];
          }
          sf = __fmaf_rn(x, x, sf);
        }
        for (int o = 16; o > 0; o >>= 1) sf += __shfl_xor_sync(0xffffffffu, sf, o);
        dropped = drop_rule_f(sf, ni, nk, tf);
        key = norm_key(sf);
      } else {
        float sf = 0.f;
        bool in = true;
#pragma unroll 1
        for (int e = lane; e < sz_m; e += 32) {
          float x;
          in = abs_f32((double)m[e], x) && in;
          sf = __fmaf_rn(x, x, sf);
        }
        for (int o = 16; o > 0; o >>= 1) sf += __shfl_xor_sync(0xffffffffu, sf, o);
        int d = drop_f32(sf, __all_sync(0xffffffffu, in) && sz_m <= 4096, ni, nk, tf, t == 0.0);
        if (d < 0) {  // too near the threshold: the oracle's summation order
          double f2 = 0.0;
          if (lane == 0) f2 = fro2_batched(m, sz_m);
          f2 = __shfl_sync(0xffffffffu, f2, 0);
          d = drop_rule(f2, ni, nk, t);
        }
        dropped = d != 0;
      }
      // this record came ahead of its step: the next one's, if its row was
      // published at the start of the step and a buffer is free
      if (want_pf && !fetched) {
        const int ob = btag0 < 0 ? 0 : (btag1 < 0 ? 1 : -1);
        w2 = __shfl_sync(0xffffffffu, w2, 0);
        if (ob >= 0 && w2 != 0 && w2 != kRowFailed && (int64_t)(w2 & 0xFFFFFFull) * 16 <= g.stage) {
          asm volatile("fence.acq_rel.gpu;" ::: "memory");
          __syncwarp();
          record_fetch(ob ? stage1 : stage0, upool + (int64_t)(w2 >> 24) * 16, (int)((w2 & 0xFFFFFFull) * 16), lane);
          (ob ? btag1 : btag0) = knext;
        }
      }
      if (dropped) {
        if (lane == 0) sstate[sk] = SL_DEAD;
        __syncwarp();
        if (btag0 == (int)k) btag0 = -1;
        if (btag1 == (int)k) btag1 = -1;
        continue;
      }
      if (lane == 0) {
        sstate[sk] = SL_LKEPT;
        if (F32) sf2[sk] = key;
      }
      __syncwarp();
      // U row k in chunks of 32 blocks: look up or create the target blocks
      // (probe, then place, separated by __syncwarp), then update.
#pragma unroll 1
      for (int q0 = 0; q0 < ucnt && status_local == 0; q0 += 32) {
        const int q = q0 + lane;
        const int nq = min(32, ucnt - q0);
        int32_t j = -1;
        int slot = -1;
        int cst = 0, nj = 0;
        bool missing = false, bad = false;
        if (q < ucnt) {
          j = staged ? rcol[q] : __ldcg(rcol + q);
          cst = staged ? rcst[q] : __ldcg(rcst + q);
          nj = staged ? rnj[q] : __ldcg(rnj + q);
          // a published U block lies right of k inside its record
          bad = j <= k || j >= A.nbr || cst < 0 || nj <= 0 || (int64_t)cst + nj > ncol;
          if (!bad) {
            slot = ws_lookup(keys, scol, hmask, j);
            missing = slot < 0;
          }
        }
        if (__any_sync(0xffffffffu, bad)) {
          status_local = DEV_INTERNAL;
          break;
        }
        const unsigned mm = __ballot_sync(0xffffffffu, missing);
        int off = 0;
        if (mm) {  // new blocks: slots and values in the order of the columns
          int incl = missing ? ni * nj : 0;
          for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
          }
          const int add_v = __shfl_sync(0xffffffffu, incl, 31), add_s = __popc(mm);
          // A shared working row that the new blocks would overflow moves to
          // the warp's global workspace first: slot numbers (so the pending L
          // columns and the lookups above), value offsets and the multiplier's
          // values stay as they are; the global hash is rebuilt.
          if (in_sh && (ns + add_s > smax_c || nval + add_v > vmax_c) && ns + add_s <= ws.smax &&
              nval + add_v <= ws.vmax) {
            int* const gh = ws.hpos + wid * ws.smax;
            int* const gc = ws.scol + wid * ws.smax;
            int* const go = ws.soff + wid * ws.smax;
            int* const gs = ws.sstate + wid * ws.smax;
            long long* const gf = ws.sf2 + wid * ws.smax;
            int* const gn = ws.sncl + wid * ws.smax;
            T* const gv = wvals_all + wid * ws.vmax;
#pragma unroll 1
            for (int x = lane; x < ns; x += 32) {
              gc[x] = scol[x];
              go[x] = soff[x];
              gs[x] = sstate[x];
              gf[x] = sf2[x];
              gn[x] = sncl[x];
            }
            warp_copy(gv, (const T*)wv, nval, lane);
            __syncwarp();
            const uint32_t gmask = (uint32_t)ws.ht - 1;
#pragma unroll 1
            for (int x = lane; x < ns; x += 32) gh[x] = ws_place(gkeys, gmask, x, gc[x]);
#pragma unroll 1
            for (int x = lane; x < g.hash; x += 32) sh_keys[x] = -1;
            __syncwarp();
            keys = gkeys, hpos = gh, scol = gc, soff = go, sstate = gs, sf2 = gf, sncl = gn;
            wv = gv;
            smax_c = ws.smax, vmax_c = ws.vmax, hmask = gmask;
            in_sh = false;
            m = wv + soff[sk];
          }
          if (ns + add_s > smax_c || nval + add_v > vmax_c) {
            status_local = DEV_OVERFLOW;
            ask_s = ns + add_s;
            ask_v = nval + add_v;
            break;
          }
          if (missing) {
            slot = ns + __popc(mm & lt);
            off = (int)nval + incl - ni * nj;
            scol[slot] = j;
            soff[slot] = off;
            sstate[slot] = SL_LIVE;
            sncl[slot] = nj;
            hpos[slot] = ws_place(keys, hmask, slot, j);
          }
          // fill in the L part: pending for a later step
          const unsigned low = __ballot_sync(0xffffffffu, missing && j < i);
          if (missing && j < i) {
            const int pq = nl + __popc(low & lt);
            if (pq < g.lcap) {
              lc[pq] = j;
              ls[pq] = slot;
            }
          }
          const unsigned dia = __ballot_sync(0xffffffffu, missing && j == i);
          if (dia) dslot = __shfl_sync(0xffffffffu, slot, __ffs(dia) - 1);
          nl += __popc(low);
          ns += add_s;
          nval += add_v;
        }
        if (slot >= 0 && !missing) off = soff[slot];
        const int cst0 = __shfl_sync(0xffffffffu, cst, 0);
        const int cols = __shfl_sync(0xffffffffu, cst + nj, nq - 1) - cst0;
        if (mb && cols <= MCOLS) {
          if (lane < nq) {
            qinfo[lane] = make_int4(off, cst - cst0, nj, missing ? 1 : 0);
#pragma unroll 1
            for (int c = 0; c < nj; ++c) cmap[cst - cst0 + c] = (unsigned char)lane;
          }
          __syncwarp();
          const T* U = reinterpret_cast<const T*>(rs + RL.val) + nk * cst0;
          if (mall) {
            update_columns(qinfo, cmap, cols, M.mt, 0, ni, nk, np, U, wv, lane);
          } else {
#pragma unroll 1
            for (int a0 = 0; a0 < ni; a0 += np) {
              const int na = min(np, ni - a0);
#pragma unroll 1
              for (int e = lane; e < nk * np; e += 32) {
                const int r = e >> (np == 16 ? 4 : 3), a = e & (np - 1);
                M.mt[e] = a < na ? m[(a0 + a) * nk + r] : (T)0;
              }
              __syncwarp();
              update_columns(qinfo, cmap, cols, M.mt, a0, na, nk, np, U, wv, lane);
              __syncwarp();
            }
          }
        } else {
          update_general<T>(tab, nq, off, cst, nj, missing, ni, nk, m, rval, staged, wv, lane);
        }
        __syncwarp();
      }
      if (btag0 == (int)k) btag0 = -1;
      if (btag1 == (int)k) btag1 = -1;
    }
    record_wait<0>();  // every record fetched ahead has been used, unless the row failed
    // A row that ends in the global workspace has its slot metadata copied to the
    // end of the shared working-row region (unused by such a row) when it fits, so
    // that the scans of the finish read on-chip data; its values stay in the global
    // workspace.  The rest of the region, right behind the stage buffers, takes a
    // large pivot block (200 block rows of 33 to 40 scalars FP32 181 ms, 156 with it).
    int region_end = in_sh ? g.o_vals : g.o_lc;  // end of what is free behind the stage buffers
    if (!in_sh && status_local == 0) {
      const int region = g.o_lc - g.o_vals;  // vals, hash and slot arrays of the shared workspace
      if (ns * 24 <= region) {
        region_end = g.o_vals + ((region - ns * 24) & ~15);
        long long* mf2 = reinterpret_cast<long long*>(wb + region_end);
        int* mcol = reinterpret_cast<int*>(mf2 + ns);
        int* mst = mcol + ns;
        int* mncl = mst + ns;
        int* moff = mncl + ns;
#pragma unroll 1
        for (int q = lane; q < ns; q += 32) {
          mf2[q] = sf2[q];
          mcol[q] = scol[q];
          mst[q] = sstate[q];
          mncl[q] = sncl[q];
          moff[q] = soff[q];
        }
        __syncwarp();
        sf2 = mf2, scol = mcol, sstate = mst, sncl = mncl, soff = moff;
      }
    }
    // ---- finish the row: what its dependants read first (the U part, the
    // pivot block, the record), then publish, then the L part.
    if (status_local == 0 && dslot < 0) status_local = DEV_ESINGULAR;
    // candidate list of the blocks right of the diagonal, in the stage buffers
    // when it fits beside its sorted form, else in the warp's global space
    int nU = 0;
    int* candU = nullptr;
    unsigned long long* srtU = nullptr;
    int gb_at = 0;  // first free byte of the stage buffers
    if (status_local == 0) {
      int p2u = 1;
      while (p2u < ns) p2u <<= 1;
      const int64_t need = ((4LL * ns + 15) & ~15LL) + 8LL * p2u;
      if (need <= 2LL * g.stage) {
        candU = reinterpret_cast<int*>(stage0);
        srtU = reinterpret_cast<unsigned long long*>(stage0 + ((4LL * ns + 15) & ~15LL));
        gb_at = (int)((need + 15) & ~15LL);
      } else {
        candU = ws.fin + wid * 2 * ws.smax;
        srtU = ws.srt + wid * 4 * ws.smax;
      }
#pragma unroll 1
      for (int q0 = 0; q0 < ns; q0 += 32) {
        const int q = q0 + lane;
        const bool isU = q < ns && sstate[q] == SL_LIVE && scol[q] > i;
        const unsigned bU = __ballot_sync(0xffffffffu, isU);
        if (isU) candU[nU + __popc(bU & lt)] = q;
        nU += __popc(bU);
      }
      __syncwarp();
      // threshold (in FP32: the norms are the lfil keys; in FP64 the keys are
      // formed when lfil has to choose), survivors compacted
      int kept = 0;
#pragma unroll 1
      for (int c0 = 0; c0 < nU; c0 += 32) {
        const int c = c0 + lane;
        const int q = c < nU ? candU[c] : -1;
        bool keep = false;
        if (q >= 0) {
          const int nc = sncl[q], n = ni * nc;
          const T* v = wv + soff[q];
          if constexpr (F32) {
            const float f2 = fro2_f32(v, n);
            keep = !drop_rule_f(f2, ni, nc, tf);
            sf2[q] = norm_key(f2);
          } else {
            float sf = 0.f;
            bool in = n <= 4096;
#pragma unroll 4
            for (int e = 0; e < n; ++e) {
              float x;
              in = abs_f32((double)v[e], x) && in;
              sf = __fmaf_rn(x, x, sf);
            }
            const int d = drop_f32(sf, in, ni, nc, tf, t == 0.0);
            keep = !(d < 0 ? drop_rule(fro2_batched(v, n), ni, nc, t) : d != 0);
          }
          if (!keep) sstate[q] = SL_DEAD;
        }
        const unsigned bk = __ballot_sync(0xffffffffu, keep);
        if (keep) candU[kept + __popc(bk & lt)] = q;
        kept += __popc(bk);
        __syncwarp();
      }
      nU = kept;
      if (lfil >= 0 && nU > lfil) {
        if (!F32) {
#pragma unroll 1
          for (int c = lane; c < nU; c += 32) {
            const int q = candU[c];
            sf2[q] = norm_key(fro2_batched(wv + soff[q], ni * sncl[q]));
          }
          __syncwarp();
        }
        nU = lfil_cut(candU, nU, lfil, sf2, scol, sstate, M.buf, TS, lane);
      }
      sort_by_column(candU, nU, scol, srtU, lane);
    }
    // the record's size and, while the pivot block is factored, its space
    // (with an FP64 pivot LU when the factor's type or a large block asks for
    // one; a small FP32 block that turns out to need one takes a second space)
    int ucols = 0;
    unsigned long long roff16 = 0;
    int64_t rbytes = 0;
    int lu64r = F32 && ni <= 32 ? 0 : 1;
    if (status_local == 0) {
#pragma unroll 1
      for (int p = lane; p < nU; p += 32) ucols += sncl[(int)(srtU[p] & 0xffffffffu)];
      ucols = __reduce_add_sync(0xffffffffu, ucols);
      rbytes = rec_layout<int64_t>(nU, ni, lu64r, ucols, TS).bytes;
      if (lane == 0) roff16 = atomicAdd(P.ctr + 2, (unsigned long long)(rbytes / 16));
    }
    // GEPP of the diagonal block, in registers, in shared memory when it fits
    // (the stage buffers' free part, and the space behind them), else in place.  FP64 factor: FP64 in the
    // oracle's operation order.  Mixed factor: FP32 GEPP and 1-norm condition
    // estimate (explicit inverse columns); a block above the threshold, larger
    // than 32, or singular in FP32 is factored again in FP64 and tagged.
    bool tag64 = !F32;
    bool lu_sm = false;  // the pivot LU and its reciprocals are in M
    const T* lu_g = nullptr;  // else: the FP32 pivot LU, rows lu_str apart
    int lu_str = ni;
    const double* lu_g64 = nullptr;
    if (status_local == 0) {
      const T* srcd = wv + soff[dslot];
      unsigned char* gb = stage0 + gb_at;
      const int gcap = region_end - g.o_stage - gb_at;
      int* pvs = ni <= PVMAX ? M.pv : nullptr;
      int32_t* gpiv = piv + A.roff[i];
      bool ok = true;
      if constexpr (F32) {
        tag64 = true;
        float norm1 = 0.f;  // (a larger block is factored in FP64)
        if (lane < ni && ni <= 32) {
          float sum = 0.f;
#pragma unroll 1
          for (int ii = 0; ii < ni; ++ii) sum += fabsf(srcd[ii * ni + lane]);
          norm1 = fmaxf(norm1, sum);
        }
        norm1 = warp_max_f(norm1);
        float inv1 = 0.f;
        if (ni <= NSMALL) {
          if (gepp_cond_small(srcd, ni, M.lu, M.ry, M.rz, M.pv, M.perm, gpiv, lane, &inv1)) {
            tag64 = !(norm1 * inv1 <= condf);
            lu_sm = !tag64;
          }
        } else if (ni <= NPIV && (ni <= 16 ? 1024 : 4096) <= gcap) {
          float* a = reinterpret_cast<float*>(gb);
          lu_str = ni <= 16 ? 16 : 32;
          if (ni <= 16 ? gepp_cond<16>(srcd, ni, a, M.ry, M.rz, M.pv, M.perm, gpiv, lane, &inv1)
                       : gepp_cond<32>(srcd, ni, a, M.ry, M.rz, M.pv, M.perm, gpiv, lane, &inv1)) {
            tag64 = !(norm1 * inv1 <= condf);
            lu_g = a;
          }
        } else if (ni <= 32) {
          float* a = dg32 + dgoff[i];
          lu_str = ni;
#pragma unroll 1
          for (int e = lane; e < ni * ni; e += 32) a[e] = srcd[e];
          __syncwarp();
          if (gepp_warp<float>(a, ni, pvs, gpiv, lane)) {
            tag64 = !(norm1 * inv_norm1_f32(a, ni, pvs, lane) <= condf);
            lu_g = a;
          }
        }
        __syncwarp();
      }
      if (tag64) {
        const bool far = ni * ni * 8 > gcap;
        double* a = far ? dg + dgoff[i] : reinterpret_cast<double*>(gb);
#pragma unroll 4
        for (int e = lane; e < ni * ni; e += 32) a[e] = (double)srcd[e];
        __syncwarp();
        ok = far ? gepp_warp<double, true>(a, ni, pvs, gpiv, lane) : gepp_warp<double>(a, ni, pvs, gpiv, lane);
        lu_g64 = a;
      }
      __syncwarp();
      if (!ok)
        status_local = DEV_ESINGULAR;
      else if ((tag64 || lu_str == ni) && !lu_sm && ni <= PVMAX)
        perm_of(M.pv, ni, M.perm, lane);
    }
    // the space, with what the pivot block turned out to need
    if (status_local == 0) {
      if (F32 && tag64 && !lu64r) {
        lu64r = 1;
        rbytes = rec_layout<int64_t>(nU, ni, lu64r, ucols, TS).bytes;
        if (lane == 0) roff16 = atomicAdd(P.ctr + 2, (unsigned long long)(rbytes / 16));
      }
      roff16 = __shfl_sync(0xffffffffu, roff16, 0);
      if ((int64_t)roff16 + rbytes / 16 > P.ucap16 || rbytes / 16 > kRecMaxUnits) status_local = DEV_OVERFLOW;
    }
    // the record
    if (status_local == 0) {
      const RecLayout<int> RL = rec_layout<int>(nU, ni, lu64r, ucols, TS);
      unsigned char* r = upool + (int64_t)roff16 * 16;
      if (lane == 0) *reinterpret_cast<int4*>(r) = make_int4(nU, ni, 2 * (maxdep + 1) + lu64r, ucols);
      int* rp = reinterpret_cast<int*>(r + RL.perm);
      if (ni <= PVMAX) {
#pragma unroll 1
        for (int a = lane; a < ni; a += 32) rp[a] = M.perm[a];
      } else if (lane == 0) {  // a block of more than PVMAX rows: in place
        const int32_t* gpiv = piv + A.roff[i];
#pragma unroll 1
        for (int a = 0; a < ni; ++a) rp[a] = a;
#pragma unroll 1
        for (int a = 0; a < ni; ++a) {
          const int q = gpiv[a], v = rp[a];
          rp[a] = rp[q];
          rp[q] = v;
        }
      }
      if (lu_sm) {
        T* o = reinterpret_cast<T*>(r + RL.lu);
#pragma unroll 1
        for (int e = lane; e < ni * NSMALL; e += 32) o[e] = M.lu[e];
        T* y = reinterpret_cast<T*>(r + RL.rcp);
        if (lane < ni) {
          y[lane] = M.ry[lane];
          y[ni + lane] = M.rz[lane];
        }
      } else if (lu64r) {
        put_pivot(lu_g64, ni, ni, reinterpret_cast<double*>(r + RL.lu), reinterpret_cast<double*>(r + RL.rcp), lane);
      } else {
        put_pivot(lu_g, lu_str, ni, reinterpret_cast<T*>(r + RL.lu), reinterpret_cast<T*>(r + RL.rcp), lane);
      }
      int* rcol = reinterpret_cast<int*>(r + RL.ucol);
      int* rcst = reinterpret_cast<int*>(r + RL.ucst);
      int* rnjw = reinterpret_cast<int*>(r + RL.unj);
      T* rv = reinterpret_cast<T*>(r + RL.val);
      int carry = 0;
#pragma unroll 1
      for (int p0 = 0; p0 < nU; p0 += 32) {
        const int p = p0 + lane;
        int nc = 0, so = 0;
        if (p < nU) {
          const int c = (int)(srtU[p] >> 32), q = (int)(srtU[p] & 0xffffffffu);
          nc = sncl[q];
          so = soff[q];
          rcol[p] = c;
          rnjw[p] = nc;
        }
        int incl = nc;
        for (int o = 1; o < 32; o <<= 1) {
          const int v = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += v;
        }
        const int cst = carry + incl - nc;
        if (p < nU) rcst[p] = cst;
        copy_blocks<T>(min(32, nU - p0), ni * nc, so, (long long)ni * cst, wv, rv, lane);
        carry += __shfl_sync(0xffffffffu, incl, 31);
      }
    }
    if (status_local != 0 && lane == 0) {
      dev_fail(st, status_local);
      atomicExch(P.abort, 1);
    }
    // publish the row: every lane's writes are made visible device-wide
    // before lane 0 sets the word
    __threadfence();
    __syncwarp();
    if (lane == 0) {
      const unsigned long long w = status_local == 0
                                       ? ((unsigned long long)roff16 << 24) | (unsigned long long)(rbytes / 16)
                                       : kRowFailed;
      asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(P.done + i), "l"(w) : "memory");
      if (ask_s) {  // to size a retry
        atomicMax(P.ctr + 5, (unsigned long long)ask_v);
        atomicMax(P.ctr + 6, (unsigned long long)ask_s);
      }
      if (P.depth) P.depth[i] = maxdep + 1;
    }
    // ---- what no other row reads: the pivot block as the solve takes it, then
    // the L part
    if (status_local == 0) {
      if (!lu_sm && tag64) {
        double* d = dg + dgoff[i];
        if (lu_g64 != d) {
#pragma unroll 1
          for (int e = lane; e < ni * ni; e += 32) d[e] = lu_g64[e];
        }
        if (mixed) {
#pragma unroll 4
          for (int e = lane; e < ni * ni; e += 32) dg32[dgoff[i] + e] = (float)lu_g64[e];
        }
      } else {
#pragma unroll 1
        for (int e = lane; e < ni * ni; e += 32) {
          const int a = e / ni;
          const float v = lu_sm ? (float)M.lu[a * NSMALL + e - a * ni] : (float)lu_g[a * lu_str + e - a * ni];
          dg32[dgoff[i] + e] = v;
          dg[dgoff[i] + e] = (double)v;
        }
      }
      if (mixed && lane == 0) ptag[i] = tag64 ? 1 : 0;
      __syncwarp();  // the stage buffers are free now
    }
    int nL = 0;
    int* candL = nullptr;
    unsigned long long* srtL = nullptr;
    unsigned long long lb = 0, lvv = 0;
    if (status_local == 0) {
      int cl = 0;
#pragma unroll 1
      for (int q0 = 0; q0 < ns; q0 += 32) {
        const int q = q0 + lane;
        cl += __popc(__ballot_sync(0xffffffffu, q < ns && sstate[q] == SL_LKEPT));
      }
      int p2l = 1;
      while (p2l < cl) p2l <<= 1;
      if (((4LL * cl + 15) & ~15LL) + 8LL * p2l <= 2LL * g.stage) {
        candL = reinterpret_cast<int*>(stage0);
        srtL = reinterpret_cast<unsigned long long*>(stage0 + ((4LL * cl + 15) & ~15LL));
      } else {
        candL = ws.fin + wid * 2 * ws.smax;
        srtL = ws.srt + wid * 4 * ws.smax;
      }
#pragma unroll 1
      for (int q0 = 0; q0 < ns; q0 += 32) {
        const int q = q0 + lane;
        const bool isL = q < ns && sstate[q] == SL_LKEPT;
        const unsigned bL = __ballot_sync(0xffffffffu, isL);
        if (isL) candL[nL + __popc(bL & lt)] = q;
        nL += __popc(bL);
      }
      __syncwarp();
      if (lfil >= 0 && nL > lfil) {
        if (!F32) {
#pragma unroll 1
          for (int c = lane; c < nL; c += 32) {
            const int q = candL[c];
            sf2[q] = norm_key(fro2_batched(wv + soff[q], ni * sncl[q]));
          }
          __syncwarp();
        }
        nL = lfil_cut(candL, nL, lfil, sf2, scol, sstate, M.buf, TS, lane);
      }
      sort_by_column(candL, nL, scol, srtL, lane);
      long long vl = 0;
#pragma unroll 1
      for (int p = lane; p < nL; p += 32) vl += (long long)ni * sncl[(int)(srtL[p] & 0xffffffffu)];
      vl = warp_sum_ll(vl);
      if (lane == 0) {
        lb = atomicAdd(P.ctr + 0, (unsigned long long)nL);
        lvv = atomicAdd(P.ctr + 1, (unsigned long long)vl);
      }
      lb = __shfl_sync(0xffffffffu, lb, 0);
      lvv = __shfl_sync(0xffffffffu, lvv, 0);
      if ((int64_t)(lb + nL) > P.lbcap || (int64_t)(lvv + vl) > P.lvcap) {
        status_local = DEV_OVERFLOW;
        if (lane == 0) {
          dev_fail(st, status_local);
          atomicExch(P.abort, 1);
        }
      }
    }
    if (status_local == 0) {
      long long carry = 0;
#pragma unroll 1
      for (int p0 = 0; p0 < nL; p0 += 32) {
        const int p = p0 + lane;
        int sz = 0, so = 0;
        if (p < nL) {
          const int c = (int)(srtL[p] >> 32), q = (int)(srtL[p] & 0xffffffffu);
          sz = ni * sncl[q];
          so = soff[q];
          P.lcol[lb + p] = c;
        }
        int incl = sz;
        for (int o = 1; o < 32; o <<= 1) {
          const int v = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += v;
        }
        const long long dof = (long long)lvv + carry + incl - sz;
        if (p < nL) P.lvo[lb + p] = dof;
        copy_blocks<T>(min(32, nL - p0), sz, so, dof, wv, lval, lane);
        carry += __shfl_sync(0xffffffffu, incl, 31);
      }
    }
    if (lane == 0) {
      P.lstart[i] = status_local == 0 ? (int64_t)lb : 0;
      P.lcnt[i] = status_local == 0 ? nL : 0;
    }
    // clear the shared hash, over which the finish of a row in global memory
    // staged its metadata and its pivot block, and the positions such a row used
#pragma unroll 1
    for (int q = lane; q < g.hash; q += 32) sh_keys[q] = -1;
    if (!in_sh) {
#pragma unroll 1
      for (int q = lane; q < ns; q += 32)
        if (hpos[q] >= 0) keys[hpos[q]] = -1;
    }
    __syncwarp();
  }
}

// Gather the pooled L rows into VBCSR (warp per row).
template <typename T>
__global__ void k_pool_to_vb(int64_t nbr, const int64_t* __restrict__ start, const int32_t* __restrict__ pcol,
                             const int64_t* __restrict__ pvo, const T* __restrict__ pval,
                             const int64_t* __restrict__ bptr, const int64_t* __restrict__ voff,
                             int32_t* __restrict__ bcol, T* __restrict__ val) {
  const int lane = threadIdx.x & 31;
  const int64_t wpb = blockDim.x >> 5;
  for (int64_t i = blockIdx.x * wpb + (threadIdx.x >> 5); i < nbr; i += (int64_t)gridDim.x * wpb) {
    const int64_t n = bptr[i + 1] - bptr[i];
    if (!voff) {  // first pass: columns only (the value offsets do not exist yet)
      for (int64_t q = lane; q < n; q += 32) bcol[bptr[i] + q] = pcol[start[i] + q];
      continue;
    }
    for (int64_t q = 0; q < n; ++q) {
      const int64_t d = bptr[i] + q;
      const int64_t sz = voff[d + 1] - voff[d];
      const int64_t src = pvo[start[i] + q];
      for (int64_t e = lane; e < sz; e += 32) val[voff[d] + e] = pval[src + e];
    }
  }
}

// U rows from the published records: counts (pass 0), columns (pass 1, after
// the row pointers), values (pass 2, after the value offsets).  A record's
// values are its row's blocks in column order, the VBCSR layout of the row.
template <typename T>
__global__ void k_rec_to_vb(int64_t nbr, int pass, const unsigned long long* __restrict__ done,
                            const unsigned char* __restrict__ upool, int32_t* __restrict__ cnt,
                            const int64_t* __restrict__ bptr, const int64_t* __restrict__ voff,
                            int32_t* __restrict__ bcol, T* __restrict__ val) {
  const int lane = threadIdx.x & 31;
  const int64_t wpb = blockDim.x >> 5;
  for (int64_t i = blockIdx.x * wpb + (threadIdx.x >> 5); i < nbr; i += (int64_t)gridDim.x * wpb) {
    const unsigned char* r = upool + (int64_t)(done[i] >> 24) * 16;
    const int* h = reinterpret_cast<const int*>(r);
    const int ucnt = h[0];
    if (pass == 0) {
      if (lane == 0) cnt[i] = ucnt;
      continue;
    }
    const RecLayout<int> RL = rec_layout<int>(ucnt, h[1], h[2] & 1, h[3], (int)sizeof(T));
    if (pass == 1) {
      for (int q = lane; q < ucnt; q += 32) bcol[bptr[i] + q] = reinterpret_cast<const int*>(r + RL.ucol)[q];
      continue;
    }
    const T* src = reinterpret_cast<const T*>(r + RL.val);
    T* dst = val + voff[bptr[i]];
    const int64_t n = (int64_t)h[3] * h[1];
    for (int64_t e = lane; e < n; e += 32) dst[e] = src[e];
  }
}

__global__ void k_sq_sizes(int64_t n, const int32_t* __restrict__ sz, int64_t* __restrict__ out) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = (int64_t)sz[i] * sz[i];
}

__global__ void k_count_to_i64(int64_t n, const int32_t* __restrict__ c, int64_t* __restrict__ out) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = c[i];
}

__global__ void k_iota(int64_t n, int64_t* __restrict__ bptr, int32_t* __restrict__ bcol) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i <= n; i += (int64_t)gridDim.x * blockDim.x) {
    bptr[i] = i;
    if (i < n) bcol[i] = (int32_t)i;
  }
}

// Row statistics of the last-level matrix for the choice of the workspace:
// [0] block rows with more than 24 blocks, [1] largest row in blocks.
__global__ void k_row_stats(int64_t nbr, const int64_t* __restrict__ bptr, unsigned long long* __restrict__ out) {
  unsigned long long big = 0, mx = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nbr; i += (int64_t)gridDim.x * blockDim.x) {
    const unsigned long long nb = (unsigned long long)(bptr[i + 1] - bptr[i]);
    big += nb > 24;
    mx = nb > mx ? nb : mx;
  }
  for (int o = 16; o > 0; o >>= 1) {
    big += __shfl_xor_sync(0xffffffffu, big, o);
    const unsigned long long v = __shfl_xor_sync(0xffffffffu, mx, o);
    mx = v > mx ? v : mx;
  }
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(out, big);
    atomicMax(out + 1, mx);
  }
}

}  // namespace

// Shared workspace of one warp: slots, value bytes, stage-buffer bytes and
// pending-column capacity, every part 16-byte aligned.
template <typename T>
static IlutGeom make_geom(int slots, int vbytes, int stage, int lcap) {
  IlutGeom G{};
  G.slots = slots;
  G.hash = 1;
  while (G.hash < 2 * slots) G.hash <<= 1;
  G.vbytes = vbytes;
  G.stage = stage;
  G.lcap = lcap;
  auto up = [](int v, int a) { return (v + a - 1) / a * a; };
  int o = 0;
  G.o_misc = o;
  o = up(o + (int)sizeof(IlutMisc<T>), 128);
  G.o_stage = o;
  o += 2 * stage;
  G.o_vals = o;
  o = up(o + vbytes, 16);
  G.o_keys = o;
  o = up(o + 4 * G.hash, 16);
  G.o_hpos = o;
  o = up(o + 4 * slots, 16);
  G.o_scol = o;
  o = up(o + 4 * slots, 16);
  G.o_soff = o;
  o = up(o + 4 * slots, 16);
  G.o_sst = o;
  o = up(o + 4 * slots, 16);
  G.o_sf2 = o;
  o = up(o + 8 * slots, 16);
  G.o_sncl = o;
  o = up(o + 4 * slots, 16);
  G.o_lc = o;
  o = up(o + 4 * lcap, 16);
  G.o_ls = o;
  o = up(o + 4 * lcap, 128);
  G.bytes = o;
  return G;
}



namespace {
// m = the largest a[i]
__global__ void k_max_i32(int64_t n, const int32_t* __restrict__ a, unsigned long long* __restrict__ m) {
  unsigned long long v = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    v = max(v, (unsigned long long)a[i]);
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0 && v) atomicMax(m, v);
}

}  // namespace

template <typename T>
void ilut_last(LastDev<T>& X, double t, int lfil, bool mixed, double cond_thr, uint64_t wait_limit, cudaStream_t s,
               int* dst, const int32_t* order) {
  IlutInfo* info = &X.info;
  const VBDev<T>& A = X.A;
  const int64_t p = A.nbr;
  const int64_t n = p ? d2h(A.roff.p + p, s) : 0;
  // pivot blocks: block diagonal structure
  set_partitions(X.Dg, A.rsz.p, p, A.rsz.p, p, s);
  X.Dg.bptr.alloc(p + 1, s);
  X.Dg.bcol.alloc(p, s);
  launch(k_iota, grid_for(p + 1, 256), 256, 0, s, p, X.Dg.bptr.p, X.Dg.bcol.p);
  VB_LAUNCH_CHECK();
  X.Dg.nnzb = p;
  X.Dg.voff.alloc(p + 1, s);
  {
    DBuf<int64_t> sq(p, s);
    if (p) {
      launch(k_sq_sizes, grid_for(p, 256), 256, 0, s, p, A.rsz.p, sq.p);
      VB_LAUNCH_CHECK();
    }
    scan_i64(sq.p, X.Dg.voff.p, p, s);
  }
  X.Dg.nval = p ? d2h(X.Dg.voff.p + p, s) : 0;
  X.Dg.val.alloc(X.Dg.nval, s);
  X.piv.alloc(n, s);
  X.ptag.alloc(p, s);
  X.ptag.zero();
  if (mixed) copy_vb<float, double>(X.Dg, X.Dg32, s);
  set_partitions(X.L, A.rsz.p, p, A.rsz.p, p, s);
  set_partitions(X.U, A.rsz.p, p, A.rsz.p, p, s);
  if (p == 0) {
    X.L.bptr.alloc(1, s);
    X.L.bptr.zero();
    X.U.bptr.alloc(1, s);
    X.U.bptr.zero();
    X.L.voff.alloc(1, s);
    X.L.voff.zero();
    X.U.voff.alloc(1, s);
    X.U.voff.zero();
    return;
  }

  int dev = 0;
  VB_CUDA(cudaGetDevice(&dev));
  int nsm = 0, smem_sm = 0, smem_block = 0;
  VB_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  VB_CUDA(cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev));
  VB_CUDA(cudaDeviceGetAttribute(&smem_block, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  // Shared workspace per warp ("tile shape" of the kernel): chosen by timing
  // the candidates below on a prefix of this matrix's own tickets (every
  // prefix of the ticket order is factored exactly on its own), the fastest
  // kept per device, precision and class of row sizes for the rest of the
  // process; small matrices take the first.  What counts is that records and
  // working rows stay on chip; the rows in flight then matter little.  Shapes as
  // slots / value bytes / stage bytes.  3.0 million unknowns FP32, whole
  // factorizations with an earlier finish of the rows (the chosen shape's takes 475
  // ms now): 64 / 6 144 / 3 072, 8 warps an SM, 709 ms; 128 / 8 192 / 4 096, 8
  // warps, 671; 128 / 12 288 / 4 096, 7 warps, 644; 128 / 16 384 / 6 144, 5 warps,
  // 677.  FP64 rows hold twice the bytes (360 000 unknowns: 128 / 8 192 / 6 144, 7
  // warps, 382 ms; 128 / 16 384 / 6 144, 5 warps, 339).  Rows of many small blocks
  // need slots: 48 000 unknowns at tau 0.9, this kernel, FP32 and FP64: 512 / 16 384
  // / 4 096, 4 warps, 290 and 586 ms; 768 / 16 384 / 4 096, 3 warps, 255 and 556.
  // (Fewer and larger workspaces measured shorter chains there still: 768 / 24 576 /
  // 4 096 242 and 517, 1 024 / 32 768 / 8 192, 2 warps, 239 and 486; not timed where
  // more than one chain is in flight.)  The prefix is 1/64 of the tickets (2 048 to
  // 16 384), so the timings add at most about 5 % to the first factorization of a
  // class.
  DBuf<unsigned long long> rstat(2, s);
  rstat.zero();
  launch(k_row_stats, grid_for(p, 256), 256, 0, s, p, A.bptr.p, rstat.p);
  VB_LAUNCH_CHECK();
  const std::vector<unsigned long long> rs = d2h_vec(rstat.p, 2, s);
  const bool wide = rs[0] * 4 > (unsigned long long)p;
  const bool f64 = sizeof(T) == sizeof(double);
  std::vector<IlutGeom> cands;
  if (wide) cands.push_back(make_geom<T>(768, 16384, 4096, 512));
  cands.push_back(make_geom<T>(128, f64 ? 16384 : 12288, f64 ? 6144 : 4096, wide ? 256 : 128));
  if (!wide) cands.push_back(make_geom<T>(128, 8192, f64 ? 6144 : 4096, 128));
  const int reserve = 1024;  // shared memory the system keeps per block
  // warps per block and blocks per SM of a geometry: the most warps per SM
  // (at most 8: their registers)
  auto shape = [&](const IlutGeom& G, int& wpb, int& bps) {
    wpb = 0, bps = 0;
    for (int w = 8; w >= 1; --w) {
      if (w * G.bytes > smem_block) continue;
      int b = smem_sm / (w * G.bytes + reserve);
      while (w * b > 8) --b;
      if (b >= 1 && w * b > wpb * bps) wpb = w, bps = b;
    }
    return wpb >= 1;
  };
  // L pool: the L blocks; U pool: one record per row.  L and U each hold
  // about half of the last-level matrix on the configured workloads; the
  // pools start at its full size and grow on overflow (retry)
  int64_t lbcap = std::max<int64_t>(A.nnzb, 1024), lvcap = std::max<int64_t>(A.nval, 1 << 16);
  int64_t ucap16 = (A.nval * (int64_t)sizeof(T) + X.Dg.nval * 8 + 8 * A.nnzb + 16 * n + 96 * p) / 16 + 4096;
  int smax = 1024;
  int64_t vmax = 32768;
  // buffers of one launch
  struct Run {
    DBuf<int32_t> lcol, lcnt, depth;
    DBuf<int64_t> lvo, lstart;
    DBuf<unsigned long long> done, ctr;
    DBuf<T> lval;
    DBuf<unsigned char> upool;
  };
  // one launch of the kernel over the first nticket tickets with geometry G;
  // returns the device status (the time of the launch in *ms when asked)
  auto run = [&](const IlutGeom& G, int64_t nticket, Run& R, float* ms, bool track = false) -> int {
    int wpb = 0, bps = 0;
    if (!shape(G, wpb, bps)) fail(VB_EINTERNAL, "last-level ILUT: shared workspace exceeds a block");
    const size_t smem = (size_t)wpb * G.bytes;
    const int64_t nblocks = std::max<int64_t>(1, std::min<int64_t>((int64_t)nsm * bps, (nticket + wpb - 1) / wpb));
    const int64_t nwarps = nblocks * wpb;
    int ht = 1;
    while (ht < 2 * smax) ht <<= 1;
    DBuf<int> keys(nwarps * ht, s), hpos(nwarps * smax, s), scol(nwarps * smax, s), sstate(nwarps * smax, s);
    DBuf<int> soff(nwarps * smax, s), sncl(nwarps * smax, s), fin(nwarps * 2 * smax, s);
    DBuf<long long> sf2(nwarps * smax, s);
    DBuf<unsigned long long> srt(nwarps * 4 * smax, s);
    DBuf<T> wvals(nwarps * vmax, s);
    Workspace ws{keys.p, hpos.p, scol.p, soff.p, sstate.p, sf2.p, sncl.p, fin.p, srt.p, ht, smax, vmax};
    R.lcol.alloc(lbcap, s);
    R.lcnt.alloc(p, s);
    R.lvo.alloc(lbcap, s);
    R.lstart.alloc(p, s);
    R.done.alloc(p, s);
    R.lval.alloc(lvcap, s);
    R.upool.alloc(ucap16 * 16, s);
    R.ctr.alloc(8, s);
    if (track) {
      R.depth.alloc(p, s);
      R.depth.zero();
    }
    DBuf<int> abort(1, s);
    R.ctr.zero();
    R.done.zero();
    abort.zero();
    X.piv.zero();
    Pools P{R.lcol.p, R.lvo.p, R.lstart.p, R.lcnt.p, R.done.p, R.ctr.p, lbcap, lvcap, ucap16, abort.p, order,
            nticket, R.depth.p};
    VB_CUDA(cudaFuncSetAttribute(k_ilut<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (ms) {
      VB_CUDA(cudaEventCreate(&e0));
      VB_CUDA(cudaEventCreate(&e1));
      VB_CUDA(cudaEventRecord(e0, s));
    }
    launch(k_ilut<T>, (unsigned)nblocks, wpb * 32, smem, s, A.view(), G, ws, wvals.p, P, R.lval.p, R.upool.p,
           X.Dg.voff.p, X.Dg.val.p, mixed ? X.Dg32.val.p : nullptr, X.piv.p, mixed ? X.ptag.p : nullptr,
           mixed ? 1 : 0, cond_thr, t, lfil, (unsigned long long)wait_limit, dst);
    VB_LAUNCH_CHECK();
    if (ms) {
      VB_CUDA(cudaEventRecord(e1, s));
      VB_CUDA(cudaEventSynchronize(e1));
      VB_CUDA(cudaEventElapsedTime(ms, e0, e1));
      cudaEventDestroy(e0);
      cudaEventDestroy(e1);
    }
    if (info) {
      info->warps_per_sm = wpb * bps;
    }
    return d2h(dst, s);
  };
  // the geometry: cached, tuned on a prefix, or the default
  IlutGeom G = cands[0];
  {
    int m1 = 0, m2 = 0;
    const double mb = (double)A.nnzb / (double)p, mv = (double)A.nval / (double)p;
    while ((1 << m1) < mb) ++m1;
    while ((1 << m2) < mv) ++m2;
    const long long key = ((long long)dev << 40) | ((long long)sizeof(T) << 32) | ((long long)wide << 24) |
                          ((long long)m1 << 8) | (long long)m2;
    std::lock_guard<std::mutex> lk(g_geom_mu);
    auto it = g_geom.find(key);
    if (it != g_geom.end()) {
      G = it->second;
      if (info) info->source = 2;
    } else if (p >= kTuneMinRows) {
      const int64_t m = std::min<int64_t>(std::max<int64_t>(p / 64, 2048), 16384);
      const auto t0 = std::chrono::steady_clock::now();
      float best = 0.f;
      int bi = -1;
      for (size_t c = 0; c < cands.size(); ++c) {
        Run R;
        float ms = 0.f;
        const int st = run(cands[c], m, R, &ms);
        if (st != DEV_OK) {
          VB_CUDA(cudaMemsetAsync(dst, 0, sizeof(int), s));
          if (st == DEV_ETIMEOUT || st == DEV_INTERNAL) check_status(dst, s, "last-level ILUT tuning");
          continue;
        }
        if (bi < 0 || ms < best) best = ms, bi = (int)c;
      }
      if (bi >= 0) G = cands[bi];
      g_geom[key] = G;
      if (info) {
        info->source = 1;
        info->tune_s = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
      }
    }
  }
  if (info) {
    info->slots = G.slots;
    info->vbytes = G.vbytes;
  }
  for (int attempt = 0; attempt < 6; ++attempt) {
    Run R;
    const int st = run(G, p, R, nullptr, true);
    auto& lcol = R.lcol;
    auto& lcnt = R.lcnt;
    auto& lvo = R.lvo;
    auto& lstart = R.lstart;
    auto& done = R.done;
    auto& lval = R.lval;
    auto& upool = R.upool;
    auto& ctr = R.ctr;
    if (st == DEV_OVERFLOW) {
      VB_CUDA(cudaMemsetAsync(dst, 0, sizeof(int), s));
      std::vector<unsigned long long> c = d2h_vec(ctr.p, 8, s);
      lbcap = std::max<int64_t>(2 * lbcap, (int64_t)c[0] + 1024);
      lvcap = std::max<int64_t>(2 * lvcap, (int64_t)c[1] + 4096);
      ucap16 = std::max<int64_t>(2 * ucap16, (int64_t)c[2] + 4096);
      while ((int64_t)c[5] > vmax) vmax *= 2;
      if ((int64_t)c[6] > smax) {
        while (smax < (int)c[6] && smax < MAX_SLOTS) smax *= 2;
        if ((int64_t)c[6] > MAX_SLOTS) fail(VB_ENOMEM, "last-level ILUT: a working row exceeds 4096 blocks");
      }
      continue;
    }
    check_status(dst, s, "vbarms_factor: last-level block ILUT");
    if (info) {  // the longest chain of waits
      DBuf<unsigned long long> mx(1, s);
      mx.zero();
      launch(k_max_i32, grid_for(p, 256), 256, 0, s, p, R.depth.p, mx.p);
      VB_LAUNCH_CHECK();
      info->chain = (long long)d2h(mx.p, s);
    }
    // assemble L from its pool
    {
      VBDev<T>& M = X.L;
      M.bptr.alloc(p + 1, s);
      DBuf<int64_t> c64(p, s);
      launch(k_count_to_i64, grid_for(p, 256), 256, 0, s, p, lcnt.p, c64.p);
      VB_LAUNCH_CHECK();
      scan_i64(c64.p, M.bptr.p, p, s);
      M.nnzb = d2h(M.bptr.p + p, s);
      M.bcol.alloc(M.nnzb, s);
      // bcol first (needed by the offsets), then offsets, then values
      launch(k_pool_to_vb<T>, grid_for(p, 8), 256, 0, s, p, lstart.p, lcol.p, lvo.p, lval.p, M.bptr.p, nullptr,
             M.bcol.p, nullptr);
      VB_LAUNCH_CHECK();
      finish_offsets(M, s);
      launch(k_pool_to_vb<T>, grid_for(p, 8), 256, 0, s, p, lstart.p, lcol.p, lvo.p, lval.p, M.bptr.p, M.voff.p,
             M.bcol.p, M.val.p);
      VB_LAUNCH_CHECK();
    }
    // assemble U from the records
    {
      VBDev<T>& M = X.U;
      M.bptr.alloc(p + 1, s);
      DBuf<int32_t> ucnt(p, s);
      DBuf<int64_t> c64(p, s);
      launch(k_rec_to_vb<T>, grid_for(p, 8), 256, 0, s, p, 0, done.p, upool.p, ucnt.p, nullptr, nullptr, nullptr,
             nullptr);
      launch(k_count_to_i64, grid_for(p, 256), 256, 0, s, p, ucnt.p, c64.p);
      VB_LAUNCH_CHECK();
      scan_i64(c64.p, M.bptr.p, p, s);
      M.nnzb = d2h(M.bptr.p + p, s);
      M.bcol.alloc(M.nnzb, s);
      launch(k_rec_to_vb<T>, grid_for(p, 8), 256, 0, s, p, 1, done.p, upool.p, nullptr, M.bptr.p, nullptr, M.bcol.p,
             nullptr);
      VB_LAUNCH_CHECK();
      finish_offsets(M, s);
      launch(k_rec_to_vb<T>, grid_for(p, 8), 256, 0, s, p, 2, done.p, upool.p, nullptr, M.bptr.p, M.voff.p, M.bcol.p,
             M.val.p);
      VB_LAUNCH_CHECK();
    }
    return;
  }
  fail(VB_ENOMEM, "vbarms_factor: last-level ILUT workspace could not be sized");
}



namespace {
__global__ void k_dom_start(int64_t p, int ndom, const int32_t* __restrict__ dom, int64_t* __restrict__ start) {
  for (int d = blockIdx.x * blockDim.x + threadIdx.x; d <= ndom; d += gridDim.x * blockDim.x) {
    int64_t lo = 0, hi = p;  // first row with dom >= d
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if (dom[mid] < d)
        lo = mid + 1;
      else
        hi = mid;
    }
    start[d] = lo;
  }
}

// Row r, the j-th of block d, goes to position
//   sum_{d'} min(len_d', j) + #{d' < d : len_d' > j},
// its place when the blocks' rows are dealt out one per block in turn.
__global__ void k_ticket_pos(int64_t p, int ndom, const int32_t* __restrict__ dom, const int64_t* __restrict__ start,
                             int32_t* __restrict__ order) {
  extern __shared__ int64_t lens[];
  for (int d = threadIdx.x; d < ndom; d += blockDim.x) lens[d] = start[d + 1] - start[d];
  __syncthreads();
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < p; r += (int64_t)gridDim.x * blockDim.x) {
    const int d = dom[r];
    const int64_t j = r - start[d];
    int64_t pos = 0;
    for (int e = 0; e < ndom; ++e) {
      const int64_t le = lens[e];
      pos += le < j ? le : j;
      if (e < d && le > j) ++pos;
    }
    order[pos] = (int32_t)r;
  }
}

__global__ void k_take_i32(int64_t n, const int32_t* __restrict__ src, const int32_t* __restrict__ idx,
                           int32_t* __restrict__ dst) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
    dst[k] = src[idx[k]];
}
}  // namespace

void ticket_order(const int32_t* dom, int64_t p, int ndom, DBuf<int32_t>& order, cudaStream_t s) {
  if (p == 0 || ndom <= 1 || ndom > kTicketMaxDom) {
    order = DBuf<int32_t>();
    return;
  }
  DBuf<int64_t> start(ndom + 1, s);
  launch(k_dom_start, grid_for(ndom + 1, 256), 256, 0, s, p, ndom, dom, start.p);
  VB_LAUNCH_CHECK();
  order.alloc(p, s);
  launch(k_ticket_pos, grid_for(p, 256), 256, (size_t)ndom * sizeof(int64_t), s, p, ndom, dom, start.p, order.p);
  VB_LAUNCH_CHECK();
}

void take_i32(const int32_t* src, const int32_t* idx, int64_t n, int32_t* dst, cudaStream_t s) {
  if (n == 0) return;
  launch(k_take_i32, grid_for(n, 256), 256, 0, s, n, src, idx, dst);
  VB_LAUNCH_CHECK();
}

template void ilut_last<double>(LastDev<double>&, double, int, bool, double, uint64_t, cudaStream_t, int*,
                                 const int32_t*);
template void ilut_last<float>(LastDev<float>&, double, int, bool, double, uint64_t, cudaStream_t, int*,
                                const int32_t*);

}  // namespace vb

namespace vb {

namespace {

// Level of every row in the dependency DAG of a triangular block pattern:
// lev[i] = 1 + max lev[k] over the row's block columns k (0 without
// blocks).  The warps of a persistent grid take 32 rows at a time in dependency
// order (forward, for L: ascending, every column below the row; backward, for
// U: descending, every column above), one row a lane; every turn of the warp
// each lane looks once at the column it stands at, so rows of one warp may
// depend on one another.  A row publishes lev + 1 (-1 when it failed) in its
// word with one store, so the word is both flag and value and needs no fence.
// The lanes take their columns from the far end to the near one, which is ready
// last.  The first half of the grid does L, the second U, at the same time.
//
// Bound: the DAG's depth times a hop through L2, while enough rows are in
// flight: consecutive rows depend on one another, so a window of a warp per row
// (4 864 rows a side) kept the whole at the pace of the rows' order.  With a
// lane per row (78 000 a side) 3.0 million unknowns (327 000 rows, 2 650 levels)
// take 3 ms instead of 15.7, a batch of 24 matrices 1.1
// instead of 22.4, 48 000 unknowns at tau 0.9 3.8 instead of 9.0.
struct DagSide {
  int64_t p;
  const int64_t* bptr;
  const int32_t* bcol;
  int32_t* word;  // 0 until published, then lev + 1 (or -1)
  unsigned long long* tick;
  int* depth;
};

__global__ void __launch_bounds__(256)
    k_dag_level(DagSide fw, DagSide bw, unsigned half, int* __restrict__ abort, unsigned long long limit, int* st) {
  const bool back = blockIdx.x >= half;
  const DagSide D = back ? bw : fw;
  const int lane = threadIdx.x & 31;
  int deepest = 0;
  for (;;) {
    long long t = 0;
    if (lane == 0) t = (long long)atomicAdd(D.tick, 1ULL);
    t = __shfl_sync(0xffffffffu, t, 0) * 32 + lane;
    if (!__any_sync(0xffffffffu, t < D.p)) break;
    const int64_t i = back ? D.p - 1 - t : t;
    bool wait = t < D.p;
    int64_t b = 0;
    int left = 0, l = 0;
    if (wait) {  // from the first block (L) or the last one (U) to the row's other end
      b = back ? D.bptr[i + 1] - 1 : D.bptr[i];
      left = (int)(D.bptr[i + 1] - D.bptr[i]);
    }
    unsigned long long t0 = 0;
    for (unsigned it = 1; __any_sync(0xffffffffu, wait); ++it) {
      bool moved = false;
      if (wait) {
        int v = 1;
        if (left > 0) v = ld_relaxed_gpu(D.word + D.bcol[b]);
        if (v != 0) {
          moved = true;
          if (left > 0) l = max(l, v);  // v = lev[k] + 1
          b += back ? -1 : 1;
          --left;
          if (left <= 0 || v < 0) {
            if (v > 0) deepest = max(deepest, l + 1);
            asm volatile("st.relaxed.gpu.global.b32 [%0], %1;" ::"l"(D.word + i), "r"(v < 0 ? -1 : l + 1) : "memory");
            wait = false;
          }
        }
      }
      if (__any_sync(0xffffffffu, moved)) {
        t0 = 0;
        continue;
      }
      __nanosleep(32);
      if ((it & 63) == 0) {
        if (*((volatile int*)abort) != 0) return;
        const unsigned long long now = global_ns();
        if (t0 == 0) t0 = now;
        if (now - t0 > limit) {
          dev_fail(st, DEV_ETIMEOUT);
          atomicExch(abort, 1);
          return;
        }
      }
    }
  }
  deepest = warp_max_i(deepest);
  if (lane == 0 && deepest) atomicMax(D.depth, deepest);
}

// word = lev + 1 -> lev
__global__ void k_dag_unword(int64_t n, int32_t* __restrict__ w) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    w[i] -= 1;
}

// Stable least-significant-digit radix sort of row ids by their level, 8
// bits a pass: per block of RS_T ids a digit histogram, one scan over
// (digit, block), then every id goes to its digit's range after the ids of
// earlier blocks and of earlier warps and lanes of its own block.
constexpr int RS_T = 256;

__global__ void k_rs_init(int64_t n, bool descending, int32_t* __restrict__ v) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    v[i] = (int32_t)(descending ? n - 1 - i : i);
}

__global__ void __launch_bounds__(RS_T) k_rs_hist(int64_t n, const int32_t* __restrict__ v,
                                                  const int32_t* __restrict__ key, int shift, int64_t nblk,
                                                  int32_t* __restrict__ hist) {
  __shared__ int h[256];
  for (int d = threadIdx.x; d < 256; d += blockDim.x) h[d] = 0;
  __syncthreads();
  const int64_t e = blockIdx.x * (int64_t)RS_T + threadIdx.x;
  if (e < n) atomicAdd(&h[(key[v[e]] >> shift) & 255], 1);
  __syncthreads();
  for (int d = threadIdx.x; d < 256; d += blockDim.x) hist[(int64_t)d * nblk + blockIdx.x] = h[d];
}

__global__ void __launch_bounds__(RS_T) k_rs_scatter(int64_t n, const int32_t* __restrict__ v,
                                                     const int32_t* __restrict__ key, int shift, int64_t nblk,
                                                     const int64_t* __restrict__ base, int32_t* __restrict__ out) {
  __shared__ int cnt[RS_T / 32][256];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int x = threadIdx.x; x < (RS_T / 32) * 256; x += blockDim.x) (&cnt[0][0])[x] = 0;
  __syncthreads();
  const int64_t e = blockIdx.x * (int64_t)RS_T + threadIdx.x;
  const bool has = e < n;
  const int32_t id = has ? v[e] : 0;
  const int d = has ? (key[id] >> shift) & 255 : 256;
  const unsigned peers = __match_any_sync(0xffffffffu, d);
  const int rank = __popc(peers & ((1u << lane) - 1u));
  if (has && rank == 0) cnt[warp][d] = __popc(peers);
  __syncthreads();
  if (has) {
    int off = 0;
    for (int w = 0; w < warp; ++w) off += cnt[w][d];
    out[base[(int64_t)d * nblk + blockIdx.x] + off + rank] = id;
  }
}

}  // namespace

// Level orders of the last level's L (forward sweep) and U (backward sweep)
// on the device: the levels of both dependency DAGs (k_dag_level), then each
// side's rows sorted by level, rows ascending (L) / descending (U) within a
// level.
template <typename T>
void level_orders(LastDev<T>& X, uint64_t wait_limit, int* dst, cudaStream_t s) {
  const int64_t p = X.L.nbr;
  X.lorder.alloc(std::max<int64_t>(p, 1), s);
  X.uorder.alloc(std::max<int64_t>(p, 1), s);
  X.ldepth = X.udepth = 0;
  if (p == 0) return;
  DBuf<int32_t> lev(2 * p, s);
  DBuf<unsigned long long> tick(2, s);
  DBuf<int> abort(1, s), dmax(2, s);
  lev.zero();
  tick.zero();
  abort.zero();
  dmax.zero();
  int dev = 0, nsm = 0;
  VB_CUDA(cudaGetDevice(&dev));
  VB_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  const unsigned half = (unsigned)std::max<int64_t>(1, std::min<int64_t>((int64_t)nsm * 2, (p + 255) / 256));
  DagSide fw{p, X.L.bptr.p, X.L.bcol.p, lev.p, tick.p, dmax.p};
  DagSide bw{p, X.U.bptr.p, X.U.bcol.p, lev.p + p, tick.p + 1, dmax.p + 1};
  launch(k_dag_level, 2 * half, 256, 0, s, fw, bw, half, abort.p, (unsigned long long)wait_limit, dst);
  VB_LAUNCH_CHECK();
  check_status(dst, s, "vbarms_factor: level order of the triangular sweeps");
  launch(k_dag_unword, grid_for(2 * p, 256), 256, 0, s, 2 * p, lev.p);
  VB_LAUNCH_CHECK();
  const std::vector<int> dd = d2h_vec(dmax.p, 2, s);
  X.ldepth = dd[0];
  X.udepth = dd[1];
  const int64_t nblk = (p + RS_T - 1) / RS_T;
  DBuf<int32_t> hist(256 * nblk, s);
  DBuf<int64_t> base(256 * nblk + 1, s);
  for (int side = 0; side < 2; ++side) {
    const int32_t* key = lev.p + side * p;
    const int64_t depth = side == 0 ? X.ldepth : X.udepth;
    DBuf<int32_t> a(p, s), b(p, s);
    launch(k_rs_init, grid_for(p, 256), 256, 0, s, p, side == 1, a.p);
    VB_LAUNCH_CHECK();
    for (int shift = 0; shift < 31 && (1LL << shift) < depth; shift += 8) {
      launch(k_rs_hist, (unsigned)nblk, RS_T, 0, s, p, a.p, key, shift, nblk, hist.p);
      VB_LAUNCH_CHECK();
      scan_i32_to_i64(hist.p, base.p, 256 * nblk, s);
      launch(k_rs_scatter, (unsigned)nblk, RS_T, 0, s, p, a.p, key, shift, nblk, base.p, b.p);
      VB_LAUNCH_CHECK();
      std::swap(a, b);
    }
    (side == 0 ? X.lorder : X.uorder) = std::move(a);
  }
}

template void level_orders<double>(LastDev<double>&, uint64_t, int*, cudaStream_t);
template void level_orders<float>(LastDev<float>&, uint64_t, int*, cudaStream_t);

}  // namespace vb
