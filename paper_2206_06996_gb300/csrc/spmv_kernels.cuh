// Product kernels of one and three right-hand sides and their launch dispatch
// (spmv.cu), with the parts that the products of eight right-hand sides share
// (spmm.cu).
#pragma once
#include <cuda_bf16.h>

#include "epilogue.cuh"
#include "kernels.h"
#include "launch.cuh"

namespace scr {

// ------------------------------------------------------------ SpMV
// Blocks that a lane of a product keeps in flight.  Measured on the 616k-node
// tube: FP64 rows gain from the lower register count of two, FP32 rows from
// four; with 4 or more right-hand sides a block already brings NRHS gathers
// per value: one block per lane pass keeps the registers in bounds.
template <int NRHS, typename VT>
constexpr int kBatch = NRHS > 3 ? 1 : (sizeof(VT) == 8 ? 2 : 4);

// U blocks t0, t0 + G, ... of a scalar row (BC values each, contiguous in the
// slab layout): the column indices and values are loaded together, then every
// gather of the batch, then the multiply-adds, so a lane keeps U independent
// load chains outstanding and every stored value costs one multiply-add
template <int BC, int U, int G, typename VT, typename AT>
struct RowBatch {
  int cidx[U];
  AT a[U][BC];
  __device__ __forceinline__ void load(const int* __restrict__ cr, const VT* __restrict__ vr, int t0, int k) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int t = t0 + u * G;
      cidx[u] = t < k ? __ldg(cr + t) : -1;
#pragma unroll
      for (int c = 0; c < BC; ++c) a[u][c] = t < k ? (AT)__ldg(vr + t * BC + c) : (AT)0;
    }
  }
  template <int NRHS, typename XT>
  __device__ __forceinline__ void multiply(const XT* x, AT (&acc)[NRHS]) const {
    AT xv[U][BC][NRHS];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const bool ok = cidx[u] >= 0;
      const long long xb = (long long)(ok ? cidx[u] : 0) * BC * NRHS;
#pragma unroll
      for (int c = 0; c < BC; ++c)
#pragma unroll
        for (int h = 0; h < NRHS; ++h) xv[u][c][h] = ok ? (AT)x[xb + c * NRHS + h] : (AT)0;
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int c = 0; c < BC; ++c)
#pragma unroll
        for (int h = 0; h < NRHS; ++h)
          if (cidx[u] >= 0) acc[h] = fma(a[u][c], xv[u][c][h], acc[h]);
  }
};

// L2 prefetch of the stored values (BS per block) and column indices of the
// blocks [b0, b1) in the slab layout, cut as below
template <int BS, typename VT>
__device__ __forceinline__ void l2_prefetch_blocks(const int* __restrict__ col, const VT* __restrict__ val,
                                                   long long b0, long long b1) {
  const unsigned long long v0 = __cvta_generic_to_global(val + b0 * BS) & ~15ULL;
  const unsigned long long v1 = __cvta_generic_to_global(val + b1 * BS) & ~15ULL;
  const unsigned long long c0 = __cvta_generic_to_global(col + b0) & ~15ULL;
  const unsigned long long c1 = __cvta_generic_to_global(col + b1) & ~15ULL;
  if (v1 > v0)
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(v0), "r"((unsigned)(v1 - v0)) : "memory");
  if (c1 > c0)
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(c0), "r"((unsigned)(c1 - c0)) : "memory");
}

// L2 prefetch (cp.async.bulk.prefetch.L2) of the stored values and column
// indices that the CTA with index cta (256 threads, 256 / G scalar rows)
// will read.  The range is cut to whole 16-byte lines inside it: the first
// line may start up to 15 bytes before the range (the same line as a valid
// byte), the last partial line is left out, so no line outside the arrays
// is named.
template <int BR, int BC, int G, typename VT>
__device__ __forceinline__ void l2_prefetch_rows(const int* __restrict__ rp, const int* __restrict__ col,
                                                 const VT* __restrict__ val, int nbr, long long cta) {
  const long long nrows = (long long)nbr * BR;
  const long long o0 = cta * (256 / G);
  if (o0 >= nrows) return;
  const long long o1 = o0 + 256 / G < nrows ? o0 + 256 / G : nrows;
  l2_prefetch_blocks<BR * BC>(col, val, __ldg(rp + o0 / BR), __ldg(rp + (o1 - 1) / BR + 1));
}

// v[j] for a j known at run time, without an indexed register array
template <int N, typename T>
__device__ __forceinline__ T select_of(const T (&v)[N], int j) {
  T w = v[0];
#pragma unroll
  for (int i = 1; i < N; ++i)
    if (j == i) w = v[i];
  return w;
}

// A row listed as long (DBsr::lrow), summed by a CTA of its own.  The bench
// tube has one node per cross-section, its axis, that is joined to 291 others
// where the rest have 15: a lane group walks such a row in a chain of
// dependent loads long after the other rows of its wave are done.  The long
// rows' CTAs come first in the grid.  Measured (Chebyshev step): FP32 16-byte
// kernel on the 616k-node tube 103 -> 82 us; FP64, 2 lanes per scalar row, 6000
// rows of 15 with one of 75 in 149: 8.3 us with a warp per long scalar row,
// 6.2 us with a CTA per long block row (5.0 us without any).
template <int BR, int BC, int NRHS, typename VT, typename XT, Epi E>
__device__ __forceinline__ void long_row_cta(int i, const int* __restrict__ rp, const int* __restrict__ col,
                                             const VT* __restrict__ val, const XT* x, const Epilogue<XT, E>& epi) {
  constexpr int N = BR * NRHS;
  __shared__ XT part[8][N];
  const int s = __ldg(rp + i), k = __ldg(rp + i + 1) - s;
  const VT* v = val + (long long)s * BR * BC;
  pdl_wait_prev();
  const int q = threadIdx.x;
  typename Epilogue<XT, E>::Operands op;
  if (q < N) op = epi.load((long long)i * N + q, (long long)i * BR + q / NRHS);
  XT acc[BR][NRHS];
#pragma unroll
  for (int r = 0; r < BR; ++r)
#pragma unroll
    for (int h = 0; h < NRHS; ++h) acc[r][h] = (XT)0;
  for (int t = q; t < k; t += 256) {
    const long long xb = (long long)__ldg(col + s + t) * BC * NRHS;
#pragma unroll
    for (int c = 0; c < BC; ++c) {
      XT xv[NRHS];
#pragma unroll
      for (int h = 0; h < NRHS; ++h) xv[h] = x[xb + c * NRHS + h];
#pragma unroll
      for (int r = 0; r < BR; ++r) {
        const XT a = (XT)__ldg(v + (long long)r * k * BC + t * BC + c);
#pragma unroll
        for (int h = 0; h < NRHS; ++h) acc[r][h] = fma(a, xv[h], acc[r][h]);
      }
    }
  }
#pragma unroll
  for (int r = 0; r < BR; ++r)
#pragma unroll
    for (int h = 0; h < NRHS; ++h) {
      const XT w = warp_sum(acc[r][h]);
      if ((q & 31) == 0) part[q >> 5][r * NRHS + h] = w;
    }
  __syncthreads();
  if (q < N) {
    XT w = (XT)0;
#pragma unroll
    for (int j = 0; j < 8; ++j) w += part[j][q];
    epi.store((long long)i * N + q, w, op);
  }
}

// Rows of more than two rounds of their group (eight rounds of one-column
// blocks), and of more than 32 blocks, are summed by the whole warp (the block
// operator and Algorithm 2's last line, whose rows span matrices).
template <int BC, int G, int U>
constexpr int kLongRow = (BC == 3 ? 2 : 8) * G * U > 32 ? (BC == 3 ? 2 : 8) * G * U : 32;

// the warp's long rows (lanes with lng: each G-group's lanes agree), one after
// another: the 32 lanes take the row's blocks in turn and the sum is added to
// the group's first lane (the caller sums the group's lanes); every lane of
// the warp calls it
template <int BR, int BC, int NRHS, int G, typename VT, typename XT, typename AT>
__device__ __forceinline__ void long_rows(const int* __restrict__ col, const VT* __restrict__ val,
                                          const XT* x, bool lng, int s, int k, int r,
                                          AT (&acc)[NRHS]) {
  const int wl = threadIdx.x & 31;
  unsigned todo = __ballot_sync(0xffffffffu, lng && wl % G == 0);
  while (todo) {
    const int src = __ffs(todo) - 1;
    todo &= todo - 1;
    const int ss = __shfl_sync(0xffffffffu, s, src), kk = __shfl_sync(0xffffffffu, k, src);
    const int rr = __shfl_sync(0xffffffffu, r, src);
    const VT* vr = val + (long long)ss * BR * BC + (long long)rr * kk * BC;
    AT a[NRHS];
#pragma unroll
    for (int h = 0; h < NRHS; ++h) a[h] = (AT)0;
#pragma unroll 4
    for (int t = wl; t < kk; t += 32) {
      const long long xb = (long long)__ldg(col + ss + t) * BC * NRHS;
#pragma unroll
      for (int c = 0; c < BC; ++c) {
        const AT v = (AT)__ldg(vr + t * BC + c);
#pragma unroll
        for (int h = 0; h < NRHS; ++h) a[h] = fma(v, (AT)x[xb + c * NRHS + h], a[h]);
      }
    }
#pragma unroll
    for (int h = 0; h < NRHS; ++h) {
      a[h] = warp_sum(a[h]);
      if (wl == src) acc[h] += a[h];
    }
  }
}

// the lanes of a G-group accumulate scalar row r of block row i of M into
// acc[h] (each its share: the caller adds them up); every lane of the warp
// calls it, those without a row with ok = false
template <int BR, int BC, int NRHS, int G, typename VT, typename XT, typename AT>
__device__ __forceinline__ void scalar_row_accum(const int* __restrict__ rp, const int* __restrict__ col,
                                                 const VT* __restrict__ val, const XT* x, bool ok,
                                                 int i, int r, int lane, AT (&acc)[NRHS]) {
  constexpr int U = kBatch<NRHS, VT>;
  int s = 0, k = 0;
  if (ok) s = __ldg(rp + i), k = __ldg(rp + i + 1) - s;
  const bool lng = k > kLongRow<BC, G, U>;
  const int kn = lng ? 0 : k;
  const VT* vr = val + (long long)s * BR * BC + (long long)r * k * BC;
  RowBatch<BC, U, G, VT, AT> bt;
  for (int t0 = lane; t0 < kn; t0 += G * U) {
    bt.load(col + s, vr, t0, kn);
    bt.template multiply<NRHS>(x, acc);
  }
  long_rows<BR, BC, NRHS, G>(col, val, x, lng, s, k, r, acc);
}

// One G-group of lanes per scalar row.  The matrix (row pointers, the first
// batch of column indices and values) is read before the wait for the
// predecessor: launched early, it is settled, so that in a chain of short
// products only the gathers of x, the sums and the epilogue remain after the
// wait; the epilogue's operands are read with the gathers.
template <int BR, int BC, int NRHS, int G, typename VT, typename XT, typename AT, Epi E>
__global__ void __launch_bounds__(256) k_spmv(int nbr, const int* __restrict__ rp, const int* __restrict__ col,
                                              const VT* __restrict__ val, const XT* x, Epilogue<XT, E> epi, int pf,
                                              const int* __restrict__ lrow, int nl, int lthr) {
  constexpr int U = kBatch<NRHS, VT>;
  pdl_allow_next();
  if ((int)blockIdx.x < nl) {
    long_row_cta<BR, BC, NRHS>(__ldg(lrow + blockIdx.x), rp, col, val, x, epi);
    return;
  }
  const long long cta = (long long)blockIdx.x - nl;
  const long long o = (cta * blockDim.x + threadIdx.x) / G;  // scalar row
  const int lane = threadIdx.x % G;
  const long long nrows = (long long)nbr * BR;
  const int i = o < nrows ? (int)(o / BR) : 0, r = (int)(o - (long long)i * BR);
  int s = 0, k = 0;
  if (o < nrows) s = __ldg(rp + i), k = __ldg(rp + i + 1) - s;
  const bool active = o < nrows && k <= lthr;  // the others still join the shuffles
  if (!active) k = 0;
  const VT* vr = val + (long long)s * BR * BC + (long long)r * k * BC;
  const int* cr = col + s;
  RowBatch<BC, U, G, VT, AT> bt;
  bt.load(cr, vr, lane, k);
  pdl_wait_prev();
  if (pf > 0 && threadIdx.x == 0) l2_prefetch_rows<BR, BC, G, VT>(rp, col, val, nbr, cta + pf);
  // the columns are dealt to the group's lanes for the epilogue: lane, lane + G, ...
  constexpr int Q = (NRHS + G - 1) / G;
  AT acc[NRHS];
#pragma unroll
  for (int h = 0; h < NRHS; ++h) acc[h] = (AT)0;
  typename Epilogue<XT, E>::Operands op[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q)
    if (active && lane + q * G < NRHS) op[q] = epi.load(o * NRHS + lane + q * G, o);
  for (int t0 = lane; t0 < k;) {
    bt.template multiply<NRHS>(x, acc);
    t0 += G * U;
    bt.load(cr, vr, t0, k);
  }
  if constexpr (G > 1) {
#pragma unroll
    for (int h = 0; h < NRHS; ++h) {
#pragma unroll
      for (int off = G / 2; off > 0; off >>= 1) acc[h] += __shfl_xor_sync(0xffffffffu, acc[h], off, G);
    }
  }
#pragma unroll
  for (int q = 0; q < Q; ++q)
    if (active && lane + q * G < NRHS) epi.store(o * NRHS + lane + q * G, select_of<NRHS>(acc, lane + q * G), op[q]);
}

// 3x3 blocks, one right-hand side: 3 M lanes per block row, 32 / (3 M) rows
// per warp.  A lane takes blocks of the row in turn and keeps the three row
// sums; the three lanes of a triple then exchange two partial sums each, so
// that lane r ends with scalar row r and runs its epilogue.
// What bounds FP64 products here is the FP64 pipe (2 lanes per SM and clock,
// a warp instruction takes 16 clocks whatever lanes are active), so this
// counts: for 10 rows of 15 blocks the warp issues 45 multiply-adds, 2 sums
// and 4 epilogue operations, against 24 + 1 + 4 for 5.3 rows with two lanes
// per scalar row (half of the epilogue's lanes idle), and each source value is
// loaded once for three multiply-adds instead of once for each.  Measured
// (Chebyshev step, us): 616k-node tube FP64 225 -> 181, FP32 103 -> 78 with one
// triple; FP32 77k rows of 16 blocks 20 -> 13.4 with two.  Few rows want more
// lanes (6000 rows, FP64: 6.0, 4.7, 5.9 us with 1, 2, 5 triples, 5.0 with the
// scalar-row kernel): the autotuner times them all.
template <int M, typename VT, typename XT, Epi E>
__global__ void __launch_bounds__(256) k_spmv_tri(int nbr, const int* __restrict__ rp, const int* __restrict__ col,
                                                  const VT* __restrict__ val, const XT* x, Epilogue<XT, E> epi, int pf,
                                                  const int* __restrict__ lrow, int nl, int lthr) {
  constexpr int G = 3 * M, W = 32 / G;  // lanes per row, rows per warp
  pdl_allow_next();
  if ((int)blockIdx.x < nl) {
    long_row_cta<3, 3, 1>(__ldg(lrow + blockIdx.x), rp, col, val, x, epi);
    return;
  }
  const long long cta = (long long)blockIdx.x - nl;
  const int wl = threadIdx.x & 31, g = wl / G, p = wl - g * G;
  const long long i = (cta * 8 + (threadIdx.x >> 5)) * W + g;
  int s = 0, k = 0;
  if (g < W && i < nbr) s = __ldg(rp + i), k = __ldg(rp + i + 1) - s;
  const bool active = g < W && i < nbr && k <= lthr;  // the others still join the shuffles
  if (!active) k = 0;
  const int* cr = col + s;
  const VT* vr = val + 9LL * s;
  int c = 0;
  XT a[3][3];
  auto load = [&](int t) {
    if (t < k) {
      c = __ldg(cr + t);
#pragma unroll
      for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int q = 0; q < 3; ++q) a[r][q] = (XT)__ldg(vr + 3LL * r * k + 3 * t + q);
    }
  };
  load(p);
  pdl_wait_prev();
  if (pf > 0 && threadIdx.x == 0) {
    const long long i0 = (cta + pf) * 8 * W, i1 = i0 + 8 * W < nbr ? i0 + 8 * W : nbr;
    if (i0 < nbr) l2_prefetch_blocks<9>(col, val, __ldg(rp + i0), __ldg(rp + i1));
  }
  typename Epilogue<XT, E>::Operands op;
  if (active && p < 3) op = epi.load(3 * i + p, 3 * i + p);
  XT acc[3] = {(XT)0, (XT)0, (XT)0};
  for (int t = p; t < k;) {
    XT xv[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) xv[q] = x[3LL * c + q];
#pragma unroll
    for (int q = 0; q < 3; ++q)
#pragma unroll
      for (int r = 0; r < 3; ++r) acc[r] = fma(a[r][q], xv[q], acc[r]);
    t += G;
    load(t);
  }
  // lane p of a triple collects row p: step d brings lane (p + d) % 3's share
  const int tri = wl - p % 3, p3 = p % 3;
  XT sum = select_of<3>(acc, p3);
#pragma unroll
  for (int d = 1; d < 3; ++d) {
    const XT give = select_of<3>(acc, (p3 + 3 - d) % 3);  // this lane is (receiver + d) % 3
    sum += __shfl_sync(0xffffffffu, give, (tri + (p3 + d) % 3) & 31);
  }
  // the row's M triples
#pragma unroll
  for (int m = 1; m < M; ++m) {
    const XT w = __shfl_sync(0xffffffffu, sum, (wl + 3 * m) & 31);
    if (p < 3) sum += w;
  }
  if (active && p < 3) epi.store(3 * i + p, sum, op);
}

// G lanes per BLOCK row: each lane takes blocks t = lane, lane+G, ... and
// accumulates all BR scalar rows, so the column index and the BC source
// values of a block are loaded once for its BR x BC multiply-adds; the
// BR*NRHS sums are combined over the G lanes and written by distinct lanes.
template <int BR, int BC, int NRHS, int G, typename VT, typename XT, typename AT, Epi E>
__global__ void __launch_bounds__(256) k_spmv_brow(int nbr, const int* __restrict__ rp, const int* __restrict__ col,
                                                   const VT* __restrict__ val, const XT* __restrict__ x,
                                                   Epilogue<XT, E> epi) {
  const long long i = (blockIdx.x * (long long)blockDim.x + threadIdx.x) / G;  // block row
  const int lane = threadIdx.x % G;
  const bool active = i < nbr;
  AT acc[BR][NRHS];
#pragma unroll
  for (int r = 0; r < BR; ++r)
#pragma unroll
    for (int h = 0; h < NRHS; ++h) acc[r][h] = (AT)0;
  if (active) {
    const int s = __ldg(rp + i), k = __ldg(rp + i + 1) - s;
    const VT* v0 = val + (long long)s * BR * BC;
    const int* cr = col + s;
#pragma unroll 2
    for (int t = lane; t < k; t += G) {
      const long long xb = (long long)__ldg(cr + t) * BC * NRHS;
      AT xv[BC][NRHS];
#pragma unroll
      for (int c = 0; c < BC; ++c)
#pragma unroll
        for (int h = 0; h < NRHS; ++h) xv[c][h] = (AT)__ldg(x + xb + c * NRHS + h);
#pragma unroll
      for (int r = 0; r < BR; ++r) {
        const VT* vt = v0 + (long long)r * k * BC + t * BC;
#pragma unroll
        for (int c = 0; c < BC; ++c) {
          const AT a = (AT)__ldg(vt + c);
#pragma unroll
          for (int h = 0; h < NRHS; ++h) acc[r][h] = fma(a, xv[c][h], acc[r][h]);
        }
      }
    }
  }
  if constexpr (G > 1) {
#pragma unroll
    for (int r = 0; r < BR; ++r)
#pragma unroll
      for (int h = 0; h < NRHS; ++h)
#pragma unroll
        for (int off = G / 2; off > 0; off >>= 1) acc[r][h] += __shfl_xor_sync(0xffffffffu, acc[r][h], off, G);
  }
  if (active) {
#pragma unroll
    for (int q = 0; q < BR * NRHS; ++q) {
      if (q % G != lane) continue;
      const int r = q / NRHS, h = q - r * NRHS;
      const long long o = i * BR + r;
      epi(o * NRHS + h, o, acc[r][h]);
    }
  }
}

// ------------------------------------------------------------ 16-byte products
// Products on the padded copy of DBsr::vdesc.  Each lane takes a chunk of V
// = 16 / sizeof(VT) blocks (3x3) or entries (1x1) at a time and loads it
// with 16-byte vector loads: for a 3x3 chunk one index vector (V column
// indices) and three value vectors per scalar row, against V column loads
// and 3 V value loads per scalar row in the scalar-row kernel.
// The stored values and indices go through the read-only path with plain
// 16-byte loads (the padded copy starts every chunk on a 16-byte boundary).
// Measured inside the solve on the 616k-node tube (FP32, 4 lanes per block
// row): 115.5 us per level-0 product with plain loads, 127 us with
// L1::no_allocate / L2::256B hints on the value loads: a lane's three value
// vectors of one scalar row share sectors, which L1 then has to keep.
template <typename VT>
__device__ __forceinline__ void ldg16(const VT* p, VT* a) {
  if constexpr (sizeof(VT) == 4) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(p));
    a[0] = v.x, a[1] = v.y, a[2] = v.z, a[3] = v.w;
  } else {
    const double2 v = __ldg(reinterpret_cast<const double2*>(p));
    a[0] = v.x, a[1] = v.y;
  }
}
// 16 bytes of a vector (ordinary loads)
__device__ __forceinline__ void load16(const float* p, float* a) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  a[0] = v.x, a[1] = v.y, a[2] = v.z, a[3] = v.w;
}
__device__ __forceinline__ void load16(const double* p, double* a) {
  const double2 v = *reinterpret_cast<const double2*>(p);
  a[0] = v.x, a[1] = v.y;
}
template <int U>
__device__ __forceinline__ void ldg_idx(const int* p, int* c) {
  if constexpr (U == 4) {
    const int4 v = __ldg(reinterpret_cast<const int4*>(p));
    c[0] = v.x, c[1] = v.y, c[2] = v.z, c[3] = v.w;
  } else {
    const int2 v = __ldg(reinterpret_cast<const int2*>(p));
    c[0] = v.x, c[1] = v.y;
  }
}

// L2 prefetch (cp.async.bulk.prefetch.L2) of the padded values and column
// slots of the block rows [i0, i1) of a padded copy (3x3: int4 descriptors;
// 1x1: int2, values and slots sharing their starts).  Whole 16-byte lines
// inside the allocations only.
template <typename VT, bool SQ3>
__device__ __forceinline__ void l2_prefetch_vec(const void* desc, const int* __restrict__ col, const VT* __restrict__ val, long long i0,
                                                long long i1) {
  long long c0, c1, v0, v1;
  if constexpr (SQ3) {
    const int4 a = __ldg(static_cast<const int4*>(desc) + i0), b = __ldg(static_cast<const int4*>(desc) + i1 - 1);
    constexpr int V = 16 / (int)sizeof(VT);
    c0 = a.x, c1 = b.x + (b.y + V - 1) / V * V;
    v0 = a.z, v1 = b.z + 3LL * b.w;
  } else {
    constexpr int V = 16 / (int)sizeof(VT);
    const int2 a = __ldg(static_cast<const int2*>(desc) + i0), b = __ldg(static_cast<const int2*>(desc) + i1 - 1);
    c0 = v0 = a.x;
    c1 = v1 = b.x + (b.y + V - 1) / V * V;
  }
  // runs start on 16-byte boundaries except FP64 column slots (8 bytes): round
  // down the start and up the end (the arrays carry 16 entries of slack)
  const unsigned long long vb = __cvta_generic_to_global(val + v0) & ~15ULL;
  const unsigned long long ve = (__cvta_generic_to_global(val + v1) + 15) & ~15ULL;
  const unsigned long long cb = __cvta_generic_to_global(col + c0) & ~15ULL;
  const unsigned long long ce = (__cvta_generic_to_global(col + c1) + 15) & ~15ULL;
  if (ve > vb)
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(vb), "r"((unsigned)(ve - vb)) : "memory");
  if (ce > cb)
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(cb), "r"((unsigned)(ce - cb)) : "memory");
}

// a chunk of U = V blocks of a 3x3 block row on the padded copy: one index
// vector and three value vectors per scalar row
template <typename VT>
struct Chunk33 {
  static constexpr int V = 16 / (int)sizeof(VT), U = V;
  int c[U], m;  // m: blocks of the chunk (0: none)
  VT a[3][3 * U];
  __device__ __forceinline__ void load(const int* __restrict__ cr, const VT* v0, int rl, int j, int k) {
    m = k - j < U ? (k - j > 0 ? k - j : 0) : U;
    if (m) ldg_idx<U>(cr + j, c);
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        if (q * V < 3 * m) {
          ldg16<VT>(v0 + (long long)r * rl + 3 * j + q * V, &a[r][q * V]);
        } else {
#pragma unroll
          for (int e = 0; e < V; ++e) a[r][q * V + e] = (VT)0;
        }
      }
  }
  template <typename XT>
  __device__ __forceinline__ void multiply(const XT* x, XT (&acc)[3]) const {
    XT xv[U][3];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const long long xb = 3LL * (u < m ? c[u] : 0);
#pragma unroll
      for (int cc = 0; cc < 3; ++cc) xv[u][cc] = u < m ? x[xb + cc] : (XT)0;
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int cc = 0; cc < 3; ++cc)
#pragma unroll
        for (int r = 0; r < 3; ++r)
          if (u < m) acc[r] = fma((XT)a[r][3 * u + cc], xv[u][cc], acc[r]);
  }
};

// 3x3 blocks, one right-hand side: G lanes per block row, each lane takes
// chunks of V blocks in turn and accumulates all three scalar rows, so a
// block's column index and its three source values are loaded once for its 9
// multiply-adds.  The three row sums are combined over the G lanes and
// written by lanes 0, 1, 2 (mod G).  Rows of more than lthr blocks are the CTAs'
// of long_row_cta; loads before the wait as in k_spmv.
template <int G, typename VT, typename XT, Epi E>
__global__ void __launch_bounds__(256, sizeof(VT) == 4 ? 4 : 3) k_spmv_vec33(int nbr, const int4* __restrict__ desc, const int* __restrict__ col,
                                                    const VT* __restrict__ val, const XT* x,
                                                    Epilogue<XT, E> epi, int pf, const int* __restrict__ rp,
                                                    const int* __restrict__ scol, const VT* __restrict__ sval,
                                                    const int* __restrict__ lrow, int nl, int lthr) {
  constexpr int U = Chunk33<VT>::U;
  pdl_allow_next();
  if ((int)blockIdx.x < nl) {  // long rows: from the slab copy
    long_row_cta<3, 3, 1>(__ldg(lrow + blockIdx.x), rp, scol, sval, x, epi);
    return;
  }
  const long long cta = (long long)blockIdx.x - nl;
  const long long i = (cta * blockDim.x + threadIdx.x) / G;
  const int lane = threadIdx.x % G;
  int4 d = make_int4(0, 0, 0, 0);
  if (i < nbr) d = __ldg(desc + i);
  const bool active = i < nbr && d.y <= lthr;  // the others still join the shuffles
  const int k = active ? d.y : 0;
  Chunk33<VT> ch;
  ch.load(col + d.x, val + d.z, d.w, lane * U, k);
  pdl_wait_prev();
  if (pf > 0 && threadIdx.x == 0) {
    const long long i0 = (cta + pf) * (256 / G);
    if (i0 < nbr) l2_prefetch_vec<VT, true>(desc, col, val, i0, i0 + 256 / G < nbr ? i0 + 256 / G : nbr);
  }
  constexpr int Q = (3 + G - 1) / G;
  typename Epilogue<XT, E>::Operands op[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q)
    if (active && lane + q * G < 3) op[q] = epi.load(3 * i + lane + q * G, 3 * i + lane + q * G);
  XT acc[3] = {(XT)0, (XT)0, (XT)0};
  for (int j = lane * U; j < k;) {
    ch.multiply(x, acc);
    j += G * U;
    if (j < k) ch.load(col + d.x, val + d.z, d.w, j, k);
  }
  if constexpr (G > 1) {
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int off = G / 2; off > 0; off >>= 1) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], off, G);
  }
#pragma unroll
  for (int q = 0; q < Q; ++q)
    if (active && lane + q * G < 3) epi.store(3 * i + lane + q * G, select_of<3>(acc, lane + q * G), op[q]);
}

// V entries of a 1x1 row on the padded copy
template <typename VT>
struct Chunk11 {
  static constexpr int V = 16 / (int)sizeof(VT);
  int c[V], m;
  VT a[V];
  __device__ __forceinline__ void load(const int* __restrict__ cr, const VT* __restrict__ vr, int j, int k) {
    m = k - j < V ? (k - j > 0 ? k - j : 0) : V;
    if (m) {
      ldg_idx<V>(cr + j, c);
      ldg16<VT>(vr + j, a);
    }
  }
  template <typename XT>
  __device__ __forceinline__ void multiply(const XT* x, XT& acc) const {
    XT xv[V];
#pragma unroll
    for (int u = 0; u < V; ++u) xv[u] = u < m ? x[c[u]] : (XT)0;
#pragma unroll
    for (int u = 0; u < V; ++u)
      if (u < m) acc = fma((XT)a[u], xv[u], acc);
  }
};

// 1x1 blocks, one right-hand side: G lanes per row, chunks of V entries
// (one 16-byte value load and one index load of V column indices); long rows
// as in k_spmv, from the slab copy.
template <int G, typename VT, typename XT, Epi E>
__global__ void __launch_bounds__(256) k_spmv_vec11(int nbr, const int2* __restrict__ desc, const int* __restrict__ col,
                                                    const VT* __restrict__ val, const XT* x,
                                                    Epilogue<XT, E> epi, int pf, const int* __restrict__ rp,
                                                    const int* __restrict__ scol, const VT* __restrict__ sval,
                                                    const int* __restrict__ lrow, int nl, int lthr) {
  constexpr int V = Chunk11<VT>::V;
  pdl_allow_next();
  if ((int)blockIdx.x < nl) {
    long_row_cta<1, 1, 1>(__ldg(lrow + blockIdx.x), rp, scol, sval, x, epi);
    return;
  }
  const long long cta = (long long)blockIdx.x - nl;
  const long long i = (cta * blockDim.x + threadIdx.x) / G;
  const int lane = threadIdx.x % G;
  pdl_wait_prev();
  if (pf > 0 && threadIdx.x == 0) {
    const long long i0 = (cta + pf) * (256 / G);
    if (i0 < nbr) l2_prefetch_vec<VT, false>(desc, col, val, i0, i0 + 256 / G < nbr ? i0 + 256 / G : nbr);
  }
  int2 d = make_int2(0, 0);
  if (i < nbr) d = __ldg(desc + i);
  const bool active = i < nbr && d.y <= lthr;  // the others still join the shuffles
  const int k = active ? d.y : 0;
  typename Epilogue<XT, E>::Operands op;
  if (active && lane == 0) op = epi.load(i, i);
  XT acc = (XT)0;
  for (int j = lane * V; j < k; j += G * V) {
    Chunk11<VT> ch;
    ch.load(col + d.x, val + d.x, j, k);
    ch.multiply(x, acc);
  }
  if constexpr (G > 1) {
#pragma unroll
    for (int off = G / 2; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off, G);
  }
  if (active && lane == 0) epi.store(i, acc, op);
}

// sliced block-ELL product: one lane per block row, no cross-lane sums
template <int BR, int BC, int NRHS, typename VT, typename XT, Epi E>
__global__ void __launch_bounds__(256) k_sell_spmv(DSell<VT> S, const XT* __restrict__ x, Epilogue<XT, E> epi) {
  const long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const int c = (int)(g / kChunk), lane = (int)(g % kChunk);
  if (c >= S.nchunk) return;
  const int q = c * kChunk + lane;
  if (q >= S.nbr) return;
  const int i = __ldg(S.perm + q);
  const int c0 = __ldg(S.cptr + c), L = __ldg(S.cptr + c + 1) - c0;
  const long long base = (long long)c0 * kChunk;
  const int* __restrict__ cl = S.col + base + lane;
  const VT* __restrict__ vl = S.val + base * (BR * BC) + lane;
  using AT = XT;
  AT acc[BR][NRHS];
#pragma unroll
  for (int r = 0; r < BR; ++r)
#pragma unroll
    for (int h = 0; h < NRHS; ++h) acc[r][h] = (AT)0;
#pragma unroll 2
  for (int t = 0; t < L; ++t) {
    const long long xb = (long long)__ldg(cl + (long long)t * kChunk) * BC * NRHS;
    AT xv[BC][NRHS];
#pragma unroll
    for (int cc = 0; cc < BC; ++cc)
#pragma unroll
      for (int h = 0; h < NRHS; ++h) xv[cc][h] = (AT)__ldg(x + xb + cc * NRHS + h);
    const VT* vt = vl + (long long)t * kChunk * (BR * BC);
#pragma unroll
    for (int r = 0; r < BR; ++r)
#pragma unroll
      for (int cc = 0; cc < BC; ++cc) {
        const AT a = (AT)__ldg(vt + (r * BC + cc) * kChunk);
#pragma unroll
        for (int h = 0; h < NRHS; ++h) acc[r][h] = fma(a, xv[cc][h], acc[r][h]);
      }
  }
#pragma unroll
  for (int r = 0; r < BR; ++r) {
    const long long o = (long long)i * BR + r;
#pragma unroll
    for (int h = 0; h < NRHS; ++h) epi(o * NRHS + h, o, acc[r][h]);
  }
}

// CTAs ahead for the L2 prefetch of the scalar-row kernel (0: off) and the
// forced kernel code of every product (0: per matrix); defined in spmv.cu
extern int g_l2_prefetch;

// the product kernels' launch: the long rows' CTAs first, then those of args
template <typename VT, typename... KArgs, typename... Args>
inline void launch_rows(const DBsr<VT>& M, void (*kern)(KArgs...), long long ctas, cudaStream_t s, Args... args) {
  const long long grid = ctas + M.nlong;
  launch_early(M.settled && early_grid(grid, sm_count()), kern, grid, 256, s, args..., M.lrow, M.nlong,
               M.lthr);
}

template <int BR, int BC, int NRHS, int G, typename VT, typename XT, typename AT, Epi E>
inline void launch_spmv_g(const DBsr<VT>& M, const XT* x, XT* y, const EpiArgs& e, cudaStream_t s) {
  const Epilogue<XT, E> epi = make_epilogue<XT, E>(x, y, e);
  const int blk = 256;
  bool done = false;
  if constexpr (BR == 3 && BC == 3 && NRHS == 1) {
    if (code_of(M) >= 400) {  // G: triples of lanes per block row
      constexpr int T = G > 4 ? 10 : G > 2 ? 5 : G;  // 10, 5, 2, 1, 1 rows per warp
      launch_rows(M, k_spmv_tri<T, VT, XT, E>, ceil_div(M.nbr, 8 * (32 / (3 * T))), s, M.nbr, (const int*)M.rp,
                  (const int*)M.col, (const VT*)M.val, x, epi, g_l2_prefetch);
      SCR_LAUNCH();
      return;
    }
  }
  if constexpr (sizeof(VT) >= 4 && NRHS == 1 && ((BR == 3 && BC == 3) || (BR == 1 && BC == 1))) {
    if (M.vdesc && code_of(M) >= 300 && code_of(M) < 400) {
      if constexpr (BR == 3) {
        const long long threads = (long long)M.nbr * G;
        launch_rows(M, k_spmv_vec33<G, VT, XT, E>, ceil_div(threads, blk), s, M.nbr, static_cast<const int4*>(M.vdesc),
                    (const int*)M.vcol, (const VT*)M.vval, x, epi, g_l2_prefetch, (const int*)M.rp, (const int*)M.col,
                    (const VT*)M.val);
      } else {
        const long long threads = (long long)M.nbr * G;
        launch_rows(M, k_spmv_vec11<G, VT, XT, E>, ceil_div(threads, blk), s, M.nbr, static_cast<const int2*>(M.vdesc),
                    (const int*)M.vcol, (const VT*)M.vval, x, epi, g_l2_prefetch, (const int*)M.rp, (const int*)M.col,
                    (const VT*)M.val);
      }
      done = true;
    }
  }
  if constexpr (sizeof(VT) >= 4 && NRHS <= 3) {  // BF16 values, multi-column products: scalar-row kernel only
    if (done) {
    } else if (M.sell) {
      const DSell<VT>& S = *static_cast<const DSell<VT>*>(M.sell);
      const long long threads = (long long)S.nchunk * kChunk;
      k_sell_spmv<BR, BC, NRHS, VT, XT, E><<<ceil_div(threads, blk), blk, 0, s>>>(S, x, epi);
      done = true;
    } else if (BR > 1 && code_of(M) > 0 && code_of(M) < 100) {
      const long long threads = (long long)M.nbr * G;
      k_spmv_brow<BR, BC, NRHS, G, VT, XT, AT, E><<<ceil_div(threads, blk), blk, 0, s>>>(M.nbr, M.rp, M.col,
                                                                                       M.val, x, epi);
      done = true;
    }
  }
  if (!done) {
    const long long threads = (long long)M.nbr * BR * G;
    launch_rows(M, k_spmv<BR, BC, NRHS, G, VT, XT, AT, E>, ceil_div(threads, blk), s, M.nbr, (const int*)M.rp,
                (const int*)M.col, (const VT*)M.val, x, epi, g_l2_prefetch);
  }
  SCR_LAUNCH();
}

template <int BR, int BC, int NRHS, int G, typename VT, typename XT>
inline void launch_spmv_e(const DBsr<VT>& M, const XT* x, XT* y, const EpiArgs& e, cudaStream_t s) {
  using AT = XT;  // accumulate in the vector precision
  switch (e.kind) {
    case Epi::Set: launch_spmv_g<BR, BC, NRHS, G, VT, XT, AT, Epi::Set>(M, x, y, e, s); break;
    case Epi::Axpby: launch_spmv_g<BR, BC, NRHS, G, VT, XT, AT, Epi::Axpby>(M, x, y, e, s); break;
    case Epi::Resid: launch_spmv_g<BR, BC, NRHS, G, VT, XT, AT, Epi::Resid>(M, x, y, e, s); break;
    case Epi::Jacobi: launch_spmv_g<BR, BC, NRHS, G, VT, XT, AT, Epi::Jacobi>(M, x, y, e, s); break;
    case Epi::ScaledSub: launch_spmv_g<BR, BC, NRHS, G, VT, XT, AT, Epi::ScaledSub>(M, x, y, e, s); break;
    case Epi::ChebFirst:
    case Epi::ChebStep:
    case Epi::ChebZero:
      if constexpr (BR == BC) {
        if (e.kind == Epi::ChebFirst) launch_spmv_g<BR, BC, NRHS, G, VT, XT, AT, Epi::ChebFirst>(M, x, y, e, s);
        else if (e.kind == Epi::ChebZero) launch_spmv_g<BR, BC, NRHS, G, VT, XT, AT, Epi::ChebZero>(M, x, y, e, s);
        else launch_spmv_g<BR, BC, NRHS, G, VT, XT, AT, Epi::ChebStep>(M, x, y, e, s);
      } else {
        throw CudaError{cudaErrorInvalidValue, "Chebyshev epilogue on a non-square block shape"};
      }
      break;
  }
}

// lanes per scalar row: FP64 keeps groups narrow (FP64 adds of the
// reduction compete with the products), FP32 widens them for coalescing
// M.g: lanes per block row (1..16, block-row kernel for BR > 1), 100 +
// lanes per scalar row (scalar-row kernel) or 300 + lanes per block row
// (16-byte kernels on the padded copy, when M has one) or 401, 402, 404, 408
// (3x3 blocks: 1, 2, 5, 10 triples of lanes per block row); 0 selects by row
// length
extern int g_forced;

template <typename VT>
inline int code_of(const DBsr<VT>& M) {
  return g_forced > 0 ? g_forced : M.g;
}

template <typename VT>
inline int pick_group(const DBsr<VT>& M) {
  int g = code_of(M);
  if (g >= 400) {
    if (M.br == 3 && M.bc == 3) return g - 400;  // triples of lanes per block row
    g = 0;  // other shapes: by row length
  }
  if (g >= 300) return g - 300;
  if (g > 0) return g >= 100 ? g - 100 : g;
  // measured on the 616k-node tube: FP64 3x3 rows are fastest with 2 lanes
  // per scalar row (the FP64 pipe binds), FP32 with 4 (coalescing binds)
  const double per_row = M.nbr ? (double)M.nnzb * M.bc / M.nbr : 0.0;
  int G = sizeof(VT) == 8 ? (per_row >= 24 ? 2 : 1) : (per_row >= 24 ? 4 : 2);
  // small operators (the coarse AMG levels) fill less than a wave of the GPU
  // with one group per row, and their rows are long, so each lane would walk
  // dozens of blocks one dependent L2 round trip at a time: widen the group
  // (up to 16 lanes, at least 4 values per lane) while the grid stays below
  // two waves, in FP64 below 256 lanes per SM: there every further lane of a
  // row adds a sum on the FP64 pipe (Chebyshev step, 1,200 rows of 15 blocks:
  // 4.9, 3.5, 2.9, 4.1 us with 2, 4, 8, 16 lanes, 6,000 rows 4.9, 5.0, 6.4,
  // 10.6 us).
  const long long nrows = (long long)M.nbr * M.br;
  const long long most = (long long)sm_count() * (sizeof(VT) == 8 ? 256 : 4096);
  while (G < 16 && per_row >= 8.0 * G && nrows * G * 2 <= most) G *= 2;
  return G;
}

template <int BR, int BC, int NR, typename VT, typename XT>
inline void dispatch_g(int G, const DBsr<VT>& M, const XT* x, XT* y, const EpiArgs& e, cudaStream_t s) {
  switch (G) {
    case 1: launch_spmv_e<BR, BC, NR, 1, VT, XT>(M, x, y, e, s); break;
    case 2: launch_spmv_e<BR, BC, NR, 2, VT, XT>(M, x, y, e, s); break;
    case 4: launch_spmv_e<BR, BC, NR, 4, VT, XT>(M, x, y, e, s); break;
    case 8: launch_spmv_e<BR, BC, NR, 8, VT, XT>(M, x, y, e, s); break;
    default: launch_spmv_e<BR, BC, NR, 16, VT, XT>(M, x, y, e, s); break;
  }
}

}  // namespace scr
