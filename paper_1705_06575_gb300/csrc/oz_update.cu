// oz_update.cu — FP64 factors on the FP16 tensor cores: digits of the factored panels, the external
// update of a tile by its descendants, and the trailing update inside a supernode. The arithmetic
// (fixed-point digits, exact products, 64-bit sums) is described in oz.cuh.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "kernels.h"
#include "oz.cuh"
#include "tc.cuh"

namespace cg = cooperative_groups;

namespace sym {
namespace {

__device__ __forceinline__ int64_t tile_base(int32_t i, int32_t ncols, int32_t ncb) {
  return i < ncb ? (int64_t)i * NB : (int64_t)ncols + (int64_t)(i - ncb) * NB;
}
__device__ __forceinline__ int tile_rows(int32_t i, int32_t ncols, int32_t nrows, int32_t ncb) {
  const int64_t base = tile_base(i, ncols, ncb);
  const int64_t r = (i < ncb ? ncols : nrows) - base;
  return (int)(r < NB ? r : NB);
}

// Row scales of one factorization (exps[k] from C_kk, permuted column k) and whether fixed point with
// these scales can stand for FP64 on this matrix. An entry of L is held to 2^-56 of its row's scale
// where FP64 keeps 2^-53 of the entry itself, so what reaches x only through entries far below the
// scale of their rows loses accuracy: a row whose diagonal is a large penalty passes 1 / sqrt(penalty)
// of its scale on to its neighbours, and parts of the matrix that only weak couplings join drive each
// other through those. Measured on a 14^3 7-point conductance matrix, largest relative error of a
// component of x, FP64 kernels | fixed point: penalties of 1e4 on 5% of the diagonal 3e-15 | 3e-15, 1e5
// 4e-15 | 9e-15, 1e8 5e-15 | 3e-13, 1e16 4e-15 | 3e-9; a plane of couplings scaled by 0.1 5e-15 | 1e-14,
// 0.01 4e-15 | 5e-14, 1e-6 2e-14 | 6e-10, 1e-12 4e-15 | 8e-4; one half's coefficients 1e2 times the other
// half's, which it drives alone, 5e-15 | 2e-14, 1e4 5e-15 | 2e-13 (in norm 9e-16 | 5e-15). Rows and columns
// scaled by powers of two up to 2^100 instead: 4e-15 | 2e-15, the row scales absorb them. So *wide gets
// bit 0, and every kernel of this file then works in FP64, if
//   * a value is not finite;
//   * a row's couplings |a_ij| / sqrt(a_ii a_jj) add up to less than 2^-LOOSE (a penalty on it);
//   * a coupling below 2^-WEAK in that measure joins rows whose diagonals are more than 2^SPREAD apart (the
//     27-point vector problem's jumps of 1e4 stay: 2^15.2 between an inner row and one at the border,
//     errors of 3.0e-13 | 2.1e-13);
//   * weak couplings are the only links between two parts of the matrix: couplings below 2^-WEAK of the
//     smaller of the two diagonals and below 2^-FAINT of the strongest couplings of both rows (a long
//     row's are all far below its diagonal). The others are united into components (lock-free
//     union-find on parent), and a weak one between two components decides. Weak couplings inside a
//     component (irregular meshes, media of varying coefficients have them everywhere) lose nothing
//     that matters: other paths between the same rows carry far more.
// (Exponents are compared, so a limit is exact to a factor of two.) A well-coupled matrix pays two more
// small launches, beside the scatter (run_factor): 2 of the 64^2 grid's 762 us for factor and solve,
// nothing that shows on larger ones.
constexpr int WEAK = 9, FAINT = 6, SPREAD = 16, LOOSE = 6;
constexpr int WIDE = 1, LINKS = 2;  // bits of *wide: FP64; couplings below 2^-WEAK of the diagonals present
struct OzRow {  // (sum and strongest are zero before the first kernel)
  unsigned long long sum;  // of the row's couplings |a_ij| / sqrt(a_ii a_jj), unit 2^-SUM_UNIT
  int strongest;           // exponent + 1 of its strongest coupling, 0: none
  int diagonal;            // exponent
};
constexpr int SUM_UNIT = 40;
constexpr unsigned long long COUPLED = 1ull << (SUM_UNIT - LOOSE);  // (no more is added to a sum beyond)
__device__ __forceinline__ int exponent_of(double a) { return (__double2hiint(a) >> 20) & 0x7ff; }

// x: exponent of a coupling of row r, scaled: of its measure.
__device__ __forceinline__ void add_coupling(OzRow *r, int x, int scaled) {
  if (*(volatile int *)&r->strongest < x + 1) atomicMax(&r->strongest, x + 1);
  if (*(volatile unsigned long long *)&r->sum < COUPLED) {
    const int sh = scaled + SUM_UNIT;
    if (sh >= 0) atomicAdd(&r->sum, sh < SUM_UNIT - LOOSE ? 1ull << sh : COUPLED);
  }
}

// strength[k]: exponent + 1 of entry k below the diagonal, 0: no coupling.
__global__ void k_oz_scale(const double *__restrict__ Ax, const int64_t *__restrict__ dpos,
                           const int2 *__restrict__ links, int32_t *__restrict__ exps, OzRow *rows,
                           int32_t *__restrict__ parent, int16_t *__restrict__ strength, int *wide, int64_t n,
                           int64_t nnz) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int bits = 0;
  if (k < n) {
    const double a = Ax[dpos[k]];
    exps[k] = oz::scale_exponent(a);
    parent[k] = (int32_t)k;
    rows[k].diagonal = exponent_of(a);
    if (exponent_of(a) == 0x7ff) bits = WIDE;
  }
  if (k < nnz) {
    const int2 l = links[k];
    const double a = Ax[k];
    int x = -1;
    if (l.x != l.y && a != 0.0) {
      x = exponent_of(a);
      const int er = exponent_of(Ax[dpos[l.x]]), ec = exponent_of(Ax[dpos[l.y]]);
      if (x + WEAK < min(er, ec)) bits |= LINKS;
      const int scaled = x - ((er + ec) >> 1);
      if (x == 0x7ff || (scaled + WEAK < 0 && (er - ec > SPREAD || ec - er > SPREAD))) bits |= WIDE;
      add_coupling(&rows[l.x], x, scaled);
      add_coupling(&rows[l.y], x, scaled);
    }
    strength[k] = (int16_t)(x + 1);
  }
  if (bits & ~*(volatile int *)wide) atomicOr(wide, bits);
}
// Whether entry k is a weak coupling.
__device__ __forceinline__ bool weak_link(const OzRow *rows, int2 l, int strength) {
  const OzRow &r = rows[l.x], &c = rows[l.y];
  return strength - 1 + WEAK < min(r.diagonal, c.diagonal) && strength + FAINT < min(r.strongest, c.strongest);
}

// Roots are linked in the order of a scrambled index (a bijection): linked by index, the neighbours k and
// k + 1 of a grid form chains of n links (14^3 vector problem, scatter and range check: 1.5 ms, 0.2 so).
__device__ __forceinline__ uint32_t link_order(int32_t v) {
  uint32_t h = (uint32_t)v * 0x9E3779B1u;
  h ^= h >> 15;
  h *= 0x85EBCA77u;
  return h ^ (h >> 13);
}
// The root of v: chains of parents descend in link_order, and a step moves v two links up.
__device__ __forceinline__ int32_t root_of(volatile int32_t *parent, int32_t v) {
  int32_t p = parent[v];
  while (p != v) {
    const int32_t g = parent[p];
    if (g == p) return p;
    parent[v] = g;
    v = g;
    p = parent[v];
  }
  return v;
}

// Rows against the sum of their couplings; with couplings below 2^-WEAK of the diagonals present, the
// components of the strong ones (the later of two roots becomes a child of the earlier one); weak ones get
// strength -1.
__global__ void k_oz_unite(const int2 *__restrict__ links, const OzRow *__restrict__ rows, int32_t *parent,
                           int16_t *__restrict__ strength, int *wide, int64_t n, int64_t nnz) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n && rows[k].strongest > 0 && rows[k].sum < COUPLED) atomicOr(wide, WIDE);
  if (k >= nnz || *(volatile int *)wide != LINKS || strength[k] == 0) return;
  if (weak_link(rows, links[k], strength[k])) {
    strength[k] = -1;
    return;
  }
  int32_t a = root_of(parent, links[k].x), b = root_of(parent, links[k].y);
  while (a != b) {
    if (link_order(a) < link_order(b)) {
      const int32_t c = a;
      a = b;
      b = c;
    }
    const int32_t old = atomicCAS(&parent[a], a, b);
    if (old == a) break;
    a = root_of(parent, old);
    b = root_of(parent, b);
  }
}

// Weak couplings between two components. The rows are cleared for the next matrix.
__global__ void k_oz_bridges(const int2 *__restrict__ links, OzRow *__restrict__ rows, int32_t *parent,
                             const int16_t *__restrict__ strength, int *wide, int64_t n, int64_t nnz) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) {
    rows[k].sum = 0;
    rows[k].strongest = 0;
  }
  if (k < nnz && *(volatile int *)wide == LINKS && strength[k] < 0 &&
      root_of(parent, links[k].x) != root_of(parent, links[k].y))
    atomicOr(wide, WIDE);
}

// Digits of a factored row tile (task {J, i, s} of a TRSM launch): thread (row, o) takes the eight
// columns of octet o (and o + 4) of one row. Storage: octet of columns, slice, row: sixteen bytes
// each, at sn.dg + (octet * 7 + slice) * nrows + row; an even number of octets per panel.
__global__ void __launch_bounds__(256) k_oz_split(const SNode *__restrict__ sn, const Int4 *__restrict__ tasks,
                                                  const int32_t *__restrict__ rows, const double *__restrict__ Lx,
                                                  uint4 *__restrict__ dg, const int32_t *__restrict__ exps,
                                                  const int *__restrict__ wide, int64_t toff) {
  const Int4 t = tasks[toff + blockIdx.x];
  const SNode sj = sn[t.a];
  if (sj.dg < 0 || (*wide & WIDE)) return;
  const int i = t.b, s = t.c;
  const int ts = min(NB, sj.ncols - s * NB);
  int64_t rb = tile_base(i, sj.ncols, sj.ncb);
  int tm = tile_rows(i, sj.ncols, sj.nrows, sj.ncb);
  const int half = t.d >> 16;
  if (half) {
    rb += (half - 1) * (NB / 2);
    tm = max(0, min(NB / 2, tm - (half - 1) * (NB / 2)));
  }
  const int row = threadIdx.x & (NB - 1);
  if (row >= tm) return;
  const int64_t ld = sj.nrows, r = rb + row;
  const int e = exps[rows[sj.rowp + r]];
  for (int o = threadIdx.x >> 6; 16 * (o >> 1) < ts; o += 4) {
    const double *src = Lx + sj.lx + (int64_t)(s * NB + 8 * o) * ld + r;
    double v[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) v[c] = 8 * o + c < ts ? src[c * ld] : 0.0;
    uint64_t q[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) q[c] = oz::to_fixed(v[c], e, oz::offset_of(c));
    uint4 w[oz::SL];
    oz::to_digits(q, w);
    uint4 *dst = dg + sj.dg + (int64_t)(s * (NB / 8) + o) * oz::SL * ld + r;
#pragma unroll
    for (int k = 0; k < oz::SL; ++k) dst[k * ld] = w[k];
  }
}

// ---------------------------------------------------------------------------------------------
// Factorization of full diagonal tiles and their panel solves in fixed point. The FP64 pipe takes 64
// cycles for a warp's multiply-add however many lanes work, which paces both the column chain of a
// diagonal tile (44 us) and the panel solve (32 us of FP64 time for a 64 x 64 tile); 32 x 32 bit
// integer multiply-adds into 64 bits run 13 times as fast. With the row scales every value here is
// below 1: c_ij / 2^(e_i + e_j) is held with unit 2^-60, operands as two 30-bit halves, a product
// takes three integer multiply-adds (the low halves' product is below 2^-62) and the sums are exact,
// against an error of 2^-54 of the running value for every multiply-add in FP64.
//
// The chains hold no square root and no division by the pivot: with L = U diag(l_cc), U unit lower
// triangular, y(r, c) = x(r, c) l_cc solves y_c = c_c - sum_{k<c} y_k u(c, k), and x follows at the
// end, all columns at once. Column c's exponent sg = ceil(-log2(d_c) / 2) of its pivot d_c = l_cc^2
// balances the two factors: yh = y 2^sg and uh = u 2^-sg = yh / delta, delta = d_c 2^(2 sg) in [1, 4),
// are below 2 and 1 (|y| <= l_cc and |u| <= 1 / l_cc for a positive definite matrix), and x = yh /
// sqrt(delta). An entry beyond its range (|x| > 0.9999: its row cannot have a positive pivot) is
// clamped to it, which keeps the row's sum of squares above its diagonal.
struct ZCol {
  int32_t sg;       // exponent
  int2 lam;         // 1 / sqrt(delta), halves
  int32_t pad;
  int64_t lim;      // 0.9999 l_cc: the range of y
};
constexpr int Z_THREADS = 256;

// One sum's halves += (-y) u.
__device__ __forceinline__ void z_mac(int64_t &hi, int64_t &mid, int2 ny, int2 u) {
  hi += (int64_t)ny.x * (int64_t)u.x;
  mid += (int64_t)ny.x * (int64_t)u.y;
  mid += (int64_t)ny.y * (int64_t)u.x;
}
__device__ __forceinline__ int64_t z_value(int64_t hi, int64_t mid) { return hi + ((mid + (1ll << 29)) >> 30); }
// (sums of more than 32 products of mixed halves could leave 64 bits: fold them, exactly)
__device__ __forceinline__ void z_fold(int64_t &hi, int64_t &mid) {
  hi += mid >> 30;
  mid &= (1ll << 30) - 1;
}
__device__ __forceinline__ int64_t shfl64(int64_t v, int lane) {
  return (int64_t)__shfl_sync(0xffffffffu, (unsigned long long)v, lane);
}
// The reciprocal square root of 1 <= d < 4 (see rsqrt_newton in kernels.cu).
__device__ __forceinline__ double rsqrt_delta(double d) {
  double x0;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(x0) : "d"(d));
  const double e = fma(-d * x0, x0, 1.0);
  return fma(x0 * e, fma(0.375, e, 0.5), x0);
}

// Diagonal tile s of J (33 to 64 columns), 16 warps. Columns go in blocks of four. Warp w of the first
// eight owns block w at the rows 0-31, warp w of the other eight blocks w and w + 8 at the rows 32-63
// (one row per lane). A block's owner at the rows that hold its diagonal factors it in registers (its
// own columns updated through shuffles) and publishes yh, uh and 1 / delta; the other warps then add
// its columns to their blocks. While the upper rows walk the first eight blocks, the lower rows follow
// one block behind, so the pivots' chain carries the work of one row per lane only; named barriers
// link each group's steps and hand the upper blocks to the lower group. (With both rows in one lane and
// one barrier for all, 46 us for 64 columns: 800 cycles per column; the FP64 kernel 44 us.)
constexpr size_t POTRF_SMEM = 2 * NB * NB * sizeof(int2);
constexpr int POTRF_Z_THREADS = 512;

// The same tile in FP64 (WIDE): the operations of k_potrf in their order. Warp 0 carries the chain, the
// others the trailing columns, lanes along the rows.
__device__ __noinline__ void potrf_wide(double (*a)[NB + 1], double *D, int64_t ld, int ts, int64_t g0,
                                        long long *status) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int idx = tid; idx < ts * NB; idx += POTRF_Z_THREADS) {
    const int r = idx & (NB - 1), c = idx / NB;
    a[c][r] = r >= c && r < ts ? D[(int64_t)c * ld + r] : 0.0;
  }
  __syncthreads();
  auto finish_column = [&](int c) {
    double d = a[c][c];
    if (!(d > 0.0)) {
      if (lane == 0) atomicMin(status, (long long)(g0 + c));
      d = 1.0;
    }
    const double x = d > 1e-30 && d < 1e30 ? rsqrt_delta(d) : 1.0 / sqrt(d);
    __syncwarp();
    for (int r = c + lane; r < ts; r += 32) a[c][r] = r == c ? d * x : a[c][r] * x;
  };
  if (warp == 0 && ts > 0) finish_column(0);
  __syncthreads();
  for (int c = 0; c + 1 < ts; ++c) {
    if (warp == 0) {
      const double l = a[c][c + 1];
      for (int r = c + 1 + lane; r < ts; r += 32) a[c + 1][r] = fma(-a[c][r], l, a[c + 1][r]);
      __syncwarp();
      finish_column(c + 1);
    } else {
      for (int cc = c + 1 + warp; cc < ts; cc += POTRF_Z_THREADS / 32 - 1)
        for (int r = cc + lane; r < ts; r += 32) a[cc][r] = fma(-a[c][r], a[c][cc], a[cc][r]);
    }
    __syncthreads();
  }
  for (int idx = tid; idx < ts * NB; idx += POTRF_Z_THREADS) {
    const int r = idx & (NB - 1), c = idx / NB;
    if (r < ts) D[(int64_t)c * ld + r] = a[c][r];
  }
}
__device__ __forceinline__ void bar_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int threads) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

__global__ void __launch_bounds__(POTRF_Z_THREADS) k_potrf_z(const SNode *__restrict__ sn,
                                                             const Int4 *__restrict__ tasks, double *__restrict__ Lx,
                                                             const int32_t *__restrict__ exps, int2 *__restrict__ zu,
                                                             ZCol *__restrict__ zc, long long *status,
                                                             const int *__restrict__ wide, int64_t toff) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int2(*ys)[NB] = reinterpret_cast<int2(*)[NB]>(smem_raw);                           // [c][row]: -yh
  int2(*us)[NB] = reinterpret_cast<int2(*)[NB]>(smem_raw + NB * NB * sizeof(int2));  // [c][row]: uh
  __shared__ int64_t dd[NB];  // delta / 4 of every column, unit 2^-60
  __shared__ int2 rhos[NB];   // 1 / delta, halves
  __shared__ ZCol col[NB];
  const Int4 t = tasks[toff + blockIdx.x];
  const SNode sj = sn[t.a];
  const int s = t.b;
  const int ts = min(NB, sj.ncols - s * NB);
  const int64_t ld = sj.nrows, g0 = sj.first + (int64_t)s * NB;
  double *D = Lx + sj.lx + (int64_t)(s * NB) * ld + s * NB;
  if (*wide & WIDE) {
    potrf_wide(reinterpret_cast<double(*)[NB + 1]>(smem_raw), D, ld, ts, g0, status);
    return;
  }
  const int32_t *ec = exps + g0;
  const int tid = threadIdx.x, lane = tid & 31, w = (tid >> 5) & 7, low = tid >> 8;  // low: rows 32-63
  const int row = lane + 32 * low;
  int64_t hi[2][4], mid[2][4];  // [block w, block w + 8][column]
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int c = 4 * (w + 8 * q) + k;
      int64_t v = 0;
      if (row >= c && row < ts) {
        const double x = D[(int64_t)c * ld + row];
        v = row == c && !(x > 0.0) ? -(1ll << 58) : oz::to_fixed60(x, ec[row] + ec[c]);
      }
      hi[q][k] = v;
      mid[q][k] = 0;
    }
  const int nblk = (ts + 3) >> 2;
  // this warp's block at q += the columns of block b. A diagonal entry below -1 stays there: its row
  // fails as a pivot, and further squares (at most 4 per block) must not wrap around 8 to a positive
  // value.
  auto mac = [&](auto qc, int b) {
    constexpr int q = decltype(qc)::value;
    const int c0 = 4 * (w + 8 * q);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int2 y = ys[4 * b + j][row];
      const int4 p0 = *reinterpret_cast<const int4 *>(&us[4 * b + j][c0]);
      const int4 p1 = *reinterpret_cast<const int4 *>(&us[4 * b + j][c0 + 2]);
      z_mac(hi[q][0], mid[q][0], y, make_int2(p0.x, p0.y));
      z_mac(hi[q][1], mid[q][1], y, make_int2(p0.z, p0.w));
      z_mac(hi[q][2], mid[q][2], y, make_int2(p1.x, p1.y));
      z_mac(hi[q][3], mid[q][3], y, make_int2(p1.z, p1.w));
    }
    if (q == low) {
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (row == c0 + k && hi[q][k] < -(1ll << 60)) hi[q][k] = -(1ll << 60);
    }
  };
  // One column of this warp's rows, given its pivot data: yh and uh, and the block's later columns.
  auto column = [&](auto qc, int b, int k, int64_t v, int2 rho, int sg, auto &&ucol) {
    constexpr int q = decltype(qc)::value;
    const int c = 4 * b + k;
    const int64_t yh = (int64_t)((uint64_t)v << sg);
    const int2 y = oz::split30(yh), ny = make_int2(-y.x, -y.y), u = oz::split30(oz::mul60(y, rho));
#pragma unroll
    for (int k2 = 1; k2 < 4; ++k2)
      if (k2 > k) z_mac(hi[q][k2], mid[q][k2], ny, ucol(u, 4 * b + k2));
    ys[c][row] = ny;
    us[c][row] = u;
  };
  // Block b at the rows that hold its diagonal (its owner warp).
  auto factor = [&](auto qc, int b) {
    constexpr int q = decltype(qc)::value;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int c = 4 * b + k;
      if (q == 1 && c >= ts) {  // (uniform) columns past the tile contribute nothing
        ys[c][row] = us[c][row] = make_int2(0, 0);
        continue;
      }
      int64_t v = z_value(hi[q][k], mid[q][k]);
      int64_t d = shfl64(v, c & 31);
      if (d <= 0) {
        if (lane == 0) atomicMin(status, (long long)(g0 + c));
        d = 1ll << 59;
      }
      const int sg = (61 - (63 - __clzll(d))) >> 1;
      const int64_t dq = (int64_t)((uint64_t)d << (2 * sg - 2));  // delta / 4
      float root;  // sqrt(delta) = l_cc 2^sg, to a few parts in 10^6
      asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(root) : "f"((float)(int)(dq >> 36) * (4.0f / 16777216.0f)));
      const int64_t lim = (int64_t)__float2int_rn(root * (0.9999f * 536870912.0f)) << (31 - sg);
      const int2 rho = oz::split30(oz::reciprocal60(dq));
      v = v > lim ? lim : v < -lim ? -lim : v;
      v = row == c ? d : row > c ? v : 0;
      column(qc, b, k, v, rho, sg, [&](int2 u, int c2) {
        return make_int2(__shfl_sync(0xffffffffu, u.x, c2 & 31), __shfl_sync(0xffffffffu, u.y, c2 & 31));
      });
      if (lane == 0) {
        dd[c] = dq;
        rhos[c] = rho;
        col[c].sg = sg;
        col[c].lim = lim;
      }
    }
  };
  using Q0 = std::integral_constant<int, 0>;
  using Q1 = std::integral_constant<int, 1>;
  // barriers: 1 the upper rows' steps, 2 the lower rows', 3 + b hands block b to the lower rows
  if (!low) {
    for (int b = 0; b < 8; ++b) {
      if (w == b) {
        factor(Q0(), b);
        bar_arrive(3 + b, 32 + 256);
      }
      bar_sync(1, 256);
      if (w > b) mac(Q0(), b);
    }
  } else {
    for (int b = 0; b < 8; ++b) {
      bar_sync(3 + b, 32 + 256);
      if (w == b) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int c = 4 * b + k;
          const int64_t lim = col[c].lim;
          int64_t v = z_value(hi[0][k], mid[0][k]);
          v = v > lim ? lim : v < -lim ? -lim : v;
          column(Q0(), b, k, v, rhos[c], col[c].sg, [&](int2, int c2) { return us[c][c2]; });
        }
      }
      bar_sync(2, 256);
      if (w > b) mac(Q0(), b);
      mac(Q1(), b);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) z_fold(hi[1][k], mid[1][k]);
    for (int b = 8; b < nblk; ++b) {
      if (w == b - 8) factor(Q1(), b);
      bar_sync(2, 256);
      if (w > b - 8) mac(Q1(), b);
    }
  }
  __syncthreads();
  if (tid < ts) {
    const double lam = rsqrt_delta((double)dd[tid] * (4.0 / 1152921504606846976.0));
    col[tid].lam = oz::split30(__double2ll_rn(lam * 1152921504606846976.0));
    zc[g0 + tid] = col[tid];
  }
  __syncthreads();
  // the tile in FP64 and uh for its panel solves
  int2 *zt = zu + sj.dx + (int64_t)s * NB * NB;
  for (int idx = tid; idx < ts * NB; idx += POTRF_Z_THREADS) {
    const int r = idx & (NB - 1), c = idx / NB;
    if (r >= ts) continue;
    double x = 0.0;
    if (r >= c) {
      const int2 ny = ys[c][r];
      x = oz::from_fixed60(oz::mul60(make_int2(-ny.x, -ny.y), col[c].lam), ec[r]);
    }
    D[(int64_t)c * ld + r] = x;
    zt[c * ts + r] = r > c ? us[c][r] : make_int2(0, 0);
  }
}

// Tile (i, s) <- tile * L_ss^-T, and its digits. Thread (r, g) owns row r and the column blocks g,
// g + G, ...; a tile of at most 32 rows (the halves of a short launch) spreads its rows over G = 8
// groups of one warp each, else G = 4 groups of two warps. Step b, one barrier: every thread adds the four solved columns of block b to its
// columns right of them, the owners of block b + 1 first taking that block and solving it in
// registers so that the next step can begin.
constexpr size_t TRSM_SMEM = 2 * NB * NB * sizeof(int2) + NB * sizeof(ZCol);

template <int N, int G, int C>
__device__ __forceinline__ void trsm_mac(int64_t (&hi)[C], int64_t (&mid)[C], const int2 (&x)[4], const int2 *l) {
#pragma unroll
  for (int u = 0; u < N; ++u)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int4 p = *reinterpret_cast<const int4 *>(l + j * NB + 4 * G * u);
      const int4 q = *reinterpret_cast<const int4 *>(l + j * NB + 4 * G * u + 2);
      z_mac(hi[4 * u], mid[4 * u], x[j], make_int2(p.x, p.y));
      z_mac(hi[4 * u + 1], mid[4 * u + 1], x[j], make_int2(p.z, p.w));
      z_mac(hi[4 * u + 2], mid[4 * u + 2], x[j], make_int2(q.x, q.y));
      z_mac(hi[4 * u + 3], mid[4 * u + 3], x[j], make_int2(q.z, q.w));
    }
}

template <int G>
__device__ __forceinline__ void trsm_z(unsigned char *smem_raw, const SNode &sj, int s, int64_t rb, int tm,
                                       const int32_t *__restrict__ rows, double *__restrict__ Lx,
                                       uint4 *__restrict__ dg, const int32_t *__restrict__ exps,
                                       const int2 *__restrict__ zu, const ZCol *__restrict__ zc) {
  constexpr int ROWS = Z_THREADS / G, C = NB / G;  // rows, columns per thread
  int2(*us)[NB] = reinterpret_cast<int2(*)[NB]>(smem_raw);                           // [c][row]: uh(row, c)
  int2(*xs)[NB] = reinterpret_cast<int2(*)[NB]>(smem_raw + NB * NB * sizeof(int2));  // [c][row]: -yh(row, c)
  ZCol *col = reinterpret_cast<ZCol *>(smem_raw + 2 * NB * NB * sizeof(int2));
  const int ts = min(NB, sj.ncols - s * NB);
  const int64_t ld = sj.nrows, g0 = sj.first + (int64_t)s * NB;
  double *B = Lx + sj.lx + (int64_t)(s * NB) * ld + rb;
  const int tid = threadIdx.x, r = tid & (ROWS - 1), g = tid / ROWS;
  const bool live = (r & ~31) < tm;  // warp-uniform: some row of this warp is in the tile
  const int er = r < tm ? exps[rows[sj.rowp + rb + r]] : 0;
  double bv[C];
#pragma unroll
  for (int u = 0; u < C; ++u) {
    const int c = 4 * G * (u >> 2) + 4 * g + (u & 3);
    bv[u] = (r < tm && c < ts) ? B[(int64_t)c * ld + r] : 0.0;
  }
  const int2 *zt = zu + sj.dx + (int64_t)s * NB * NB;
#pragma unroll 4
  for (int idx = tid; idx < NB * NB; idx += Z_THREADS) {
    const int rr = idx & (NB - 1), c = idx / NB;
    us[c][rr] = rr > c && rr < ts ? zt[c * ts + rr] : make_int2(0, 0);
  }
  if (tid < NB) {
    ZCol z = {0, make_int2(0, 0), 0, 0};
    col[tid] = tid < ts ? zc[g0 + tid] : z;
  }
  int64_t hi[C], mid[C];
#pragma unroll
  for (int u = 0; u < C; ++u) {
    const int c = 4 * G * (u >> 2) + 4 * g + (u & 3);
    hi[u] = r < tm && c < ts ? oz::to_fixed60(bv[u], er + exps[g0 + c]) : 0;
    mid[u] = 0;
  }
  __syncthreads();
  int bn = g;  // the block in sums 0-3
  auto solve = [&](int b) {  // the owners of block b: sums 0-3 move out
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int c = 4 * b + k;
      const int64_t lim = col[c].lim;
      int64_t v = z_value(hi[k], mid[k]);
      v = v > lim ? lim : v < -lim ? -lim : v;
      const int2 ny = oz::split30(-(int64_t)((uint64_t)v << col[c].sg));
      xs[c][r] = ny;
#pragma unroll
      for (int k2 = k + 1; k2 < 4; ++k2) z_mac(hi[k2], mid[k2], ny, us[c][4 * b + k2]);
    }
#pragma unroll
    for (int u = 0; u < C - 4; ++u) {
      hi[u] = hi[u + 4];
      mid[u] = mid[u + 4];
    }
    bn += G;
  };
  const int nblk = (ts + 3) >> 2;
  if (live && g == 0) solve(0);
  __syncthreads();
  for (int b = 0; b + 1 < nblk; ++b) {
    if (live && bn < nblk) {
      int2 x[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) x[j] = xs[4 * b + j][r];
      if (b == 8) {
#pragma unroll
        for (int u = 0; u < C; ++u) z_fold(hi[u], mid[u]);
      }
      if (bn == b + 1) {  // (warp-uniform)
        trsm_mac<1, G>(hi, mid, x, &us[4 * b][4 * bn]);
        solve(b + 1);
      }
      const int2 *l = &us[4 * b][4 * bn];
      switch ((nblk - bn + G - 1) / G) {  // blocks bn, bn + G, ... below nblk
        case 1: trsm_mac<1, G>(hi, mid, x, l); break;
        case 2: trsm_mac<2, G>(hi, mid, x, l); break;
        case 3:
          if constexpr (G == 4) trsm_mac<3, G>(hi, mid, x, l);
          break;
        case 4:
          if constexpr (G == 4) trsm_mac<4, G>(hi, mid, x, l);
          break;
        default: break;
      }
    }
    __syncthreads();
  }
  // the tile in FP64 and its digits: thread (row, o) takes octets o, o + G, ... of one row
  if (r < tm) {
    for (int o = g; 16 * (o >> 1) < ts; o += G) {
      uint64_t q[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int c = 8 * o + k;
        int64_t x = 0;
        if (c < ts) {
          const int2 ny = xs[c][r];
          x = oz::mul60(make_int2(-ny.x, -ny.y), col[c].lam);
          B[(int64_t)c * ld + r] = oz::from_fixed60(x, er);
        }
        x = (x + 15 + (x >> 5 & 1)) >> 5;  // (to even)
        x = max(min(x, (int64_t)oz::QMAX), -(int64_t)oz::QMAX);
        q[k] = (uint64_t)(x + (int64_t)oz::offset_of(k));
      }
      if (sj.dg >= 0) {
        uint4 w[oz::SL];
        oz::to_digits(q, w);
        uint4 *dst = dg + sj.dg + (int64_t)(s * (NB / 8) + o) * oz::SL * ld + rb + r;
#pragma unroll
        for (int k = 0; k < oz::SL; ++k) dst[k * ld] = w[k];
      }
    }
  }
}

// The same tile in FP64 (WIDE): the operations of k_trsm in their order, thread (row, group of columns).
__device__ __noinline__ void trsm_wide(double (*Ls)[NB], double (*X)[NB], double *dinv, double *B, const double *D,
                                       int64_t ld, int ts, int tm) {
  const int tid = threadIdx.x, r = tid & (NB - 1), g = tid / NB;
  constexpr int G = Z_THREADS / NB;
  for (int c = g; c < ts; c += G) {
    Ls[c][r] = r >= c && r < ts ? D[(int64_t)c * ld + r] : 0.0;
    X[c][r] = r < tm ? B[(int64_t)c * ld + r] : 0.0;
  }
  __syncthreads();
  if (tid < ts) dinv[tid] = 1.0 / Ls[tid][tid];
  __syncthreads();
  const bool live = (r & ~31) < tm;  // (warp-uniform)
  for (int c = 0; c < ts; ++c) {
    double xc = 0.0;
    if (live) {
      xc = X[c][r] * dinv[c];
      for (int cc = c + 1 + g; cc < ts; cc += G) X[cc][r] = fma(-xc, Ls[c][cc], X[cc][r]);
    }
    __syncthreads();  // (X[c] is not read again)
    if (live && g == 0 && r < tm) B[(int64_t)c * ld + r] = xc;
  }
}
static_assert(sizeof(double) * (2 * NB * NB + NB) <= TRSM_SMEM, "shared memory of the FP64 form");
static_assert(sizeof(double) * NB * (NB + 1) <= POTRF_SMEM, "shared memory of the FP64 form");

__global__ void __launch_bounds__(Z_THREADS) k_trsm_z(const SNode *__restrict__ sn, const Int4 *__restrict__ tasks,
                                                      const int32_t *__restrict__ rows, double *__restrict__ Lx,
                                                      uint4 *__restrict__ dg, const int32_t *__restrict__ exps,
                                                      const int2 *__restrict__ zu, const ZCol *__restrict__ zc,
                                                      const int *__restrict__ wide, int64_t toff) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const Int4 t = tasks[toff + blockIdx.x];
  const SNode sj = sn[t.a];
  int64_t rb = tile_base(t.b, sj.ncols, sj.ncb);
  int tm = tile_rows(t.b, sj.ncols, sj.nrows, sj.ncb);
  const int half = t.d >> 16;  // 0: whole tile; 1, 2: its first or second 32 rows
  if (half) {
    rb += (half - 1) * (NB / 2);
    tm = max(0, min(NB / 2, tm - (half - 1) * (NB / 2)));
  }
  if (*wide & WIDE) {
    const int64_t ld = sj.nrows, c0 = (int64_t)t.c * NB;
    double *s = reinterpret_cast<double *>(smem_raw), *P = Lx + sj.lx + c0 * ld;
    trsm_wide(reinterpret_cast<double(*)[NB]>(s), reinterpret_cast<double(*)[NB]>(s + NB * NB), s + 2 * NB * NB, P + rb,
              P + c0, ld, min(NB, sj.ncols - (int)c0), tm);
    return;
  }
  if (tm > NB / 2) trsm_z<4>(smem_raw, sj, t.c, rb, tm, rows, Lx, dg, exps, zu, zc);
  else trsm_z<8>(smem_raw, sj, t.c, rb, tm, rows, Lx, dg, exps, zu, zc);
}

// ---------------------------------------------------------------------------------------------
// The products. Two kernels share one pipeline: the external update of 64 x 64 tiles by all their
// descendant entries (UPD; every entry's rows are placed in the tile's coordinates through inverse
// row maps while they are staged, rows it does not touch are zero, so all entries of a tile add up
// in the same accumulators), and the trailing update inside a supernode (one "entry": column tile
// s of J, rows onto themselves).
//
// A tile's column groups of sixteen (over all its entries) form one sequence of chunks. A CTA
// is persistent over tiles and its warps have fixed roles, linked by mbarriers with bounded waits
// and without CTA-wide barriers:
//   * warps 16-19 stage chunks into a six-stage ring (thread = operand, row: one asynchronous copy
//     per octet and slice);
//   * warps 20 and 21 issue the MMAs, one for each half of the tile's columns, whose segments end
//     four chunks apart (an issuing thread is held until its MMA is nearly done, so one thread
//     leaves the tensor core idle whenever it does anything else);
//   * warps 0-15 read finished segments back (64-bit sums in registers), and with a half of a tile
//     complete exchange the sums of the even-slice and odd-slice lanes and update C;
//   * warps 22-23 prepare the entry descriptors and row maps of the following batches of entries
//     (of this tile or the next), so their chains of dependent loads stay off the other warps.
// One CTA per SM: the accumulators take all of tensor memory, the ring 180 KB. A stage of 16 values of K
// has the MMAs read 70 KB of shared memory and the loaders write 28 KB, 0.76k cycles at 128 bytes per
// clock, and 0.64k cycles of MMA time (measured without staging); 1.3-1.45k cycles are measured on the
// 48^3 root, the rest being the read-back (F2I runs at 16 per clock and SM) and the handshakes. The
// root level's update at 64^3: 8.9 ms, 3.5 ms with the MMAs alone.
// Measured and not kept: digits kept as bytes and converted while they are staged (half the bytes
// loaded, ~400 instructions per warp and chunk: 4.6k cycles per chunk); staging and read-back in
// the same sixteen warps with whole-tile accumulators (4.1k cycles: the read-back, limited by the
// conversions, stops both the staging and the MMAs).
// A wait that runs out (wait_ns) records -1 in *status; every role then leaves its loop. withhold
// != 0 (a failure-path test) issues no MMA and no commit.
constexpr int NSTAGE = 6, LAG = 2;
constexpr int EB = 16;      // entries per batch
constexpr int NMETA = 2;    // batches in flight, one per descriptor warp
constexpr int EPI_WARPS = 16, LOAD_WARPS = 4, MMA_WARP = EPI_WARPS + LOAD_WARPS;
constexpr int META_WARP = MMA_WARP + 2;
constexpr int OZ_THREADS = 32 * (META_WARP + NMETA);
constexpr unsigned OZ_CTAS = OZ_SMS;
struct OzBatch {
  int64_t dg[EB];          // first octet of the entry's digits
  int64_t c;               // offset of the tile in Lx (last batch of a tile)
  int32_t ld[EB], ng[EB], rlo[EB], clo[EB];
  int32_t ne, total;       // entries, groups; total = -1: no more tiles
  int32_t last, diag;      // last batch of its tile; diag - 1: first row of a diagonal tile (0: none)
  int32_t cld, tm, tn;
  int16_t erow[NB], ecol[NB];  // scale exponents of the tile's rows and columns
  int8_t inv[2][EB][NB];   // [0] rows, [1] columns: tile position -> entry row, or -1
  float sq[2][NB];         // (last batch of a diagonal tile) squares of digit 4: rows, even octets; columns, odd
};
struct OzShared {
  OzBatch eb[NMETA];
  unsigned long long red[NB * NB];  // exchanged sums
  float dred[2][8][2][32];          // [half][warp pair][even, odd slices][lane]
  uint64_t full[NSTAGE], empty[NSTAGE], done[2], drained[2], mfull[NMETA], mempty[NMETA], xch[8];
  uint32_t tmem;
  int bad;
};
constexpr size_t OZ_SMEM = NSTAGE * oz::STAGE + sizeof(OzShared) + 128;
static_assert(OZ_SMEM <= 227 * 1024, "shared memory of one SM");

// Segments of the two halves of a tile: at most SEG_STEPS steps each, half 1's first one half as
// long, so that the two halves do not wait for their read-backs at the same time.
struct Segments {
  int n[2], lim[2];
  __device__ __forceinline__ void tile() {
    n[0] = n[1] = 0;
    lim[0] = oz::SEG_STEPS;
    lim[1] = oz::SEG_STEPS / 2;
  }
  // the next chunk; tile_end: the tile's last one. Returns 1 << h: first of a segment of half h,
  // 4 << h: last of one.
  __device__ __forceinline__ uint32_t chunk(bool tile_end) {
    uint32_t info = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (n[h] == 0) info |= 1u << h;
      if (++n[h] == lim[h] || tile_end) {
        info |= 4u << h;
        n[h] = 0;
        lim[h] = oz::SEG_STEPS;
      }
    }
    if (tile_end) tile();
    return info;
  }
};

// The same tiles in FP64 (WIDE), as the SIMT kernels: an entry's elements are mapped flat onto the
// threads (a warp's multiply-add takes 64 cycles of the FP64 pipe however many lanes work, so every lane
// should), the operands of eight columns are copied while the eight before are used, the tile's sums stay
// in shared memory. Three groups of 256 threads (the SIMT kernels' three CTAs per SM) take every third
// entry of an external update, their sums and then those of a cluster's CTAs added up in order, or a
// tile each of a trailing update, so that one group's loads hide behind the others' arithmetic. Updates
// and trailing updates of 7-point grids, milliseconds here | SIMT kernels: 31^3 4.5, 3.9 | 5.4, 3.6; 64^3
// 240, 143 | 222, 132.
constexpr int WIDE_SLOTS = 8, WIDE_K = 8;
struct WideOperands {  // two chunks of columns: one in use, one on its way
  double A[2][WIDE_K][NB], B[2][WIDE_K][NB];
};
constexpr int WIDE_GROUPS = 3;
struct WideShared {
  double sum[WIDE_GROUPS][NB][NB + 1];
  WideOperands op[WIDE_GROUPS];
};
static_assert(sizeof(WideShared) <= NSTAGE * oz::STAGE, "the FP64 form uses the ring's memory");

template <int J>
__device__ __forceinline__ void wide_chunk(double (&v)[WIDE_SLOTS], const int (&ab)[WIDE_SLOTS],
                                           const double (*A)[NB], const double (*B)[NB], int nk) {
#pragma unroll J == 1 ? 4 : 2
  for (int k = 0; k < nk; ++k)
#pragma unroll
    for (int q = 0; q < J; ++q) v[q] = fma(-A[k][ab[q] & 0xff], B[k][ab[q] >> 8], v[q]);
}

template <bool UPD>
__device__ __noinline__ void update_wide(WideShared &W, const SNode *sn, const UpdTask *utasks,
                                         const UpdEntry *ents, const int32_t *rel, const Int4 *tasks, double *Lx,
                                         int64_t toff, int ntiles) {
  cg::cluster_group cluster = cg::this_cluster();
  const int cs = UPD ? (int)cluster.num_blocks() : 1, rank = UPD ? (int)cluster.block_rank() : 0;
  constexpr int NG = WIDE_GROUPS, TG = OZ_THREADS / NG;
  const int grp = threadIdx.x / TG, tid = threadIdx.x % TG, w = tid >> 5;
  double(*sum)[NB + 1] = W.sum[grp];
  WideOperands &O = W.op[grp];
  const int tile0 = UPD ? blockIdx.x / cs : blockIdx.x + grp * gridDim.x;
  const int tstep = UPD ? gridDim.x / cs : gridDim.x * NG;
  for (int round = 0; round * tstep < ntiles; ++round) {
    // (an update's tiles are sorted by work: every other round runs backwards over the CTAs)
    const int tile = round * tstep + (UPD && (round & 1) ? tstep - 1 - tile0 : tile0);
    if (tile >= ntiles) continue;
    int J, i, j, s = 0, hoff = 0, tm = NB;
    int64_t ea = 0, ez = 1;
    if (UPD) {
      const UpdTask t = utasks[toff + tile];
      J = t.J;
      i = t.bi;
      j = t.bj;
      ea = t.e0 + (t.e1 - t.e0) * rank / cs;
      ez = t.e0 + (t.e1 - t.e0) * (rank + 1) / cs;
    } else {
      const Int4 t = tasks[toff + tile];
      J = t.a;
      i = t.b;
      j = t.c;
      s = t.d & 0xffff;
      if (t.d >> 16) {
        hoff = ((t.d >> 16) - 1) * (NB / 2);
        tm = NB / 2;
      }
    }
    const SNode sj = sn[J];
    const int64_t ld = sj.nrows, rb = tile_base(i, sj.ncols, sj.ncb) + hoff;
    const int cb = j * NB, tn = min(NB, sj.ncols - cb);
    tm = max(0, min(tm, tile_rows(i, sj.ncols, sj.nrows, sj.ncb) - hoff));
    double *C = Lx + sj.lx + (int64_t)cb * ld + rb;
    for (int idx = tid; idx < NB * NB; idx += TG) {
      const int r = idx & (NB - 1), c = idx / NB;
      sum[c][r] = rank == 0 && (grp == 0 || !UPD) && r < tm && c < tn ? C[(int64_t)c * ld + r] : 0.0;
    }
    for (int64_t e = UPD ? ea + grp : ea; e < ez; e += NG) {
      bar_sync(1 + grp, TG);  // the tile's sums as the entry before left them
      const UpdEntry E = UPD ? ents[e] : UpdEntry();
      const SNode sk = UPD ? sn[E.K] : sj;
      const int m = UPD ? E.m : tm, nc = UPD ? E.n : tn, kc = UPD ? sk.ncols : min(NB, sj.ncols - s * NB);
      const bool tri = UPD && i == j;  // a diagonal tile's entry: its rows are its columns
      const int cnt = tri ? m * (m + 1) / 2 : m * nc;
      const int64_t lk = sk.nrows;
      const double *K = Lx + sk.lx + (UPD ? 0 : (int64_t)s * NB * ld);
      const double *A = K + (UPD ? E.r_lo : rb), *B = K + (UPD ? E.c_lo : cb);
      for (int e0 = 0; e0 < cnt; e0 += WIDE_SLOTS * TG) {
        int ab[WIDE_SLOTS], at[WIDE_SLOTS];
        double v[WIDE_SLOTS];
#pragma unroll
        for (int q = 0; q < WIDE_SLOTS; ++q) {
          const int el = e0 + tid + TG * q;
          int a = 0, b = 0;
          at[q] = -1;
          v[q] = 0.0;
          if (el < cnt) {
            if (tri) {
              a = (int)((sqrtf(8.0f * el + 1.0f) - 1.0f) * 0.5f);
              while ((a + 1) * (a + 2) / 2 <= el) ++a;
              while (a * (a + 1) / 2 > el) --a;
              b = el - a * (a + 1) / 2;
            } else {
              a = el % m;
              b = el / m;
            }
            const int r = UPD ? rel[E.relr + a] - (int)rb : a, c = UPD ? rel[E.relc + b] - cb : b;
            if (UPD || i != j || c <= r + hoff) {  // (not above the diagonal)
              at[q] = c * (NB + 1) + r;
              v[q] = sum[0][at[q]];
            }
          }
          ab[q] = a | (b << 8);
        }
        const int left = cnt - e0 - 32 * w;  // elements from this warp's first one on
        auto fetch = [&](int k0) {
          const int nk = min(WIDE_K, kc - k0), u = (k0 / WIDE_K) & 1;
          for (int idx = tid; idx < nk * NB; idx += TG) {
            const int r = idx & (NB - 1), k = idx / NB;
            if (r < m) oz::copy8(&O.A[u][k][r], A + (k0 + k) * lk + r);
            if (r < nc) oz::copy8(&O.B[u][k][r], B + (k0 + k) * lk + r);
          }
          oz::copies_commit();
        };
        fetch(0);
        for (int k0 = 0; k0 < kc; k0 += WIDE_K) {
          const int nk = min(WIDE_K, kc - k0), u = (k0 / WIDE_K) & 1;
          if (k0 + WIDE_K < kc) {
            fetch(k0 + WIDE_K);
            oz::copies_wait<1>();
          } else {
            oz::copies_wait<0>();
          }
          bar_sync(1 + grp, TG);
          switch (left > 0 ? (left + TG - 1) / TG : 0) {  // this warp's slots with elements
            case 0: break;
            case 1: wide_chunk<1>(v, ab, O.A[u], O.B[u], nk); break;
            case 2: wide_chunk<2>(v, ab, O.A[u], O.B[u], nk); break;
            case 3: wide_chunk<3>(v, ab, O.A[u], O.B[u], nk); break;
            case 4: wide_chunk<4>(v, ab, O.A[u], O.B[u], nk); break;
            case 5: wide_chunk<5>(v, ab, O.A[u], O.B[u], nk); break;
            case 6: wide_chunk<6>(v, ab, O.A[u], O.B[u], nk); break;
            case 7: wide_chunk<7>(v, ab, O.A[u], O.B[u], nk); break;
            default: wide_chunk<8>(v, ab, O.A[u], O.B[u], nk); break;
          }
          bar_sync(1 + grp, TG);  // (the chunk has been read)
        }
#pragma unroll
        for (int q = 0; q < WIDE_SLOTS; ++q)
          if (at[q] >= 0) sum[0][at[q]] = v[q];
      }
    }
    if (!UPD) {
      bar_sync(1 + grp, TG);
      for (int idx = tid; idx < NB * tn; idx += TG) {
        const int r = idx & (NB - 1), c = idx / NB;
        if (r < tm) C[(int64_t)c * ld + r] = sum[c][r];
      }
      continue;  // (a thread's elements of the next tile's sums are those that it has written here)
    }
    __syncthreads();
    if (cs > 1) cluster.sync();  // every rank's sums are complete
    for (int idx = threadIdx.x; idx < NB * tn; idx += OZ_THREADS) {
      const int r = idx & (NB - 1), c = idx / NB;
      if (r >= tm || c % cs != rank) continue;
      double v = 0.0;
      for (int o = 0; o < cs; ++o) {
        const double *p = cs > 1 ? cluster.map_shared_rank(&W.sum[0][0][0], o) : &W.sum[0][0][0];
        for (int q = 0; q < NG; ++q) v += p[(q * NB + c) * (NB + 1) + r];
      }
      C[(int64_t)c * ld + r] = v;
    }
    if (cs > 1) cluster.sync();  // keep the other ranks' shared memory alive until it has been read
    else __syncthreads();
  }
}

template <bool UPD>
__global__ void __launch_bounds__(OZ_THREADS, 1)
    k_oz(const SNode *__restrict__ sn, const UpdTask *__restrict__ utasks, const UpdEntry *__restrict__ ents,
         const int32_t *__restrict__ rel, const Int4 *__restrict__ tasks, const int32_t *__restrict__ rows,
         double *__restrict__ Lx, const uint4 *__restrict__ dg, const int32_t *__restrict__ exps, int64_t toff,
         int ntiles, long long *status, const int *__restrict__ wide, uint64_t wait_ns, int withhold) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *stage0 = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
  OzShared &sh = *reinterpret_cast<OzShared *>(stage0 + NSTAGE * oz::STAGE);
  if (*wide & WIDE) {
    update_wide<UPD>(*reinterpret_cast<WideShared *>(stage0), sn, utasks, ents, rel, tasks, Lx, toff, ntiles);
    return;
  }
  cg::cluster_group cluster = cg::this_cluster();
  const int cs = UPD ? (int)cluster.num_blocks() : 1, rank = UPD ? (int)cluster.block_rank() : 0;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int tile0 = blockIdx.x / cs, tstep = gridDim.x / cs;  // a cluster shares a tile's entries

  if (warp == MMA_WARP) tc::tmem_alloc(&sh.tmem, oz::TMEM_COLS);
  if (tid == 0) {
    for (int b = 0; b < NSTAGE; ++b) {
      tc::mbar_init(&sh.full[b], LOAD_WARPS);
      tc::mbar_init(&sh.empty[b], 2);
    }
    for (int b = 0; b < NMETA; ++b) {
      tc::mbar_init(&sh.mfull[b], 1);
      tc::mbar_init(&sh.mempty[b], LOAD_WARPS + EPI_WARPS + 2);
    }
    for (int h = 0; h < 2; ++h) {
      tc::mbar_init(&sh.done[h], 1);
      tc::mbar_init(&sh.drained[h], EPI_WARPS);
    }
    for (int b = 0; b < 8; ++b) tc::mbar_init(&sh.xch[b], 2);
    tc::mbar_init_fence();
    sh.bad = 0;
  }
  if (tid < 128) {  // the zero slice of every octet and stage
    for (int b = 0; b < NSTAGE; ++b)
      *reinterpret_cast<uint4 *>(stage0 + b * oz::STAGE + (tid >> 6) * oz::A_LBO + oz::SL * oz::A_SLICE +
                                 (tid & 63) * 16) = make_uint4(0, 0, 0, 0);
    tc::fence_smem_to_async();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = sh.tmem;
  volatile int *bad = &sh.bad;
  // A bounded wait of a whole warp that also records its failure; false when this CTA gives up. One
  // answer for the warp: lanes time out, and see another warp's failure, at different moments, and
  // those that went on alone would wait for the others at the next warp-wide operation for ever.
  auto wait = [&](uint64_t *bar, uint32_t parity) -> bool {
    const bool done = tc::mbar_wait(bar, parity, wait_ns);
    const bool ok = __all_sync(0xffffffffu, done && *bad == 0);
    if (!ok) *bad = 1;
    return ok;
  };

  if (warp >= META_WARP) {
    // ---- descriptors: batch number b of this CTA's sequence goes to warp b % NMETA
    const int me = warp - META_WARP;
    OzBatch &eb = sh.eb[me];
    int b = 0, uses = 0;
    bool ok = true;
    for (int round = 0; ok; ++round) {
      // (tiles are sorted by work: every other round runs backwards over the CTAs)
      const int tile = round * tstep + ((round & 1) ? tstep - 1 - tile0 : tile0);
      const bool end = tile >= ntiles;
      int64_t ea = 0, ez = 1;
      int J = 0, i = 0, j = 0, s = 0, hoff = 0, tmax = NB;
      if (!end) {
        if (UPD) {
          const UpdTask t = utasks[toff + tile];
          const int64_t etot = t.e1 - t.e0;
          ea = t.e0 + etot * rank / cs;
          ez = t.e0 + etot * (rank + 1) / cs;
          i = t.bi;
          j = t.bj;
          J = t.J;
        } else {
          const Int4 t = tasks[toff + tile];
          J = t.a;
          i = t.b;
          j = t.c;
          s = t.d & 0xffff;
          const int half = t.d >> 16;
          if (half) {
            hoff = (half - 1) * (NB / 2);
            tmax = NB / 2;
          }
        }
      }
      for (int64_t e0 = ea; e0 < ez || e0 == ea; e0 += EB, ++b) {
        if (b % NMETA != me) continue;
        if (uses > 0) ok = wait(&sh.mempty[me], (uint32_t)(uses - 1) & 1u);
        ++uses;
        if (!ok) break;
        int total = -1;
        if (!end) {
          const SNode sj = sn[J];
          const int64_t rb = tile_base(i, sj.ncols, sj.ncb) + hoff;
          const int left = tile_rows(i, sj.ncols, sj.nrows, sj.ncb) - hoff;
          const int tm = max(0, min(tmax, left)), cb = j * NB, tn = min(NB, sj.ncols - cb);
          const int ne = UPD ? (int)max((int64_t)0, min((int64_t)EB, ez - e0)) : 1;
          int ng = 0;
          if (UPD) {
            for (int idx = lane; idx < ne * (NB / 4); idx += 32) {
              reinterpret_cast<int32_t *>(&eb.inv[0][0][0])[idx] = -1;
              reinterpret_cast<int32_t *>(&eb.inv[1][0][0])[idx] = -1;
            }
            if (lane < ne) {
              const UpdEntry E = ents[e0 + lane];
              const SNode *sk = &sn[E.K];
              eb.dg[lane] = sk->dg;
              eb.ld[lane] = sk->nrows;
              eb.ng[lane] = ng = (sk->ncols + 15) >> 4;
              eb.rlo[lane] = E.r_lo;
              eb.clo[lane] = E.c_lo;
            }
            __syncwarp();
            for (int k = 0; k < ne; ++k) {
              const UpdEntry &E = ents[e0 + k];
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                const int a = lane + 32 * h;
                if (a < E.m) eb.inv[0][k][rel[E.relr + a] - (int)rb] = (int8_t)a;
                if (a < E.n) eb.inv[1][k][rel[E.relc + a] - cb] = (int8_t)a;
              }
            }
          } else {
            ng = lane == 0 ? (min(NB, sj.ncols - s * NB) + 15) >> 4 : 0;
            if (lane == 0) {
              eb.dg[0] = sj.dg + (int64_t)s * (NB / 8) * oz::SL * sj.nrows;
              eb.ld[0] = sj.nrows;
              eb.ng[0] = ng;
              eb.rlo[0] = (int32_t)rb;
              eb.clo[0] = cb;
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int a = lane + 32 * h;
              eb.inv[0][0][a] = (int8_t)(a < tm ? a : -1);
              eb.inv[1][0][a] = (int8_t)(a < tn ? a : -1);
            }
          }
          total = __reduce_add_sync(0xffffffffu, ng);
          if (e0 + EB >= ez) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int a = lane + 32 * h;
              if (a < tm) eb.erow[a] = (int16_t)exps[rows[sj.rowp + rb + a]];
              if (a < tn) eb.ecol[a] = (int16_t)exps[sj.first + cb + a];
            }
          }
          if (lane == 0) {
            eb.ne = ne;
            eb.last = e0 + EB >= ez;
            eb.diag = i == j ? hoff + 1 : 0;
            eb.c = sj.lx + (int64_t)cb * sj.nrows + rb;
            eb.cld = sj.nrows;
            eb.tm = tm;
            eb.tn = tn;
          }
        }
        if (lane == 0) eb.total = total;
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&sh.mfull[me]);
      }
      if (end) break;
    }
  } else if (warp >= MMA_WARP) {
    // ---- MMA issue, one warp per half of the tile's columns. The whole warp runs the loop on values
    // the compiler knows to be uniform (shuffles), lane 0 issues: with the loop inside one lane's
    // branch every operand of every MMA is moved to a uniform register by itself.
    const uint32_t h = __shfl_sync(0xffffffffu, (uint32_t)(warp - MMA_WARP), 0);
    const uint32_t d = __shfl_sync(0xffffffffu, tmem, 0) + 256u * h;
    const uint32_t smem0 = __shfl_sync(0xffffffffu, tc::smem_addr(stage0), 0);
    const uint64_t adesc = tc::desc(smem0, oz::A_LBO, oz::SBO);
    const uint64_t bdesc = tc::desc(smem0 + oz::A_BYTES + h * oz::B_HALF, oz::B_LBO, oz::SBO);
    Segments seg;
    seg.tile();
    uint32_t st = 0, ph = 0, segs = 0;
    bool ok = true;
    for (int b = 0; ok; ++b) {
      const int mb = b % NMETA;
      if (!(ok = wait(&sh.mfull[mb], (uint32_t)(b / NMETA) & 1u))) break;
      const int total = __shfl_sync(0xffffffffu, *(volatile int *)&sh.eb[mb].total, 0);
      const int last = __shfl_sync(0xffffffffu, *(volatile int *)&sh.eb[mb].last, 0);
      if (total < 0) break;
      if (lane == 0) tc::mbar_arrive(&sh.mempty[mb]);
#pragma unroll 1
      for (int c = 0; c < total; ++c) {
        const uint32_t info = seg.chunk(last && c + 1 == total);
        const uint32_t first = (info >> h) & 1u;
        // the accumulators are free once the half's previous segment has been read
        ok = (!first || segs == 0 || wait(&sh.drained[h], (segs - 1) & 1u)) && wait(&sh.full[st], ph);
        if (!ok) break;
        segs += first;
        const uint64_t a = adesc + st * (oz::STAGE >> 4), bd = bdesc + st * (oz::STAGE >> 4);
        if (!withhold && lane == 0) {
          tc::fence_after_sync();
          if (first) oz::mma_step<true>(d, a, bd);
          else oz::mma_step<false>(d, a, bd);
          if (info & (4u << h)) tc::commit(&sh.done[h]);
          tc::commit(&sh.empty[st]);
        }
        __syncwarp();
        if (++st == NSTAGE) {
          st = 0;
          ph ^= 1;
        }
      }
    }
  } else if (warp >= EPI_WARPS) {
    // ---- staging
    const int lt = tid - 32 * EPI_WARPS, op = lt >> 6, p = lt & (NB - 1);  // operand, row
    const uint32_t dst0 = tc::smem_addr(stage0) +
                          (op ? oz::A_BYTES + (uint32_t)(p >> 5) * oz::B_HALF + 16u * (p & 31) : 16u * p);
    const uint32_t lbo = op ? oz::B_LBO : oz::A_LBO, slice = op ? oz::B_SLICE : oz::A_SLICE;
    // A chunk is announced (one arrival per warp: an asynchronous arrival of every thread costs ~8
    // cycles each on the barrier, 1k cycles per chunk) LAG chunks after its copies were issued, or
    // when the sequence pauses.
    int it = 0, told = 0;  // chunks issued, chunks announced
    // On a diagonal tile each thread also adds up the squares of digit 4 of its row (operand A: the first
    // octet of every chunk, B: the second one), read back once its copies have landed. kinds: four bits per
    // chunk that is not announced yet (1: of a diagonal tile, 2: the tile's last one, 4: its batch's place).
    // The sum is written before the tile's last chunk is announced, so before its MMAs are issued and
    // before the read-back learns that they are done.
    const uint8_t *digit4 = stage0 + (op ? oz::A_BYTES + (p >> 5) * oz::B_HALF + 16 * (p & 31) + 4 * oz::B_SLICE + oz::B_LBO
                                         : 16 * p + 4 * oz::A_SLICE);
    float sq = 0.f;
    uint32_t kinds = 0;
    auto announce = [&]() {
      const uint32_t kind = kinds & 15u;
      kinds >>= 4;
      if (kind & 1u) {
        sq += oz::square_sum(*reinterpret_cast<const uint4 *>(digit4 + (told % NSTAGE) * oz::STAGE));
        if ((kind & 2u) && cs == 1) {
          sh.eb[kind >> 2].sq[op][p] = sq;
          sq = 0.f;
        }
      }
      tc::fence_smem_to_async();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&sh.full[told % NSTAGE]);
      ++told;
    };
    bool ok = true;
    for (int b = 0; ok; ++b) {
      const int mb = b % NMETA;
      if (told < it && !__all_sync(0xffffffffu, tc::mbar_test(&sh.mfull[mb], (uint32_t)(b / NMETA) & 1u))) {
        oz::copies_wait<0>();
        while (told < it) announce();
      }
      if (!(ok = wait(&sh.mfull[mb], (uint32_t)(b / NMETA) & 1u))) break;
      const OzBatch &eb = sh.eb[mb];
      const int total = eb.total, ne = eb.ne;
      if (total < 0) break;
      int ci = 0, cgp = 0;  // position in the sequence of groups: entry, group
      const uint4 *src = dg;
      int64_t ld = 0;
      int r = -1;
      auto enter = [&]() {  // the row of entry ci at this thread's tile position
        r = ci < ne ? eb.inv[op][ci][p] : -1;
        ld = 0;
        src = dg;
        if (r >= 0) {
          ld = eb.ld[ci];
          src += eb.dg[ci] + (op ? eb.clo[ci] : eb.rlo[ci]) + r;
        }
      };
      if (total > 0) enter();
      for (int c = 0; c < total; ++c, ++it) {
        const int st = it % NSTAGE;
        if (it >= NSTAGE && !(ok = wait(&sh.empty[st], (uint32_t)(it / NSTAGE - 1) & 1u))) break;
        const uint32_t dst = dst0 + (uint32_t)st * oz::STAGE;
#pragma unroll
        for (int o = 0; o < 2; ++o)
#pragma unroll
          for (int k = 0; k < oz::SL; ++k) {
            oz::copy16(dst + o * lbo + k * slice, src, r >= 0);
            src += ld;
          }
        oz::copies_commit();
        kinds |= ((eb.diag ? 1u : 0u) | (eb.last && c + 1 == total ? 2u : 0u) | (uint32_t)mb << 2) << (4 * (it - told));
        if (it - told >= LAG) {
          oz::copies_wait<LAG>();
          announce();
        }
        if (++cgp == eb.ng[ci]) {
          cgp = 0;
          ++ci;
          enter();
        }
      }
      if (!ok) break;
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&sh.mempty[mb]);
    }
    oz::copies_wait<0>();
    while (told < it) announce();
    if (UPD && cs > 1) sh.eb[0].sq[op][p] = sq;  // (for the end)
  } else {
    // ---- read-back: lanes 32 (warp & 3) .. of tensor memory, columns 8 (warp >> 2) .. of each
    // half of the tile
    const int row = 32 * (warp & 1) + lane, g8 = 8 * (warp >> 2);
    const bool up = (warp & 2) != 0;
    const int pair = (warp & 1) | ((warp >> 2) << 1);  // this warp and the one with the other slices' sums
    const uint32_t addr0 = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)g8;
    unsigned long long acc0[8], acc1[8];  // (one set where a segment is a whole tile)
    float ds0 = 0.f, ds1 = 0.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) acc0[q] = acc1[q] = 0;
    Segments seg;
    seg.tile();
    int segs[2] = {0, 0}, nx = 0;
    // The finished segment of half h; fin: the tile's last one.
    auto segment = [&](auto hc, unsigned long long(&acc)[8], float &dsum, const OzBatch &eb, bool fin) -> bool {
      constexpr int h = decltype(hc)::value;
      const int dtop = eb.diag - 1;          // (dtop >= 0: a diagonal tile)
      const int c0 = 32 * h + g8, drow = row + dtop;
      const bool here = dtop >= 0 && (drow & ~7) == c0;
      const int k0 = c0 + (up ? 4 : 0);      // the four columns this thread finishes
      double *C = Lx + eb.c + (int64_t)k0 * eb.cld + row;
      double cv[4];
      const int tm = eb.tm, tn = eb.tn;
      if (!UPD) {  // C's entries, loaded while the MMAs run
#pragma unroll
        for (int q = 0; q < 4; ++q) cv[q] = (row < tm && k0 + q < tn) ? C[(int64_t)q * eb.cld] : 0.0;
      }
      if (!wait(&sh.done[h], (uint32_t)segs[h] & 1u)) return false;
      ++segs[h];
      __syncwarp();
      tc::fence_after_sync();
      oz::drain<!UPD>(addr0 + 256u * h, up, acc, here, drow & 7, dsum);
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&sh.drained[h]);
      if (!fin || cs > 1) return true;
      if (UPD) {
#pragma unroll
        for (int q = 0; q < 4; ++q) cv[q] = (row < tm && k0 + q < tn) ? C[(int64_t)q * eb.cld] : 0.0;
      }
      // hand four columns' sums to the other warp of the pair (its buffer of this half has been
      // read: it has arrived for the other half since), keep four
      unsigned long long *buf = sh.red + (pair * 2 + h) * 8 * 32 + lane;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        buf[(up ? q : q + 4) * 32] = up ? acc[q] : acc[q + 4];
        acc[q] = up ? acc[q + 4] : acc[q];
      }
      if (here) sh.dred[h][pair][up][lane] = dsum;
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&sh.xch[pair]);
      if (!wait(&sh.xch[pair], (uint32_t)nx & 1u)) return false;
      ++nx;
      if (row < tm) {
        const int ei = eb.erow[row];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int c = k0 + q;
          if (c < tn && !(dtop >= 0 && c > drow)) {
            unsigned long long v = acc[q] + buf[(up ? q + 4 : q) * 32];
            if (dtop >= 0 && c == drow) v += oz::dropped_squares(eb.sq[0][row] + eb.sq[1][c]);
            C[(int64_t)q * eb.cld] =
                dtop >= 0 && c == drow && sh.dred[h][pair][0][lane] + sh.dred[h][pair][1][lane] > 1.5f
                    ? -1.0
                    : oz::apply(cv[q], (long long)v, ei, eb.ecol[c]);
          }
        }
      }
#pragma unroll
      for (int q = 0; q < 8; ++q) acc[q] = 0;
      dsum = 0.f;
      return true;
    };
    bool ok = true;
    for (int b = 0; ok; ++b) {
      const int mb = b % NMETA;
      if (!(ok = wait(&sh.mfull[mb], (uint32_t)(b / NMETA) & 1u))) break;
      const OzBatch &eb = sh.eb[mb];
      const int total = eb.total, last = eb.last;
      if (total < 0) break;
      for (int c = 0; c < total && ok; ++c) {
        const bool fin = last && c + 1 == total;
        const uint32_t info = seg.chunk(fin);
        if (info & 4u) ok = segment(std::integral_constant<int, 0>(), acc0, ds0, eb, fin);
        if (ok && (info & 8u)) {
          if (UPD) ok = segment(std::integral_constant<int, 1>(), acc1, ds1, eb, fin);
          else ok = segment(std::integral_constant<int, 1>(), acc0, ds0, eb, fin);
        }
      }
      if (!ok) break;
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&sh.mempty[mb]);
    }
    if (UPD && cs > 1 && ok) {  // the even-slice and odd-slice sums of this rank meet in shared memory
      if (!up) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          sh.red[(g8 + q) * NB + row] = acc0[q];
          sh.red[(32 + g8 + q) * NB + row] = acc1[q];
        }
      }
      if ((row & 24) == g8) {  // the eight columns that hold the row's diagonal entry
        sh.dred[0][pair][up][lane] = ds0;
        sh.dred[1][pair][up][lane] = ds1;
      }
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&sh.xch[pair]);
      if (up && wait(&sh.xch[pair], 0)) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          sh.red[(g8 + q) * NB + row] += acc0[q];
          sh.red[(32 + g8 + q) * NB + row] += acc1[q];
        }
      }
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == MMA_WARP) {
    // (with a wait that ran out the last MMAs may still be in flight: let them finish, bounded, so
    // that tensor memory is not given back under them)
    if (sh.bad && !withhold) __nanosleep(100000);
    tc::fence_after_sync();
    tc::tmem_free(tmem, oz::TMEM_COLS);
  }
  if (tid == 0 && sh.bad) atomicMin(status, -1ll);
  if (UPD && cs > 1) {
    cluster.sync();  // every rank's sums of the whole tile are in its shared memory
    const UpdTask t = utasks[toff + tile0];
    const SNode sj = sn[t.J];
    const int64_t rb = tile_base(t.bi, sj.ncols, sj.ncb);
    const int tm = tile_rows(t.bi, sj.ncols, sj.nrows, sj.ncb), cb = t.bj * NB, tn = min(NB, sj.ncols - cb);
    const bool diag = t.bi == t.bj;
    double *C = Lx + sj.lx + (int64_t)cb * sj.nrows + rb;
    // rank r finishes the columns c = r mod cs, adding the ranks in order (whole numbers)
    for (int idx = tid; idx < NB * (NB / cs) && !sh.bad; idx += OZ_THREADS) {
      const int r = idx & (NB - 1), c = (idx / NB) * cs + rank;
      if (r >= tm || c >= tn || (diag && c > r)) continue;
      double *x = C + (int64_t)c * sj.nrows + r;
      const double old = *x;
      unsigned long long v = 0;
      float d = 0.f, sq = 0.f;
      for (int o = 0; o < cs; ++o) {
        v += cluster.map_shared_rank(sh.red, o)[c * NB + r];
        if (diag && c == r) {
          const float *dr = cluster.map_shared_rank(&sh.dred[c >> 5][(r >> 5) | ((c >> 3 & 3) << 1)][0][0], o);
          d += dr[r & 31] + dr[32 + (r & 31)];
          const float *q = cluster.map_shared_rank(&sh.eb[0].sq[0][0], o);
          sq += q[r] + q[NB + c];
        }
      }
      v += oz::dropped_squares(sq);
      *x = d > 1.5f ? -1.0 : oz::apply(old, (long long)v, exps[rows[sj.rowp + rb + r]], exps[sj.first + cb + c]);
    }
    cluster.sync();  // keep the other ranks' shared memory alive until it has been read
  }
}

template <typename... KArgs, typename... Args>
cudaError_t launch_oz(void (*kernel)(KArgs...), unsigned grid, int threads, size_t smem, int cs, cudaStream_t st,
                      int prio, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  cfg.gridDim = dim3(grid * (unsigned)cs, 1, 1);
  cfg.blockDim = dim3(threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributePriority;
  attr[0].val.priority = prio;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)cs;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cs > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace

cudaError_t prepare_oz() {
  cudaError_t e0 = cudaFuncSetAttribute(k_trsm_z, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TRSM_SMEM);
  if (e0 != cudaSuccess) return e0;
  e0 = cudaFuncSetAttribute(k_potrf_z, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)POTRF_SMEM);
  if (e0 != cudaSuccess) return e0;
  cudaError_t e = cudaFuncSetAttribute(k_oz<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)OZ_SMEM);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_oz<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)OZ_SMEM);
}
cudaError_t launch_oz_scale(cudaStream_t st, const DevPlan &d, const double *Ax) {
  const unsigned grid = (unsigned)((std::max(d.n, d.nnz_a) + 255) / 256);
  k_oz_scale<<<grid, 256, 0, st>>>(Ax, d.dpos, d.links, d.exps, (OzRow *)d.oz_rows, d.parent, d.strength, d.wide, d.n,
                                   d.nnz_a);
  return cudaGetLastError();
}
cudaError_t launch_oz_range(cudaStream_t st, const DevPlan &d) {
  const unsigned grid = (unsigned)((std::max(d.n, d.nnz_a) + 255) / 256);
  k_oz_unite<<<grid, 256, 0, st>>>(d.links, (const OzRow *)d.oz_rows, d.parent, d.strength, d.wide, d.n, d.nnz_a);
  k_oz_bridges<<<grid, 256, 0, st>>>(d.links, (OzRow *)d.oz_rows, d.parent, d.strength, d.wide, d.n, d.nnz_a);
  return cudaGetLastError();
}
cudaError_t launch_oz_split(unsigned tasks, cudaStream_t st, int prio, const DevPlan &d, const double *Lx,
                            int64_t toff) {
  return launch_oz(k_oz_split, tasks, 256, 0, 1, st, prio, d.sn, d.tasks, d.rows, Lx, d.dg, (const int32_t *)d.exps,
                   (const int *)d.wide, toff);
}
size_t oz_column_bytes() { return sizeof(ZCol); }
size_t oz_row_bytes() { return sizeof(OzRow); }
cudaError_t launch_potrf_z(unsigned tasks, cudaStream_t st, int prio, const DevPlan &d, double *Lx, int64_t toff,
                           long long *status) {
  return launch_oz(k_potrf_z, tasks, POTRF_Z_THREADS, POTRF_SMEM, 1, st, prio, d.sn, d.tasks, Lx, (const int32_t *)d.exps,
                   d.zu, (ZCol *)d.zc, status, (const int *)d.wide, toff);
}
cudaError_t launch_trsm_z(unsigned tasks, cudaStream_t st, int prio, const DevPlan &d, double *Lx, int64_t toff) {
  return launch_oz(k_trsm_z, tasks, Z_THREADS, TRSM_SMEM, 1, st, prio, d.sn, d.tasks, d.rows, Lx, d.dg,
                   (const int32_t *)d.exps, (const int2 *)d.zu, (const ZCol *)d.zc, (const int *)d.wide, toff);
}
cudaError_t launch_update_oz(unsigned tasks, int cluster, cudaStream_t st, int prio, const DevPlan &d, double *Lx,
                             int64_t toff, long long *status) {
  const unsigned grid = cluster > 1 ? tasks : tasks < OZ_CTAS ? tasks : OZ_CTAS;
  return launch_oz(k_oz<true>, grid, OZ_THREADS, OZ_SMEM, cluster, st, prio, d.sn, d.upd_tasks, d.upd_entries, d.rel,
                   d.tasks, d.rows, Lx, (const uint4 *)d.dg, (const int32_t *)d.exps, toff, (int)tasks, status,
                   (const int *)d.wide, d.tc_wait_ns, (int)d.tc_withhold);
}
cudaError_t launch_gemm_oz(unsigned tasks, cudaStream_t st, int prio, const DevPlan &d, double *Lx, int64_t toff,
                           long long *status) {
  return launch_oz(k_oz<false>, tasks < OZ_CTAS ? tasks : OZ_CTAS, OZ_THREADS, OZ_SMEM, 1, st, prio, d.sn,
                   d.upd_tasks, d.upd_entries, d.rel, d.tasks, d.rows, Lx, (const uint4 *)d.dg,
                   (const int32_t *)d.exps, toff, (int)tasks, status, (const int *)d.wide,
                   d.tc_wait_ns, (int)d.tc_withhold);
}

}  // namespace sym
