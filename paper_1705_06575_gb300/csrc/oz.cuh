// oz.cuh — FP64 products on the FP16 tensor cores: device building blocks shared by the external
// update and the in-supernode trailing update of FP64 factors (oz_update.cu).
//
// Fixed point. In a Cholesky factor every entry obeys |l_ik| <= sqrt(a_ii). Row i of the factor
// gets the scale 2^e_i with sqrt(a_ii) < 0.986 * 2^e_i (e_i from the diagonal of A alone, known
// before the factorization), and v = l_ik / 2^e_i is held as a 56-bit fixed-point number
// v = sum_{s<7} d_s 2^(-7 - 8 s), the digits d_s integers in [-128, 128] (rounding error at most
// 2^-56). A digit is exact in FP16, a product of digits is an integer of magnitude <= 2^14, and
// an FP32 accumulator is exact while its sum stays below 2^24.
//
// Products (Ozaki's error-free splitting, with one exponent per row as in its integer variants: Ozaki,
// Ogita, Oishi, Rump, Numer. Algorithms 59, 2012; Ootomo, Ozaki, Yokota 2024).
// sum_k v_ik v_jk = sum_p 2^(-14 - 8 p) sum_{s+t=p} sum_k d_s(i,k) d_t(j,k). All pairs s + t <= 7 are
// formed (34 products of digit matrices). Errors per term, in units of sqrt(a_ii a_jj): the rounding of
// one operand's digits is at most 2^-56 times the other operand (to even, so without a preferred sign),
// the dropped pairs are 2^-64.4 (root mean square; at most 2^-61.7). Off the diagonal the dropped pairs
// have no preferred sign either once the columns' offsets alternate (OFFSET_ODD), so a sum's error grows
// like sqrt(K), as FP64's does with one rounding of 2^-54 of the running value per step. On the diagonal
// the pair s = t = 4 is a square, 2^-65.6 on average: these are added up apart (dropped_squares). A
// bias would be invisible in residual norms and for random solutions; in a smooth solution of a nearly
// singular matrix it adds up over a row. Row sums of L L^T - A of 7-point grids, mean over the supernodes
// wider than 512 | standard deviation / sqrt(rows): here, 48^3, 1.3e-16 | 7e-17 (the FP64 kernels 0 |
// 1.8e-16); with one offset for all columns, 40^3, 2.0e-15 | 1e-16. Errors of x = 1, geometric means over
// seeds, FP64 kernels | here | without the squares, one offset, halves rounded up: 31^3 3.4e-14 | 1.2e-14
// | 4.5e-14, 40^3 1.0e-14 | 8.3e-15 | 2.3e-13, 48^3 1.4e-14 | 1.6e-14 | 5.6e-13, 27-point 28^3 7.4e-14 |
// 2.8e-14 | 6.8e-13. Random x: 31^3 9.5e-15 | 7.2e-15, 48^3 2.1e-14 | 1.0e-14, 27-point 28^3 1.2e-13 |
// 2.7e-14. The accumulators are combined in 64-bit integers
// (unit 2^-62: the sum is below 2^62 by Cauchy-Schwarz, intermediate wrap-around cancels), whole tiles are
// summed without any rounding but the last digits' (2^-63 per segment), and the tile is updated with one
// FP64 rounding per entry.
//
// Layout. The digits of a factored panel are kept in FP16 as the tensor core reads them: octets of
// eight columns, per octet the seven slices, per slice the rows, sixteen bytes each. A stage holds
// 16 values of k of 64 rows per operand in the K-major core-matrix layout with the row groups 128
// bytes apart and the octets LBO apart, so rows are copied as they are, two consecutive slices of
// the A operand form one M = 128 operand, and consecutive slices of 32 rows of the B operand (a
// half of the tile's columns) one operand of N = 32 per slice. The MMA of A slices (2a, 2a+1) with
// B slices 0..T-1 adds to the half's accumulator column blocks 2a .. 2a+T-1 (32 columns each):
// block c holds weight p = c in lanes 0-63 (even s) and p = c + 1 in lanes 64-127 (odd s). Four
// MMAs per 16 values of k and half (N = 224, 192, 128, 64), 256 columns of tensor memory per half:
// one half is read back while the other one accumulates. Each accumulator lane sums at most four
// pairs per k, so 256 values of k (4 * 256 * 2^14 = 2^24) are exact; a segment of that length is
// then read back.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "plan.h"
#include "tc.cuh"

namespace sym {
namespace oz {

constexpr int SL = 7;                       // digits per value
constexpr uint32_t A_SLICE = 64 * 16;       // one octet of k of one slice: 64 rows of 16 bytes
constexpr uint32_t B_SLICE = 32 * 16;       // the same of half the tile's columns
constexpr uint32_t B_HALF = SL * B_SLICE;   // the other half of the columns
constexpr uint32_t SBO = 128;               // next 8 rows
constexpr uint32_t A_LBO = 8 * A_SLICE;     // next octet of k: seven slices and one of zeros (the
constexpr uint32_t B_LBO = 2 * B_HALF;      // partner of slice 6) for A, two halves for B
constexpr uint32_t A_BYTES = 2 * A_LBO;
constexpr uint32_t B_BYTES = 2 * B_LBO;
constexpr uint32_t STAGE = A_BYTES + B_BYTES;
constexpr uint32_t TMEM_COLS = 512;
constexpr int SEG_STEPS = 16;               // K = 16 steps per segment (256 values of k)
// Digit 0 is stored as byte 128 in even columns (digits -128 .. 127), as byte 127 in odd ones (-127 ..
// 128). A column's lower digits average -1/2 or 1/2; where they meet leading digits of one sign (the
// entries of an M-matrix's factor) in pairs that are dropped, a single offset leaves a bias that grows
// with K. Digit 6 has the other offset of its column: of the five dropped pairs of weight 8, each worth 1/4
// on average if both digits have the same offset, the two with digit 6 then cancel two others.
constexpr uint64_t OFFSET = 0x008080808080807Full, OFFSET_ODD = 0x007F7F7F7F7F7F80ull;
constexpr uint64_t QMAX = 0x007F7F7F7F7F7F7Full;
__device__ __forceinline__ constexpr uint64_t offset_of(int column) { return column & 1 ? OFFSET_ODD : OFFSET; }

// Scale exponent of a row from its diagonal entry a of A: sqrt(a) <= 0.986 * 2^e. Rows whose
// diagonal is not a positive finite number fail as pivots whatever their scale.
__device__ __forceinline__ int scale_exponent(double a) {
  if (!(a > 0.0)) return 0;
  if (!(a < 1.7e308)) return 513;
  int x;
  frexp(a, &x);  // a < 2^x; 1.03 a < 2^(x + 1)
  double f = ldexp(a, -x);
  if (f * 1.03 > 1.0) ++x;
  return (x + 1) >> 1;
}

// |v| / 2^e as a fixed-point number with unit 2^-U, rounded to nearest even (few bits are dropped where
// |v| is large, so halves are frequent; rounded up they would lengthen every row), at most `most` (a
// saturated row fails as a pivot: its sum of squares exceeds its diagonal; so does a NaN's row).
template <int U>
__device__ __forceinline__ uint64_t fixed_magnitude(double v, int e, uint64_t most) {
  const uint64_t bits = (uint64_t)__double_as_longlong(v);
  const int E = (int)(bits >> 52) & 0x7ff;
  const uint64_t m = (bits & 0xFFFFFFFFFFFFFull) | (E ? 0x10000000000000ull : 0ull);
  const int sh = (E ? E : 1) - (1075 - U) - e;  // q = m 2^sh
  uint64_t q;
  if (E == 0x7ff || sh > U - 53) q = most;
  else if (sh >= 0) q = m << sh;
  else if (sh >= -54) q = (m + (1ull << (-sh - 1)) - 1 + (m >> (-sh) & 1)) >> (-sh);
  else q = 0;
  return q < most ? q : most;
}
// v / 2^e with unit 2^-55 plus a column's offset: the digits' bytes.
__device__ __forceinline__ uint64_t to_fixed(double v, int e, uint64_t offset) {
  const uint64_t q = fixed_magnitude<55>(v, e, QMAX);
  return v < 0.0 ? offset - q : offset + q;
}
// v / 2^e with unit 2^-60 (the panel solve's arithmetic).
constexpr int64_t Q60MAX = (int64_t)(QMAX << 5);
__device__ __forceinline__ int64_t to_fixed60(double v, int e) {
  const int64_t q = (int64_t)fixed_magnitude<60>(v, e, (uint64_t)Q60MAX);
  return v < 0.0 ? -q : q;
}
// x = h 2^30 + l with |l| <= 2^29.
__device__ __forceinline__ int2 split30(int64_t x) {
  const int64_t l = (int64_t)((uint64_t)x << 34) >> 34;
  return make_int2((int)((x - l) >> 30), (int)l);
}
// The double x 2^(e - 60) (the exponent stays normal: |x| <= 2^60, -537 <= e <= 513).
__device__ __forceinline__ double from_fixed60(int64_t x, int e) {
  const double d = (double)x;
  return x ? __hiloint2double(__double2hiint(d) + ((e - 60) << 20), __double2loint(d)) : 0.0;
}

// a b / 2^60 rounded, for halves a = (h, l) and b: the low halves' product is left out.
__device__ __forceinline__ int64_t mul60(int2 a, int2 b) {
  const int64_t m = (int64_t)a.x * (int64_t)b.y + (int64_t)a.y * (int64_t)b.x;
  return (int64_t)a.x * (int64_t)b.x + ((m + (1ll << 29)) >> 30);
}
// 1 / (4 D / 2^60) with unit 2^-60 for 2^58 <= D < 2^60: an FP32 reciprocal r0 of D / 2^60 (24 bits),
// held with unit 2^-22, e = 1 - (D / 2^60) r0 formed exactly modulo 2^64 (|e| < 2^-21.4, unit 2^-82),
// and r0 (1 + e + e^2) / 4, Newton's series through second order: the error is below 2^-59.
__device__ __forceinline__ int64_t reciprocal60(int64_t D) {
  const float f = (float)(int)((D + (1ll << 35)) >> 36) * (1.0f / 16777216.0f);
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(f));
  const int R = __float2int_rn(r * 4194304.0f);
  const int64_t P = (D >> 30) * (int64_t)R, Q = (int64_t)((int)D & 0x3fffffff) * (int64_t)R;
  const int64_t e = (int64_t)(0ull - (((uint64_t)P << 30) + (uint64_t)Q));
  const float ef = (float)(int)(e >> 31) * (1.0f / 262144.0f);  // e 2^33 (unit 2^-51 to unit 2^-33)
  const int64_t c = e + ((int64_t)__float2int_rn(ef * ef) << 16);
  const int64_t h = (int64_t)(int)(c >> 30) * (int64_t)R, l = (int64_t)((int)c & 0x3fffffff) * (int64_t)R;
  return ((int64_t)R << 36) + ((h + (l >> 30) + (1ll << 15)) >> 16);
}

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t r;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
  return r;
}
// Byte transpose of four words: out[k] = byte k of w0, w1, w2, w3.
__device__ __forceinline__ void transpose4(uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3, uint32_t (&out)[4]) {
  const uint32_t t0 = prmt(w0, w1, 0x5140), t1 = prmt(w2, w3, 0x5140);
  const uint32_t t2 = prmt(w0, w1, 0x7362), t3 = prmt(w2, w3, 0x7362);
  out[0] = prmt(t0, t1, 0x5410);
  out[1] = prmt(t0, t1, 0x7632);
  out[2] = prmt(t2, t3, 0x5410);
  out[3] = prmt(t2, t3, 0x7632);
}
// Two digits (bytes 128 + d, 127 + d) to FP16: the byte under the exponent byte 0x64 is 1024 + 128 + d,
// exact; minus 1152 (1151).
__device__ __forceinline__ uint32_t half2_of(uint32_t w, uint32_t sel, uint32_t offsets) {
  uint32_t h = prmt(w, 0x64646464u, sel), r;
  asm("sub.f16x2 %0, %1, %2;" : "=r"(r) : "r"(h), "r"(offsets));
  return r;
}
// The FP16 digits of eight values (fixed-point numbers with their columns' offsets), one slice per
// element of w.
__device__ __forceinline__ void to_digits(const uint64_t (&q)[8], uint4 (&w)[SL]) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t lo[4], hi[4], b[SL];  // b[s]: digit s of the four values, one byte each
    transpose4((uint32_t)q[4 * h], (uint32_t)q[4 * h + 1], (uint32_t)q[4 * h + 2], (uint32_t)q[4 * h + 3], lo);
    transpose4((uint32_t)(q[4 * h] >> 32), (uint32_t)(q[4 * h + 1] >> 32), (uint32_t)(q[4 * h + 2] >> 32),
               (uint32_t)(q[4 * h + 3] >> 32), hi);
#pragma unroll
    for (int k = 0; k < 4; ++k) b[6 - k] = lo[k];
#pragma unroll
    for (int k = 0; k < 3; ++k) b[2 - k] = hi[k];
#pragma unroll
    for (int s = 0; s < SL; ++s) {
      const uint32_t offsets = s == 6 ? 0x6480647Fu : 0x647F6480u;
      const uint32_t x = half2_of(b[s], 0x4140, offsets), y = half2_of(b[s], 0x4342, offsets);
      if (h == 0) {
        w[s].x = x;
        w[s].y = y;
      } else {
        w[s].z = x;
        w[s].w = y;
      }
    }
  }
}

// Copy sixteen bytes of global memory to shared memory without registers (zeros where !in); groups
// of copies of this thread, and a wait until at most N groups are in flight.
__device__ __forceinline__ void copy16(uint32_t dst, const void *src, bool in) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(in ? 16u : 0u) : "memory");
}
__device__ __forceinline__ void copy8(double *dst, const double *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(tc::smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copies_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// The MMAs of one K = 16 step of one half of the tile's columns, accumulating in the half's
// column blocks at d. a, b: descriptors of the step's octets (slice 0; b: the half's rows). INIT:
// first step of a segment, whose first two MMAs together cover all eight column blocks and
// overwrite them.
template <bool INIT>
__device__ __forceinline__ void mma_step(uint32_t d, uint64_t a, uint64_t b) {
  constexpr uint64_t AS = A_SLICE >> 4, BS = B_SLICE >> 4;
  tc::mma_f16(d + 32 * 4, a + 4 * AS, b, tc::idesc_f16<128>(), INIT ? 0u : 1u);  // s 4,5: t 0-3
  if (INIT) {
    tc::mma_f16(d, a, b, tc::idesc_f16<128>(), 0u);                              // s 0,1: t 0-3
    tc::mma_f16(d + 32 * 4, a, b + 4 * BS, tc::idesc_f16<96>(), 1u);             // s 0,1: t 4-6
  } else {
    tc::mma_f16(d, a, b, tc::idesc_f16<224>(), 1u);                              // s 0,1: t 0-6
  }
  tc::mma_f16(d + 32 * 2, a + 2 * AS, b, tc::idesc_f16<192>(), 1u);              // s 2,3: t 0-5
  tc::mma_f16(d + 32 * 6, a + 6 * AS, b, tc::idesc_f16<64>(), 1u);               // s 6: t 0-1
}

// Read a finished segment of one half back and add it to the 64-bit sums, unit 2^-62: this warp's
// 32 lanes, eight columns from addr (of block 0). Weight p sits in block p (lanes 0-63) or p - 1
// (lanes 64-127, up). SHORT: a segment of at most 64 values of k, whose sums are at most 2^22 in
// magnitude: adding 1.5 * 2^23 leaves the integer in the low bits (a conversion runs at 16 per
// clock and SM, an addition at 128), and pairs of weights combine in 32 bits. diag: this lane's
// row has its diagonal entry here, in column q0; dsum gets its approximate sum of squares.
template <bool SHORT>
__device__ __forceinline__ void drain(uint32_t addr, bool up, unsigned long long (&acc)[8], bool diag, int q0,
                                      float &dsum) {
  const uint32_t base = addr - (up ? 32u : 0u);
#pragma unroll
  for (int p = 0; p < 8; p += 2) {
    uint32_t v[8], w[8];
    tc::ld8x2(base + (p == 0 && up ? 32u : 32u * p), base + 32u * (p + 1), v, w);
    if (p == 0 && up) {  // (weight 0 has no odd slice)
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = 0u;
    }
    if (diag && p < 4) {
      float x = 0.f, y = 0.f;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        x = q == q0 ? __uint_as_float(v[q]) : x;
        y = q == q0 ? __uint_as_float(w[q]) : y;
      }
      const float u = 1.0f / (float)(1ll << (14 + 8 * p));
      dsum += x * u + y * (u / 256.0f);
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      int x, y;
      if constexpr (SHORT) {
        x = __float_as_int(__uint_as_float(v[q]) + 12582912.0f) - 0x4B400000;
        y = __float_as_int(__uint_as_float(w[q]) + 12582912.0f) - 0x4B400000;
      } else {
        x = __float2int_rn(__uint_as_float(v[q]));
        y = __float2int_rn(__uint_as_float(w[q]));
      }
      if (p == 0) acc[q] += (unsigned long long)((unsigned)x * 65536u + (unsigned)y * 256u) << 32;
      else if (p == 2) acc[q] += ((unsigned long long)(unsigned)x << 32) + (unsigned long long)((long long)y * (1 << 24));
      else if (p == 4) acc[q] += SHORT ? (unsigned long long)((long long)(x * 256 + y) * 256)
                                       : (unsigned long long)((long long)x * (1 << 16)) +
                                             (unsigned long long)((long long)y * 256);
      else acc[q] += (unsigned long long)(long long)(x + ((y + 127 + (y >> 8 & 1)) >> 8));  // (halves to even)
    }
  }
}

// The sum of the squares of eight digits.
__device__ __forceinline__ float square_sum(uint4 w) {
  const uint32_t u[4] = {w.x, w.y, w.z, w.w};
  float s[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&u[k]));
    s[k] = fmaf(f.x, f.x, f.y * f.y);
  }
  return (s[0] + s[1]) + (s[2] + s[3]);
}
// Squares of digit 4 (unit 2^-78) in the unit of the 64-bit sums.
__device__ __forceinline__ unsigned long long dropped_squares(float sq) {
  return (unsigned long long)__float2ll_rn(sq * (1.0f / 65536.0f));
}

// c - q 2^(-62) 2^ei 2^ej with one rounding of the product's conversion and one of the sum.
__device__ __forceinline__ double apply(double c, long long q, int ei, int ej) {
  const int x = ei + ej - 62;
  if (x > -1000 && x < 1000) return fma(-(double)q, __hiloint2double((x + 1023) << 20, 0), c);
  return c - ldexp((double)q, x);
}

}  // namespace oz
}  // namespace sym
