// 1-D contractions of FP64 data on the tensor cores in integer digits.
//
// GB300 issues one FP64 multiply-add per warp and SM every 16 cycles, but an FP16
// mma.sync m16n8k16 (2,048 multiply-adds) every 2.4 and an IMAD.WIDE every 0.4 (measured). So
// the (N+1)-wide contractions run on integers: an element's values, as 64-bit fixed-point numbers
// with one common exponent, are cut into eight 8-bit digits, the entries of the 1-D matrix into
// eight signed 8-bit digits, the products of digits are summed by mma.sync in FP32 (all sums are
// integers below 2^22, so they are exact), and the sums of equal weight are put together in
// 64-bit integers. The digits of weight 2^-8 .. 2^-64 of the product are kept (36 digit products of
// 64), which leaves an error of about 2^-60 of the element's largest term, against 2^-53 of every
// partial sum in FP64.
//
// * Digits of a value. 128 is added to every byte (one 64-bit addition), and a byte b = digit + 128 is put into an FP16
//   register half as it is: as a subnormal its value is b 2^-24, so one byte permute gives two digits, with no
//   conversion. What the 128s add to an output is a constant of the matrix row, which dig_merge's nk takes out again
//   (exactly: an all-zero line gives zero).
// * Two digits of a value lie beside each other along the mma's depth (16 = 8 points x 2 digits),
//   the two matrix digits that belong with them likewise, and the sixteen rows are the eight outputs
//   twice, with the matrix digits shifted by one: rows 0-7 give the odd weights 2q+1, rows 8-15 the even
//   ones 2q. Ten mma.sync are 36 digit products of eight outputs on eight lines, with no padding.
// * The sums start at 0.75 = 1.5 2^23 ulp: the low bits of the FP32 result are the integer sum (its unit
//   is 2^-24), so that no conversion is needed (F2I runs at 16 lanes per clock).
#pragma once

#include <stdint.h>

#include <cuda_runtime.h>

namespace sem {

constexpr int DIG_SH1 = 46, DIG_SH2 = 47;   // scale 2^SH of the leading digit products in a merged sum, per stage

// One order's matrices in digits: stage 0 multiplies by D (scaled by c1), stage 1 by 2^-a D^T 2^a (scaled by
// c2), c1 c2 = 2^k; 2^a_i is the power of two next to (rho_i / max rho)^(3/4), rho the GLL weights (see ax_dig.cu).
struct DigTab {
  uint4 frag[2][4][32];          // [stage][m][lane (g, c)]: (odd, even) rows of output g for input points 2c, 2c+1
  unsigned long long nk0[8];     // stage 0: minus the merged sum of an all-zero line, per output
  unsigned long long nk1t[8];    // stage 1, one direction
  unsigned long long nk1rs[64];  // stage 1, the sum of two directions: outputs (j, i) at 8 j + i
  int32_t a[8];                  // exponents a_i
};

__device__ __forceinline__ void dig_mma(float (&d)[4], const uint32_t a0, const uint32_t a1, const uint32_t a2,
                                        const uint32_t a3, const uint32_t b0, const uint32_t b1, const float c0,
                                        const float c1, const float c2, const float c3) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%12,%13};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(c0), "f"(c1), "f"(c2), "f"(c3));
}

// A fixed-point value is kept with 128 added to each of its bytes (dig_flip; x < 2^63 (1 - 2^-8) keeps that in 64 bits, and every
// use says what bounds its operand): its digits, byte - 128, lie in -128..127 around zero, so that the digit products that are dropped have no mean. dig_pair(x, n) is
// the bytes 2n+1 (low half) and 2n (high half) in FP16.
__device__ __forceinline__ unsigned long long dig_flip(const long long x) {
  return (unsigned long long)x + 0x8080808080808080ull;
}
__device__ __forceinline__ uint32_t dig_pair(const unsigned long long x, const int n) {
  return __byte_perm(n < 2 ? (uint32_t)(x >> 32) : (uint32_t)x, 0, n & 1 ? 0x4140 : 0x4342);
}

struct DigPack {
  uint32_t p[4];
  __device__ __forceinline__ explicit DigPack(const unsigned long long x)
      : p{dig_pair(x, 0), dig_pair(x, 1), dig_pair(x, 2), dig_pair(x, 3)} {}
};

// 0.75 in four registers that the compiler cannot rebuild: as the first product's addend they cost no
// instruction, while constants would be moved into place for every one.
struct DigStart {
  float z[4];
  __device__ __forceinline__ DigStart() {
#pragma unroll
    for (int i = 0; i < 4; ++i) asm volatile("mov.b32 %0, 0x3F400000;" : "=f"(z[i]));
  }
};

constexpr __host__ __device__ int dig_q(const int H, const int h) { return H == 0 ? 3 - 3 * h : 2 - h; }   // {3, 0}, {2, 1}

// Digit sums of four outputs a lane. A result needs the weights q = 0..3 (2q and 2q+1) of q + 1 chained products each;
// q runs through {3, 0} and then {2, 1} (H = 0, 1), and two fields go together, so that four to eight independent products
// are in flight (one product's latency is several times its issue time) while 32 registers hold their sums.
//
// Lines as columns: out[h][p] = weights 2q+1 ([0], [1]) and 2q ([2], [3]) of output g for
// lines 2c and 2c+1 of field p; b[p][x]: the digits of point 2c+x of line g. START: the sums begin at 0.75, else at 0.
template <bool START, int H>
__device__ __forceinline__ void dig_cols(float (&out)[2][2][4], const uint4 (&D)[4], const DigPack (&b)[2][2],
                                         const DigStart& z) {
#pragma unroll
  for (int m = 0; m <= 3 - H; ++m)
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        const int n = dig_q(H, h) - m;
        float(&o)[4] = out[h][p];
        if (n < 0) {
        } else if (m > 0)
          dig_mma(o, D[m].x, D[m].y, D[m].z, D[m].w, b[p][0].p[n], b[p][1].p[n], o[0], o[1], o[2], o[3]);
        else if (START)
          dig_mma(o, D[0].x, D[0].y, D[0].z, D[0].w, b[p][0].p[n], b[p][1].p[n], z.z[0], z.z[1], z.z[2], z.z[3]);
        else
          dig_mma(o, D[0].x, D[0].y, D[0].z, D[0].w, b[p][0].p[n], b[p][1].p[n], 0.f, 0.f, 0.f, 0.f);
      }
}

// Lines as rows (two sets of eight): out[h][0] (weight 2q) and out[h][1] (2q+1) of outputs 2c, 2c+1 for line g of the first
// set ([0], [1]) and the second ([2], [3]); a[s][x]: the digits of point 2c+x of line g of set s.
template <int H>
__device__ __forceinline__ void dig_rows(float (&out)[2][2][4], const uint4 (&D)[4], const DigPack (&a)[2][2],
                                         const DigStart& z) {
#pragma unroll
  for (int m = 0; m <= 3 - H; ++m)
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int o = 0; o < 2; ++o) {
        const int n = dig_q(H, h) - m;
        float(&t)[4] = out[h][o];
        const uint32_t b0 = o ? D[m].x : D[m].y, b1 = o ? D[m].z : D[m].w;
        if (n < 0) {
        } else if (m > 0)
          dig_mma(t, a[0][0].p[n], a[1][0].p[n], a[0][1].p[n], a[1][1].p[n], b0, b1, t[0], t[1], t[2], t[3]);
        else
          dig_mma(t, a[0][0].p[n], a[1][0].p[n], a[0][1].p[n], a[1][1].p[n], b0, b1, z.z[0], z.z[1], z.z[2], z.z[3]);
      }
}

__device__ __forceinline__ long long mad_wide_s(const int a, const int b, const long long c) {
  long long d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
}
__device__ __forceinline__ long long mul_wide_s(const int a, const int b) {
  long long d;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
  return d;
}

// A result's merged sum, sum_d f_d 2^(SH - 8d). Pairs of weights first, p_q = 256 f_2q + f_2q+1 (as the integers of
// the sums' bits: no carry is lost, a sum is below 2^21), then v = 2^(SH-40) (2^32 p_0 + 2^16 p_1 + p_2) + 2^(SH-56) p_3 + nk
// by shifts and additions: IMAD.WIDE, which would need one instruction a weight, runs at 1.4 cycles a warp and SM
// and not beside mma.sync (measured), these at 0.3 and 0.5.
struct DigAcc {
  uint32_t p0, p3;
};
__device__ __forceinline__ uint32_t dig_two(const float fe, const float fo) {
  return (__float_as_uint(fe) << 8) + __float_as_uint(fo);
}
template <int SH>
__device__ __forceinline__ unsigned long long dig_merge(const DigAcc a, const uint32_t p1, const uint32_t p2,
                                                        const unsigned long long nk) {
  // written out: as 64-bit shifts the compiler would make IMAD.WIDE of them
  uint32_t lo, hi, l6, h6;
  asm("{\n .reg .u32 a, b;\n shl.b32 a, %2, 16;\n shr.u32 b, %2, 16;\n add.cc.u32 %0, %3, a;\n addc.u32 %1, %4, b;\n}"
      : "=r"(lo), "=r"(hi)
      : "r"(p1), "r"(p2), "r"(a.p0));
  asm("shl.b32 %0, %1, %2;" : "=r"(l6) : "r"(lo), "n"(SH - 40));
  asm("shf.l.wrap.b32 %0, %1, %2, %3;" : "=r"(h6) : "r"(lo), "r"(hi), "n"(SH - 40));
  return (((unsigned long long)h6 << 32) | l6) + nk + (a.p3 >> (56 - SH));
}

// A pair of result r = 2p + x: columns, and columns on top of rows.
__device__ __forceinline__ uint32_t dig_two_cols(const float (&f)[2][4], const int r) {
  return dig_two(f[r >> 1][2 + (r & 1)], f[r >> 1][r & 1]);
}
__device__ __forceinline__ uint32_t dig_two_both(const float (&t)[2][4], const float (&f)[2][4], const int r) {
  return dig_two(t[0][r] + f[r >> 1][2 + (r & 1)], t[1][r] + f[r >> 1][r & 1]);
}

// The merged results of two planes, v[2p + x] = output x of plane p: along rows (nk.x, nk.y for x = 0, 1), along
// columns (one nk), and the sum of both.
template <int SH>
__device__ __forceinline__ void dig_lines_rows(unsigned long long (&v)[4], const uint4 (&D)[4], const DigPack (&a)[2][2],
                                               const DigStart& z, const ulonglong2 nk) {
  float f[2][2][4];
  DigAcc s[4];
  dig_rows<0>(f, D, a, z);
#pragma unroll
  for (int r = 0; r < 4; ++r) s[r] = {dig_two(f[1][0][r], f[1][1][r]), dig_two(f[0][0][r], f[0][1][r])};
  dig_rows<1>(f, D, a, z);
#pragma unroll
  for (int r = 0; r < 4; ++r)
    v[r] = dig_merge<SH>(s[r], dig_two(f[1][0][r], f[1][1][r]), dig_two(f[0][0][r], f[0][1][r]), r & 1 ? nk.y : nk.x);
}
template <int SH>
__device__ __forceinline__ void dig_lines_cols(unsigned long long (&v)[4], const uint4 (&D)[4], const DigPack (&b)[2][2],
                                               const DigStart& z, const unsigned long long nk) {
  float f[2][2][4];
  DigAcc s[4];
  dig_cols<true, 0>(f, D, b, z);
#pragma unroll
  for (int r = 0; r < 4; ++r) s[r] = {dig_two_cols(f[1], r), dig_two_cols(f[0], r)};
  dig_cols<true, 1>(f, D, b, z);
#pragma unroll
  for (int r = 0; r < 4; ++r) v[r] = dig_merge<SH>(s[r], dig_two_cols(f[1], r), dig_two_cols(f[0], r), nk);
}
template <int SH>
__device__ __forceinline__ void dig_lines_both(unsigned long long (&v)[4], const uint4 (&D)[4], const DigPack (&a)[2][2],
                                               const DigPack (&b)[2][2], const DigStart& z, const ulonglong2 nk) {
  float t[2][2][4], f[2][2][4];
  DigAcc s[4];
  dig_rows<0>(t, D, a, z);
  dig_cols<false, 0>(f, D, b, z);
#pragma unroll
  for (int r = 0; r < 4; ++r) s[r] = {dig_two_both(t[1], f[1], r), dig_two_both(t[0], f[0], r)};
  dig_rows<1>(t, D, a, z);
  dig_cols<false, 1>(f, D, b, z);
#pragma unroll
  for (int r = 0; r < 4; ++r) v[r] = dig_merge<SH>(s[r], dig_two_both(t[1], f[1], r), dig_two_both(t[0], f[0], r), r & 1 ? nk.y : nk.x);
}

// One group of eight lines as columns, all weights at once: f[q] = weights 2q+1 ([0], [1]) and 2q ([2], [3]) of output g for
// lines 2c and 2c+1; b[x]: the digits of point 2c+x of line g. START: the sums begin at 0.75, else they go on.
template <bool START>
__device__ __forceinline__ void dig_sums(float (&f)[4][4], const uint4 (&D)[4], const DigPack (&b)[2],
                                         const DigStart& z) {
#pragma unroll
  for (int m = 0; m < 4; ++m)
#pragma unroll
    for (int q = 3; q >= m; --q) {
      const int n = q - m;
      float(&o)[4] = f[q];
      if (START && m == 0)
        dig_mma(o, D[0].x, D[0].y, D[0].z, D[0].w, b[0].p[n], b[1].p[n], z.z[0], z.z[1], z.z[2], z.z[3]);
      else
        dig_mma(o, D[m].x, D[m].y, D[m].z, D[m].w, b[0].p[n], b[1].p[n], o[0], o[1], o[2], o[3]);
    }
}
template <int SH>
__device__ __forceinline__ unsigned long long dig_merge4(const float (&f)[4][4], const int x,
                                                         const unsigned long long nk) {
  const DigAcc a = {dig_two(f[0][2 + x], f[0][x]), dig_two(f[3][2 + x], f[3][x])};
  return dig_merge<SH>(a, dig_two(f[1][2 + x], f[1][x]), dig_two(f[2][2 + x], f[2][x]), nk);
}

// |x| as a fixed-point number of 63 bits with binary exponent `top` (the biased exponent of the
// element's largest value) at bit 62, the sign applied; the bits below are dropped.
__device__ __forceinline__ long long dig_fix(const double x, const int top) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  const int d = min(top - ((hi >> 20) & 0x7ff), 63);
  const unsigned long long m =
      (((unsigned long long)(uint32_t)((hi & 0xfffff) | 0x100000) << 32) | (uint32_t)lo) << 10;
  const long long s = hi >> 31;
  return ((long long)(m >> d) ^ s) - s;
}

// high word of |v| (of its one's complement where v < 0)
__device__ __forceinline__ uint32_t dig_size(const unsigned long long v) {
  const int h = (int)(v >> 32);
  return (uint32_t)(h ^ (h >> 31));
}

// hi and lo of a 64-bit integer v = hi 2^32 + lo with a signed lo
__device__ __forceinline__ int dig_lo(const long long v) { return (int)(uint32_t)v; }
__device__ __forceinline__ int dig_hi(const long long v) {
  return (int)(uint32_t)((unsigned long long)v >> 32) + (int)((uint32_t)v >> 31);
}

// ---- host ----------------------------------------------------------------------------------------

// FP16 bits of an integer |v| <= 2048
inline uint16_t half_of(int v) {
  if (v == 0) return 0;
  const int a = v < 0 ? -v : v, ex = 31 - __builtin_clz((unsigned)a);
  return (uint16_t)((v < 0 ? 0x8000 : 0) | ((ex + 15) << 10) | ((a << 10 >> ex) & 0x3ff));
}

// What a merge gives, without nk, where every value is zero (bytes 128): r[d] = the sum of the row's matrix digits d.
inline unsigned long long dig_merge_zero(const int64_t (&r0)[8], int SH) {
  int64_t s[8], c = 0;
  for (int d = 0; d < 8; ++d) s[d] = 128 * (c += r0[d]);
  auto two = [&](int q) { return (uint32_t)(((0x3f400000 + s[2 * q]) << 8) + 0x3f400000 + s[2 * q + 1]); };
  const unsigned long long r = (((unsigned long long)two(0) << 32) | two(2)) + ((unsigned long long)two(1) << 16);
  return (r << (SH - 40)) + (two(3) >> (56 - SH));
}

}  // namespace sem
