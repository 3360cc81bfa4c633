// The element operator in integer digits (ax_dig.cu says how) as the body of a block: one element, DigShape<NP>::T threads.
#pragma once

#include <cmath>

#include "dig.cuh"
#include "eo.cuh"

namespace sem {

namespace {

constexpr int DIG_BAD = INT32_MIN;   // gexp of an element whose factors fixed point cannot hold

template <int NP>
struct DigShape {
  static constexpr int NW = (NP + 1) / 2;         // warps: two planes each
  static constexpr int T = 32 * NW;
  static constexpr int NPE = (NP + 1) / 2 * 2;    // i extent of the stored factors
  static constexpr int GE = NP * NP * NPE;        // stored values per element and component
  static constexpr int FLD = 2 * NW * 64;         // 64-bit values of a field in shared memory
  static constexpr int SMEM = 3 * FLD > 3 * Pad3<NP>::ES ? 3 * FLD : 3 * Pad3<NP>::ES;   // of the block
};

// round(x num/den 2^s) in integers, half away from zero
inline __int128 dig_scaled(double x, int num, int den, int s) {
  int ex;
  const __int128 m = (__int128)std::llround(std::ldexp(std::frexp(x, &ex), 53)) * num;
  const int sh = ex - 53 + s;
  const bool neg = m < 0;
  __int128 a = neg ? -m : m;
  __int128 b = den;
  if (sh >= 0) a <<= sh;
  else b <<= -sh;
  a = (2 * a + b) / (2 * b);
  return neg ? -a : a;
}

// A nodal h1 is kept in 61 bits below the element's largest, so its values keep FP64's 53 bits down to 2^-8 of that, and the pairs' 48
// down to 2^-13; an element whose h1 spans more (a jump of a material, say) is computed in FP64, which keeps every value's own bits.
// That is slow for a pair call (N = 7, 32^3, every element: 1,555 us against 351 in digits and 448 in pairs). dig_h1_low is largest for
// the smallest |h1| that is not zero (a zero is exact in both); dig_h1_wide takes the block's largest high word of |h1| and dig_h1_low.
inline int dig_h1_span(bool pairs) { return 61 - (pairs ? 48 : 53); }
__device__ __forceinline__ uint32_t dig_h1_low(const double h1) {
  const uint32_t a = (uint32_t)__double2hiint(h1) & 0x7fffffffu;
  return (a | (uint32_t)__double2loint(h1)) ? 0x7fffffffu - a : 0u;
}
__device__ __forceinline__ bool dig_h1_wide(const uint32_t high, const uint32_t low, const int span) {
  return (int)(high >> 20) - (int)((0x7fffffffu - low) >> 20) > span;
}

// exponent of a scalar h1, as the kernel takes it (4096: not a normal number, the elements go to the FP64 form)
inline int dig_h1_exp(double h1) { return h1 == 0.0 ? 0 : std::isnormal(h1) ? std::ilogb(h1) : 4096; }

// Elements the fixed-point form does not take. nil: no high word of u is set and h1 and G are finite: the element is zero, unless some
// value is below 2^-1042.
template <int NP, bool VARH1>
__device__ __noinline__ void dig_fallback(double* A, int e, const double* u, double* w, const double* G,
                                          const EOMat<ArF64>& Df, const EOMat<ArF64>& Dt, double h1, double h2,
                                          const double* h1L, bool nil) {
  constexpr int NP2 = NP * NP, NP3 = NP2 * NP;
  if (nil) {
    const size_t eb = (size_t)e * NP3;
    int lo = 0;
    for (int p = threadIdx.x; p < NP3; p += blockDim.x) lo |= __double2loint(u[eb + p]);
    if (!__syncthreads_or(lo != 0)) {
      for (int p = threadIdx.x; p < NP3; p += blockDim.x)
        w[eb + p] = h2 != 0.0 ? h2 * G[7 * eb + 6 * NP3 + p] * u[eb + p] : 0.0;
      return;
    }
  }
  const bool on = threadIdx.x < NP2;
  const int ij = on ? threadIdx.x : 0;
  eo_element<ArF64, NP, VARH1>(on, on, ij % NP, ij / NP, (size_t)e * NP2 * NP, u, w, G + (size_t)e * 7 * NP2 * NP, Df,
                               Dt, h1, h2, h1L, A, A + Pad3<NP>::ES, A + 2 * Pad3<NP>::ES);
}

// w = A^e u of element e. HELD: the block holds the element's u at its own points (uv, zero at points that do not exist;
// also in memory, for an element that fixed point cannot hold) and gets the result there in o too, unless false is returned
// (then the result is in memory only, written by other threads of the block).
// smem: digits of u, then of the s-flux; t-exchange of the derivatives, then digits of the t-flux; t-exchange of the result
// (the even-odd form of an element uses the whole).
template <int NP, bool VARH1, bool HELD>
__device__ __forceinline__ bool dig_element(const int e, const double* __restrict__ u, double* __restrict__ w,
                                            const int2* __restrict__ Gx, const int32_t* __restrict__ gexp,
                                            const double* __restrict__ G, const DigTab* __restrict__ tab,
                                            const int kexp, const double h1, const double h2,
                                            const double* __restrict__ h1L, const int span, const int vec, const int mass, const int e1,
                                            const EOMat<ArF64>& Df, const EOMat<ArF64>& Dt, unsigned long long* smem,
                                            uint32_t (*s_max)[4], double (&uv)[2][2], double (&o)[2][2]) {
  using S = DigShape<NP>;
  constexpr int NP2 = NP * NP, NP3 = NP2 * NP;
  unsigned long long *sA = smem, *sB = smem + S::FLD, *sY = smem + 2 * S::FLD;
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const int g = lane >> 2, c = lane & 3;
  const int k0 = 2 * wp, i0 = 2 * c;
  const int loc = (k0 * NP + g) * NP + i0;   // point (i0, g, k0)
  u += (size_t)e * NP3 + loc;
  w += (size_t)e * NP3 + loc;
  if (VARH1) h1L += (size_t)e * NP3 + loc;
  const double* Bp = G + ((size_t)e * 7 + 6) * NP3 + loc;
  const int2* Gp = Gx + (size_t)e * 6 * S::GE + (k0 * NP + g) * S::NPE + i0;
  const uint4* Dp = &tab->frag[0][0][lane];
  const bool row = NP == 8 || (g < NP && i0 < NP);
  auto has = [&](int p, int x) { return row && (NP % 2 == 0 || (k0 + p < NP && i0 + x < NP)); };
  auto ld2 = [&](const double* v, int p, double (&o)[2]) {
    if (NP % 2 == 0 && vec) {
      const double2 t = has(p, 0) ? *reinterpret_cast<const double2*>(v + p * NP2) : make_double2(0.0, 0.0);
      o[0] = t.x;
      o[1] = t.y;
    } else {
      o[0] = has(p, 0) ? v[p * NP2] : 0.0;
      o[1] = has(p, 1) ? v[p * NP2 + 1] : 0.0;
    }
  };
  // Position of point (i, j, k) in a digit field: 64 k + 16 (j >> 1) + 8 b3 + 4 b2 + (i & 3), b3 = bit 0 of
  // j ^ (j >> 2) ^ (k >> 2), b2 = bit 0 of (i >> 2) ^ (j >> 1) ^ (k >> 1); in an exchange: 64 k + 16 (j >> 1) +
  // 8 ((j ^ k) & 1) + i. The lanes of every access then fall on distinct banks. As the accesses need them:
  const int b23 = ((((c ^ wp) >> 1) & 1) << 3) + ((((g >> 2) ^ c ^ wp) & 1) << 2) + (g & 3);
  const int w0 = k0 * 64 + (g >> 1) * 16 + (((g ^ (g >> 2) ^ (wp >> 1)) & 1) << 3) +
                 ((((c >> 1) ^ (g >> 1) ^ wp) & 1) << 2) + (i0 & 3);   // own points (2c, g, k0 + p): + 64 p
  const int s0 = k0 * 64 + c * 16 + b23;                              // (g, 2c + y, k0 + p): + 64 p, ^ 8 y
  const int t0 = i0 * 64 + wp * 16 + b23;                             // (g, k0 + p, 2c + y): + 64 y, ^ 8 p
  const int xw = g * 64 + wp * 16 + ((g & 1) << 3) + i0;              // exchange, (2c, k0 + p, g): ^ 8 p
  const int xr = k0 * 64 + (g >> 1) * 16 + ((g & 1) << 3) + i0;       // exchange, (2c, g, k0 + p): + 64 p, ^ 8 p

  // the element's factors on their way into L2 before the threads ask for them
  if (!HELD && threadIdx.x == 0) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(Gx + (size_t)e * 6 * S::GE), "r"(6 * S::GE * 8)
                 : "memory");
    if (NP % 2 == 0 && mass)
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(G + ((size_t)e * 7 + 6) * NP3), "r"(NP3 * 8)
                   : "memory");
  }
  // the element's exponents
  double hv[2][2];
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    if (!HELD) ld2(u, p, uv[p]);
    if (VARH1) ld2(h1L, p, hv[p]);
  }
  const int ge = gexp[e];
  uint32_t um = 0, hm = 0, hl = 0;
#pragma unroll
  for (int p = 0; p < 2; ++p)
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      um = max(um, (uint32_t)__double2hiint(uv[p][x]) & 0x7fffffffu);
      if (VARH1) {
        hm = max(hm, (uint32_t)__double2hiint(hv[p][x]) & 0x7fffffffu);
        hl = max(hl, dig_h1_low(hv[p][x]));
      }
    }
  um = __reduce_max_sync(0xffffffffu, um);
  if (VARH1) {
    hm = __reduce_max_sync(0xffffffffu, hm);
    hl = __reduce_max_sync(0xffffffffu, hl);
  }
  if (lane == 0) {
    s_max[0][wp] = um;
    if (VARH1) {
      s_max[1][wp] = hm;
      s_max[3][wp] = hl;
    }
  }
  uint4 D[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) D[m] = Dp[m * 32];
  __syncthreads();
#pragma unroll
  for (int t = 0; t < S::NW; ++t) {
    um = max(um, s_max[0][t]);
    if (VARH1) {
      hm = max(hm, s_max[1][t]);
      hl = max(hl, s_max[3][t]);
    }
  }
  // biased exponent of the largest |u|, one more where its fixed-point form would reach 2^63 (1 - 2^-7)
  const int eu = (int)((um + 0x4000) >> 20);   // no high word set: 0, not held
  const int eh = VARH1 ? (hm ? (int)(hm >> 20) - 1022 : 0) : 0;   // |h1| < 2^eh
  // exponent of the result's unit before the shift by the derivatives' size (at most 32)
  const int ex = ge + eh + eu - 1023 - kexp - DIG_SH2 - 12;
  if (um >= 0x7ff00000u || hm >= 0x7ff00000u || ge == DIG_BAD || abs(ex) > 800 || abs(ex + e1) > 800 ||
      abs(eh) > 800 || abs(eu - 1023) > 800 || (VARH1 && dig_h1_wide(hm, hl, span))) {
    const bool nil = um == 0 && hm < 0x7ff00000u && ge != DIG_BAD && e1 < 4096;
    const ptrdiff_t at = (ptrdiff_t)e * NP3 + loc;
    dig_fallback<NP, VARH1>(reinterpret_cast<double*>(smem), e, u - at, w - at, G, Df, Dt, h1, h2,
                            VARH1 ? h1L - at : nullptr, nil);
    return false;
  }

  // digits of u (below 2^63 (1 - 2^-7): eu); derivatives along r from the lane's own digits
  const DigStart zs;
  unsigned long long Vr[4], Vs[4], Vt[4];   // derivatives at point 2c + x of plane p: [2p + x], two's complement
  {
    unsigned long long X[2][2];
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      X[p][0] = dig_flip(dig_fix(uv[p][0], eu));
      X[p][1] = dig_flip(dig_fix(uv[p][1], eu));
      *reinterpret_cast<ulonglong2*>(&sA[w0 + 64 * p]) = make_ulonglong2(X[p][0], X[p][1]);
    }
    const DigPack a[2][2] = {{DigPack(X[0][0]), DigPack(X[0][1])}, {DigPack(X[1][0]), DigPack(X[1][1])}};
    const ulonglong2 nk = *reinterpret_cast<const ulonglong2*>(&tab->nk0[i0]);
    dig_lines_rows<DIG_SH1>(Vr, D, a, zs, nk);
  }
  __syncthreads();
  // derivatives along s (the warp's planes) and t (rows j = k0, k0 + 1 of every plane)
  uint32_t vm = 0;
  const unsigned long long nkg = tab->nk0[g];
  {
    const DigPack b[2][2] = {{DigPack(sA[s0]), DigPack(sA[s0 ^ 8])},
                             {DigPack(sA[s0 + 64]), DigPack(sA[(s0 ^ 8) + 64])}};
    dig_lines_cols<DIG_SH1>(Vs, D, b, zs, nkg);
#pragma unroll
    for (int r = 0; r < 4; ++r) vm |= dig_size(Vr[r]) | dig_size(Vs[r]);
  }
  const bool in = S::NW == 4 || i0 < 2 * S::NW, tout = S::NW == 4 || g < 2 * S::NW;   // planes that exist
  auto t_digits = [&](const unsigned long long* F, int at) { return DigPack(in ? F[at] : dig_flip(0)); };
  {
    const DigPack b[2][2] = {{t_digits(sA, t0), t_digits(sA, t0 + 64)},
                             {t_digits(sA, t0 ^ 8), t_digits(sA, (t0 ^ 8) + 64)}};
    unsigned long long v[4];
    dig_lines_cols<DIG_SH1>(v, D, b, zs, nkg);
    vm |= dig_size(v[0]) | dig_size(v[1]) | dig_size(v[2]) | dig_size(v[3]);
    if (tout) {
      *reinterpret_cast<ulonglong2*>(&sB[xw]) = make_ulonglong2(v[0], v[1]);
      *reinterpret_cast<ulonglong2*>(&sB[xw ^ 8]) = make_ulonglong2(v[2], v[3]);
    }
  }
  vm = __reduce_or_sync(0xffffffffu, vm);
  if (lane == 0) s_max[2][wp] = vm;
  __syncthreads();

  // fluxes
#pragma unroll
  for (int t = 0; t < S::NW; ++t) vm |= s_max[2][t];
  const int sv = __clz(vm) - 3;   // the largest derivative below 2^61
#pragma unroll
  for (int m = 0; m < 4; ++m) D[m] = Dp[(4 + m) * 32];
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    const ulonglong2 vt = *reinterpret_cast<const ulonglong2*>(&sB[(xr ^ (8 * p)) + 64 * p]);
    Vt[2 * p] = vt.x;
    Vt[2 * p + 1] = vt.y;
  }
  __syncwarp();   // the warp writes its planes of sB next
  unsigned long long fr[2][2];
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    int4 G6[6];
#pragma unroll
    for (int q = 0; q < 6; ++q)
            G6[q] = (NP % 2 == 0 ? row : (row && k0 + p < NP))
                  ? *reinterpret_cast<const int4*>(Gp + q * S::GE + p * NP * S::NPE)
                  : make_int4(0, 0, 0, 0);
    unsigned long long fs[2], ft[2];
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      int ah[3], al[3];
      int Hh = 0, Hl = 0;
      if (VARH1) {
        const long long h = dig_fix(hv[p][x], eh + 1022) >> 2;   // below 2^61
        Hh = dig_hi(h);
        Hl = dig_lo(h);
      }
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        long long v = (long long)((d == 0 ? Vr : d == 1 ? Vs : Vt)[2 * p + x] << sv);
        if (VARH1) {
          const int vh = dig_hi(v), vl = dig_lo(v);
          v = (mul_wide_s(vh, Hh) << 3) + (mad_wide_s(vl, Hh, mul_wide_s(vh, Hl)) >> 29);
        }
        ah[d] = dig_hi(v);
        al[d] = dig_lo(v);
      }
      auto gh = [&](int q) { return x ? G6[q].w : G6[q].y; };
      auto gl = [&](int q) { return x ? G6[q].z : G6[q].x; };
      auto flux = [&](int q0, int q1, int q2) {
        const long long hh =
            mad_wide_s(ah[2], gh(q2), mad_wide_s(ah[1], gh(q1), mul_wide_s(ah[0], gh(q0))));
        const long long m = mad_wide_s(
            al[2], gh(q2),
            mad_wide_s(ah[2], gl(q2),
                       mad_wide_s(al[1], gh(q1),
                                  mad_wide_s(ah[1], gl(q1), mad_wide_s(al[0], gh(q0), mul_wide_s(ah[0], gl(q0)))))));
        // a derivative (times h1) below 2^61, factors below 2^62 / (1 + 2^-5) in sum (k_dig_factors): below 2^63 / (1 + 2^-5)
        return dig_flip((hh << 4) + (m >> 28));
      };
      fr[p][x] = flux(0, 1, 2);
      fs[x] = flux(1, 3, 4);
      ft[x] = flux(2, 4, 5);
    }
    *reinterpret_cast<ulonglong2*>(&sA[w0 + 64 * p]) = make_ulonglong2(fs[0], fs[1]);
    *reinterpret_cast<ulonglong2*>(&sB[w0 + 64 * p]) = make_ulonglong2(ft[0], ft[1]);
  }
  __syncthreads();

  // 2^-a D^T 2^a along t into the exchange, along r and s together
  {
    const unsigned long long nkt = tab->nk1t[g];
    const DigPack b[2][2] = {{t_digits(sB, t0), t_digits(sB, t0 + 64)},
                             {t_digits(sB, t0 ^ 8), t_digits(sB, (t0 ^ 8) + 64)}};
    unsigned long long v[4];
    dig_lines_cols<DIG_SH2>(v, D, b, zs, nkt);
    if (tout) {
      *reinterpret_cast<ulonglong2*>(&sY[xw]) = make_ulonglong2(v[0], v[1]);
      *reinterpret_cast<ulonglong2*>(&sY[xw ^ 8]) = make_ulonglong2(v[2], v[3]);
    }
  }
  unsigned long long W[4];
  {
    const ulonglong2 nk = *reinterpret_cast<const ulonglong2*>(&tab->nk1rs[g * 8 + i0]);
    const DigPack a[2][2] = {{DigPack(fr[0][0]), DigPack(fr[0][1])}, {DigPack(fr[1][0]), DigPack(fr[1][1])}};
    const DigPack b[2][2] = {{DigPack(sA[s0]), DigPack(sA[s0 ^ 8])},
                             {DigPack(sA[s0 + 64]), DigPack(sA[(s0 ^ 8) + 64])}};
    dig_lines_both<DIG_SH2>(W, D, a, b, zs, nk);
  }
  __syncthreads();

  // w = h1 2^(S + a_i + a_j + a_k) W + h2 B u
  const int hs = VARH1 ? 0x3ff00000 : __double2hiint(h1), ls = VARH1 ? 0 : __double2loint(h1);
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    const ulonglong2 wt = *reinterpret_cast<const ulonglong2*>(&sY[(xr ^ (8 * p)) + 64 * p]);
    const int sp = ex - sv + tab->a[k0 + p] + tab->a[g];
#pragma unroll
    for (int x = 0; x < 2; ++x)
      o[p][x] = (double)(long long)(W[2 * p + x] + (x ? wt.y : wt.x)) *
             __hiloint2double(hs + (hs << 1 == 0 ? 0 : (sp + tab->a[i0 + x]) << 20), ls);
    if (mass) {
      double Bv[2];
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        Bv[x] = has(p, x) ? Bp[p * NP2 + x] : 0.0;
        o[p][x] = fma(h2 * Bv[x], uv[p][x], o[p][x]);
      }
    }
    if (NP % 2 == 0 && vec) {
      if (has(p, 0)) *reinterpret_cast<double2*>(w + p * NP2) = make_double2(o[p][0], o[p][1]);
    } else {
      if (has(p, 0)) w[p * NP2] = o[p][0];
      if (has(p, 1)) w[p * NP2 + 1] = o[p][1];
    }
  }
  return true;
}

}  // namespace

}  // namespace sem
