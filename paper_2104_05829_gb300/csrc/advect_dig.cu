// The dealiased advection operator of FP64 data (see advect.cu) in integer digits on the tensor cores
// (dig.cuh), for 4 <= N <= 7.
//
// What bounds it: the FP64 form executes about 620 FP64 instructions a nodal point and component at 16 cycles a warp and
// SM. Here an element of N = 7 with three components costs 10,320 mma.sync (2.3 cycles each, a third of the time), 49,000
// merged sums of eleven 32-bit instructions, and 124 KB of factors; the rest is the latency of chains at the 16 warps an SM that
// the intermediate fields leave room for (88 KB a block, two blocks; twelve warps a block with fewer registers were slower, 0.95
// against 0.85 ms). 16^3, three components: N = 7 3.52 ms in FP64 and 2.27 ms in FP32 pairs -> 0.83 ms; 18^3, N = 6 3.41 and
// 1.42 -> 1.09; 21^3, N = 5 3.07 and 1.33 -> 1.28; 25^3, N = 4 2.71 (pairs 0.95, kept) -> 1.03.
//
// Per element (one block), with the interpolation I (GLL -> Gauss, nq x (N+1)), its derivative DI = Dq I and
// B = 2^-a I^T 2^b (the powers of two next to the quadrature weights, as in ax_dig.cu):
//   wind:    c_m at the Gauss points by three passes of I, chat_d = sum_m G_dm c_m, kept in shared memory;
//   each u:  r: I, DI; s: I and DI on the first, I on the second; t: I, I, DI give u_r, u_s, u_t, every pass eight points long
//            (differentiating on the Gauss points would take passes of nq = 12 points, padded to 16);
//            conv = sum_d chat_d u_d in registers; three passes of B back to the GLL points.
// A warp takes a group of eight lines and a tile of eight outputs (lane (g, c): output g of lines 2c, 2c+1). Every pass writes
// its results with the next pass's direction contiguous, so that a lane reads its two points of a line as 16 bytes.
// All values stay below their first bound (c 2^61, u 2^62) through the passes: each scales its matrix by a power of two so that no
// row sum exceeds 2, and a pass halves the unit. c, chat and conv are shifted up by their largest values before the
// products and the passes back, where few bits would be left otherwise.
//
// Elements that fixed point cannot hold go to the FP64 form in the same block.
#include <algorithm>
#include <cmath>
#include <vector>

#include "advect.cuh"
#include "dig.cuh"

namespace sem {

namespace {

constexpr int ADV_SH = 48;
// The factors and the wind have one exponent each, so where chat comes out 2^-k of what the two could give, it keeps 61 - k bits: the
// wind along a thin element, with one large and one small component and the metric the other way round. FP64 keeps every
// product's own bits. Elements that lose more than these go to the FP64 form (53 bits, less the one that a bound may be off; 48).
// Smooth data, elements 2^-k of their width thick, 2-norm error against 128-bit arithmetic at k = 0, 6, 8, 10, 14, 20: N = 7 2.5e-15, 2.4e-15,
// 2.9e-15, 9.5e-15, 1.5e-13, 9.9e-12 in digits throughout and at most 3.9e-15, the FP64 form's at any k, with the line here
// (N = 4: up to 1.0e-11, and 3.3e-15). What it costs a call without such elements: nothing (24^3, N = 7: 2.84 ms before and after).
constexpr int ADV_LOSS = 61 - 53 - 1, ADV_LOSS_PAIRS = 61 - 48;

template <int NP>
struct DigAdv {
  static constexpr int NQ = nq_of(NP), NQ2 = NQ * NQ, NP2 = NP * NP, NP3 = NP2 * NP;
  static constexpr int LQ = (NQ2 + 7) / 8 * 8;      // (r, s) lines at the Gauss points, padded to groups of eight
  static constexpr int TQ = NQ > 8 ? 2 : 1;         // tiles of Gauss outputs; depth steps of the passes back
  static constexpr int CS = (NQ + 1) / 2 * 2;       // line stride of the passes back
  static constexpr int G5 = (NP * NQ + 7) / 8;      // groups of (t, r) lines in the s-pass back
  static constexpr int W = 8;                       // warps
  static constexpr int T = 32 * W;
  // shared memory, in 64-bit values
  static constexpr int X = 0, T1 = NP * 64, D1 = T1 + NQ * 64;                 // u; after the r-pass
  static constexpr int R0 = D1 + NQ * 64;
  static constexpr int TT = R0, SD = TT + LQ * 8, RD = SD + LQ * 8;            // after the s-pass (wind: components 0..2)
  static constexpr int CH = RD + LQ * 8, CZS = LQ + 8;                         // chat [3][NQ][CZS]
  static constexpr int END = CH + 3 * NQ * CZS;
  static constexpr int CV = 0, V1 = 0, V2 = TT;                                // conv; passes back
  static_assert(LQ * CS + 16 <= R0 && NP * 8 * CS + 16 <= R0 && G5 * 8 * CS + 16 <= 3 * LQ * 8, "shared memory regions");
  static constexpr size_t SMEM = 8 * (size_t)END;
};

// Tiles of matrix rows: I 0..7, DI 0..7, I 8..11 with DI 8..11, I 8.., DI 8.., B (two depth steps)
enum { F_I, F_D, F_ID, F_I8, F_D8, F_B0, F_B1, F_N };

}  // namespace

struct AdvDigTab {
  uint4 frag[F_N][4][32];
  unsigned long long nk[F_N][8];   // B: at F_B0
  int32_t a[8];                    // 2^a next to the GLL weights
};

namespace {

__device__ __forceinline__ void adv_load(uint4 (&D)[4], const AdvDigTab* tab, const int f, const int lane) {
#pragma unroll
  for (int m = 0; m < 4; ++m) D[m] = tab->frag[f][m][lane];
}

// the lane's two results of a line group whose points 2c, 2c + 1 are at p
__device__ __forceinline__ ulonglong2 adv_line(const uint4 (&D)[4], const unsigned long long* p, const DigStart& z,
                                               const unsigned long long nk) {
  const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p);
  const DigPack b[2] = {DigPack(v.x), DigPack(v.y)};
  float f[4][4];
  dig_sums<true>(f, D, b, z);
  return make_ulonglong2(dig_merge4<ADV_SH>(f, 0, nk), dig_merge4<ADV_SH>(f, 1, nk));
}

// the same for two groups (twice the independent products in flight, one set of matrix digits)
__device__ __forceinline__ void adv_line2(ulonglong2 (&o)[2], const uint4 (&D)[4], const unsigned long long* p0,
                                          const unsigned long long* p1, const DigStart& z, const unsigned long long nk) {
  const ulonglong2 v0 = *reinterpret_cast<const ulonglong2*>(p0), v1 = *reinterpret_cast<const ulonglong2*>(p1);
  const DigPack b0[2] = {DigPack(v0.x), DigPack(v0.y)}, b1[2] = {DigPack(v1.x), DigPack(v1.y)};
  float f[4][4], h[4][4];
  dig_sums<true>(f, D, b0, z);
  dig_sums<true>(h, D, b1, z);
  o[0] = make_ulonglong2(dig_merge4<ADV_SH>(f, 0, nk), dig_merge4<ADV_SH>(f, 1, nk));
  o[1] = make_ulonglong2(dig_merge4<ADV_SH>(h, 0, nk), dig_merge4<ADV_SH>(h, 1, nk));
}

// the same over TQ depth steps of eight points (B); shift >= 0: plain values, shifted up first
template <int TQ>
__device__ __forceinline__ ulonglong2 adv_back(const AdvDigTab* tab, const int lane, const unsigned long long* p,
                                               const DigStart& z, const unsigned long long nk, const int shift = -1) {
  float f[4][4];
#pragma unroll
  for (int s = 0; s < TQ; ++s) {
    uint4 D[4];
    adv_load(D, tab, F_B0 + s, lane);
    ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p + 8 * s);
    if (shift >= 0) v = make_ulonglong2(dig_flip((long long)(v.x << shift)), dig_flip((long long)(v.y << shift)));
    const DigPack b[2] = {DigPack(v.x), DigPack(v.y)};
    if (s == 0) dig_sums<true>(f, D, b, z);
    else dig_sums<false>(f, D, b, z);
  }
  return make_ulonglong2(dig_merge4<ADV_SH>(f, 0, nk), dig_merge4<ADV_SH>(f, 1, nk));
}

__device__ __forceinline__ ulonglong2 flip2(const ulonglong2 v) {
  return make_ulonglong2(dig_flip((long long)v.x), dig_flip((long long)v.y));
}

template <int NP>
__device__ __noinline__ void adv_fallback(unsigned char* smem, int e, int ncomp, int64_t nL, const double* cv,
                                          const double* uv, const double* Gq, const double* Im, const double* Dq,
                                          double* wv, const AdvOps<double, NP>& P) {
  constexpr int NQ = nq_of(NP);
  const int t = threadIdx.x < NQ * NQ ? threadIdx.x : 0;
  __syncthreads();
  advect_element<AdvPlain<double>, NP>(threadIdx.x < NQ * NQ, t % NQ, t / NQ, e, smem, ncomp, nL, cv, uv, Gq, Im, Dq, wv,
                                       P);
}

template <int NP>
__global__ void __launch_bounds__(DigAdv<NP>::T, 2)
    k_advect_dig(const int ncomp, const int64_t nL, const double* __restrict__ cv, const double* __restrict__ uv,
                 const int2* __restrict__ Gx, const int32_t* __restrict__ gexp, const AdvDigTab* __restrict__ tab,
                 const int ebase, const int loss, double* __restrict__ wv, const double* __restrict__ Gq, const double* __restrict__ Im,
                 const double* __restrict__ Dq, const __grid_constant__ AdvOps<double, NP> P) {
  using S = DigAdv<NP>;
  constexpr int NQ = S::NQ, NP2 = S::NP2, NP3 = S::NP3, W = S::W, LQ = S::LQ;
  extern __shared__ __align__(16) unsigned char s_raw[];
  unsigned long long* sm = reinterpret_cast<unsigned long long*>(s_raw);
  __shared__ uint32_t s_max[2][W];
  const int e = blockIdx.x;
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const int g = lane >> 2, c = lane & 3;
  const size_t eb = (size_t)e * NP3;
  const DigStart zs;
  // largest |value| of n fields (high words, at least 1 for a value that is not zero) over the element; one barrier
  int par = 0;
  auto largest = [&](const double* v, int n) {
    uint32_t m = 0;
    for (int f = 0; f < n; ++f)
      for (int q = threadIdx.x; q < NP3; q += S::T) {
        const double x = v[(size_t)f * nL + eb + q];
        m = max(m, ((uint32_t)__double2hiint(x) & 0x7fffffffu) | (__double2loint(x) != 0));
      }
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0) s_max[par][wp] = m;
    __syncthreads();
#pragma unroll
    for (int t = 0; t < W; ++t) m = max(m, s_max[par][t]);
    par ^= 1;
    return m;
  };
  // or of the block's values (sizes of results); one barrier
  auto merged = [&](uint32_t m) {
    m = __reduce_or_sync(0xffffffffu, m);
    if (lane == 0) s_max[par][wp] = m;
    __syncthreads();
#pragma unroll
    for (int t = 0; t < W; ++t) m |= s_max[par][t];
    par ^= 1;
    return m;
  };
  // a field as sign-flipped fixed point, its largest value's exponent at bit 62 - down: |u| < 2^62, |c| < 2^61. A pass's row sums
  // are below 2 and its unit is doubled, so every later operand of dig_flip keeps that bound; conv, at most 1.16 2^61 (the row
  // sums of I, I, DI over the three directions, N = 6), is below 2^62 once shifted.
  auto load = [&](const double* v, int ex, int down) {
    for (int q = threadIdx.x; q < NP3; q += S::T) {
      const int k = q / NP2, j = q / NP % NP, i = q % NP;
      sm[S::X + (k * 8 + j) * 8 + i] = dig_flip(dig_fix(v[eb + q], ex) >> down);
    }
  };
  // position of (j = 2c, k) behind output a of the r-pass
  auto t1 = [&](int a, int k) { return a * 64 + (((k * 4 + c) ^ (4 * (a & 1))) * 2); };
  const uint32_t cm = largest(cv, 3);
  const int ge = gexp[e];
  const int ec = cm ? (int)((cm + 0x4000) >> 20) : 1023;
  bool bad = cm >= 0x7ff00000u || ge == INT32_MIN || abs(ec - 1023) > 400;

  // 1. wind at the Gauss points
  for (int m = 0; m < 3 && !bad; ++m) {
    load(cv + (size_t)m * nL, ec, 2);
    __syncthreads();
    for (int it = wp; it < S::TQ * NP; it += W) {
      const int t = it / NP, k = it - t * NP;
      uint4 D[4];
      adv_load(D, tab, t ? F_I8 : F_I, lane);
      const ulonglong2 v = flip2(adv_line(D, sm + S::X + (k * 8 + g) * 8 + 2 * c, zs, tab->nk[t ? F_I8 : F_I][g]));
      const int a = 8 * t + g;
      if (a < NQ) *reinterpret_cast<ulonglong2*>(sm + S::T1 + t1(a, k)) = v;
    }
    __syncthreads();
    for (int it = wp; it < S::TQ * NQ; it += W) {
      const int t = it / NQ, a = it - t * NQ;
      uint4 D[4];
      adv_load(D, tab, t ? F_I8 : F_I, lane);
      const ulonglong2 v = flip2(
          adv_line(D, sm + S::T1 + a * 64 + (((g * 4 + c) ^ (4 * (a & 1))) * 2), zs, tab->nk[t ? F_I8 : F_I][g]));
      const int b = 8 * t + g;
      if (b < NQ) *reinterpret_cast<ulonglong2*>(sm + S::TT + m * LQ * 8 + (a * NQ + b) * 8 + 2 * c) = v;
    }
    // the next component's r-pass waits at the barrier after its load
  }
  __syncthreads();
  // 2. contravariant wind: the t-pass, then c and chat shifted up to 61 bits by their largest values, as unit-normalised
  // factors of the products that follow (lane by lane on its own points)
  int sc = 0;   // binary digits by which chat was shifted
  if (!bad) {
    auto points = [&](auto f) {   // f(cz, l0, valid points x of lines l0 + 2c + x)
      for (int it = wp; it < S::TQ * (LQ / 8); it += W) {
        const int t = it / (LQ / 8), l0 = (it - t * (LQ / 8)) * 8;
        f(t, l0, 8 * t + g);
      }
    };
    auto size2 = [&](int l0, const ulonglong2 v) {
      return (l0 + 2 * c < S::NQ2 ? dig_size(v.x) : 0u) | (l0 + 2 * c + 1 < S::NQ2 ? dig_size(v.y) : 0u);
    };
    uint32_t vm = 0;
    points([&](int t, int l0, int cz) {
      uint4 D[4];
      adv_load(D, tab, t ? F_I8 : F_I, lane);
      const unsigned long long nk = tab->nk[t ? F_I8 : F_I][g];
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        const ulonglong2 v = adv_line(D, sm + S::TT + m * LQ * 8 + (l0 + g) * 8 + 2 * c, zs, nk);
        if (cz < NQ) {
          *reinterpret_cast<ulonglong2*>(sm + S::CH + (m * NQ + cz) * S::CZS + l0 + 2 * c) = v;
          vm |= size2(l0, v);
        }
      }
    });
    const int s1 = __clz(merged(vm)) - 3;
    vm = 0;
    points([&](int t, int l0, int cz) {
      if (cz >= NQ) return;
      ulonglong2* ch = reinterpret_cast<ulonglong2*>(sm + S::CH + cz * S::CZS + l0 + 2 * c);
      int vh[3][2], vl[3][2];
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        const ulonglong2 v = ch[m * (NQ * S::CZS / 2)];
        vh[m][0] = dig_hi((long long)(v.x << s1));
        vl[m][0] = dig_lo((long long)(v.x << s1));
        vh[m][1] = dig_hi((long long)(v.y << s1));
        vl[m][1] = dig_lo((long long)(v.y << s1));
      }
      const int2* Gp = Gx + ((size_t)e * 9 * NQ + cz) * LQ + l0 + 2 * c;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        long long h[2], l[2];
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          const int4 G2 = *reinterpret_cast<const int4*>(Gp + (size_t)(3 * d + m) * NQ * LQ);
#pragma unroll
          for (int x = 0; x < 2; ++x) {
            const int gl = x ? G2.z : G2.x, gh = x ? G2.w : G2.y;
            h[x] = m ? mad_wide_s(vh[m][x], gh, h[x]) : mul_wide_s(vh[m][x], gh);
            l[x] = mad_wide_s(vl[m][x], gh, m ? mad_wide_s(vh[m][x], gl, l[x]) : mul_wide_s(vh[m][x], gl));
          }
        }
        const ulonglong2 v = make_ulonglong2((h[0] << 2) + (l[0] >> 30), (h[1] << 2) + (l[1] >> 30));
        ch[d * (NQ * S::CZS / 2)] = v;
        vm |= size2(l0, v);
      }
    });
    const int s2 = __clz(merged(vm)) - 3;
    points([&](int t, int l0, int cz) {
      if (cz >= NQ) return;
      ulonglong2* ch = reinterpret_cast<ulonglong2*>(sm + S::CH + cz * S::CZS + l0 + 2 * c);
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const ulonglong2 v = ch[d * (NQ * S::CZS / 2)];
        const long long x = (long long)(v.x << s2), y = (long long)(v.y << s2);
        *reinterpret_cast<int4*>(&ch[d * (NQ * S::CZS / 2)]) = make_int4(dig_lo(x), dig_hi(x), dig_lo(y), dig_hi(y));
      }
    });
    sc = s1 + s2;
    bad = s2 > loss && cm != 0;
  }

  // 3. every advected component
  for (int comp = 0; comp < ncomp; ++comp) {
    const double* u = uv + (size_t)comp * nL;
    const uint32_t um = largest(u, 1);
    const int eu = um ? (int)((um + 0x4000) >> 20) : 1023;
    const int ex = ebase + ge + (ec - 1023) + (eu - 1023) - sc;   // exponent of the result's unit, before conv is shifted
    if (bad || um >= 0x7ff00000u || abs(eu - 1023) > 400 || abs(ex) > 900) {
      adv_fallback<NP>(s_raw, e, ncomp, nL, cv, uv, Gq, Im, Dq, wv, P);
      return;
    }
    load(u, eu, 1);
    __syncthreads();
    // r: I and DI
    {
      constexpr int NT = S::TQ == 2 ? 3 : 2;
      const int i0 = wp * (NT * NP) / W, i1 = (wp + 1) * (NT * NP) / W;
      uint4 D[4];
      int cur = -1;
      for (int it = i0; it < i1; ++it) {
        const int t = it / NP, k = it - t * NP;
        if (t != cur) adv_load(D, tab, t, lane);
        cur = t;
        const ulonglong2 v = flip2(adv_line(D, sm + S::X + (k * 8 + g) * 8 + 2 * c, zs, tab->nk[t][g]));
        const int a = t == F_ID ? 8 + (g & 3) : g;
        const int to = t == F_D || (t == F_ID && g >= 4) ? S::D1 : S::T1;
        if (a < NQ) *reinterpret_cast<ulonglong2*>(sm + to + t1(a, k)) = v;
      }
    }
    __syncthreads();
    // s: I and DI on the first, I on the second
    {
      constexpr int NT = S::TQ == 2 ? 5 : 3;
      const int i0 = wp * (NT * NQ) / W, i1 = (wp + 1) * (NT * NQ) / W;
      uint4 D[4];
      int cur = -1;
      for (int it = i0; it < i1; ++it) {
        const int kind = it / NQ, a = it - kind * NQ;
        const bool two = it + 1 < i1 && a + 1 < NQ;   // the next group has the same matrix
        // tile of kind: TQ = 2: F_I, F_D, F_ID on T1, F_I, F_I8 on D1; TQ = 1: F_I, F_D on T1, F_I on D1
        const bool second = kind >= S::TQ + 1;
        const int t = !second ? kind : kind == S::TQ + 1 ? F_I : F_I8;
        if (kind != cur) adv_load(D, tab, t, lane);
        cur = kind;
        const int b = t == F_ID ? 8 + (g & 3) : t == F_I8 ? 8 + g : g;
        unsigned long long* to =
            sm + (second ? S::RD : t == F_D || (t == F_ID && g >= 4) ? S::SD : S::TT) + (a * NQ + b) * 8 + 2 * c;
        const unsigned long long* from = sm + (second ? S::D1 : S::T1) + a * 64;
        const int p0 = ((g * 4 + c) ^ (4 * (a & 1))) * 2;
        const unsigned long long nk = tab->nk[t][g];
        if (two) {
          ulonglong2 v[2];
          adv_line2(v, D, from + p0, from + 64 + (p0 ^ 8), zs, nk);
          if (b < NQ) {
            *reinterpret_cast<ulonglong2*>(to) = flip2(v[0]);
            *reinterpret_cast<ulonglong2*>(to + NQ * 8) = flip2(v[1]);
          }
          ++it;
        } else {
          const ulonglong2 v = flip2(adv_line(D, from + p0, zs, nk));
          if (b < NQ) *reinterpret_cast<ulonglong2*>(to) = v;
        }
      }
    }
    __syncthreads();
    // t: I, I, DI, and the product with the wind
    uint32_t vm = 0;
    for (int it = wp; it < S::TQ * (LQ / 8); it += W) {
      const int t = it / (LQ / 8), l0 = (it - t * (LQ / 8)) * 8, cz = 8 * t + g;
      long long h[2], l[2];
      const int4* ch = reinterpret_cast<const int4*>(sm + S::CH + (cz < NQ ? cz : 0) * S::CZS + l0 + 2 * c);
      // below 2^62 x 2^61 in three terms: h, the cross terms l and the signed high words of the low ones stay in 64 bits
      auto add = [&](const ulonglong2 v, const int4 C2, bool first) {
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          const long long s = (long long)(x ? v.y : v.x);
          const int sh = dig_hi(s), sl = dig_lo(s), cl = x ? C2.z : C2.x, chh = x ? C2.w : C2.y;
          h[x] = first ? mul_wide_s(sh, chh) : mad_wide_s(sh, chh, h[x]);
          l[x] = mad_wide_s(sl, chh, first ? mul_wide_s(sh, cl) : mad_wide_s(sh, cl, l[x])) + __mulhi(sl, cl);
        }
      };
      {
        uint4 D[4];
        adv_load(D, tab, t ? F_I8 : F_I, lane);
        const unsigned long long nk = tab->nk[t ? F_I8 : F_I][g];
        ulonglong2 v[2];
        adv_line2(v, D, sm + S::RD + (l0 + g) * 8 + 2 * c, sm + S::SD + (l0 + g) * 8 + 2 * c, zs, nk);
        add(v[0], ch[0], true);
        add(v[1], ch[NQ * S::CZS / 2], false);
      }
      {
        uint4 D[4];
        adv_load(D, tab, t ? F_D8 : F_D, lane);
        add(adv_line(D, sm + S::TT + (l0 + g) * 8 + 2 * c, zs, tab->nk[t ? F_D8 : F_D][g]), ch[NQ * S::CZS], false);
      }
      if (cz < NQ) {
        const unsigned long long v0 = (h[0] << 2) + (l[0] >> 30), v1 = (h[1] << 2) + (l[1] >> 30);
        sm[S::CV + (l0 + 2 * c) * S::CS + cz] = v0;
        sm[S::CV + (l0 + 2 * c + 1) * S::CS + cz] = v1;
        vm |= (l0 + 2 * c < S::NQ2 ? dig_size(v0) : 0u) | (l0 + 2 * c + 1 < S::NQ2 ? dig_size(v1) : 0u);
      }
    }
    const int s3 = __clz(merged(vm)) - 2;   // conv fills 62 bits on its way into the passes back
    // back along t
    const unsigned long long nkb = tab->nk[F_B0][g];
    for (int it = wp; it < LQ / 8; it += W) {
      const ulonglong2 v = flip2(adv_back<S::TQ>(tab, lane, sm + S::CV + (it * 8 + g) * S::CS + 2 * c, zs, nkb, s3));
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const int ln = it * 8 + 2 * c + x, a = ln / NQ, b = ln - a * NQ;
        if (g < NP && ln < S::NQ2) sm[S::V2 + (g * NQ + a) * S::CS + b] = x ? v.y : v.x;
      }
    }
    __syncthreads();
    // back along s
    for (int it = wp; it < S::G5; it += W) {
      const ulonglong2 v = flip2(adv_back<S::TQ>(tab, lane, sm + S::V2 + (it * 8 + g) * S::CS + 2 * c, zs, nkb));
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const int ln = it * 8 + 2 * c + x, k = ln / NQ, a = ln - k * NQ;
        if (g < NP && ln < NP * NQ) sm[S::V1 + (k * 8 + g) * S::CS + a] = x ? v.y : v.x;
      }
    }
    __syncthreads();
    // back along r, to FP64
    for (int k = wp; k < NP; k += W) {
      const ulonglong2 v = adv_back<S::TQ>(tab, lane, sm + S::V1 + (k * 8 + g) * S::CS + 2 * c, zs, nkb);
      double* o = wv + (size_t)comp * nL + eb + k * NP2 + g;
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const int j = 2 * c + x;
        if (g < NP && j < NP)
          o[j * NP] = (double)(long long)(x ? v.y : v.x) *
                      __hiloint2double((ex - s3 + 1023 + tab->a[k] + tab->a[j] + tab->a[g]) << 20, 0);
      }
    }
    // the next component's maximum has a barrier before X is written again
  }
}


// Fixed-point factors of one element per block: Gq 2^-(b_a + b_b + b_c) 2^(62 - gexp), gexp the exponent of the largest row sum
// |G_d0| + |G_d1| + |G_d2|, lines (a, b) contiguous behind the t index, as (signed low word, high word).
template <int NP>
__global__ void __launch_bounds__(256)
    k_adv_factors(const double* __restrict__ Gq, const int* __restrict__ bexp, int2* __restrict__ Gx,
                  int32_t* __restrict__ gexp) {
  using S = DigAdv<NP>;
  constexpr int NQ = S::NQ, NQ2 = S::NQ2, NQ3 = NQ2 * NQ;
  __shared__ double s_m[8];
  const int e = blockIdx.x;
  const double* Ge = Gq + (size_t)e * 9 * NQ3;
  double m = 0.0;
  bool ok = true;
  for (int t = threadIdx.x; t < NQ3; t += 256) {   // t = (c NQ + b) NQ + a
    const double r = ldexp(1.0, -(bexp[t % NQ] + bexp[t / NQ % NQ] + bexp[t / NQ2]));
    for (int d = 0; d < 3; ++d) {
      const double v = (fabs(Ge[(3 * d) * NQ3 + t]) + fabs(Ge[(3 * d + 1) * NQ3 + t]) + fabs(Ge[(3 * d + 2) * NQ3 + t])) * r;
      ok = ok && isfinite(v);
      m = fmax(m, v);
    }
  }
  for (int o = 16; o; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) s_m[threadIdx.x >> 5] = m;
  ok = __syncthreads_and(ok);
  for (int t = 0; t < 8; ++t) m = fmax(m, s_m[t]);
  const int ge = ok && m > 0.0 ? ilogb(m) + 1 : 0;
  const bool take = ok && m > 0.0 && abs(ge) < 400;
  if (threadIdx.x == 0) gexp[e] = take ? ge : INT32_MIN;
  const double sc = take ? ldexp(1.0, 62 - ge) : 0.0;
  int2* Gxe = Gx + (size_t)e * 9 * NQ * S::LQ;
  for (int t = threadIdx.x; t < 9 * NQ * S::LQ; t += 256) {
    const int l = t % S::LQ, cz = t / S::LQ % NQ, dm = t / (S::LQ * NQ);
    long long v = 0;
    if (take && l < NQ2) {
      const int a = l / NQ, b = l - a * NQ;
      const double r = ldexp(1.0, -(bexp[a] + bexp[b] + bexp[cz]));
      v = __double2ll_rn(Ge[dm * NQ3 + (cz * NQ + b) * NQ + a] * r * sc);
    }
    Gxe[t] = make_int2(dig_lo(v), dig_hi(v));
  }
}

// ---- host: digit tables ------------------------------------------------------------------------------

// Unevaluated sums of two doubles (Dekker's and Knuth's error-free products and sums): the tables hold 63 bits.
struct Dd {
  double h, l;
  Dd(double a = 0, double b = 0) : h(a + b), l(b - (h - a)) {}   // |a| >= |b|
};
Dd operator+(const Dd a, const Dd b) {
  const double s = a.h + b.h, t = s - a.h;
  return Dd(s, (a.h - (s - t)) + (b.h - t) + a.l + b.l);
}
Dd operator-(const Dd a) { return Dd(-a.h, -a.l); }
Dd operator-(const Dd a, const Dd b) { return a + -b; }
Dd operator*(const Dd a, const Dd b) {
  const double p = a.h * b.h;
  return Dd(p, std::fma(a.h, b.h, -p) + a.h * b.l + a.l * b.h);
}
Dd operator/(const Dd a, const Dd b) {
  const double q = a.h / b.h;
  const Dd r = a - b * Dd(q);
  return Dd(q, r.h / b.h);
}

// P_n and P_n-1 at x
void legendre(int n, const Dd x, Dd& p, Dd& pm) {
  pm = Dd(1);
  p = x;
  for (int k = 1; k < n; ++k) {
    const Dd t = (Dd(2 * k + 1) * x * p - Dd(k) * pm) / Dd(k + 1);
    pm = p;
    p = t;
  }
}

// Gauss-Legendre nodes (ascending) by Newton's method from cos(pi (4i - 1) / (4n + 2)); GLL nodes of order N likewise from the
// level's: P_N' = N (x P_N - P_N-1) / (x^2 - 1), P_N'' from Legendre's equation.
void gauss_nodes(int n, Dd* z) {
  for (int i = 1; i <= n; ++i) {
    Dd x(std::cos(M_PI * (4.0 * i - 1.0) / (4.0 * n + 2.0))), p, pm;
    for (int it = 0; it < 8; ++it) {
      legendre(n, x, p, pm);
      x = x - p * (x * x - Dd(1)) / (Dd(n) * (x * p - pm));
    }
    z[n - i] = x;
  }
}
void gll_nodes(int N, const double* xi, Dd* x) {
  for (int i = 0; i <= N; ++i) {
    x[i] = Dd(xi[i]);
    for (int it = 0; it < 3 && i > 0 && i < N; ++it) {
      Dd p, pm;
      legendre(N, x[i], p, pm);
      const Dd d = Dd(N) * (x[i] * p - pm) / (x[i] * x[i] - Dd(1));
      x[i] = x[i] - d * (Dd(1) - x[i] * x[i]) / (Dd(2) * x[i] * d - Dd(N * (N + 1)) * p);
    }
  }
}

struct AdvMat {   // a matrix of up to 14 x 14 entries hi + lo
  int rows, cols;
  double hi[14][14], lo[14][14];
};

// Power-of-two scale 2^-s that keeps the entries up to 1 and the row sums below 2.
int scale_of(const AdvMat& M) {
  double row = 0, mx = 0;
  for (int a = 0; a < M.rows; ++a) {
    double r = 0;
    for (int b = 0; b < M.cols; ++b) {
      r += std::fabs(M.hi[a][b]);
      mx = std::fmax(mx, std::fabs(M.hi[a][b]));
    }
    row = std::fmax(row, r);
  }
  int s = 0;
  while (mx > std::ldexp(1.0, s) || row >= std::ldexp(2.0 - 0x1p-5, s)) ++s;
  return s;
}

// the eight digits of M[a][b] 2^(63 - s); zeros outside the matrix
void digits_of(const AdvMat& M, int s, int a, int b, int (&x)[8]) {
  for (int t = 0; t < 8; ++t) x[t] = 0;
  if (a >= M.rows || b >= M.cols) return;
  const double t = std::ldexp(M.hi[a][b], 63 - s);   // an entry of 1 (a Gauss node that is a GLL node): the largest value
  __int128 v = t >= 0x1p63 ? INT64_MAX : std::llrint(t) + std::llrint(std::ldexp(M.lo[a][b], 63 - s));
  for (int t = 7; t > 0; --t) {
    x[t] = (int)(((v + 128) & 255) - 128);
    v = (v - x[t]) >> 8;
  }
  x[0] = (int)v;
}

template <int NP>
int adv_dig_build_np(AdvData& A, const Level& L, cudaStream_t s) {
  using S = DigAdv<NP>;
  constexpr int NQ = S::NQ;
  // powers of two next to the quadrature weights
  double wmax = 0, rmax = 0;
  for (int q = 0; q < NQ; ++q) wmax = std::fmax(wmax, A.hwq[q]);
  for (int i = 0; i < NP; ++i) rmax = std::fmax(rmax, L.rho[i]);
  int bexp[14], aexp[14];
  for (int q = 0; q < NQ; ++q) bexp[q] = (int)std::lround(0.5 * std::log2(A.hwq[q] / wmax));
  for (int i = 0; i < NP; ++i) aexp[i] = (int)std::lround(0.5 * std::log2(L.rho[i] / rmax));
  // the cardinal polynomials of the GLL nodes and their derivatives at the Gauss nodes, to 63 bits: the FP64 forms work with matrices
  // in FP64, whose roundings make most of their error (N = 7, smooth data: 5e-15 of the result)
  AdvMat I{NQ, NP, {}, {}}, DI{NQ, NP, {}, {}}, B{NP, NQ, {}, {}};
  Dd z14[14], x14[14];
  gauss_nodes(NQ, z14);
  gll_nodes(L.N, L.xi, x14);
  for (int q = 0; q < NQ; ++q)
    for (int i = 0; i < NP; ++i) {
      Dd v(1), d(0);
      for (int c = 0; c < NP; ++c) {
        if (c == i) continue;
        const Dd den = Dd(1) / (x14[i] - x14[c]);
        d = d * (z14[q] - x14[c]) * den + v * den;   // product rule
        v = v * (z14[q] - x14[c]) * den;
      }
      I.hi[q][i] = v.h;
      I.lo[q][i] = v.l;
      B.hi[i][q] = std::ldexp(v.h, bexp[q] - aexp[i]);
      B.lo[i][q] = std::ldexp(v.l, bexp[q] - aexp[i]);
      DI.hi[q][i] = d.h;
      DI.lo[q][i] = d.l;
    }
  const int sI = scale_of(I), sD = scale_of(DI), sB = scale_of(B);
  std::vector<AdvDigTab> tabs(1);
  AdvDigTab& T = tabs[0];
  struct Row {
    const AdvMat* M;
    int s, r;
  };
  bool exact = true;
  // fragment of eight rows on the eight points from column c0 on, and the constants of an all-zero line
  auto tile = [&](int f, auto row, int c0, bool first, bool last, int64_t (&z)[8][8]) {
    for (int m = 0; m < 4; ++m)
      for (int lane = 0; lane < 32; ++lane) {
        const int g = lane >> 2, c = lane & 3;
        const Row r = row(g);
        auto pair = [&](int in, int d) -> uint32_t {
          int x[8];
          digits_of(*r.M, r.s, r.r, c0 + in, x);
          return (uint32_t)(d < 0 ? 0 : half_of(x[d])) | ((uint32_t)half_of(x[d + 1]) << 16);
        };
        T.frag[f][m][lane] = make_uint4(pair(2 * c, 2 * m), pair(2 * c, 2 * m - 1), pair(2 * c + 1, 2 * m),
                                        pair(2 * c + 1, 2 * m - 1));
      }
    for (int g = 0; g < 8; ++g) {
      if (first)
        for (int d = 0; d < 8; ++d) z[g][d] = 0;
      const Row r = row(g);
      int64_t sum = 0;
      for (int b = 0; b < r.M->cols; ++b) {
        int x[8];
        digits_of(*r.M, r.s, r.r, b, x);
        for (int d = 0; d < 8; ++d) {
          if (b >= c0 && b < c0 + 8) z[g][d] += x[d];
          sum += std::abs(x[d]);
        }
      }
      if (255 * sum >= (1 << 21)) exact = false;
      if (last) T.nk[f][g] = 0ull - dig_merge_zero(z[g], ADV_SH);
    }
  };
  int64_t z[8][8];
  tile(F_I, [&](int g) { return Row{&I, sI, g}; }, 0, true, true, z);
  tile(F_D, [&](int g) { return Row{&DI, sD, g}; }, 0, true, true, z);
  tile(F_ID, [&](int g) { return g < 4 ? Row{&I, sI, 8 + g} : Row{&DI, sD, 4 + g}; }, 0, true, true, z);
  tile(F_I8, [&](int g) { return Row{&I, sI, 8 + g}; }, 0, true, true, z);
  tile(F_D8, [&](int g) { return Row{&DI, sD, 8 + g}; }, 0, true, true, z);
  tile(F_B1, [&](int g) { return Row{&B, sB, g}; }, 8, true, true, z);
  tile(F_B0, [&](int g) { return Row{&B, sB, g}; }, 0, S::TQ == 1, true, z);
  for (int i = 0; i < 8; ++i) T.a[i] = i < NP ? aexp[i] : 0;
  if (!exact) return SEM_OK;
  const size_t ng = (size_t)L.E * 9 * NQ * S::LQ;
  int2* gx = nullptr;
  int32_t* ge = nullptr;
  AdvDigTab* dt = nullptr;
  int* be = nullptr;
  // without the memory the FP64 (or FP32-pair) form runs
  if (cudaMalloc((void**)&gx, ng * sizeof(int2)) != cudaSuccess ||
      cudaMalloc((void**)&ge, (size_t)L.E * sizeof(int32_t)) != cudaSuccess ||
      cudaMalloc((void**)&dt, sizeof(AdvDigTab)) != cudaSuccess || cudaMalloc((void**)&be, sizeof(bexp)) != cudaSuccess) {
    cudaGetLastError();
    for (void* p : {(void*)gx, (void*)ge, (void*)dt})
      if (p) cudaFree(p);
    return SEM_OK;
  }
  cudaError_t err = cudaMemcpyAsync(dt, &T, sizeof(AdvDigTab), cudaMemcpyHostToDevice, s);
  if (err == cudaSuccess) err = cudaMemcpyAsync(be, bexp, sizeof(bexp), cudaMemcpyHostToDevice, s);
  if (err == cudaSuccess) {
    k_adv_factors<NP><<<L.E, 256, 0, s>>>(A.Gq, be, gx, ge);
    err = cudaGetLastError();
  }
  if (err == cudaSuccess) err = cudaStreamSynchronize(s);
  cudaFree(be);
  if (err != cudaSuccess) {
    for (void* p : {(void*)gx, (void*)ge, (void*)dt}) cudaFree(p);
    set_detail("advection digit factors: %s", cudaGetErrorString(err));
    return SEM_ECUDA;
  }
  A.Gqx = gx;
  A.gqexp = ge;
  A.dig = dt;
  A.dig_ebase = -59 + (1 + sD) + 5 * (1 + sI) + 3 * (1 + sB);
  return SEM_OK;
}

}  // namespace

// The digit tables and fixed-point factors (first FP64 or FP32-pair evaluation; synchronous), where the kernel is compiled.
int advect_dig_build(AdvData& A, const Level& L, cudaStream_t s) {
  if (A.dig_tried) return SEM_OK;
  A.dig_tried = true;
  switch (L.NP) {
    case 5: return adv_dig_build_np<5>(A, L, s);
    case 6: return adv_dig_build_np<6>(A, L, s);
    case 7: return adv_dig_build_np<7>(A, L, s);
    case 8: return adv_dig_build_np<8>(A, L, s);
    default: return SEM_OK;
  }
}

int advect_dig_apply(const Level& L, const AdvData& A, const double* c, const double* u, double* w, int ncomp,
                     bool pairs, cudaStream_t s) {
  const int loss = pairs ? ADV_LOSS_PAIRS : ADV_LOSS;
  switch (L.NP) {
#define CASE(NP)                                                                                                      \
  case NP: {                                                                                                          \
    using S = DigAdv<NP>;                                                                                             \
    constexpr size_t smem = std::max(S::SMEM, advect_smem<AdvPlain<double>, NP>());                                   \
    static PerDevice<bool> attr;                                                                                      \
    SEM_TRY(smem_attr_once(attr, (const void*)k_advect_dig<NP>, smem));                                               \
    k_advect_dig<NP><<<L.E, S::T, smem, s>>>(ncomp, L.nL, c, u, A.Gqx, A.gqexp, A.dig, A.dig_ebase, loss, w, A.Gq,     \
                                             A.Im, A.Dq, adv_ops<AdvPlain<double>, NP>(A));                           \
    SEM_LAUNCH_CHECK();                                                                                               \
    return SEM_OK;                                                                                                    \
  }
    CASE(5) CASE(6) CASE(7) CASE(8)
#undef CASE
  }
  set_detail("order %d not compiled", L.N);
  return SEM_EINVAL;
}

}  // namespace sem
