// FP64 element operator in integer digits (dig.cuh, ax_dig.cu) for 8 <= N <= 11, with even-odd lines.
//
// What bounds it: the FP64 form (ax_eo.cu) issues an FP64 instruction every 16 cycles: 2,368 us at 26^3, N = 9, against 187 us
// for its bytes. Here it is instruction issue and the mma.sync chains (ncu, 16^3, N = 9: issue 56 %, tensor pipe 30 %, 758 warp
// instructions for 32 points; 917 with one loop over all groups and 8-byte stores). Element kernel, about 16 million points, FP64 form ->
// this: N = 8 1841 -> 675 us, N = 9 2368 -> 603, N = 10 1872 -> 654, N = 11 2460 -> 491. (The FP32-pair kernel: 458, 634, 495, 682.)
// Error against 128-bit arithmetic, 2-norm, 4x3x4 warped elements: random u 0.57e-16 to 0.7e-16 (FP64 form 1.4e-16 to 1.65e-16); linear,
// quadratic and smooth u 0.54e-15 (N = 8) to 5.3e-15 (N = 11) (FP64 form 2.9e-15 to 1.8e-14).
//
// A line of NP = 9..12 points is two contractions of at most six: the sums v[b] + v[N-b] with the even part of the matrix, the
// differences with the odd part. Each fits an mma's eight points and eight outputs, where the lines as they are would take
// four mma of half-empty tiles. A group of eight lines is a warp's task (dig_sums, lines as columns): lane (g, c) reads the
// points 2c, 2c+1 and N-2c, N-2c-1 of line g and gets outputs g and N-g of lines 2c and 2c+1.
// One element per block; its fields stay in shared memory as 64-bit integers: u, then three derivatives, which become fluxes
// point by point and are transformed in place (a line belongs to one warp). Values have one bit less than in
// ax_dig.cu, for the sums; fluxes are shifted up to the element's largest, which takes random u from up to 3.9e-16 (N = 10) to the
// figures above. Exponents, factors, the weights 2^a and the elements that go to the FP64 form are as there.
#include <cmath>
#include <cstddef>
#include <vector>

#include "ax_dig.cuh"
#include "sem_internal.cuh"

namespace sem {

// One order's matrices in digits: stage 0 by D, stage 1 by 2^-a D^T 2^a; parity 0 even, 1 odd.
struct DigEoTab {
  uint4 frag[2][2][4][32];
  unsigned long long nk[2][2][8];
  int32_t a[12];
};

namespace {

template <int NP>
struct DigEoShape {
  static constexpr int NW = NP == 12 ? 6 : 4;              // warps: 3 LG tasks go into them with little rest
  static constexpr int T = 32 * NW;
  static constexpr int LG = (NP * NP + 7) / 8;             // groups of eight lines a direction
  static constexpr int NPE = (NP + 1) / 2 * 2;             // i extent of the stored factors
  static constexpr int GE = NP * NP * NPE;
  static constexpr int RS = NP <= 10 ? 10 : 14;            // row and plane strides: 2 mod 4, so that lanes of a t- or s-line
  static constexpr int PS = (NP * RS + 1) / 4 * 4 + 2;     // group read distinct banks
  static constexpr int FLD = PS * NP;
  static constexpr int EO = 3 * Pad3<NP>::ES;              // of the FP64 form
  static constexpr size_t SMEM = 8 * (size_t)(4 * FLD > EO ? 4 * FLD : EO);
};

// Blocks an SM, as many as the fields let in: the warps wait on mma.sync chains (each before the room for mirror sums, which costs
// two microseconds at any: N = 9, 26^3: 648, 617, 600 us at four, five, six; N = 11, 21^3: 535 at two, 490 at three; N = 10, 23^3: 775 at
// three, 652 at four).
template <int NP>
constexpr int dig_eo_min_blocks() {
  return NP == 12 ? 3 : NP == 11 ? 4 : 6;
}

// The lines of direction DIR (0: i, 1: j, 2: k), group by group: src and dst may be the same field. g0: this warp's first group.
// Bounds: u comes below 2^62 (1 - 2^-7) (half of what the exponent eu leaves), a flux shifted by sh below 2^62 / (1 + 2^-6), so the
// sums s and d that dig_flip takes are below 2^63 (1 - 2^-7) and 2^63 / (1 + 2^-6). ev and od together stay below 2^60 (derivatives)
// and 2^62 / 3 (each direction of the result) by the scales of the matrices.
template <int NP, int SH, int DIR>
__device__ __forceinline__ uint32_t dig_eo_lines(const unsigned long long* src, unsigned long long* dst, const int g0,
                                                 const uint4 (&De)[4], const uint4 (&Do)[4], const unsigned long long nke,
                                                 const unsigned long long nko, const int sh, const DigStart& z) {
  using S = DigEoShape<NP>;
  constexpr int H = NP / 2, N = NP - 1, NP2 = NP * NP;
  constexpr int sa = DIR == 0 ? S::RS : 1, sb = DIR == 2 ? S::RS : S::PS, st = DIR == 0 ? 1 : DIR == 1 ? S::RS : S::PS;
  const int lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;
  auto at = [&](int l) { return (l / NP) * sb + (l % NP) * sa; };
  uint32_t vm = 0;
#pragma unroll 1
  for (int gi = g0; gi < S::LG; gi += S::NW) {
    const int lg = 8 * gi + g, lo = 8 * gi + 2 * c;
    const bool on = lg < NP2;
    const int base = at(lg);
    unsigned long long s[2] = {0, 0}, d[2] = {0, 0};
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      const int b = 2 * c + x;
      if (on && b < H) {
        const unsigned long long p = src[base + b * st], q = src[base + (N - b) * st];
        s[x] = (p + q) << sh;
        d[x] = (p - q) << sh;
      } else if (NP % 2 == 1 && on && b == H) {
        s[x] = src[base + H * st] << sh;
      }
    }
    unsigned long long ev[2], od[2];
    float f[4][4];
    {
      const DigPack b[2] = {DigPack(dig_flip((long long)s[0])), DigPack(dig_flip((long long)s[1]))};
      dig_sums<true>(f, De, b, z);
      ev[0] = dig_merge4<SH>(f, 0, nke);
      ev[1] = dig_merge4<SH>(f, 1, nke);
    }
    {
      const DigPack b[2] = {DigPack(dig_flip((long long)d[0])), DigPack(dig_flip((long long)d[1]))};
      dig_sums<true>(f, Do, b, z);
      od[0] = dig_merge4<SH>(f, 0, nko);
      od[1] = dig_merge4<SH>(f, 1, nko);
    }
    __syncwarp();   // the group's lines are read
    const int out = at(lo);
    if (NP % 2 == 0 && DIR > 0) {   // two lines side by side: 16-byte words
      if (lo < NP2 && g < H) {
        const ulonglong2 a = make_ulonglong2(od[0] + ev[0], od[1] + ev[1]), b = make_ulonglong2(od[0] - ev[0], od[1] - ev[1]);
        *reinterpret_cast<ulonglong2*>(&dst[out + g * st]) = a;
        *reinterpret_cast<ulonglong2*>(&dst[out + (N - g) * st]) = b;
        if (SH == DIG_SH1) vm |= dig_size(a.x) | dig_size(a.y) | dig_size(b.x) | dig_size(b.y);
      }
    } else {
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const int o = x == 0 ? out : NP % 2 == 0 ? out + sa : at(lo + 1);
        const unsigned long long a = od[x] + ev[x], b = od[x] - ev[x];
        if (lo + x < NP2 && g < H) {
          dst[o + g * st] = a;
          dst[o + (N - g) * st] = b;
          if (SH == DIG_SH1) vm |= dig_size(a) | dig_size(b);
        } else if (NP % 2 == 1 && lo + x < NP2 && g == H) {
          dst[o + H * st] = od[x];
          if (SH == DIG_SH1) vm |= dig_size(od[x]);
        }
      }
    }
  }
  return vm;
}

// All lines of the three directions: from U into the fields F + d FLD (ST = 0), or each field in place. The groups of the
// three directions are dealt out to the warps in one round.
template <int NP, int ST>
__device__ __forceinline__ uint32_t dig_eo_pass(const unsigned long long* U, unsigned long long* F,
                                                const DigEoTab* __restrict__ tab, const int sh, const DigStart& z) {
  using S = DigEoShape<NP>;
  constexpr int SH = ST ? DIG_SH2 : DIG_SH1;
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, g = lane >> 2;
  uint4 De[4], Do[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    De[m] = tab->frag[ST][0][m][lane];
    Do[m] = tab->frag[ST][1][m][lane];
  }
  const unsigned long long nke = tab->nk[ST][0][g], nko = tab->nk[ST][1][g];
  constexpr int R1 = (S::NW - S::LG % S::NW) % S::NW, R2 = (S::NW - 2 * S::LG % S::NW) % S::NW;
  const int g1 = (wp + R1) % S::NW, g2 = (wp + R2) % S::NW;
  uint32_t vm = dig_eo_lines<NP, SH, 0>(ST ? F : U, F, wp, De, Do, nke, nko, sh, z);
  vm |= dig_eo_lines<NP, SH, 1>(ST ? F + S::FLD : U, F + S::FLD, g1, De, Do, nke, nko, sh, z);
  vm |= dig_eo_lines<NP, SH, 2>(ST ? F + 2 * S::FLD : U, F + 2 * S::FLD, g2, De, Do, nke, nko, sh, z);
  return vm;
}

template <int NP, bool VARH1>
__global__ void __launch_bounds__(DigEoShape<NP>::T, dig_eo_min_blocks<NP>())
    k_ax_dig_eo(const double* __restrict__ u, double* __restrict__ w, const int2* __restrict__ Gx,
                const int32_t* __restrict__ gexp, const double* __restrict__ G, const DigEoTab* __restrict__ tab,
                const int kexp, const double h1, const double h2, const double* __restrict__ h1L, const int span,
                const double* skip, const int mass, const int e1, const __grid_constant__ EOMat<ArF64> Df,
                const __grid_constant__ EOMat<ArF64> Dt) {
  using S = DigEoShape<NP>;
  constexpr int NP2 = NP * NP, NP3 = NP2 * NP;
  if (skip && *skip != 0.0) return;
  extern __shared__ __align__(16) unsigned long long dig_eo_smem[];
  __shared__ uint32_t s_max[4][S::NW];
  unsigned long long *U = dig_eo_smem, *F = dig_eo_smem + S::FLD;
  const int e = blockIdx.x, lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const double* ue = u + (size_t)e * NP3;
  const double* he = VARH1 ? h1L + (size_t)e * NP3 : nullptr;
  const int2* Ge = Gx + (size_t)e * 6 * S::GE;
  auto at = [&](int p) { return (p / NP2) * S::PS + (p / NP % NP) * S::RS + p % NP; };
  if (threadIdx.x == 0)
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(Ge), "r"(6 * S::GE * 8) : "memory");
  // the element's exponents
  constexpr int PT = (NP3 + S::T - 1) / S::T;
  uint32_t um = 0, hm = 0, hl = 0;
  double uv[PT];
#pragma unroll
  for (int q = 0; q < PT; ++q) {
    const int p = threadIdx.x + q * S::T;
    uv[q] = p < NP3 ? ue[p] : 0.0;
  }
#pragma unroll
  for (int q = 0; q < PT; ++q) um = max(um, (uint32_t)__double2hiint(uv[q]) & 0x7fffffffu);
  if (VARH1)
    for (int p = threadIdx.x; p < NP3; p += S::T) {
      const double h = he[p];
      hm = max(hm, (uint32_t)__double2hiint(h) & 0x7fffffffu);
      hl = max(hl, dig_h1_low(h));
    }
  const int ge = gexp[e];
  um = __reduce_max_sync(0xffffffffu, um);
  if (VARH1) {
    hm = __reduce_max_sync(0xffffffffu, hm);
    hl = __reduce_max_sync(0xffffffffu, hl);
  }
  if (lane == 0) {
    s_max[0][wp] = um;
    s_max[1][wp] = hm;
    s_max[3][wp] = hl;
  }
  __syncthreads();
#pragma unroll
  for (int t = 0; t < S::NW; ++t) {
    um = max(um, s_max[0][t]);
    if (VARH1) {
      hm = max(hm, s_max[1][t]);
      hl = max(hl, s_max[3][t]);
    }
  }
  const int eu = (int)((um + 0x4000) >> 20);
  const int eh = VARH1 ? (hm ? (int)(hm >> 20) - 1022 : 0) : 0;   // |h1| < 2^eh
  const int ex = ge + eh + eu - 1023 - kexp - DIG_SH2 - 12 + 2;   // values and fluxes carry half
  if (um >= 0x7ff00000u || hm >= 0x7ff00000u || ge == DIG_BAD || abs(ex) > 800 || abs(ex + e1) > 800 ||
      abs(eh) > 800 || abs(eu - 1023) > 800 || (VARH1 && dig_h1_wide(hm, hl, span))) {
    const bool nil = um == 0 && hm < 0x7ff00000u && ge != DIG_BAD && e1 < 4096;
    dig_fallback<NP, VARH1>(reinterpret_cast<double*>(dig_eo_smem), e, u, w, G, Df, Dt, h1, h2, h1L, nil);
    return;
  }
#pragma unroll
  for (int q = 0; q < PT; ++q) {
    const int p = threadIdx.x + q * S::T;
    if (p < NP3) U[at(p)] = (unsigned long long)(dig_fix(uv[q], eu) >> 1);
  }
  __syncthreads();

  // derivatives
  const DigStart zs;
  uint32_t vm = __reduce_or_sync(0xffffffffu, dig_eo_pass<NP, 0>(U, F, tab, 0, zs));
  if (lane == 0) s_max[2][wp] = vm;
  __syncthreads();
#pragma unroll
  for (int t = 0; t < S::NW; ++t) vm |= s_max[2][t];
  const int sv = __clz(vm) - 3;   // the largest derivative below 2^61

  // fluxes
  uint32_t fm = 0;
#pragma unroll 2
  for (int p = threadIdx.x; p < NP3; p += S::T) {
    const int i = at(p), pg = NP % 2 == 0 ? p : p / NP * S::NPE + p % NP;
    int2 G6[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) G6[q] = Ge[q * S::GE + pg];
    int ah[3], al[3];
    int Hh = 0, Hl = 0;
    if (VARH1) {
      const long long h = dig_fix(he[p], eh + 1022) >> 2;   // below 2^61
      Hh = dig_hi(h);
      Hl = dig_lo(h);
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      long long v = (long long)(F[d * S::FLD + i] << sv);
      if (VARH1) {
        const int vh = dig_hi(v), vl = dig_lo(v);
        v = (mul_wide_s(vh, Hh) << 3) + (mad_wide_s(vl, Hh, mul_wide_s(vh, Hl)) >> 29);
      }
      ah[d] = dig_hi(v);
      al[d] = dig_lo(v);
    }
    auto flux = [&](int q0, int q1, int q2) {
      const long long hh =
          mad_wide_s(ah[2], G6[q2].y, mad_wide_s(ah[1], G6[q1].y, mul_wide_s(ah[0], G6[q0].y)));
      const long long m = mad_wide_s(
          al[2], G6[q2].y,
          mad_wide_s(ah[2], G6[q2].x,
                     mad_wide_s(al[1], G6[q1].y,
                                mad_wide_s(ah[1], G6[q1].x, mad_wide_s(al[0], G6[q0].y, mul_wide_s(ah[0], G6[q0].x))))));
      return (unsigned long long)((hh << 3) + (m >> 29));
    };
    const unsigned long long f0 = flux(0, 1, 2), f1 = flux(1, 3, 4), f2 = flux(2, 4, 5);
    F[i] = f0;
    F[S::FLD + i] = f1;
    F[2 * S::FLD + i] = f2;
    fm = max(max(fm, dig_size(f0)), max(dig_size(f1), dig_size(f2)));
  }
  fm = __reduce_max_sync(0xffffffffu, fm);
  if (lane == 0) s_max[0][wp] = fm;
  __syncthreads();
#pragma unroll
  for (int t = 0; t < S::NW; ++t) fm = max(fm, s_max[0][t]);
  // |flux| < (fm + 1) 2^32, and fm + fm / 64 + 1 below 2^(30 - sf) makes (fm + 1) (1 + 2^-6) at most 2^(30 - sf): shifted by sf, a
  // flux stays below 2^62 / (1 + 2^-6), and the sum or difference of two mirror points (dig_eo_lines), 0.9847 2^63 at most, within
  // dig_flip's bound. Mirror fluxes are equal wherever u is linear, so that the sums do come this close. Unshifted (sf = 0) a flux
  // is below 2^62 / (1 + 2^-5) by the exponent of the factors.
  const int sf = max(__clz(fm + (fm >> 6) + 1) - 2, 0);
  dig_eo_pass<NP, 1>(U, F, tab, sf, zs);
  __syncthreads();

  // w = h1 2^(ex + a_i + a_j + a_k) W + h2 B u
  const int hs = VARH1 ? 0x3ff00000 : __double2hiint(h1), ls = VARH1 ? 0 : __double2loint(h1);
  const double* Be = G + ((size_t)e * 7 + 6) * NP3;
#pragma unroll
  for (int q = 0; q < PT; ++q) {
    const int p = threadIdx.x + q * S::T;
    if (p >= NP3) break;
    const int i = at(p);
    const unsigned long long W = F[i] + F[S::FLD + i] + F[2 * S::FLD + i];
    const int sp = ex - sv - sf + tab->a[p / NP2] + tab->a[p / NP % NP] + tab->a[p % NP];
    double o = (double)(long long)W * __hiloint2double(hs + (hs << 1 == 0 ? 0 : sp << 20), ls);
    if (mass) o = fma(h2 * Be[p], ue[p], o);
    w[(size_t)e * NP3 + p] = o;
  }
}

using i128 = __int128;

}  // namespace

// The digit tables of an order on the device (scales and exponents: dig_scales); *tab null where it has none, or no memory.
int dig_eo_tables(const Level& L, const int* a, int k, int m2, int q2, DigEoTab** tab, cudaStream_t s) {
  const int NP = L.NP, H = NP / 2, N = NP - 1;
  *tab = nullptr;
  std::vector<DigEoTab> tv(1);
  DigEoTab& T = tv[0];
  int dg[8][8][8];
  for (int st = 0; st < 2; ++st)
    for (int par = 0; par < 2; ++par) {
      const int rows = H + (par == 1 ? NP % 2 : 0), cols = H + (par == 0 ? NP % 2 : 0);
      for (int r = 0; r < 8; ++r)
        for (int c = 0; c < 8; ++c) {
          i128 v = 0;
          if (r < rows && c < cols) {
            auto entry = [&](int i, int j) -> i128 {
              const double d = st ? std::ldexp(L.D.a[j * NP + i], a[j] - a[i]) : L.D.a[i * NP + j];
              return st ? dig_scaled(d, m2, 1, 63 + q2 - 8) : dig_scaled(d, 1, m2, 63 + k - (q2 - 8));
            };
            if (c == H) {
              v = entry(r, H);
            } else {
              v = par ? entry(r, c) - entry(r, N - c) : entry(r, c) + entry(r, N - c);
              v = (v + (v >= 0 ? 1 : 0)) >> 1;   // half, rounded
            }
          }
          for (int t = 7; t > 0; --t) {
            const int x = (int)(((v + 128) & 255) - 128);
            dg[r][c][t] = x;
            v = (v - x) >> 8;
          }
          dg[r][c][0] = (int)v;
          if (v < -128 || v > 128) return SEM_OK;
        }
      for (int r = 0; r < 8; ++r) {
        int64_t z[8] = {}, sum = 0;
        for (int t = 0; t < 8; ++t)
          for (int c = 0; c < 8; ++c) {
            z[t] += dg[r][c][t];
            sum += std::abs(dg[r][c][t]);
          }
        if (255 * sum >= (1 << 21)) return SEM_OK;   // a digit sum stays exact and below 2^21 for every u
        T.nk[st][par][r] = 0ull - dig_merge_zero(z, st ? DIG_SH2 : DIG_SH1);
      }
      for (int m = 0; m < 4; ++m)
        for (int lane = 0; lane < 32; ++lane) {
          const int g = lane >> 2, c = lane & 3;
          auto pair = [&](int in, int d) -> uint32_t {   // digits d (low half), d + 1 (high half) of entry (g, in)
            const int* x = dg[g][in];
            return (uint32_t)(d < 0 ? 0 : half_of(x[d])) | ((uint32_t)half_of(x[d + 1]) << 16);
          };
          T.frag[st][par][m][lane] =
              make_uint4(pair(2 * c, 2 * m), pair(2 * c, 2 * m - 1), pair(2 * c + 1, 2 * m), pair(2 * c + 1, 2 * m - 1));
        }
    }
  for (int i = 0; i < 12; ++i) T.a[i] = i < NP ? a[i] : 0;
  DigEoTab* dt = nullptr;
  if (cudaMalloc((void**)&dt, sizeof(DigEoTab)) != cudaSuccess) {
    cudaGetLastError();
    return SEM_OK;
  }
  *tab = dt;
  SEM_CUDA_TRY(cudaMemcpyAsync(dt, &T, sizeof(DigEoTab), cudaMemcpyHostToDevice, s));
  SEM_CUDA_TRY(cudaStreamSynchronize(s));   // T goes out of scope
  return SEM_OK;
}

const int32_t* dig_eo_exponents(const DigEoTab* tab) {
  return reinterpret_cast<const int32_t*>(reinterpret_cast<const char*>(tab) + offsetof(DigEoTab, a));
}

// Elements [e0, e0 + E) of the level; u, w, h1L already at e0.
int ax_dig_eo_apply(const Level& L, int e0, int E, const double* u, double* w, double h1, double h2, const double* h1L,
                    int span, const double* skip, const EOMat<ArF64>& Df, const EOMat<ArF64>& Dt, cudaStream_t s) {
  const size_t off = (size_t)e0 * L.NP * L.NP * L.NP;
  const int mass = h2 != 0.0 ? 1 : 0, e1 = dig_h1_exp(h1);
  switch (L.NP) {
#define CASE(NP)                                                                                                       \
  case NP: {                                                                                                           \
    using S = DigEoShape<NP>;                                                                                          \
    const int2* Gx = L.Gx + (size_t)e0 * 6 * S::GE;                                                                    \
    if (h1L) {                                                                                                         \
      SEM_CUDA_TRY(cudaFuncSetAttribute(k_ax_dig_eo<NP, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,            \
                                        (int)S::SMEM));                                                                \
      k_ax_dig_eo<NP, true><<<E, S::T, S::SMEM, s>>>(u, w, Gx, L.gexp + e0, L.G + 7 * off, L.dig_eo, L.dig_kexp, 1.0,  \
                                                     h2, h1L, span, skip, mass, 0, Df, Dt);                            \
    } else {                                                                                                           \
      SEM_CUDA_TRY(cudaFuncSetAttribute(k_ax_dig_eo<NP, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,           \
                                        (int)S::SMEM));                                                                \
      k_ax_dig_eo<NP, false><<<E, S::T, S::SMEM, s>>>(u, w, Gx, L.gexp + e0, L.G + 7 * off, L.dig_eo, L.dig_kexp, h1,  \
                                                      h2, nullptr, 0, skip, mass, e1, Df, Dt);                         \
    }                                                                                                                  \
    SEM_LAUNCH_CHECK();                                                                                                \
    return SEM_OK;                                                                                                     \
  }
    CASE(9) CASE(10) CASE(11) CASE(12)
#undef CASE
  }
  set_detail("order %d not compiled", L.N);
  return SEM_EINVAL;
}

}  // namespace sem
