// FP64 element operator A^e = D^T h1 G D + h2 B (eq. Ae) with the contractions in integer
// digits on the tensor cores (dig.cuh), for 4 <= N <= 7.
//
// What bounds it: the FP64 form (ax_eo.cu) issues about 50 FP64 instructions a point at 16 cycles a warp and SM each, eight
// times the time of its bytes. Here 32 points cost 30 mma.sync (2.3 cycles each), 27 IMAD.WIDE (1.3, and not beside an
// mma.sync), about 280 other 32-bit instructions and four FP64 ones (16): 184 cycles at 24 warps an SM, of which
// the tensor and wide-multiply pipes need 110 and the bytes 107. Element kernel at 32^3, N = 7: 1576 -> 309 us (3.9 TB/s); 43^3,
// N = 5: 1444 -> 608 us (padded to 64 lines of 8 points); the FP32-pair kernel takes 366 and 353 us there.
//
// One element per block, one warp per two planes k = 2w, 2w+1; lane (g, c) holds the points
// (i, j) = (2c, g), (2c+1, g) of both planes all the way, the layout of an mma's rows and results:
// * r-lines (i): the lane's own digits are the mma's A fragment, no exchange at all;
// * s-lines (j) and t-lines (k): the values go through shared memory and are cut into digits by their readers (a value has
//   8 bytes, its digits 16), at positions that keep rows, columns and planes free of bank conflicts; the t-direction's
//   results come back through shared memory as 64-bit integers;
// * fluxes F = G (D u): 64 x 64-bit products by IMAD.WIDE (the low x low parts are dropped) on factors that are stored as
//   62-bit fixed-point numbers with one exponent per element, the same 8 bytes a value as FP64.
// The element's exponent comes from its largest |u| (block maximum), and the derivatives are shifted to 61 bits by
// their largest, so that the result does not depend on the scale of u.
//
// The GLL weights make G, and the result, a hundred times smaller at an element's edges and corners than inside. So G is stored
// over 2^(a_i + a_j + a_k), 2^a_i near rho_i^(3/4) (a power of two: no rounding), the second contraction uses
// 2^-a D^T 2^a, and the result gets 2^(a_i + a_j + a_k) back in the exponent of its scale: edges and corners then keep the
// relative error of the interior (2-norm error against 128-bit arithmetic, N = 4 and 7: random u 0.5e-16 and 0.6e-16 of the result,
// 1.3e-16 and 1.4e-16 for the FP64 form; linear, quadratic and smooth u 0.6e-16 to 2.6e-16, FP64 form 0.9e-15 to 8.5e-15).
//
// Elements that fixed point cannot hold (an Inf or NaN in u, h1 or G, exponents near the ends of the FP64 range, or a nodal h1
// that spans more than 2^8) are computed by the even-odd FP64 code in the same block. The look at h1's span costs a nodal call 0.4 to
// 0.8 % (N = 7, 32^3: 348 -> 351 us; N = 9, 26^3: 680 -> 683).
#include <cmath>
#include <cstddef>
#include <vector>

#include "ax_dig.cuh"

namespace sem {

int dig_eo_tables(const Level& L, const int* a, int k, int m2, int q2, DigEoTab** tab, cudaStream_t s);
const int32_t* dig_eo_exponents(const DigEoTab* tab);
int ax_dig_eo_apply(const Level& L, int e0, int E, const double* u, double* w, double h1, double h2, const double* h1L, int span,
                    const double* skip, const EOMat<ArF64>& Df, const EOMat<ArF64>& Dt, cudaStream_t s);

namespace {

// Blocks an SM. The warps wait on mma.sync chains and on each other, so more of them pay for a few spilled registers
// (N = 7, 32^3, with the kernel at 306 us: 327 us at five blocks, 306 at six (80 registers), 316 at seven; N = 5, 43^3: 648, 643, 617, 615 at 5..8).
template <int NP>
constexpr int dig_min_blocks() {
  return NP <= 6 ? 7 : 6;
}

template <int NP, bool VARH1>
__global__ void __launch_bounds__(DigShape<NP>::T, dig_min_blocks<NP>())
    k_ax_dig(const double* __restrict__ u, double* __restrict__ w, const int2* __restrict__ Gx,
             const int32_t* __restrict__ gexp, const double* __restrict__ G, const DigTab* __restrict__ tab,
             const int kexp, const double h1, const double h2,
             const double* __restrict__ h1L, const int span, const double* skip, const int vec, const int mass, const int e1,
             const __grid_constant__ EOMat<ArF64> Df, const __grid_constant__ EOMat<ArF64> Dt) {
  if (skip && *skip != 0.0) return;
  __shared__ __align__(16) unsigned long long smem[DigShape<NP>::SMEM];
  __shared__ uint32_t s_max[4][4];
  double uv[2][2], o[2][2];
  dig_element<NP, VARH1, false>(blockIdx.x, u, w, Gx, gexp, G, tab, kexp, h1, h2, h1L, span, vec, mass, e1, Df, Dt, smem,
                                s_max, uv, o);
}

// Fixed-point factors of one element per block: G 2^-(a_i + a_j + a_k) 2^(62 - gexp), gexp the exponent of the largest
// row sum |G_m1| + |G_m2| + |G_m3| of its points, as (signed low word, high word).
template <int NP>
__global__ void __launch_bounds__(128)
    k_dig_factors(const double* __restrict__ G, const int32_t* __restrict__ a, int2* __restrict__ Gx,
                  int32_t* __restrict__ gexp) {
  using S = DigShape<NP>;
  constexpr int NP3 = NP * NP * NP;
  __shared__ double s_m[4];
  const int e = blockIdx.x;
  const double* Ge = G + (size_t)e * 7 * NP3;
  auto weight = [&](int i, int kj) { return ldexp(1.0, -(a[i] + a[kj % NP] + a[kj / NP])); };
  double m = 0.0;
  bool ok = true;
  for (int t = threadIdx.x; t < NP3; t += 128) {
    double v[6];
    const double r = weight(t % NP, t / NP);
    for (int q = 0; q < 6; ++q) v[q] = fabs(Ge[q * NP3 + t]) * r;
    const double r0 = v[0] + v[1] + v[2], r1 = v[1] + v[3] + v[4], r2 = v[2] + v[4] + v[5];
    ok = ok && isfinite(r0) && isfinite(r1) && isfinite(r2);
    m = fmax(m, fmax(r0, fmax(r1, r2)));
  }
  for (int o = 16; o; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) s_m[threadIdx.x >> 5] = m;
  ok = __syncthreads_and(ok);
  m = fmax(fmax(s_m[0], s_m[1]), fmax(s_m[2], s_m[3]));
  const int ge = ok && m > 0.0 ? ilogb(m * (1.0 + 0x1p-5)) + 1 : DIG_BAD;   // the fluxes stay below 2^63 (1 - 2^-7)
  const bool take = ge != DIG_BAD && abs(ge) < 400;
  if (threadIdx.x == 0) gexp[e] = take ? ge : DIG_BAD;
  const double sc = take ? ldexp(1.0, 62 - ge) : 0.0;
  int2* Gxe = Gx + (size_t)e * 6 * S::GE;
  for (int t = threadIdx.x; t < 6 * S::GE; t += 128) {
    const int q = t / S::GE, kj = (t % S::GE) / S::NPE, i = t % S::NPE;
    const long long v = take && i < NP ? __double2ll_rn(Ge[q * NP3 + kj * NP + i] * weight(i, kj) * sc) : 0;
    Gxe[t] = make_int2(dig_lo(v), dig_hi(v));
  }
}

// ---- host: the digit tables of an order ----------------------------------------------------------

struct DigHost {
  int dg[2][12][12][8];   // digits of the scaled matrices [stage][out][in]
  int kexp;               // c1 c2 = 2^kexp
  int a[12];              // 2^a next to the GLL weights^(3/4)
};

// D scaled by c1 = 2^k / c2 and 2^-a D^T 2^a by c2: every entry below 1 (eight digits), a line's derivative below 2 max|u|
// (61 bits after the merge), the sum of the three directions within 64 bits; c2 = m2 2^(q2 - 8) has eight significant
// bits, so that the divisions are exact in 128-bit integers.
double dig_entry(const double* Dm, int NP, const int* A, int st, int a, int b) {
  return st ? std::ldexp(Dm[b * NP + a], A[b] - A[a]) : Dm[a * NP + b];
}
void dig_scales(const double* Dm, const double* rho, int NP, int* A, int* k, int* m2, int* q2) {
  double row[2] = {0, 0}, mx[2] = {0, 0};
  double rm = 0;
  for (int a = 0; a < NP; ++a) rm = std::fmax(rm, rho[a]);
  for (int a = 0; a < NP; ++a) A[a] = (int)std::lround(0.75 * std::log2(rho[a] / rm));
  for (int st = 0; st < 2; ++st)
    for (int a = 0; a < NP; ++a) {
      double r = 0;
      for (int b = 0; b < NP; ++b) {
        r += std::fabs(dig_entry(Dm, NP, A, st, a, b));
        mx[st] = std::fmax(mx[st], std::fabs(dig_entry(Dm, NP, A, st, a, b)));
      }
      row[st] = std::fmax(row[st], r);
    }
  const double g = 1.0 - 0x1p-10;
  const double c1m = std::fmin(2.0 / row[0], 1.0 / mx[0]) * g, c2m = std::fmin(4.0 / (3.0 * row[1]), 1.0 / mx[1]) * g;
  *m2 = (int)std::floor(std::ldexp(std::frexp(c2m, q2), 8));
  *k = (int)std::floor(std::log2(c1m * std::ldexp((double)*m2, *q2 - 8)));
}

// The digits of an order up to 7; false when the sums of digits would not stay exact.
bool dig_digits(const double* Dm, const double* rho, int NP, DigHost& H) {
  int k, m2, q2;
  dig_scales(Dm, rho, NP, H.a, &k, &m2, &q2);
  H.kexp = k;
  for (int st = 0; st < 2; ++st)
    for (int a = 0; a < NP; ++a)
      for (int b = 0; b < NP; ++b) {
        const double d = dig_entry(Dm, NP, H.a, st, a, b);
        __int128 v = st ? dig_scaled(d, m2, 1, 63 + q2 - 8) : dig_scaled(d, 1, m2, 63 + k - (q2 - 8));
        for (int t = 7; t > 0; --t) {
          const int x = (int)(((v + 128) & 255) - 128);
          H.dg[st][a][b][t] = x;
          v = (v - x) >> 8;
        }
        H.dg[st][a][b][0] = (int)v;
        if (v < -128 || v > 128) return false;
      }
  // a digit sum of two directions stays below 2^22 for every u (digits 0..255)
  for (int st = 0; st < 2; ++st)
    for (int a = 0; a < NP; ++a) {
      int64_t s = 0;
      for (int b = 0; b < NP; ++b)
        for (int t = 0; t < 8; ++t) s += std::abs(H.dg[st][a][b][t]);
      if (2 * 255 * s >= (1 << 22)) return false;
    }
  return true;
}

// The level's fixed-point factors; a: the exponents on the device. The stream is synchronised (the tables' host copies go).
template <int NP>
int dig_factors(Level& L, const int32_t* a, int kexp, cudaStream_t s) {
  using S = DigShape<NP>;
  int2* Gx = nullptr;
  int32_t* ge = nullptr;
  if (cudaMalloc((void**)&Gx, (size_t)L.E * 6 * S::GE * sizeof(int2)) != cudaSuccess ||
      cudaMalloc((void**)&ge, (size_t)L.E * sizeof(int32_t)) != cudaSuccess) {
    cudaGetLastError();
    if (Gx) cudaFree(Gx);
    SEM_CUDA_TRY(cudaStreamSynchronize(s));
    return SEM_OK;
  }
  L.Gx = Gx;
  L.gexp = ge;
  L.dig_kexp = kexp;
  k_dig_factors<NP><<<L.E, 128, 0, s>>>(L.G, a, Gx, ge);
  SEM_LAUNCH_CHECK();
  SEM_CUDA_TRY(cudaStreamSynchronize(s));
  return SEM_OK;
}

template <int NP>
int dig_build_np(Level& L, cudaStream_t s) {
  DigHost H;
  if (!dig_digits(L.D.a, L.rho, NP, H)) return SEM_OK;
  std::vector<DigTab> tab(1);
  DigTab& T = tab[0];
  for (int st = 0; st < 2; ++st)
    for (int m = 0; m < 4; ++m)
      for (int lane = 0; lane < 32; ++lane) {
        const int g = lane >> 2, c = lane & 3;
        auto pair = [&](int in, int d) -> uint32_t {   // digits d (low half), d + 1 (high half) of entry (g, in)
          if (g >= NP || in >= NP) return 0;
          const int* x = H.dg[st][g][in];
          return (uint32_t)(d < 0 ? 0 : half_of(x[d])) | ((uint32_t)half_of(x[d + 1]) << 16);
        };
        T.frag[st][m][lane] = make_uint4(pair(2 * c, 2 * m), pair(2 * c, 2 * m - 1), pair(2 * c + 1, 2 * m),
                                         pair(2 * c + 1, 2 * m - 1));
      }
  int64_t z[2][8][8] = {};
  for (int st = 0; st < 2; ++st)
    for (int a = 0; a < NP; ++a)
      for (int d = 0; d < 8; ++d)
        for (int b = 0; b < NP; ++b) z[st][a][d] += H.dg[st][a][b][d];
  for (int a = 0; a < 8; ++a) {
    T.a[a] = a < NP ? H.a[a] : 0;
    T.nk0[a] = 0ull - dig_merge_zero(z[0][a], DIG_SH1);
    T.nk1t[a] = 0ull - dig_merge_zero(z[1][a], DIG_SH2);
    for (int b = 0; b < 8; ++b) {
      int64_t t[8];
      for (int d = 0; d < 8; ++d) t[d] = z[1][a][d] + z[1][b][d];
      T.nk1rs[a * 8 + b] = 0ull - dig_merge_zero(t, DIG_SH2);
    }
  }
  DigTab* dt = nullptr;
  // without the memory the even-odd form runs
  if (cudaMalloc((void**)&dt, sizeof(DigTab)) != cudaSuccess) {
    cudaGetLastError();
    return SEM_OK;
  }
  L.dig = dt;
  SEM_CUDA_TRY(cudaMemcpyAsync(dt, &T, sizeof(DigTab), cudaMemcpyHostToDevice, s));
  return dig_factors<NP>(L, reinterpret_cast<const int32_t*>(reinterpret_cast<const char*>(dt) + offsetof(DigTab, a)),
                         H.kexp, s);
}

// 8 <= N <= 11
template <int NP>
int dig_build_eo(Level& L, cudaStream_t s) {
  int A[12], k, m2, q2;
  dig_scales(L.D.a, L.rho, NP, A, &k, &m2, &q2);
  SEM_TRY(dig_eo_tables(L, A, k, m2, q2, &L.dig_eo, s));
  if (!L.dig_eo) return SEM_OK;
  return dig_factors<NP>(L, dig_eo_exponents(L.dig_eo), k, s);
}

}  // namespace

// The fixed-point factors and digit tables of a level, where the digit kernel is compiled for its order.
int dig_build(Level& L, cudaStream_t s) {
  switch (L.NP) {
    case 5: return dig_build_np<5>(L, s);
    case 6: return dig_build_np<6>(L, s);
    case 7: return dig_build_np<7>(L, s);
    case 8: return dig_build_np<8>(L, s);
    case 9: return dig_build_eo<9>(L, s);
    case 10: return dig_build_eo<10>(L, s);
    case 11: return dig_build_eo<11>(L, s);
    case 12: return dig_build_eo<12>(L, s);
    default: return SEM_OK;
  }
}

// The element operator on elements [e0, e0 + E) (u, w, h1L: whole-level L-vectors). Needs L.Gx.
int ax_dig_apply(const Level& L, int e0, int E, const double* u, double* w, double h1, double h2, const double* h1L,
                 bool pairs, const double* skip, cudaStream_t s) {
  EOMat<ArF64> Df, Dt;
  make_eo<ArF64>(L.D.a, L.NP, false, Df);
  make_eo<ArF64>(L.D.a, L.NP, true, Dt);
  const size_t off = (size_t)e0 * L.NP * L.NP * L.NP;
  u += off;
  w += off;
  if (h1L) h1L += off;
  const int vec = (((uintptr_t)u | (uintptr_t)w | (uintptr_t)h1L) & 15u) == 0;
  const int mass = h2 != 0.0 ? 1 : 0;                         // h2 B u is added
  const int e1 = dig_h1_exp(h1), span = dig_h1_span(pairs);
  switch (L.NP) {
#define CASE(NP)                                                                                                   \
  case NP: {                                                                                                       \
    using S = DigShape<NP>;                                                                                        \
    const int2* Gx = L.Gx + (size_t)e0 * 6 * S::GE;                                                                \
    if (h1L)                                                                                                       \
      k_ax_dig<NP, true><<<E, S::T, 0, s>>>(u, w, Gx, L.gexp + e0, L.G + 7 * off, L.dig, L.dig_kexp, 1.0,   \
                                            h2, h1L, span, skip, vec, mass, 0, Df, Dt);                             \
    else                                                                                                           \
      k_ax_dig<NP, false><<<E, S::T, 0, s>>>(u, w, Gx, L.gexp + e0, L.G + 7 * off, L.dig, L.dig_kexp, h1,   \
                                             h2, nullptr, 0, skip, vec, mass, e1, Df, Dt);                          \
    SEM_LAUNCH_CHECK();                                                                                            \
    return SEM_OK;                                                                                                 \
  }
    CASE(5) CASE(6) CASE(7) CASE(8)
#undef CASE
  }
  if (L.dig_eo) return ax_dig_eo_apply(L, e0, E, u, w, h1, h2, h1L, span, skip, Df, Dt, s);
  set_detail("order %d not compiled", L.N);
  return SEM_EINVAL;
}

}  // namespace sem
