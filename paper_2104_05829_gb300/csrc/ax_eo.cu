// Local operator A^e = D^T h1 G D + h2 B (eq. Ae) with even-odd
// (centro-antisymmetric) 1-D contractions, in FP64 or in FP32-pair arithmetic.
//
// On GB300 both variants are bound by instruction throughput (the FP64 pipe,
// or the FP32 pipes for the pair arithmetic), so their speed is set by how
// many arithmetic instructions they issue. D_hat on symmetric GLL nodes
// satisfies D[N-a][N-b] = -D[a][b] exactly (also in floating point: the nodes
// are exactly antisymmetric and P_N(-x) = (-1)^N P_N(x)). Writing a line v as
// s_b = v_b + v_{N-b}, d_b = v_b - v_{N-b} (b < H = (N+1)/2),
//   out_a = ev_a + od_a,  out_{N-a} = od_a - ev_a,
//   ev_a = sum_b E[a][b] s_b (+ D[a][m] v_m for the middle point m when N is even),
//   od_a = sum_b O[a][b] d_b,  E = (D[a][b] + D[a][N-b]) / 2, O = (D[a][b] - D[a][N-b]) / 2,
// and, when N is even, out_m = sum_b D[m][b] d_b. A line of N+1 outputs costs
// (N+1)^2/2 multiply-adds and 2(N+1) additions instead of (N+1)^2 multiply-adds.
// The same holds for D^T.
//
// Every thread of the (N+1)^2 plane of an element transforms whole lines: its
// own t-line in registers, and one r-row and one s-column of shared memory.
// h1 multiplies the stiffness sum once per point instead of each factor.
//
// The pair variant keeps every value as an unevaluated sum of two floats
// (pairs.cuh); the factors are stored pre-split as float2 (hi, lo).
#include "eo.cuh"

namespace sem {

namespace {

template <class Ar, int NP, bool VARH1>
__global__ void __launch_bounds__(NP* NP* eo_epb<NP>(), (eo_min_blocks<Ar, NP>()))
    k_ax_eo(int E, const double* __restrict__ u, double* __restrict__ w, const typename Ar::GT* __restrict__ G,
            EOMat<Ar> Df, EOMat<Ar> Dt, typename Ar::V h1, typename Ar::V h2, const double* __restrict__ h1L,
            const double* skip) {
  using V = typename Ar::V;
  constexpr int EPB = eo_epb<NP>();
  constexpr int NP2 = NP * NP, NP3 = NP2 * NP;
  constexpr int ES = Pad3<NP>::ES;
  if (skip && *skip != 0.0) return;
  __shared__ V s_a[EPB * ES];
  __shared__ V s_b[EPB * ES];
  __shared__ V s_c[EPB * ES];
  const int tid = threadIdx.x;
  const int le = tid / NP2;
  const int ij = tid - le * NP2;
  const int j = ij / NP, i = ij - j * NP;
  const int e = blockIdx.x * EPB + le;
  eo_element<Ar, NP, VARH1>(true, e < E, i, j, (size_t)e * NP3, u, w, G + (size_t)e * 7 * NP3, Df, Dt, h1, h2, h1L,
                            s_a + le * ES, s_b + le * ES, s_c + le * ES);
}

template <class Ar>
int eo_launch(const Level& L, const double* u, double* w, const typename Ar::GT* G, double h1, double h2,
              const double* h1L, const double* skip, cudaStream_t s) {
  EOMat<Ar> Df, Dt;
  make_eo<Ar>(L.D.a, L.NP, false, Df);
  make_eo<Ar>(L.D.a, L.NP, true, Dt);
  const typename Ar::V vh1 = Ar::host(h1), vh2 = Ar::host(h2);
  switch (L.NP) {
#define CASE(NP)                                                                                      \
  case NP: {                                                                                          \
    constexpr int EPB = eo_epb<NP>();                                                                 \
    const dim3 grid((L.E + EPB - 1) / EPB), block(NP * NP * EPB);                                     \
    if (h1L)                                                                                          \
      k_ax_eo<Ar, NP, true><<<grid, block, 0, s>>>(L.E, u, w, G, Df, Dt, vh1, vh2, h1L, skip);         \
    else                                                                                              \
      k_ax_eo<Ar, NP, false><<<grid, block, 0, s>>>(L.E, u, w, G, Df, Dt, vh1, vh2, nullptr, skip);    \
    SEM_LAUNCH_CHECK();                                                                               \
    return SEM_OK;                                                                                    \
  }
    CASE(2) CASE(3) CASE(4) CASE(5) CASE(6) CASE(7) CASE(8) CASE(9) CASE(10) CASE(11) CASE(12)
#undef CASE
  }
  set_detail("order %d not compiled", L.N);
  return SEM_EINVAL;
}

__global__ void k_split_pairs(int64_t n, const double* __restrict__ G, float2* __restrict__ G2) {
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
    const ff v = ff_split(G[q]);
    G2[q] = make_float2(v.h, v.l);
  }
}

}  // namespace

// FP64 element operator: in digits where the level has fixed-point factors (ax_dig.cu), else, or with eo, by even-odd
// contractions.
int ax_eo_apply(const Level& L, const double* u, double* w, double h1, double h2, const double* h1L,
                const double* skip, cudaStream_t s, bool eo) {
  if (L.Gx && !eo) return ax_dig_apply(L, 0, L.E, u, w, h1, h2, h1L, false, skip, s);
  return eo_launch<ArF64>(L, u, w, L.G, h1, h2, h1L, skip, s);
}

// FP64-accurate element operator in FP32-pair arithmetic (scalar h1, or a nodal h1L, split
// into pairs as it is read); in digits where those are faster, unless eo.
int ax_pairs_apply(const Level& L, const double* u, double* w, double h1, double h2, const double* h1L,
                   cudaStream_t s, bool eo) {
  if (!L.pairs) {
    set_detail("FP32-pair factors were not built");
    return SEM_EINVAL;
  }
  if (dig_for_pairs(L) && !eo) return ax_dig_apply(L, 0, L.E, u, w, h1, h2, h1L, true, nullptr, s);
  return eo_launch<ArPair>(L, u, w, L.G2, h1, h2, h1L, nullptr, s);
}

// The element operator on elements [e0, e1) only (FP64 or FP32 pairs, scalar or nodal h1):
// the same kernels on a view of the level whose pointers start at element e0.
int ax_eo_apply_range(const Level& L, int e0, int e1, const double* u, double* w, double h1, double h2,
                      const double* h1L, bool pairs, cudaStream_t s) {
  if (e1 <= e0) return SEM_OK;
  if (pairs && !L.pairs) {
    set_detail("FP32-pair factors not built");
    return SEM_EINVAL;
  }
  if (pairs ? dig_for_pairs(L) : L.Gx != nullptr) return ax_dig_apply(L, e0, e1 - e0, u, w, h1, h2, h1L, pairs, nullptr, s);
  const size_t off = (size_t)e0 * L.NP * L.NP * L.NP;
  Level V = L;
  V.E = e1 - e0;
  V.nL = (int64_t)V.E * L.NP * L.NP * L.NP;
  if (pairs)
    return eo_launch<ArPair>(V, u + off, w + off, L.G2 + 7 * off, h1, h2, h1L ? h1L + off : nullptr, nullptr, s);
  return eo_launch<ArF64>(V, u + off, w + off, L.G + 7 * off, h1, h2, h1L ? h1L + off : nullptr, nullptr, s);
}

// (hi, lo) FP32 split of the FP64 factors for the pair kernel.
int pairs_build(Level& L, cudaStream_t s) {
  L.pairs = true;
  if (!L.G2) {
    cudaError_t e = cudaMalloc((void**)&L.G2, 7 * L.nL * sizeof(float2) + 16);
    if (e != cudaSuccess) {
      cudaGetLastError();
      L.G2 = nullptr;
      set_detail("cudaMalloc of the FP32-pair factors: %s", cudaGetErrorString(e));
      return SEM_ENOMEM;
    }
  }
  const int64_t n = 7 * L.nL;
  int64_t nb = (n + 255) / 256;
  if (nb > 152 * 32) nb = 152 * 32;
  k_split_pairs<<<(unsigned)nb, 256, 0, s>>>(n, L.G, L.G2);
  SEM_LAUNCH_CHECK();
  return SEM_OK;
}

}  // namespace sem
