// Dealiased advection operator (Section 2.1, the nonlinear term of eq. stdadv
// and the hyperbolic substeps of eq. hyp; Section 3.3 "High-Order Kernels":
// the term is evaluated on N_q^3 quadrature points with a 2-D thread plane and
// one register line per thread).
//
// For an advecting field c (three components) and ncomp advected fields u:
//   (C u)_i = sum_q w_q J_q phi_i(x_q) (c . grad u)(x_q),
// q over nq^3 Gauss-Legendre points, nq = ceil(3 (N+1) / 2). Per element:
//   1. each c_m is interpolated to the Gauss points (three sum-factorised
//      passes, the last one into the thread's register line along t);
//   2. the contravariant wind chat_d = sum_m Gq[d][m] c_m with the cubature
//      factors Gq = w J dr_d/dx_m (stored per point, set up once) -- kept in
//      registers and reused for every advected component (Section 3.3);
//   3. for each u: interpolation as in 1, derivatives on the Gauss points
//      (t along the thread's register line; r and s on lines of the Gauss-point
//      array in shared memory, each thread differentiating one whole line; all
//      three in even-odd form with the coefficients as kernel parameters), the
//      pointwise product sum_d chat_d du/dr_d, and the transposed interpolation
//      back to the GLL points (three passes).
// Thread (a, b) of the nq x nq plane owns the Gauss points (a, b, *).
#include <algorithm>
#include <cmath>
#include <vector>

#include "advect.cuh"

namespace sem {

namespace {

// Gauss-Legendre nodes (ascending) and weights: roots of P_n by Newton's method
// from x = cos(pi (4i - 1) / (4n + 2)), weights 2 / ((1 - x^2) P_n'(x)^2).
void host_gauss(int n, double* z, double* w) {
  for (int i = 1; i <= n; ++i) {
    double x = std::cos(M_PI * (4.0 * i - 1.0) / (4.0 * n + 2.0));
    double dp = 1.0;
    for (int it = 0; it < 100; ++it) {
      double p0 = 1.0, p1 = x;
      for (int k = 1; k < n; ++k) {
        const double p2 = ((2 * k + 1) * x * p1 - k * p0) / (k + 1);
        p0 = p1;
        p1 = p2;
      }
      const double pn = n == 0 ? 1.0 : p1, pm1 = n == 0 ? 0.0 : p0;
      dp = n * (x * pn - pm1) / (x * x - 1.0);
      const double step = pn / dp;
      x -= step;
      if (std::fabs(step) < 1e-16) break;
    }
    z[n - i] = x;
    w[n - i] = 2.0 / ((1.0 - x * x) * dp * dp);
  }
  for (int i = 0; i < n / 2; ++i) {   // exact symmetry
    const double a = 0.5 * (z[n - 1 - i] - z[i]), b = 0.5 * (w[i] + w[n - 1 - i]);
    z[n - 1 - i] = a;
    z[i] = -a;
    w[i] = w[n - 1 - i] = b;
  }
  if (n % 2 == 1) z[n / 2] = 0.0;
}

// Dq[a][b] = h_b'(z_a) for the cardinal polynomials on the nodes z (barycentric form).
void host_deriv(int n, const double* z, double* D) {
  std::vector<double> lam(n, 1.0);
  for (int b = 0; b < n; ++b)
    for (int c = 0; c < n; ++c)
      if (c != b) lam[b] /= (z[b] - z[c]);
  for (int a = 0; a < n; ++a) {
    double diag = 0.0;
    for (int b = 0; b < n; ++b) {
      if (a == b) continue;
      D[a * n + b] = lam[b] / lam[a] / (z[a] - z[b]);
      diag -= D[a * n + b];
    }
    D[a * n + a] = diag;
  }
}

// resident blocks requested from the register allocator: four in FP32 up to N = 7 (18
// warps per SM, 96 registers with a 128-byte spill: measured 1.63 ms against 1.74 ms at
// three blocks with no spill on the 32^3 box), two at N = 8; two in FP64 (a few hundred
// bytes of spills, measured 1.26x faster at N = 7 than one block with no spills)
template <class Ar, int NP>
__host__ __device__ constexpr int adv_min_blocks() {
  return sizeof(typename Ar::V) == 4 ? (NP <= 8 ? 4 : 2) : 2;
}

template <class Ar, int NP>
__global__ void __launch_bounds__(AdvShape<NP>::T, (adv_min_blocks<Ar, NP>()))
    k_advect(int E, int ncomp, int64_t nL, const typename Ar::S* __restrict__ cv, const typename Ar::S* __restrict__ uv,
             const typename Ar::G* __restrict__ Gq, const typename Ar::G* __restrict__ Im,
             const typename Ar::G* __restrict__ Dq, typename Ar::S* __restrict__ wv, AdvOps<typename Ar::V, NP> P) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  constexpr int NQ = AdvShape<NP>::NQ;
  advect_element<Ar, NP>(true, threadIdx.x % NQ, threadIdx.x / NQ, blockIdx.x, s_raw, ncomp, nL, cv, uv, Gq, Im, Dq, wv, P);
}

// Cubature factors Gq[e][d][m][point] = w_q J_q dr_d/dx_m at the Gauss points:
// the coordinates (relative to the element's first node) interpolated and
// differentiated on the Gauss points, the 3x3 metric inverted by cofactors.
template <int NP>
__global__ void __launch_bounds__(AdvShape<NP>::T)
    k_cub_geom(int E, const double* __restrict__ x, const double* __restrict__ y, const double* __restrict__ z,
               const double* __restrict__ Im, const double* __restrict__ Dq, const double* __restrict__ wq,
               double* __restrict__ Gq, float* __restrict__ Gq32, int* bad) {
  constexpr int NQ = AdvShape<NP>::NQ, NP3 = NP * NP * NP, NQ2 = NQ * NQ, NQ3 = NQ2 * NQ;
  __shared__ double sI[NQ * NP];
  __shared__ double sD[NQ * NQ];
  __shared__ double s_src[NP3];
  __shared__ double s_t1[NP * NP * NQ];
  __shared__ double s_X[NQ3];
  const int e = blockIdx.x;
  const int a = threadIdx.x % NQ, b = threadIdx.x / NQ;
  load_ops<AdvPlain<double>, NP, NQ>(Im, Dq, sI, sD);
  const size_t eb = (size_t)e * NP3;
  double Jl[3][3][NQ];   // Jl[m][d][c] = dx_m / dr_d at Gauss point (a, b, c)
  const double* X[3] = {x, y, z};
  for (int m = 0; m < 3; ++m) {
    __syncthreads();
    const double x0 = X[m][eb];
    for (int q = threadIdx.x; q < NP3; q += blockDim.x) s_src[q] = X[m][eb + q] - x0;
    __syncthreads();
    double line[NQ];
    to_gauss<AdvPlain<double>, NP, NQ>(true, s_src, s_t1, sI, sI, a, b, line);
#pragma unroll
    for (int c = 0; c < NQ; ++c) s_X[(c * NQ + b) * NQ + a] = line[c];
    __syncthreads();
#pragma unroll
    for (int c = 0; c < NQ; ++c) {
      double dr = 0, ds = 0, dt = 0;
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        dr = fma(sD[a * NQ + q], s_X[(c * NQ + b) * NQ + q], dr);
        ds = fma(sD[b * NQ + q], s_X[(c * NQ + q) * NQ + a], ds);
        dt = fma(sD[c * NQ + q], line[q], dt);
      }
      Jl[m][0][c] = dr;
      Jl[m][1][c] = ds;
      Jl[m][2][c] = dt;
    }
  }
#pragma unroll
  for (int c = 0; c < NQ; ++c) {
    double J[3][3];   // J[m][d] = dx_m / dr_d
#pragma unroll
    for (int m = 0; m < 3; ++m)
#pragma unroll
      for (int d = 0; d < 3; ++d) J[m][d] = Jl[m][d][c];
    const double c00 = J[1][1] * J[2][2] - J[1][2] * J[2][1];
    const double c01 = J[1][2] * J[2][0] - J[1][0] * J[2][2];
    const double c02 = J[1][0] * J[2][1] - J[1][1] * J[2][0];
    const double det = J[0][0] * c00 + J[0][1] * c01 + J[0][2] * c02;
    if (!(det > 0.0)) atomicExch(bad, 1);
    // R[d][m] = det * dr_d/dx_m (the adjugate); w J dr_d/dx_m = w R[d][m]
    double R[3][3];
    R[0][0] = c00;
    R[1][0] = c01;
    R[2][0] = c02;
    R[0][1] = J[0][2] * J[2][1] - J[0][1] * J[2][2];
    R[1][1] = J[0][0] * J[2][2] - J[0][2] * J[2][0];
    R[2][1] = J[0][1] * J[2][0] - J[0][0] * J[2][1];
    R[0][2] = J[0][1] * J[1][2] - J[0][2] * J[1][1];
    R[1][2] = J[0][2] * J[1][0] - J[0][0] * J[1][2];
    R[2][2] = J[0][0] * J[1][1] - J[0][1] * J[1][0];
    const double wgt = wq[a] * wq[b] * wq[c];
    const size_t pt = (size_t)e * 9 * NQ3 + (c * NQ + b) * NQ + a;
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        const double v = wgt * R[d][m];
        Gq[pt + (d * 3 + m) * NQ3] = v;
        if (Gq32) Gq32[pt + (d * 3 + m) * NQ3] = (float)v;
      }
  }
}

template <int NP>
int cub_geom_launch(const Level& L, const double* Im, const double* Dq, const double* wq, double* Gq, float* Gq32,
                    int* bad, cudaStream_t s) {
  k_cub_geom<NP><<<L.E, AdvShape<NP>::T, 0, s>>>(L.E, L.x, L.y, L.z, Im, Dq, wq, Gq, Gq32, bad);
  SEM_LAUNCH_CHECK();
  return SEM_OK;
}

template <class Ar, int NP>
int advect_launch(const Level& L, const AdvData& A, const typename Ar::S* c, const typename Ar::S* u,
                  typename Ar::S* w, int ncomp, const typename Ar::G* Gq, const typename Ar::G* Im,
                  const typename Ar::G* Dq, cudaStream_t s) {
  const AdvOps<typename Ar::V, NP> P = adv_ops<Ar, NP>(A);
  constexpr size_t smem = advect_smem<Ar, NP>();
  static PerDevice<bool> attr;
  SEM_TRY(smem_attr_once(attr, (const void*)k_advect<Ar, NP>, smem));
  k_advect<Ar, NP><<<L.E, AdvShape<NP>::T, smem, s>>>(L.E, ncomp, L.nL, c, u, Gq, Im, Dq, w, P);
  SEM_LAUNCH_CHECK();
  return SEM_OK;
}

#define ADV_DISPATCH(NPV, CALL) \
  case NPV: return CALL;

#define GRID_LOOP_ADV(l, n) \
  for (int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; l < (n); l += (int64_t)gridDim.x * blockDim.x)

inline unsigned vgrid_adv(int64_t n) {
  int64_t b = (n + 255) / 256;
  if (b > 152 * 16) b = 152 * 16;
  if (b < 1) b = 1;
  return (unsigned)b;
}

// m = B_L, the local GLL mass (component 6 of the geometric factors)
__global__ void k_mass_local(int64_t n, int np3, const double* __restrict__ G, double* __restrict__ m) {
  GRID_LOOP_ADV(l, n) {
    const int64_t e = l / np3;
    m[l] = G[(e * 7 + 6) * np3 + (l - e * np3)];
  }
}

// minv = 1 / (QQ^T B) from the gathered mass in m (in place), FP64 and FP32 copies
__global__ void k_minv(int64_t n, double* __restrict__ m, float* __restrict__ m32) {
  GRID_LOOP_ADV(l, n) {
    const double v = 1.0 / m[l];
    m[l] = v;
    m32[l] = (float)v;
  }
}

// c(t) = c0 + th (c1 - c0) over the three wind components
template <typename T>
__global__ void k_wind(int64_t n, const T* __restrict__ c0, const T* __restrict__ c1, T th, T* __restrict__ c) {
  GRID_LOOP_ADV(l, n) c[l] = c0[l] + th * (c1[l] - c0[l]);
}

// (hi, lo) FP32 split of FP64 values
__global__ void k_split_adv(int64_t n, const double* __restrict__ a, float2* __restrict__ b) {
  GRID_LOOP_ADV(q, n) {
    const ff v = ff_split(a[q]);
    b[q] = make_float2(v.h, v.l);
  }
}

// One RK4 stage on ncomp components: k = -minv z (z = QQ^T C w_stage);
// mode 0: acc = k, ws = w + cw k; mode 1: acc += 2k, ws = w + cw k; mode 2: w += cw (acc + k).
template <typename T>
__global__ void k_rk_stage(int64_t n, int64_t nL, const T* __restrict__ z, const T* __restrict__ minv,
                           T* __restrict__ w, T* __restrict__ ws, T* __restrict__ acc, T cw, int mode) {
  GRID_LOOP_ADV(q, n) {
    const T k = -minv[q % nL] * z[q];
    if (mode == 0) {
      acc[q] = k;
      ws[q] = w[q] + cw * k;
    } else if (mode == 1) {
      acc[q] += T(2) * k;
      ws[q] = w[q] + cw * k;
    } else {
      w[q] += cw * (acc[q] + k);
    }
  }
}

}  // namespace

// Build the cubature data of level 0 (Gauss rule, interpolation and derivative
// matrices, Gq in FP64 and FP32). Synchronous.
int advect_build(Ctx& C, cudaStream_t s) {
  Level& L = C.lev[0];
  if (C.adv.ready) return SEM_OK;
  if (L.N < 2 || L.N > 8) {
    set_detail("the dealiased advection operator is compiled for 2 <= N <= 8 (order %d)", L.N);
    return SEM_EINVAL;
  }
  const int NP = L.NP, NQ = nq_of(NP);
  std::vector<double> z(NQ), w(NQ), Im(NQ * NP), Dq(NQ * NQ);
  host_gauss(NQ, z.data(), w.data());
  host_interp(NP, L.xi, NQ, z.data(), Im.data());
  host_deriv(NQ, z.data(), Dq.data());
  std::vector<float> Im32(Im.begin(), Im.end()), Dq32(Dq.begin(), Dq.end());
  AdvData& A = C.adv;
  A.nq = NQ;
  for (size_t q = 0; q < Im.size(); ++q) A.hIm[q] = Im[q];
  for (size_t q = 0; q < Dq.size(); ++q) A.hDq[q] = Dq[q];
  for (int q = 0; q < NQ; ++q) A.hwq[q] = w[q];
  const size_t ng = (size_t)L.E * 9 * NQ * NQ * NQ;
  auto dm = [&](void** p, size_t bytes) -> int {
    if (cudaMalloc(p, bytes) != cudaSuccess) {
      *p = nullptr;
      cudaGetLastError();
      set_detail("cudaMalloc of %zu bytes failed (advection cubature data)", bytes);
      return SEM_ENOMEM;
    }
    return SEM_OK;
  };
  SEM_TRY(dm((void**)&A.Gq, ng * 8));
  SEM_TRY(dm((void**)&A.Gq32, ng * 4));
  SEM_TRY(dm((void**)&A.Im, Im.size() * 8));
  SEM_TRY(dm((void**)&A.Dq, Dq.size() * 8));
  SEM_TRY(dm((void**)&A.wq, NQ * 8));
  SEM_TRY(dm((void**)&A.Im32, Im.size() * 4));
  SEM_TRY(dm((void**)&A.Dq32, Dq.size() * 4));
  SEM_CUDA_TRY(cudaMemcpyAsync(A.Im, Im.data(), Im.size() * 8, cudaMemcpyHostToDevice, s));
  SEM_CUDA_TRY(cudaMemcpyAsync(A.Dq, Dq.data(), Dq.size() * 8, cudaMemcpyHostToDevice, s));
  SEM_CUDA_TRY(cudaMemcpyAsync(A.wq, w.data(), NQ * 8, cudaMemcpyHostToDevice, s));
  SEM_CUDA_TRY(cudaMemcpyAsync(A.Im32, Im32.data(), Im32.size() * 4, cudaMemcpyHostToDevice, s));
  SEM_CUDA_TRY(cudaMemcpyAsync(A.Dq32, Dq32.data(), Dq32.size() * 4, cudaMemcpyHostToDevice, s));
  int* bad = nullptr;
  SEM_TRY(dm((void**)&bad, sizeof(int)));
  SEM_CUDA_TRY(cudaMemsetAsync(bad, 0, sizeof(int), s));
  int rc = SEM_OK;
  switch (NP) {
    case 3: rc = cub_geom_launch<3>(L, A.Im, A.Dq, A.wq, A.Gq, A.Gq32, bad, s); break;
    case 4: rc = cub_geom_launch<4>(L, A.Im, A.Dq, A.wq, A.Gq, A.Gq32, bad, s); break;
    case 5: rc = cub_geom_launch<5>(L, A.Im, A.Dq, A.wq, A.Gq, A.Gq32, bad, s); break;
    case 6: rc = cub_geom_launch<6>(L, A.Im, A.Dq, A.wq, A.Gq, A.Gq32, bad, s); break;
    case 7: rc = cub_geom_launch<7>(L, A.Im, A.Dq, A.wq, A.Gq, A.Gq32, bad, s); break;
    case 8: rc = cub_geom_launch<8>(L, A.Im, A.Dq, A.wq, A.Gq, A.Gq32, bad, s); break;
    default: rc = cub_geom_launch<9>(L, A.Im, A.Dq, A.wq, A.Gq, A.Gq32, bad, s); break;
  }
  int h_bad = 0;
  if (rc == SEM_OK) {
    if (cudaMemcpyAsync(&h_bad, bad, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess) {
      set_detail("advection cubature setup failed: %s", cudaGetErrorString(cudaGetLastError()));
      rc = SEM_ECUDA;
    }
  }
  cudaFree(bad);
  if (rc != SEM_OK) return rc;
  if (h_bad) {
    set_detail("non-positive Jacobian at a Gauss point");
    return SEM_EMESH;
  }
  A.ready = true;
  return SEM_OK;
}

// The FP32-pair copies of the cubature factors and the 1-D matrices (first pair evaluation).
int advect_pairs_build(AdvData& A, const Level& L, cudaStream_t s) {
  if (A.Gq2) return SEM_OK;
  const int NQ = A.nq, NP = L.NP;
  const size_t ng = (size_t)L.E * 9 * NQ * NQ * NQ;
  float2 *g2 = nullptr, *i2 = nullptr, *d2 = nullptr;
  if (cudaMalloc((void**)&g2, ng * sizeof(float2)) != cudaSuccess ||
      cudaMalloc((void**)&i2, (size_t)NQ * NP * sizeof(float2)) != cudaSuccess ||
      cudaMalloc((void**)&d2, (size_t)NQ * NQ * sizeof(float2)) != cudaSuccess) {
    cudaGetLastError();
    if (g2) cudaFree(g2);
    if (i2) cudaFree(i2);
    set_detail("cudaMalloc of %zu bytes failed (FP32-pair cubature factors)", ng * sizeof(float2));
    return SEM_ENOMEM;
  }
  k_split_adv<<<vgrid_adv((int64_t)ng), 256, 0, s>>>((int64_t)ng, A.Gq, g2);
  k_split_adv<<<1, 256, 0, s>>>((int64_t)NQ * NP, A.Im, i2);
  k_split_adv<<<1, 256, 0, s>>>((int64_t)NQ * NQ, A.Dq, d2);
  SEM_LAUNCH_CHECK();
  A.Gq2 = g2;
  A.Im2 = i2;
  A.Dq2 = d2;
  return SEM_OK;
}

void advect_free(AdvData& A) {
  void* ptrs[] = {A.Gq, A.Gq32, A.Gq2, A.Im, A.Dq, A.wq, A.Im32, A.Dq32, A.Im2, A.Dq2, A.minv, A.minv32, A.ws,
                  A.Gqx, A.gqexp, A.dig};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  A = AdvData();
}

int advect_apply(Ctx& C, int prec, const void* c, const void* u, void* w, int ncomp, cudaStream_t s) {
  const Level& L = C.lev[0];
  AdvData& A = C.adv;
  if (prec != SEM_FP32) {
    SEM_TRY(advect_dig_build(A, L, s));
    // at N = 4 (lines and outputs padded from five and eight points) the pair form is the faster one
    if (A.Gqx && (prec == SEM_FP64 || L.N >= 5)) return advect_dig_apply(L, A, (const double*)c, (const double*)u, (double*)w, ncomp, prec == SEM_FP64P, s);
  }
  if (prec == SEM_FP64P) {
    SEM_TRY(advect_pairs_build(A, L, s));
    const double *cc = (const double*)c, *uu = (const double*)u;
    double* ww = (double*)w;
    switch (L.NP) {
      ADV_DISPATCH(3, (advect_launch<AdvPair, 3>(L, A, cc, uu, ww, ncomp, A.Gq2, A.Im2, A.Dq2, s)))
      ADV_DISPATCH(4, (advect_launch<AdvPair, 4>(L, A, cc, uu, ww, ncomp, A.Gq2, A.Im2, A.Dq2, s)))
      ADV_DISPATCH(5, (advect_launch<AdvPair, 5>(L, A, cc, uu, ww, ncomp, A.Gq2, A.Im2, A.Dq2, s)))
      ADV_DISPATCH(6, (advect_launch<AdvPair, 6>(L, A, cc, uu, ww, ncomp, A.Gq2, A.Im2, A.Dq2, s)))
      ADV_DISPATCH(7, (advect_launch<AdvPair, 7>(L, A, cc, uu, ww, ncomp, A.Gq2, A.Im2, A.Dq2, s)))
      ADV_DISPATCH(8, (advect_launch<AdvPair, 8>(L, A, cc, uu, ww, ncomp, A.Gq2, A.Im2, A.Dq2, s)))
      ADV_DISPATCH(9, (advect_launch<AdvPair, 9>(L, A, cc, uu, ww, ncomp, A.Gq2, A.Im2, A.Dq2, s)))
      default: break;
    }
  } else if (prec == SEM_FP64) {
    const double *cc = (const double*)c, *uu = (const double*)u;
    double* ww = (double*)w;
    switch (L.NP) {
      ADV_DISPATCH(3, (advect_launch<AdvPlain<double>, 3>(L, A, cc, uu, ww, ncomp, A.Gq, A.Im, A.Dq, s)))
      ADV_DISPATCH(4, (advect_launch<AdvPlain<double>, 4>(L, A, cc, uu, ww, ncomp, A.Gq, A.Im, A.Dq, s)))
      ADV_DISPATCH(5, (advect_launch<AdvPlain<double>, 5>(L, A, cc, uu, ww, ncomp, A.Gq, A.Im, A.Dq, s)))
      ADV_DISPATCH(6, (advect_launch<AdvPlain<double>, 6>(L, A, cc, uu, ww, ncomp, A.Gq, A.Im, A.Dq, s)))
      ADV_DISPATCH(7, (advect_launch<AdvPlain<double>, 7>(L, A, cc, uu, ww, ncomp, A.Gq, A.Im, A.Dq, s)))
      ADV_DISPATCH(8, (advect_launch<AdvPlain<double>, 8>(L, A, cc, uu, ww, ncomp, A.Gq, A.Im, A.Dq, s)))
      ADV_DISPATCH(9, (advect_launch<AdvPlain<double>, 9>(L, A, cc, uu, ww, ncomp, A.Gq, A.Im, A.Dq, s)))
      default: break;
    }
  } else {
    const float *cc = (const float*)c, *uu = (const float*)u;
    float* ww = (float*)w;
    switch (L.NP) {
      ADV_DISPATCH(3, (advect_launch<AdvPlain<float>, 3>(L, A, cc, uu, ww, ncomp, A.Gq32, A.Im32, A.Dq32, s)))
      ADV_DISPATCH(4, (advect_launch<AdvPlain<float>, 4>(L, A, cc, uu, ww, ncomp, A.Gq32, A.Im32, A.Dq32, s)))
      ADV_DISPATCH(5, (advect_launch<AdvPlain<float>, 5>(L, A, cc, uu, ww, ncomp, A.Gq32, A.Im32, A.Dq32, s)))
      ADV_DISPATCH(6, (advect_launch<AdvPlain<float>, 6>(L, A, cc, uu, ww, ncomp, A.Gq32, A.Im32, A.Dq32, s)))
      ADV_DISPATCH(7, (advect_launch<AdvPlain<float>, 7>(L, A, cc, uu, ww, ncomp, A.Gq32, A.Im32, A.Dq32, s)))
      ADV_DISPATCH(8, (advect_launch<AdvPlain<float>, 8>(L, A, cc, uu, ww, ncomp, A.Gq32, A.Im32, A.Dq32, s)))
      ADV_DISPATCH(9, (advect_launch<AdvPlain<float>, 9>(L, A, cc, uu, ww, ncomp, A.Gq32, A.Im32, A.Dq32, s)))
      default: break;
    }
  }
  set_detail("the dealiased advection operator is compiled for 2 <= N <= 8");
  return SEM_EINVAL;
}

// RK4 substeps of dw/dt = -M^-1 QQ^T C(c(t)) w (the hyperbolic subproblem of the
// characteristics scheme, Section 2.1 eq. hyp): c(t) linear between c0 at t0 and
// c1 at t1 (c1 null: frozen), nsub classical Runge-Kutta steps, w in place.
int char_advance(Ctx& C, int prec, const void* c0, const void* c1, void* w, int ncomp, double t0, double t1,
                 int nsub, cudaStream_t s) {
  const Level& L = C.lev[0];
  AdvData& A = C.adv;
  const int64_t nL = L.nL, n = (int64_t)ncomp * nL;
  const int vp = prec == SEM_FP32 ? SEM_FP32 : SEM_FP64;   // the vectors' type (FP64 with the pair operator)
  const size_t esz = vp == SEM_FP64 ? 8 : 4;
  if (!A.minv) {
    if (cudaMalloc(&A.minv, nL * 8) != cudaSuccess || cudaMalloc(&A.minv32, nL * 4) != cudaSuccess) {
      cudaGetLastError();
      set_detail("cudaMalloc of the inverse mass failed");
      return SEM_ENOMEM;
    }
    k_mass_local<<<vgrid_adv(nL), 256, 0, s>>>(nL, L.NP * L.NP * L.NP, L.G, A.minv);
    SEM_LAUNCH_CHECK();
    SEM_TRY(gs_apply(L, SEM_FP64, A.minv, false, s));
    k_minv<<<vgrid_adv(nL), 256, 0, s>>>(nL, A.minv, A.minv32);
    SEM_LAUNCH_CHECK();
  }
  const size_t need = (3 * (size_t)n + 3 * (size_t)nL) * esz;
  if (A.ws_bytes < need) {
    if (A.ws) cudaFree(A.ws);
    A.ws = nullptr;
    A.ws_bytes = 0;
    if (cudaMalloc(&A.ws, need) != cudaSuccess) {
      cudaGetLastError();
      set_detail("cudaMalloc of %zu bytes failed (characteristics workspace)", need);
      return SEM_ENOMEM;
    }
    A.ws_bytes = need;
  }
  char* base = static_cast<char*>(A.ws);
  void* zb = base;                       // QQ^T C w_stage
  void* wsb = base + n * esz;            // w_stage
  void* accb = base + 2 * n * esz;       // sum of the weighted stages
  void* cb = base + 3 * n * esz;         // c(t)
  const double h = (t1 - t0) / nsub;
  auto wind = [&](double t) -> const void* {
    if (!c1) return c0;
    const double th = (t - t0) / (t1 - t0);
    if (vp == SEM_FP64)
      k_wind<double><<<vgrid_adv(3 * nL), 256, 0, s>>>(3 * nL, (const double*)c0, (const double*)c1, th, (double*)cb);
    else
      k_wind<float><<<vgrid_adv(3 * nL), 256, 0, s>>>(3 * nL, (const float*)c0, (const float*)c1, (float)th,
                                                     (float*)cb);
    return cb;
  };
  auto eval = [&](double t, const void* win) -> int {   // z = QQ^T C(c(t)) win
    const void* c = wind(t);
    SEM_LAUNCH_CHECK();
    SEM_TRY(advect_apply(C, prec, c, win, zb, ncomp, s));
    for (int q = 0; q < ncomp; ++q) SEM_TRY(gs_apply(L, vp, static_cast<char*>(zb) + q * nL * esz, false, s));
    return SEM_OK;
  };
  auto stage = [&](double cw, int mode) -> int {
    if (vp == SEM_FP64)
      k_rk_stage<double><<<vgrid_adv(n), 256, 0, s>>>(n, nL, (const double*)zb, A.minv, (double*)w, (double*)wsb,
                                                      (double*)accb, cw, mode);
    else
      k_rk_stage<float><<<vgrid_adv(n), 256, 0, s>>>(n, nL, (const float*)zb, A.minv32, (float*)w, (float*)wsb,
                                                     (float*)accb, (float)cw, mode);
    SEM_LAUNCH_CHECK();
    return SEM_OK;
  };
  for (int q = 0; q < nsub; ++q) {
    const double t = t0 + q * h;
    SEM_TRY(eval(t, w));
    SEM_TRY(stage(0.5 * h, 0));
    SEM_TRY(eval(t + 0.5 * h, wsb));
    SEM_TRY(stage(0.5 * h, 1));
    SEM_TRY(eval(t + 0.5 * h, wsb));
    SEM_TRY(stage(h, 1));
    SEM_TRY(eval(t + h, wsb));
    SEM_TRY(stage(h / 6.0, 2));
  }
  return SEM_OK;
}

}  // namespace sem
