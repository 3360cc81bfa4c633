// Even-odd element operator A^e = D^T h1 G D + h2 B (eq. Ae): the arithmetic back ends, the
// 1-D transforms and one element's work, for the kernels of ax_eo.cu and for the elements
// that the digit kernel (ax_dig.cu) does not take. The even-odd form is described in ax_eo.cu.
#pragma once

#include "pairs.cuh"
#include "sem_internal.cuh"

namespace sem {

// ---- arithmetic back ends ------------------------------------------------------
struct ArF64 {
  static constexpr bool kPairs = false;
  using V = double;
  using GT = double;
  __device__ static V in(const double* u, size_t i) { return u[i]; }
  __device__ static void out(double* w, size_t i, V v) { w[i] = v; }
  __device__ static V gl(const GT* G, size_t i) { return G[i]; }
  __device__ static V zero() { return 0.0; }
  __device__ static V add(V a, V b) { return a + b; }
  __device__ static V sub(V a, V b) { return a - b; }
  __device__ static V add_u(V a, V b) { return a + b; }
  __device__ static V sub_u(V a, V b) { return a - b; }
  __device__ static V mul(V a, V b) { return a * b; }
  __device__ static V mac(V acc, V a, V b) { return fma(a, b, acc); }
  __device__ static V tidy(V a) { return a; }
  __device__ static V tidy_before_add(V a) { return a; }
  static V host(double x) { return x; }
};

struct ArPair {
  static constexpr bool kPairs = true;
  using V = ff;
  using GT = float2;
  __device__ static V in(const double* u, size_t i) { return ff_split(u[i]); }
  // the FP64 addition in ff_join rounds hi + lo correctly without renormalising first
  __device__ static void out(double* w, size_t i, V v) { w[i] = ff_join(v); }
  __device__ static V gl(const GT* G, size_t i) {
    const float2 g = G[i];
    return {g.x, g.y};
  }
  __device__ static V zero() { return {0.f, 0.f}; }
  __device__ static V add(V a, V b) { return ff_add(a, b); }
  __device__ static V sub(V a, V b) { return ff_sub(a, b); }
  // the additions inside the even-odd line transforms, whose results only enter further
  // error-free additions and products, skip the renormalisation
  __device__ static V add_u(V a, V b) { return ff_add_u(a, b); }
  __device__ static V sub_u(V a, V b) { return ff_sub_u(a, b); }
  __device__ static V mul(V a, V b) { return ff_mul(a, b); }
  __device__ static V mac(V acc, V a, V b) { return ff_mac(acc, a, b); }
  __device__ static V tidy(V a) { return ff_norm(a); }
  // values that next enter the error-free additions of eo_apply need no renormalising
  __device__ static V tidy_before_add(V a) { return a; }
  static V host(double x) { return ff_host_split(x); }
};

template <class Ar>
struct EOMat {
  typename Ar::V ep[36];   // E[a][b], a, b < H
  typename Ar::V op[36];   // O[a][b]
  typename Ar::V mc[6];    // D[a][m]: the middle input's weight in ev_a (N even)
  typename Ar::V mr[6];    // D[m][b]: the middle output's weights on d_b (N even)
};

template <int NP>
struct Pad3 {
  // row stride NP+1 for even NP; plane stride chosen so that rows of
  // successive planes start on different banks
  static constexpr int RS = (NP % 2 == 0) ? NP + 1 : NP;
  static constexpr int PS = NP * RS + ((NP * RS) % 2 == 0 ? 2 : 1);
  static constexpr int ES = NP * PS;
};

// Blocks per SM requested from the register allocator: at N = 7 four 192-thread blocks (at
// most 85 registers; five made the pair kernel spill and run slower). The pair kernel at other
// orders: three blocks, four at N = 9 (one 100-thread element per block there), against the
// register allocator's default of one or two blocks of up to 255 registers: at 16.8M points
// N = 3, 5, 11 took 0.390, 0.416, 1.347 ms with one block and 0.334, 0.371, 0.749 ms with three,
// and N = 8, 9, 10 took 0.518, 0.848, 0.625 ms with two blocks and 0.453, 0.634 (four),
// 0.492 ms; the FP64 kernel is bound by its pipe at any occupancy.
template <class Ar, int NP>
__host__ __device__ constexpr int eo_min_blocks() {
  return NP == 8 ? 4 : (Ar::kPairs ? (NP == 10 ? 4 : 3) : 1);
}

template <int NP>
__host__ __device__ constexpr int eo_epb() {
  int e = 256 / (NP * NP);
  if (e < 1) e = 1;
  while (e > 1 && (size_t)(3 * e * Pad3<NP>::ES) * 8 > 46 * 1024) --e;
  return e;
}

template <class Ar, int NP>
__device__ __forceinline__ void eo_apply(const EOMat<Ar>& M, const typename Ar::V (&v)[NP],
                                         typename Ar::V (&o)[NP]) {
  using V = typename Ar::V;
  constexpr int H = NP / 2, N = NP - 1;
  V s[H], d[H];
#pragma unroll
  for (int b = 0; b < H; ++b) {
    s[b] = Ar::add_u(v[b], v[N - b]);
    d[b] = Ar::sub_u(v[b], v[N - b]);
  }
#pragma unroll
  for (int a = 0; a < H; ++a) {
    V ev = Ar::mul(M.ep[a * H], s[0]);
    V od = Ar::mul(M.op[a * H], d[0]);
#pragma unroll
    for (int b = 1; b < H; ++b) {
      ev = Ar::mac(ev, M.ep[a * H + b], s[b]);
      od = Ar::mac(od, M.op[a * H + b], d[b]);
    }
    if (NP % 2 == 1) ev = Ar::mac(ev, M.mc[a], v[H]);
    o[a] = Ar::add_u(ev, od);
    o[N - a] = Ar::sub_u(od, ev);
  }
  if (NP % 2 == 1) {
    V m = Ar::mul(M.mr[0], d[0]);
#pragma unroll
    for (int b = 1; b < H; ++b) m = Ar::mac(m, M.mr[b], d[b]);
    o[H] = Ar::tidy(m);
  }
}

// One element by the even-odd transforms: thread (i, j) of its plane holds the t-line; A, B, Cc
// are its padded shared arrays of Pad3<NP>::ES values. Every thread of the block calls it
// (block barriers); `on`: the thread owns lines, `active`: the element exists.
template <class Ar, int NP, bool VARH1>
__device__ __forceinline__ void eo_element(bool on, bool active, int i, int j, size_t ebase,
                                           const double* __restrict__ u, double* __restrict__ w,
                                           const typename Ar::GT* __restrict__ Ge0, const EOMat<Ar>& Df,
                                           const EOMat<Ar>& Dt, typename Ar::V h1, typename Ar::V h2,
                                           const double* __restrict__ h1L, typename Ar::V* A, typename Ar::V* B,
                                           typename Ar::V* Cc) {
  using V = typename Ar::V;
  constexpr int NP2 = NP * NP, NP3 = NP2 * NP;
  constexpr int RS = Pad3<NP>::RS, PS = Pad3<NP>::PS;
  const int ij = j * NP + i;

  // phase 0: the element into registers (own t-line) and shared memory
  V ru[NP];
  if (on) {
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      ru[k] = active ? Ar::in(u, ebase + k * NP2 + ij) : Ar::zero();
      A[k * PS + j * RS + i] = ru[k];
    }
  }
  __syncthreads();

  // phase 1: u_t (own line), u_r (row k = i, j), u_s (column k = i, i' = j)
  V ut[NP];
  if (on) {
    eo_apply<Ar, NP>(Df, ru, ut);
    V v[NP], o[NP];
#pragma unroll
    for (int l = 0; l < NP; ++l) v[l] = A[i * PS + j * RS + l];
    eo_apply<Ar, NP>(Df, v, o);
#pragma unroll
    for (int l = 0; l < NP; ++l) B[i * PS + j * RS + l] = o[l];
#pragma unroll
    for (int l = 0; l < NP; ++l) v[l] = A[i * PS + l * RS + j];
    eo_apply<Ar, NP>(Df, v, o);
#pragma unroll
    for (int l = 0; l < NP; ++l) Cc[i * PS + l * RS + j] = o[l];
  }
  __syncthreads();

  // phase 2: pointwise G-combine, in place
  if (active) {
    const typename Ar::GT* Ge = Ge0 + ij;
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      const int o = k * NP2;
      const V ur = B[k * PS + j * RS + i], us = Cc[k * PS + j * RS + i], uq = ut[k];
      const V g11 = Ar::gl(Ge, 0 * NP3 + o), g12 = Ar::gl(Ge, 1 * NP3 + o), g13 = Ar::gl(Ge, 2 * NP3 + o);
      const V g22 = Ar::gl(Ge, 3 * NP3 + o), g23 = Ar::gl(Ge, 4 * NP3 + o), g33 = Ar::gl(Ge, 5 * NP3 + o);
      V wr = Ar::mac(Ar::mac(Ar::mul(g11, ur), g12, us), g13, uq);
      V ws = Ar::mac(Ar::mac(Ar::mul(g12, ur), g22, us), g23, uq);
      V wt = Ar::mac(Ar::mac(Ar::mul(g13, ur), g23, us), g33, uq);
      if (VARH1) {
        const V hh = Ar::in(h1L, ebase + o + ij);
        wr = Ar::mul(wr, hh);
        ws = Ar::mul(ws, hh);
        wt = Ar::mul(wt, hh);
      }
      B[k * PS + j * RS + i] = Ar::tidy_before_add(wr);
      Cc[k * PS + j * RS + i] = Ar::tidy_before_add(ws);
      ut[k] = Ar::tidy_before_add(wt);
    }
  }
  __syncthreads();

  // phase 3a: D_t^T on the own line, D_r^T on row (k = i, j) -> A
  V ot[NP];
  if (on) {
    eo_apply<Ar, NP>(Dt, ut, ot);
    V v[NP], o[NP];
#pragma unroll
    for (int l = 0; l < NP; ++l) v[l] = B[i * PS + j * RS + l];
    eo_apply<Ar, NP>(Dt, v, o);
#pragma unroll
    for (int l = 0; l < NP; ++l) A[i * PS + j * RS + l] = o[l];
  }
  __syncthreads();
  // phase 3b: D_s^T on column (k = i, i' = j) -> B
  if (on) {
    V v[NP], o[NP];
#pragma unroll
    for (int l = 0; l < NP; ++l) v[l] = Cc[i * PS + l * RS + j];
    eo_apply<Ar, NP>(Dt, v, o);
#pragma unroll
    for (int l = 0; l < NP; ++l) B[i * PS + l * RS + j] = o[l];
  }
  __syncthreads();

  // phase 4: w = h1 (D^T G D u) + h2 B u
  if (active) {
    const typename Ar::GT* Be = Ge0 + 6 * NP3 + ij;
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      const V st = Ar::add_u(Ar::add_u(A[k * PS + j * RS + i], B[k * PS + j * RS + i]), ot[k]);
      const V hb = Ar::mul(Ar::mul(h2, Ar::gl(Be, k * NP2)), ru[k]);
      Ar::out(w, ebase + k * NP2 + ij, VARH1 ? Ar::add(st, hb) : Ar::mac(hb, h1, st));
    }
  }
}

template <class Ar>
void make_eo(const double* D, int NP, bool transpose, EOMat<Ar>& M) {
  const int H = NP / 2, N = NP - 1, m = NP / 2;
  auto at = [&](int a, int b) { return transpose ? D[b * NP + a] : D[a * NP + b]; };
  for (int q = 0; q < 36; ++q) M.ep[q] = M.op[q] = Ar::host(0.0);
  for (int q = 0; q < 6; ++q) M.mc[q] = M.mr[q] = Ar::host(0.0);
  for (int a = 0; a < H; ++a)
    for (int b = 0; b < H; ++b) {
      M.ep[a * H + b] = Ar::host(0.5 * (at(a, b) + at(a, N - b)));
      M.op[a * H + b] = Ar::host(0.5 * (at(a, b) - at(a, N - b)));
    }
  if (NP % 2 == 1)
    for (int a = 0; a < H; ++a) {
      M.mc[a] = Ar::host(at(a, m));
      M.mr[a] = Ar::host(at(m, a));
    }
}

}  // namespace sem
