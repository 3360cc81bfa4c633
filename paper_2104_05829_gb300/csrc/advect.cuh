// The dealiased advection operator, element by element (see advect.cu): the arithmetics, the 1-D passes
// and one element's work, for the kernel of advect.cu and for the elements that the digit kernel (advect_dig.cu)
// does not take.
#pragma once

#include "pairs.cuh"
#include "sem_internal.cuh"

namespace sem {

// Arithmetics of the advection kernel: V the working value, S the stored vectors (c, u, w), G
// the stored cubature factors and 1-D matrices. Plain FMA in FP64 or FP32; or FP32 pairs
// (pairs.cuh, about 48 significant bits) on FP64 vectors with pre-split factors. The pair
// form keeps its sums unnormalised (lo may exceed ulp(hi)/2): each value only enters the
// error-free additions and products of pairs.cuh and the FP64 join at the store. Where two
// computed values meet in a product the dropped lo * lo term then grows: errors rose from
// 1.5e-13 to 6.2e-13 against the oracle (N = 2..8), still far below the 3e-11 bar, for a
// 16 % faster kernel (normalising the derivatives alone cost more than it saved).
template <typename T>
struct AdvPlain {
  using V = T;
  using S = T;
  using G = T;
  __device__ static V ld(const S* p, size_t i) { return p[i]; }
  __device__ static void st(S* p, size_t i, V v) { p[i] = v; }
  __device__ static V lg(const G* p, size_t i) { return p[i]; }
  __device__ static V zero() { return T(0); }
  __device__ static V mac(V acc, V a, V b) { return fma(a, b, acc); }
  __device__ static V mul(V a, V b) { return a * b; }
  __device__ static V add(V a, V b) { return a + b; }
  __device__ static V sub(V a, V b) { return a - b; }
  __device__ static V norm(V a) { return a; }
  static V host(double x) { return (T)x; }
};

struct AdvPair {
  using V = ff;
  using S = double;
  using G = float2;
  __device__ static V ld(const S* p, size_t i) { return ff_split(p[i]); }
  __device__ static void st(S* p, size_t i, V v) { p[i] = ff_join(v); }
  __device__ static V lg(const G* p, size_t i) {
    const float2 g = p[i];
    return {g.x, g.y};
  }
  __device__ static V zero() { return {0.f, 0.f}; }
  __device__ static V mac(V acc, V a, V b) { return ff_mac(acc, a, b); }
  __device__ static V mul(V a, V b) { return ff_mul(a, b); }
  __device__ static V add(V a, V b) { return ff_add_u(a, b); }
  __device__ static V sub(V a, V b) { return ff_sub_u(a, b); }
  __device__ static V norm(V a) { return a; }
  static V host(double x) { return ff_host_split(x); }
};

__host__ __device__ constexpr int nq_of(int NP) { return (3 * NP + 1) / 2; }

template <int NP>
struct AdvShape {
  static constexpr int NQ = nq_of(NP);
  static constexpr int T = NQ * NQ;                      // threads per element
  static constexpr int RS = NQ % 2 == 0 ? NQ + 1 : NQ;   // padded row stride of the Gauss-point arrays
  static constexpr int PS = NQ * RS;                     // plane stride
};

// dynamic shared memory of k_advect<Ar, NP>
template <class Ar, int NP>
constexpr size_t advect_smem() {
  constexpr int NQ = AdvShape<NP>::NQ, PS = AdvShape<NP>::PS;
  return sizeof(typename Ar::V) * ((size_t)NQ * NP + NQ * NQ + NP * NP * NP + NP * NP * NQ + 2 * NQ * PS + 3 * NQ * NQ * NQ);
}

// 1-D operators in shared memory: Im [NQ][NP] (GLL -> Gauss), Dq [NQ][NQ]
template <class Ar, int NP, int NQ>
__device__ __forceinline__ void load_ops(const typename Ar::G* __restrict__ Im, const typename Ar::G* __restrict__ Dq,
                                         typename Ar::V* sI, typename Ar::V* sD) {
  for (int q = threadIdx.x; q < NQ * NP; q += blockDim.x) sI[q] = Ar::lg(Im, q);
  for (int q = threadIdx.x; q < NQ * NQ; q += blockDim.x) sD[q] = Ar::lg(Dq, q);
}

// Interpolate the element's nodal field src (in shared memory, [k][j][i]) to the
// Gauss points; thread (a, b) receives its t-line out[c] = f(z_a, z_b, z_c).
// Uses t1 [NP][NP][NQ] in shared memory.
template <class Ar, int NP, int NQ>
__device__ __forceinline__ void to_gauss(bool on, const typename Ar::V* src, typename Ar::V* t1, const typename Ar::V* sI,
                                         const typename Ar::V* cI, int a, int b, typename Ar::V (&out)[NQ]) {
  using T = typename Ar::V;
  // r-pass: t1[k][j][a] for j < NP (threads with b < NP); row a of I held in registers
  if (on && b < NP) {
    T ia[NP];
#pragma unroll
    for (int i = 0; i < NP; ++i) ia[i] = sI[a * NP + i];
#pragma unroll 2
    for (int k = 0; k < NP; ++k) {
      T acc = Ar::zero();
#pragma unroll
      for (int i = 0; i < NP; ++i) acc = Ar::mac(acc, ia[i], src[(k * NP + b) * NP + i]);
      t1[(k * NP + b) * NQ + a] = Ar::norm(acc);
    }
  }
  __syncthreads();
  if (!on) return;
  // s-pass into registers: t2[k] = sum_j I[b][j] t1[k][j][a]; row b of I in registers
  T t2[NP];
  {
    T ib[NP];
#pragma unroll
    for (int j = 0; j < NP; ++j) ib[j] = sI[b * NP + j];
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      T acc = Ar::zero();
#pragma unroll
      for (int j = 0; j < NP; ++j) acc = Ar::mac(acc, ib[j], t1[(k * NP + j) * NQ + a]);
      t2[k] = Ar::norm(acc);
    }
  }
  // t-pass in registers (cI: the interpolation matrix at compile-time indices)
#pragma unroll
  for (int c = 0; c < NQ; ++c) {
    T acc = Ar::zero();
#pragma unroll
    for (int k = 0; k < NP; ++k) acc = Ar::mac(acc, cI[c * NP + k], t2[k]);
    out[c] = Ar::norm(acc);
  }
}

// 1-D operators passed by value (kernel parameters: with fully unrolled loops the
// coefficients become constant-bank operands, no shared-memory loads): the
// interpolation Im [NQ][NP] and the even-odd pieces of the Gauss derivative Dq,
// which is centro-antisymmetric (Dq[NQ-1-a][NQ-1-b] = -Dq[a][b]): with
// H = NQ / 2, s_b = v_b + v_{NQ-1-b} and d_b = v_b - v_{NQ-1-b},
//   ev_a = sum_b ep[a][b] s_b (+ mc[a] v_H if NQ is odd), od_a = sum_b op[a][b] d_b,
//   (Dq v)_a = ev_a + od_a, (Dq v)_{NQ-1-a} = od_a - ev_a, (Dq v)_H = sum_b mr[b] d_b (NQ odd),
// ep = (Dq[a][b] + Dq[a][NQ-1-b]) / 2, op = (Dq[a][b] - Dq[a][NQ-1-b]) / 2.
template <typename T, int NP>
struct AdvOps {
  static constexpr int NQ = nq_of(NP), H = NQ / 2;
  T Im[NQ * NP];
  T ep[H * H], op[H * H], mc[H > 0 ? H : 1], mr[H > 0 ? H : 1];
};

template <class Ar, int NP>
__device__ __forceinline__ void eo_deriv(const AdvOps<typename Ar::V, NP>& P, const typename Ar::V (&v)[nq_of(NP)],
                                         typename Ar::V (&o)[nq_of(NP)]) {
  using T = typename Ar::V;
  constexpr int NQ = nq_of(NP), H = NQ / 2, N = NQ - 1;
  T sm[H], df[H];
#pragma unroll
  for (int b = 0; b < H; ++b) {
    sm[b] = Ar::add(v[b], v[N - b]);
    df[b] = Ar::sub(v[b], v[N - b]);
  }
#pragma unroll
  for (int a = 0; a < H; ++a) {
    T ev = Ar::zero(), od = Ar::zero();
#pragma unroll
    for (int b = 0; b < H; ++b) {
      ev = Ar::mac(ev, P.ep[a * H + b], sm[b]);
      od = Ar::mac(od, P.op[a * H + b], df[b]);
    }
    if (NQ % 2 == 1) ev = Ar::mac(ev, P.mc[a], v[H]);
    o[a] = Ar::add(ev, od);
    o[N - a] = Ar::sub(od, ev);
  }
  if (NQ % 2 == 1) {
    T m = Ar::zero();
#pragma unroll
    for (int b = 0; b < H; ++b) m = Ar::mac(m, P.mr[b], df[b]);
    o[H] = Ar::norm(m);
  }
}

// One element: thread (a, b) of the nq x nq plane (`on`; a block's other threads only meet the barriers).
// s_raw: advect_smem<Ar, NP>() bytes of shared memory.
template <class Ar, int NP>
__device__ __forceinline__ void advect_element(bool on, int a, int b, int e, unsigned char* s_raw, int ncomp, int64_t nL,
                                               const typename Ar::S* __restrict__ cv,
                                               const typename Ar::S* __restrict__ uv,
                                               const typename Ar::G* __restrict__ Gq,
                                               const typename Ar::G* __restrict__ Im,
                                               const typename Ar::G* __restrict__ Dq, typename Ar::S* __restrict__ wv,
                                               const AdvOps<typename Ar::V, NP>& P) {
  using T = typename Ar::V;
  constexpr int NQ = AdvShape<NP>::NQ, NP3 = NP * NP * NP, NQ2 = NQ * NQ, NQ3 = NQ2 * NQ;
  constexpr int RS = AdvShape<NP>::RS, PS = AdvShape<NP>::PS;
  // dynamic shared memory (advect_smem<Ar, NP>() bytes):
  T* sI = reinterpret_cast<T*>(s_raw);   // [NQ * NP] interpolation, runtime-indexed rows and columns
  T* sD = sI + NQ * NP;                  // [NQ * NQ]
  T* s_src = sD + NQ * NQ;               // [NP3] nodal field
  T* s_t1 = s_src + NP3;                 // [NP * NP * NQ] first interpolation pass; last projection pass
  T* s_U = s_t1 + NP * NP * NQ;          // [NQ * PS] u on the Gauss points; later the t-projected planes
  T* s_R = s_U + NQ * PS;                // [NQ * PS] a derivative, one direction at a time
  T* s_ch = s_R + NQ * PS;               // [3 * NQ3] the contravariant wind
  load_ops<Ar, NP, NQ>(Im, Dq, sI, sD);
  const size_t eb = (size_t)e * NP3;
  const typename Ar::G* G = Gq + (size_t)e * 9 * NQ3 + b * NQ + a;
  // 1-2. contravariant wind at this thread's points, kept in shared memory
  const int pt0 = b * NQ + a;   // point (a, b, c) at pt0 + c * NQ2
  if (on)
#pragma unroll
  for (int c = 0; c < NQ; ++c)
    s_ch[pt0 + c * NQ2] = s_ch[NQ3 + pt0 + c * NQ2] = s_ch[2 * NQ3 + pt0 + c * NQ2] = Ar::zero();
  for (int m = 0; m < 3; ++m) {
    __syncthreads();
    for (int q = threadIdx.x; q < NP3; q += blockDim.x) s_src[q] = Ar::ld(cv, (size_t)m * nL + eb + q);
    __syncthreads();
    T cf[NQ];
    to_gauss<Ar, NP, NQ>(on, s_src, s_t1, sI, P.Im, a, b, cf);
    if (on)
#pragma unroll
    for (int c = 0; c < NQ; ++c) {
      const int pt = pt0 + c * NQ2;
#pragma unroll
      for (int d = 0; d < 3; ++d)
        s_ch[d * NQ3 + pt] = Ar::mac(s_ch[d * NQ3 + pt], Ar::lg(G, (d * 3 + m) * NQ3 + c * NQ2), cf[c]);
    }
  }
  // 3. every advected component
  for (int comp = 0; comp < ncomp; ++comp) {
    __syncthreads();
    for (int q = threadIdx.x; q < NP3; q += blockDim.x) s_src[q] = Ar::ld(uv, (size_t)comp * nL + eb + q);
    __syncthreads();
    T uf[NQ];
    to_gauss<Ar, NP, NQ>(on, s_src, s_t1, sI, P.Im, a, b, uf);
    T conv[NQ];
    if (on) {
#pragma unroll
      for (int c = 0; c < NQ; ++c) s_U[c * PS + b * RS + a] = uf[c];
      T ut[NQ];
      eo_deriv<Ar, NP>(P, uf, ut);   // t-derivative along this thread's line
#pragma unroll
      for (int c = 0; c < NQ; ++c) conv[c] = Ar::mul(s_ch[2 * NQ3 + pt0 + c * NQ2], ut[c]);
    }
    __syncthreads();
    // r-derivative on the line (plane c = b, row j = a) -> s_R
    if (on) {
      T v[NQ], o[NQ];
      const int rb = a, rc = b;
#pragma unroll
      for (int m = 0; m < NQ; ++m) v[m] = s_U[rc * PS + rb * RS + m];
      eo_deriv<Ar, NP>(P, v, o);
#pragma unroll
      for (int m = 0; m < NQ; ++m) s_R[rc * PS + rb * RS + m] = o[m];
    }
    __syncthreads();
    if (on)
#pragma unroll
      for (int c = 0; c < NQ; ++c) conv[c] = Ar::mac(conv[c], s_ch[pt0 + c * NQ2], s_R[c * PS + b * RS + a]);
    __syncthreads();
    // s-derivative on the column (plane c = b, column i = a) -> s_R
    if (on) {
      T v[NQ], o[NQ];
      const int sa = a, sc = b;
#pragma unroll
      for (int m = 0; m < NQ; ++m) v[m] = s_U[sc * PS + m * RS + sa];
      eo_deriv<Ar, NP>(P, v, o);
#pragma unroll
      for (int m = 0; m < NQ; ++m) s_R[sc * PS + m * RS + sa] = o[m];
    }
    __syncthreads();
    if (on) {
#pragma unroll
      for (int c = 0; c < NQ; ++c)
        conv[c] = Ar::norm(Ar::mac(conv[c], s_ch[NQ3 + pt0 + c * NQ2], s_R[c * PS + b * RS + a]));
      // back to the GLL points: t-pass from registers into v2[k][b][a] (s_U reused)
#pragma unroll
      for (int k = 0; k < NP; ++k) {
        T acc = Ar::zero();
#pragma unroll
        for (int c = 0; c < NQ; ++c) acc = Ar::mac(acc, P.Im[c * NP + k], conv[c]);
        s_U[k * PS + b * RS + a] = Ar::norm(acc);
      }
    }
    __syncthreads();
    // s-pass: v1[k][j][a] = sum_b I[b][j] v2[k][b][a] (threads with b < NP own j = b)
    if (on && b < NP) {
      T cb[NQ];   // column b of I
#pragma unroll
      for (int q = 0; q < NQ; ++q) cb[q] = sI[q * NP + b];
#pragma unroll 2
      for (int k = 0; k < NP; ++k) {
        T acc = Ar::zero();
#pragma unroll
        for (int q = 0; q < NQ; ++q) acc = Ar::mac(acc, cb[q], s_U[k * PS + q * RS + a]);
        s_t1[(k * NP + b) * NQ + a] = Ar::norm(acc);
      }
    }
    __syncthreads();
    // r-pass: w[k][j][i] = sum_a I[a][i] v1[k][j][a] (threads (i, j) = (a, b) with a, b < NP)
    if (on && a < NP && b < NP) {
      typename Ar::S* out = wv + (size_t)comp * nL + eb;
      T ca[NQ];   // column a of I
#pragma unroll
      for (int q = 0; q < NQ; ++q) ca[q] = sI[q * NP + a];
#pragma unroll 2
      for (int k = 0; k < NP; ++k) {
        T acc = Ar::zero();
#pragma unroll
        for (int q = 0; q < NQ; ++q) acc = Ar::mac(acc, ca[q], s_t1[(k * NP + b) * NQ + q]);
        Ar::st(out, (size_t)(k * NP + b) * NP + a, acc);
      }
    }
  }
}

// the 1-D operators as kernel parameters
template <class Ar, int NP>
AdvOps<typename Ar::V, NP> adv_ops(const AdvData& A) {
  constexpr int NQ = nq_of(NP), H = NQ / 2, N = NQ - 1;
  AdvOps<typename Ar::V, NP> P{};
  for (int q = 0; q < NQ * NP; ++q) P.Im[q] = Ar::host(A.hIm[q]);
  auto d = [&](int r, int q) { return A.hDq[r * NQ + q]; };
  for (int r = 0; r < H; ++r)
    for (int q = 0; q < H; ++q) {
      P.ep[r * H + q] = Ar::host(0.5 * (d(r, q) + d(r, N - q)));
      P.op[r * H + q] = Ar::host(0.5 * (d(r, q) - d(r, N - q)));
    }
  if (NQ % 2 == 1)
    for (int r = 0; r < H; ++r) {
      P.mc[r] = Ar::host(d(r, H));
      P.mr[r] = Ar::host(d(H, r));
    }
  return P;
}

}  // namespace sem
