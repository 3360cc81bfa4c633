// Jacobi-PCG of a small mesh in one cooperative launch: every element's block stays on the chip for the whole solve.
//
// What bounds a small solve is the chain of launches: on a 4^3 box of order 7 (32,768 points) an iteration as five kernels
// (operator, gather-scatter, two reductions, direction) takes 34 us, of which the operator's own chain is about 5.
// Here a block (DigShape<NP>::T threads) owns an element: x, r, p and D^-1 of its points stay in registers, the operator is
// the digit form (ax_dig.cuh), and an iteration has two grid barriers:
//   1. p -> w = A^e p, stored; the element's part of (p, A p) = sum over the copies of p w (w not yet summed), stored;
//   barrier; the gather-scatter as a gather (each point adds its copies in ascending order, as gs.cu does); alpha;
//   2. x, r updated; the element's parts of (r, r) and (r, D^-1 r), stored;
//   barrier; beta, p.
// Every block adds all the parts in the same fixed order, so all take the same alpha and beta and leave in the same
// iteration. A wait is bounded (sem_opts.spin_limit). x, r and the scalars are written only once all blocks are through (jac_commit); when
// a wait gives up, all blocks leave without a write to them, and the kernels without waits take the solve over from there.
// Measured, an iteration: N = 7, one element 32.8 -> 11 to 12 us, 4^3 36.9 -> 14.7, 6^3 42.5 -> 18.2, 8^3 55.0 -> 25.4 (the manufactured
// 4^3 solve 6.9 -> 2.73 ms). What is left at one element is latency: the operator's chain, two barriers and four
// reductions; at four elements an SM the FP64 instructions of the vector work (about 400 a block, 16 cycles each), so sums
// are formed by one warp where one is enough and the quotients by one lane.
#include "ax_dig.cuh"
#include "sem_internal.cuh"

namespace sem {

namespace {

struct JacArgs {
  double *x, *r, *p, *w;
  const double *dinv, *h1L, *G;
  const int2* Gx;
  const int32_t* gexp;
  const DigTab* tab;
  const uint8_t* own;
  const int2* seg;       // per point: position of its node's copies in idx, count (0: the only copy); Dirichlet: bit 31
  const int32_t* idx;
  double *part, *sc;
  unsigned* bar;         // arrivals so far; then blocks that are through
  int* state;            // 0: under way, JAC_GIVEN_UP, JAC_THROUGH
  long long spin;
  double h1, h2;
  int kexp, span, mass, e1, maxit;
};

constexpr int JAC_DIR = INT32_MIN;
constexpr int JAC_GIVEN_UP = 1, JAC_THROUGH = 2;

// Blocks an SM: registers for the vectors next to the operator's.
constexpr int JAC_MIN_BLOCKS = 4;

__global__ void k_jac_seg(int64_t nseg, const int32_t* __restrict__ off, const int32_t* __restrict__ idx,
                          const uint8_t* __restrict__ sdir, int2* __restrict__ seg) {
  const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (q >= nseg) return;
  const int b = off[q], e = off[q + 1];
  for (int t = b; t < e; ++t) seg[idx[t]] = make_int2(b, sdir[q] ? JAC_DIR : e - b);
}

// Arrive at the grid barrier (one thread, its block's stores behind a block barrier) and wait for the others: false when a
// wait gave up here or in another block.
__device__ __forceinline__ bool jac_arrive_wait(const JacArgs& a, unsigned target) {
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(a.bar) : "memory");
  const long long t0 = clock64();
  unsigned polls = 0, v;
  while (true) {
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a.bar) : "memory");
    if ((int)(v - target) >= 0) return true;
    const bool late = clock64() - t0 > a.spin;
    if (late) atomicCAS(a.state, 0, JAC_GIVEN_UP);
    if ((late || (++polls & 63u) == 0) && *(volatile int*)a.state != 0) return false;
  }
}

// Whether this launch's result counts, the same answer in every block (one thread each): `state` leaves 0 once, to JAC_THROUGH by
// the last block that is through its iterations, to JAC_GIVEN_UP by the first wait that gives up, here or at a barrier.
__device__ __forceinline__ bool jac_commit(const JacArgs& a, unsigned* through, unsigned E) {
  if (atomicAdd(through, 1u) == E - 1) atomicCAS(a.state, 0, JAC_THROUGH);
  const long long t0 = clock64();
  int v;
  while ((v = *(volatile int*)a.state) == 0)
    if (clock64() - t0 > a.spin) atomicCAS(a.state, 0, JAC_GIVEN_UP);
  return v == JAC_THROUGH;
}

__device__ __forceinline__ double jac_warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// the sum of E parts, by one warp, in every lane
__device__ __forceinline__ double jac_sum_parts(const double* part, int E) {
  double v = 0.0;
#pragma unroll 4
  for (int q = threadIdx.x & 31; q < E; q += 32) v += __ldcg(part + q);
  return jac_warp_sum(v);
}

template <int NP, bool VARH1>
__global__ void __launch_bounds__(DigShape<NP>::T, JAC_MIN_BLOCKS)
    k_jacobi_dig(const __grid_constant__ JacArgs a, const __grid_constant__ EOMat<ArF64> Df,
                 const __grid_constant__ EOMat<ArF64> Dt) {
  using S = DigShape<NP>;
  constexpr int NP2 = NP * NP, NP3 = NP2 * NP;
  __shared__ __align__(16) unsigned long long smem[S::SMEM];
  __shared__ uint32_t s_max[4][4];
  __shared__ double s_red[2][4], s_bc[4];
  __shared__ int s_ok;
  if (a.sc[S_DONE] != 0.0) return;
  const int e = blockIdx.x, E = gridDim.x;
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const int g = lane >> 2, k0 = 2 * wp, i0 = 2 * (lane & 3);
  const int64_t at = (int64_t)e * NP3 + (k0 * NP + g) * NP + i0;
  auto has = [&](int p, int x) { return g < NP && i0 + x < NP && k0 + p < NP; };
  double xv[2][2], rv[2][2], pv[2][2], dv[2][2], zv[2][2] = {};
  bool ov[2][2];
#pragma unroll
  for (int p = 0; p < 2; ++p)
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      const bool h = has(p, x);
      const int64_t l = at + p * NP2 + x;
      xv[p][x] = h ? a.x[l] : 0.0;
      rv[p][x] = h ? a.r[l] : 0.0;
      pv[p][x] = h ? a.p[l] : 0.0;
      dv[p][x] = h ? a.dinv[l] : 0.0;
      ov[p][x] = h && a.own[l] != 0;
    }
  const double tol2 = a.sc[S_TOL2], rz0 = a.sc[S_RZ];
  double rz = rz0, rr = a.sc[S_RR], alpha = 0.0, beta = 0.0, pw = 0.0;
  bool done = false, bad = false, ok = true;
  int it = 0;
  unsigned target = 0;
  while (it < a.maxit && !done && !bad) {
    // p in memory for elements that fixed point cannot hold
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
      for (int x = 0; x < 2; ++x)
        if (has(p, x)) a.p[at + p * NP2 + x] = pv[p][x];
    double o[2][2];
    const bool held = dig_element<NP, VARH1, true>(e, a.p, a.w, a.Gx, a.gexp, a.G, a.tab, a.kexp, a.h1, a.h2, a.h1L, a.span, 0,
                                                   a.mass, a.e1, Df, Dt, smem, s_max, pv, o);
    if (!held) __syncthreads();
    double s1 = 0.0;
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        if (!has(p, x)) continue;
        if (!held) o[p][x] = __ldcg(a.w + at + p * NP2 + x);
        s1 = fma(pv[p][x], o[p][x], s1);
      }
    s1 = jac_warp_sum(s1);
    if (lane == 0) s_red[0][wp] = s1;
    target += E;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = s_red[0][0];
#pragma unroll
      for (int q = 1; q < S::NW; ++q) t += s_red[0][q];
      a.part[e] = t;
      s_ok = jac_arrive_wait(a, target);
    }
    __syncthreads();
    if (!(ok = s_ok != 0)) break;
    // (p, A p) and alpha by one warp, for the others to read
    if (wp == 0) {
      const double t = jac_sum_parts(a.part, E);
      if (lane == 0) {
        s_bc[0] = t;
        s_bc[1] = rz / t;
      }
    }
    // the sums of the copies
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const int2 sg = has(p, x) ? a.seg[at + p * NP2 + x] : make_int2(0, 0);
        const int few = sg.y <= 8 ? sg.y : 0;
        double v[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) v[t] = t < few ? __ldcg(a.w + a.idx[sg.x + t]) : 0.0;
        const int most = __reduce_max_sync(0xffffffffu, few);   // fewer FP64 instructions where no lane needs them
        if (few > 0) {
          double t1 = v[0] + v[1];
          if (most > 2) {
#pragma unroll
            for (int t = 2; t < 4; ++t)
              if (t < few) t1 += v[t];
            if (most > 4) {
#pragma unroll
              for (int t = 4; t < 8; ++t)
                if (t < few) t1 += v[t];
            }
          }
          o[p][x] = t1;
        } else if (sg.y > 8) {
          double t1 = __ldcg(a.w + a.idx[sg.x]);
          for (int t = 1; t < sg.y; ++t) t1 += __ldcg(a.w + a.idx[sg.x + t]);
          o[p][x] = t1;
        } else if (sg.y == JAC_DIR) {
          o[p][x] = 0.0;
        }
      }
    __syncthreads();
    pw = s_bc[0];
    if (!(pw > 0.0) || !isfinite(pw)) {
      bad = true;
      alpha = 0.0;
      break;
    }
    alpha = s_bc[1];
    double s2[2] = {0.0, 0.0};
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        if (!has(p, x)) continue;
        xv[p][x] = fma(alpha, pv[p][x], xv[p][x]);
        const double rl = fma(-alpha, o[p][x], rv[p][x]);
        rv[p][x] = rl;
        zv[p][x] = dv[p][x] * rl;
        if (ov[p][x]) {
          s2[0] = fma(rl, rl, s2[0]);
          s2[1] = fma(rl, zv[p][x], s2[1]);
        }
      }
    // both sums in one set of additions: the lower half-warp carries (r, r), the upper (r, D^-1 r)
    double t2 = lane < 16 ? s2[0] : s2[1];
    t2 += __shfl_xor_sync(0xffffffffu, lane < 16 ? s2[1] : s2[0], 16);
#pragma unroll
    for (int q = 8; q > 0; q >>= 1) t2 += __shfl_xor_sync(0xffffffffu, t2, q);
    if ((lane & 15) == 0) s_red[lane >> 4][wp] = t2;
    target += E;
    __syncthreads();
    if (wp == 0) {
      if (lane < 2) {
        double t = s_red[lane][0];
#pragma unroll
        for (int q = 1; q < S::NW; ++q) t += s_red[lane][q];
        a.part[(1 + lane) * E + e] = t;
      }
      __syncwarp();
      if (lane == 0) s_ok = jac_arrive_wait(a, target);
    }
    __syncthreads();
    if (!(ok = s_ok != 0)) break;
    if (wp == 0) {
      const double t = jac_sum_parts(a.part + E, E);
      if (lane == 0) s_bc[2] = t;
    } else if (wp == 1) {
      const double t = jac_sum_parts(a.part + 2 * E, E);
      if (lane == 0) {
        s_bc[0] = t;
        s_bc[3] = t / rz;
      }
    }
    __syncthreads();
    rr = s_bc[2];
    rz = s_bc[0];
    beta = s_bc[3];
    ++it;
    bad = !isfinite(rr);
    done = rr <= tol2;
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
      for (int x = 0; x < 2; ++x) pv[p][x] = fma(beta, pv[p][x], zv[p][x]);
  }
  if (!ok) return;
  if (threadIdx.x == 0) s_ok = jac_commit(a, a.bar + 2, E);
  __syncthreads();
  if (!s_ok) return;
#pragma unroll
  for (int p = 0; p < 2; ++p)
#pragma unroll
    for (int x = 0; x < 2; ++x)
      if (has(p, x)) {
        const int64_t l = at + p * NP2 + x;
        a.x[l] = xv[p][x];
        a.r[l] = rv[p][x];
        a.p[l] = pv[p][x];
      }
  if (e == 0 && threadIdx.x == 0) {
    a.sc[S_PW] = pw;
    a.sc[S_ALPHA] = alpha;
    a.sc[S_BETA] = beta;
    a.sc[S_RZ] = rz;
    a.sc[S_RR] = rr;
    a.sc[S_ITER] += it;
    a.sc[S_TOTAL] += it;
    if (bad) a.sc[S_BREAK] = 1.0;
    if (bad || done) a.sc[S_DONE] = 1.0;
  }
}

}  // namespace

// Iterations of a started Jacobi-PCG (pcg_begin_tol), at most maxit >= 1 of them, in one cooperative launch, where the mesh's
// blocks fit on the device together. seg: room for 2 nL 32-bit words. *used: false when the solve takes the launches. A launch whose
// waits gave up leaves x, r and the scalars as they were (S_ITER and S_DONE tell) and p undefined: jacobi_dig_resume makes it D^-1 r.
//
// The rule. All blocks must be resident, four on an SM: up to 608 elements on 152 SMs. It is the faster form over that whole
// range (N = 7, 8 x 8 x 9 elements: 27.1 against 57.2 us an iteration; N = 4, 5, 6, 8^3: 21.2, 22.4, 24.6 against 43.0, 44.1, 49.1).
// A spin limit under a millisecond could run out in an ordinary solve: it keeps the launches, which have no waits. A limit of
// zero does not: every barrier gives up at the first poll that finds a block missing, and the launches take over.
int jacobi_dig_solve(Ctx& C, const Level& L, double* x, double* r, double* p, double* w, const double* dinv, double h1,
                     double h2, const double* h1L, bool pairs, int2* seg, double* sc, int maxit, bool start, cudaStream_t s,
                     bool* used) {
  *used = false;
  if (!L.Gx || (L.spin_limit != 0 && L.spin_limit < (1ll << 21)) || L.E > JAC_MAX_E) return SEM_OK;
  int dev = 0, nsm = 0, coop = 0, per_sm = 0;
  SEM_CUDA_TRY(cudaGetDevice(&dev));
  SEM_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  SEM_CUDA_TRY(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
  if (!coop || L.E > JAC_MIN_BLOCKS * nsm) return SEM_OK;
  const void* f = nullptr;
  int threads = 0;
  switch (L.NP) {
#define CASE(NP)                                                                                     \
  case NP:                                                                                           \
    f = h1L ? (const void*)k_jacobi_dig<NP, true> : (const void*)k_jacobi_dig<NP, false>;            \
    threads = DigShape<NP>::T;                                                                       \
    break;
    CASE(5) CASE(6) CASE(7) CASE(8)
#undef CASE
    default: return SEM_OK;
  }
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, threads, 0) != cudaSuccess) {
    cudaGetLastError();
    return SEM_OK;
  }
  if (L.E > per_sm * nsm) return SEM_OK;
  JacArgs a;
  a.x = x;
  a.r = r;
  a.p = p;
  a.w = w;
  a.dinv = dinv;
  a.h1L = h1L;
  a.G = L.G;
  a.Gx = L.Gx;
  a.gexp = L.gexp;
  a.tab = L.dig;
  a.own = L.owner;
  a.seg = seg;
  a.idx = L.seg_idx;
  a.part = C.jac;
  a.sc = sc;
  unsigned* sync = reinterpret_cast<unsigned*>(C.jac + 3 * JAC_MAX_E);
  a.bar = sync;
  a.state = reinterpret_cast<int*>(sync + 1);
  a.spin = L.spin_limit;
  a.h1 = h1L ? 1.0 : h1;
  a.h2 = h2;
  a.kexp = L.dig_kexp;
  a.span = dig_h1_span(pairs);
  a.mass = h2 != 0.0 ? 1 : 0;
  a.e1 = h1L ? 0 : dig_h1_exp(h1);
  a.maxit = maxit;
  EOMat<ArF64> Df, Dt;
  make_eo<ArF64>(L.D.a, L.NP, false, Df);
  make_eo<ArF64>(L.D.a, L.NP, true, Dt);
  if (start) {
    SEM_CUDA_TRY(cudaMemsetAsync(seg, 0, (size_t)L.nL * sizeof(int2), s));
    if (L.n_seg)
      k_jac_seg<<<(unsigned)((L.n_seg + 255) / 256), 256, 0, s>>>(L.n_seg, L.seg_off, L.seg_idx, L.seg_dir, seg);
    SEM_LAUNCH_CHECK();
  }
  SEM_CUDA_TRY(cudaMemsetAsync(sync, 0, 3 * sizeof(unsigned), s));
  void* args[] = {&a, &Df, &Dt};
  const cudaError_t rc = cudaLaunchCooperativeKernel(f, dim3(L.E), dim3(threads), args, 0, s);
  if (rc == cudaErrorCooperativeLaunchTooLarge) {   // a part of the device only (MPS, green contexts): the launches
    cudaGetLastError();
    return SEM_OK;
  }
  SEM_CUDA_TRY(rc);
  *used = true;
  return SEM_OK;
}

// p = D^-1 r, the start of the iteration from x and r, after a launch that gave up.
int jacobi_dig_resume(const Level& L, double* p, const double* r, const double* dinv, double* sc, cudaStream_t s) {
  SEM_CUDA_TRY(cudaMemsetAsync(p, 0, (size_t)L.nL * sizeof(double), s));
  SEM_CUDA_TRY(cudaMemsetAsync(sc + S_BETA, 0, sizeof(double), s));
  return kr_direction_jacobi(L, SEM_FP64, p, r, dinv, sc, s);   // D^-1 r + beta 0
}

}  // namespace sem
