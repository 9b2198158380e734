// Time steps of a small batch kept on chip: one warp holds one simulation in
// registers through all steps of a call (the partitioned solve of partition.h, lane c
// owning chunk c of L rows).
//
// Why.  On GB300 a warp issues at most one FP64 operation every 64 cycles, whatever its
// instruction-level parallelism (measured: one chain or eight, 32 lanes or one, the
// same 64), and one SM's FP64 unit serves four such warps at once.  The one-thread-
// per-simulation step (stepper.cu) gives a batch of 64 simulations two warps, each
// walking 2N dependent rows with a trip to memory at every row: 123 us for a step of
// N = 256, all latency.  Here the 32 lanes share the rows of a simulation, so the chain
// is 2L + corrections + the boundary reduction instead of 2N, the state never leaves
// the registers between steps and the steps of a call are one launch: systems are
// independent, so no step needs a grid-wide wait.
//
// One step, per lane (rows cL .. cL+L-1):
//   r = C (+ E phi(C), phi of the neighbouring rows by shuffles)
//   y_c = A_c^{-1} r_c (chunk sweeps), boundary unknowns by cyclic reduction over the
//   lanes (5 levels at most; levels whose couplings have decayed below 2^-100 are left
//   off), x = y - W lam - V rho, and for periodic ends the rank-1 or rank-2 correction.
//   Crank-Nicolson: B = 2 I - A, so C^{n+1} = A^{-1} B C = 2 A^{-1} C - C: the
//   right-hand side costs one operation per row instead of a 3- or 5-point stencil.
// Measured: periodic Crank-Nicolson diffusion, N = 256, 64 simulations, 200 steps:
// 24.6 ms before, 0.70 ms (3.4 us a step; its ~90 FP64 operations alone take 2.8 us).
// Coefficients sit in shared memory with the lane as the fastest index (row j of every
// chunk side by side), so a coefficient read is one conflict-free 256-byte access.
#include <algorithm>
#include <cmath>
#include <mutex>
#include <type_traits>
#include <vector>

#include "arith.cuh"
#include "partition.h"
#include "sb_internal.h"

namespace sb {
namespace {

constexpr int kLanes = 32;
constexpr int kMaxWarps = 8;
constexpr int kStepsPerLaunch = 4096;  // bounds the length of one launch

// Offsets (in doubles) of the image's sections; every row section is [j][value][lane].
struct ResidentLayout {
  int fwd, bwd, cor, cyc, e, T0, M, total;
};

__host__ __device__ inline ResidentLayout resident_layout(int PB, int L, int rank, bool ch, int NL) {
  const int Q = 2 * PB, R = L * kLanes;
  ResidentLayout l;
  int o = 0;
  l.fwd = o, o += (PB + 1) * R;
  l.bwd = o, o += PB * R;
  l.cor = o, o += Q * R;
  l.cyc = o, o += rank * R;
  l.e = o, o += (ch ? 3 : 0) * R;
  l.T0 = o, o += Q * Q * kLanes;
  l.M = o, o += NL * (Q * Q + 2 * Q * PB) * kLanes;
  l.total = o;
  return l;
}

// Scalars of the periodic correction: rank 1 uses v[0] = beta, v[1] = alpha; rank 2 the
// twelve values P, Q, S^{-1} of the factor.
struct CycScalars {
  double v[12];
};

__device__ __forceinline__ double shfl(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }

template <int PB, int L, int RANK, bool CN, bool CH>
__global__ void __launch_bounds__(kMaxWarps * 32, 1)
resident_steps_kernel(const double* __restrict__ image, int NL, int N, int64_t M, int64_t ld, double* state,
                      int nsteps, const __grid_constant__ CycScalars cs) {
  constexpr int Q = 2 * PB, W = PB + 1, K = kLanes - 1;
  extern __shared__ __align__(16) double img[];
  const ResidentLayout lay = resident_layout(PB, L, RANK, CH, NL);
  for (int k = threadIdx.x; k < lay.total; k += blockDim.x) img[k] = image[k];
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const double* fw = img + lay.fwd + lane;
  const double* bw = img + lay.bwd + lane;
  const double* co = img + lay.cor + lane;
  const double* cy = img + lay.cyc + lane;
  const double* ee = img + lay.e + lane;
  const int r0 = lane * L;
  const int cl = (N - 1) / L, jl = (N - 1) % L;  // lane and slot of row N-1
  const int cl2 = N > 1 ? (N - 2) / L : 0, jl2 = N > 1 ? (N - 2) % L : 0;
  // slot j (uniform over the warp) of lane `src`
  auto pick = [&](const double (&v)[L], int src, int j) {
    double t = 0.0;
#pragma unroll
    for (int k = 0; k < L; ++k)
      if (k == j) t = v[k];
    return shfl(t, src);
  };

  const int nw = blockDim.x >> 5;
  for (int64_t m = (int64_t)blockIdx.x + (int64_t)gridDim.x * (threadIdx.x >> 5); m < M;
       m += (int64_t)gridDim.x * nw) {
    double* base = state + m;
    double c[L];
#pragma unroll
    for (int j = 0; j < L; ++j) c[j] = r0 + j < N ? base[(int64_t)(r0 + j) * ld] : 0.0;
#pragma unroll 1
    for (int n = 0; n < nsteps; ++n) {
      double y[L];
      if constexpr (CH) {
        // r_j = C_j + E_j (phi_{j-1}, phi_j, phi_{j+1})
        const double p_first = NativeArith<double>::cubic(c[0]), p_last = NativeArith<double>::cubic(c[L - 1]);
        double pl = __shfl_up_sync(0xffffffffu, p_last, 1), pr = __shfl_down_sync(0xffffffffu, p_first, 1);
        double wrap = 0.0;
        if constexpr (RANK != 0) {
          const double p_end = NativeArith<double>::cubic(pick(c, cl, jl));
          wrap = shfl(p_first, 0);
          if (lane == 0) pl = p_end;
        } else {
          if (lane == 0) pl = 0.0;
        }
        if (lane == K) pr = 0.0;
        double pm = pl, p0 = p_first;
#pragma unroll
        for (int j = 0; j < L; ++j) {
          double pp = j + 1 < L ? (j + 2 == L ? p_last : NativeArith<double>::cubic(c[j + 1 < L ? j + 1 : j])) : pr;
          double pu = pp;
          if constexpr (RANK != 0)
            if (r0 + j == N - 1) pu = wrap;
          const double* e = ee + (size_t)j * 3 * kLanes;
          double r = fma(e[0], pm, c[j]);
          r = fma(e[kLanes], p0, r);
          y[j] = fma(e[2 * kLanes], pu, r);
          pm = p0;
          p0 = pp;
        }
      } else {
#pragma unroll
        for (int j = 0; j < L; ++j) y[j] = c[j];
      }
      // chunk sweeps
      {
        double u1 = 0.0, u2 = 0.0;
#pragma unroll
        for (int j = 0; j < L; ++j) {
          const double* f = fw + (size_t)j * W * kLanes;
          double t = y[j] * f[0];
          if constexpr (PB == 2) t = fma(-f[2 * kLanes], u2, t);
          t = fma(-f[kLanes], u1, t);
          y[j] = t;
          u2 = u1;
          u1 = t;
        }
        double x1 = 0.0, x2 = 0.0;
#pragma unroll
        for (int j = L - 1; j >= 0; --j) {
          const double* b = bw + (size_t)j * PB * kLanes;
          double t = y[j];
          if constexpr (PB == 2) t = fma(-b[kLanes], x2, t);
          t = fma(-b[0], x1, t);
          y[j] = t;
          x2 = x1;
          x1 = t;
        }
      }
      // boundary k of lane k: tail of chunk k, head of chunk k + 1
      double d[Q];
      {
        double r[Q];
#pragma unroll
        for (int u = 0; u < PB; ++u) {
          r[u] = y[L - PB + u];
          r[PB + u] = __shfl_down_sync(0xffffffffu, y[u], 1);
        }
        const double* T0 = img + lay.T0 + lane;
#pragma unroll
        for (int i = 0; i < Q; ++i) {
          double t = T0[i * Q * kLanes] * r[0];
#pragma unroll
          for (int j = 1; j < Q; ++j) t = fma(T0[(i * Q + j) * kLanes], r[j], t);
          d[i] = t;
        }
      }
      const double* Mb = img + lay.M + lane;
#pragma unroll 1
      for (int l = 0; l < NL; ++l) {
        const int st = 1 << l;
        double dl[PB], dr[PB];
#pragma unroll
        for (int u = 0; u < PB; ++u) {
          // entries that reach outside 0 .. K-1 have zero coefficients
          dl[u] = __shfl_up_sync(0xffffffffu, d[u], st);
          dr[u] = __shfl_down_sync(0xffffffffu, d[PB + u], st);
        }
        const double* M1 = Mb + Q * Q * kLanes;
        const double* M2 = M1 + Q * PB * kLanes;
        double nd[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) {
          double t = Mb[i * Q * kLanes] * d[0];
#pragma unroll
          for (int j = 1; j < Q; ++j) t = fma(Mb[(i * Q + j) * kLanes], d[j], t);
#pragma unroll
          for (int j = 0; j < PB; ++j) {
            t = fma(-M1[(i * PB + j) * kLanes], dl[j], t);
            t = fma(-M2[(i * PB + j) * kLanes], dr[j], t);
          }
          nd[i] = t;
        }
#pragma unroll
        for (int i = 0; i < Q; ++i) d[i] = nd[i];
        Mb += (Q * Q + 2 * Q * PB) * kLanes;
      }
      // x_j = y_j - W_j lam - V_j rho (the end lanes' missing sides have zero spikes)
      {
        double lam[PB], rho[PB];
#pragma unroll
        for (int u = 0; u < PB; ++u) {
          lam[u] = __shfl_up_sync(0xffffffffu, d[u], 1);
          rho[u] = d[PB + u];
        }
#pragma unroll
        for (int j = 0; j < L; ++j) {
          const double* w = co + (size_t)j * Q * kLanes;
          double t = y[j];
#pragma unroll
          for (int u = 0; u < PB; ++u) {
            t = fma(-w[u * kLanes], lam[u], t);
            t = fma(-w[(PB + u) * kLanes], rho[u], t);
          }
          y[j] = t;
        }
      }
      if constexpr (RANK == 1) {
        const double f = cs.v[0] * fma(cs.v[1], pick(y, cl, jl), shfl(y[0], 0));
#pragma unroll
        for (int j = 0; j < L; ++j) y[j] = fma(cy[(size_t)j * kLanes], f, y[j]);
      }
      if constexpr (RANK == 2) {
        const double ya = shfl(y[0], 0), yb = shfl(y[1 % L], 0), yc = pick(y, cl2, jl2), yd = pick(y, cl, jl);
        const double t0 = fma(cs.v[0], ya, fma(cs.v[1], yb, fma(cs.v[4], yc, cs.v[5] * yd)));
        const double t1 = fma(cs.v[2], ya, fma(cs.v[3], yb, fma(cs.v[6], yc, cs.v[7] * yd)));
        const double g0 = fma(cs.v[8], t0, cs.v[9] * t1), g1 = fma(cs.v[10], t0, cs.v[11] * t1);
#pragma unroll
        for (int j = 0; j < L; ++j) {
          const double* z = cy + (size_t)j * 2 * kLanes;
          y[j] = fma(z[kLanes], g1, fma(z[0], g0, y[j]));
        }
      }
#pragma unroll
      for (int j = 0; j < L; ++j) c[j] = CN ? fma(2.0, y[j], -c[j]) : y[j];
    }
#pragma unroll
    for (int j = 0; j < L; ++j)
      if (r0 + j < N) base[(int64_t)(r0 + j) * ld] = c[j];
  }
}

// ------------------------------------------------------------------ host side

int chunk_rows(int64_t N) {
  for (int L : {4, 8, 16, 32})
    if ((int64_t)L * kLanes >= N) return L;
  return 0;
}

template <int PB, int L, int RANK, bool CN, bool CH>
int launch(const sb_stepper* st, double* state, int64_t M, int64_t ld, int64_t nsteps, cudaStream_t stream) {
  const sb_factor* f = st->fac;
  const ResidentLayout lay = resident_layout(PB, L, RANK, CH, st->res_NL);
  const size_t smem = (size_t)lay.total * sizeof(double);
  CycScalars cs{};
  if constexpr (RANK == 1) {
    cs.v[0] = f->cyc_beta[0];
    cs.v[1] = f->cyc_alpha[0];
  }
  if constexpr (RANK == 2) std::copy_n(f->h_cyc.begin() + 4 * f->N, 12, cs.v);
  auto k = resident_steps_kernel<PB, L, RANK, CN, CH>;
  const int sms = std::max(1, sm_count(f->device));
  // one warp per simulation; as few warps per CTA as still puts every simulation on an
  // SM at once, since four warps or fewer per SM do not slow each other down
  const int warps = (int)std::min<int64_t>(kMaxWarps, std::max<int64_t>(1, (M + sms - 1) / sms));
  int nb = 0;
  SB_TRY(kernel_occupancy(reinterpret_cast<const void*>(k), f->device, warps * 32, smem, &nb));
  const int64_t grid = std::min<int64_t>((M + warps - 1) / warps, (int64_t)nb * sms);
  for (int64_t done = 0; done < nsteps; done += kStepsPerLaunch) {
    const int n = (int)std::min<int64_t>(kStepsPerLaunch, nsteps - done);
    k<<<(unsigned)grid, warps * 32, smem, stream>>>(st->res_img, st->res_NL, (int)st->N, M, ld, state, n, cs);
    SB_TRY(cuda_check(cudaGetLastError(), "resident step launch"));
  }
  return SB_OK;
}

template <int PB, int L>
int dispatch(const sb_stepper* st, double* state, int64_t M, int64_t ld, int64_t nsteps, cudaStream_t s) {
  constexpr int RANK = PB;  // periodic tridiagonal: rank 1, cyclic pentadiagonal: rank 2
  const bool per = st->fac->periodic, cn = st->NB > 0;
  if constexpr (PB == 2)
    if (st->has_e)
      return per ? launch<PB, L, RANK, false, true>(st, state, M, ld, nsteps, s)
                 : launch<PB, L, 0, false, true>(st, state, M, ld, nsteps, s);
  if (per)
    return cn ? launch<PB, L, RANK, true, false>(st, state, M, ld, nsteps, s)
              : launch<PB, L, RANK, false, false>(st, state, M, ld, nsteps, s);
  return cn ? launch<PB, L, 0, true, false>(st, state, M, ld, nsteps, s)
            : launch<PB, L, 0, false, false>(st, state, M, ld, nsteps, s);
}

}  // namespace

namespace {

// The batch up to which these steps beat the one-thread-per-simulation ones, with chunks of
// L rows and NL reduction levels.  Those take a latency of about N (430 + 71 n) cycles for n
// FP64 operations a row, whatever the batch; these take 17 cycles of an SM's FP64 unit per
// operation of each simulation's warp.  Microseconds per step there | here (the rule's line
// for M):
//   diffusion, CN, periodic, N = 256:  M = 4096 124 | 21, 16384 132 | 79, 32768 146 | 156 (21700)
//   hyperdiffusion, CN, periodic, N = 100:  M = 4096 70 | 55, 8192 70 | 105 (4600)
//   Cahn-Hilliard, no flux, N = 512:  M = 8192 261 | 134, 16384 275 | 269 (10700)
int64_t batch_limit(const sb_stepper* st, int L, int NL) {
  const int PB = st->fac->P, Q = 2 * PB, rank = st->fac->periodic ? st->fac->periodic_rank : 0;
  const int row_there = 2 * PB + 2 * rank + (st->has_e ? 5 : st->NB);
  const int row_here = 1 + 2 * PB + Q + rank + (st->has_e ? 5 : st->NB > 0 ? 1 : 0);
  const int ops = L * row_here + Q * Q + NL * (Q * Q + 2 * Q * PB) + 6 * rank;
  return (int64_t)(0.9 * sm_count(st->fac->device) * st->N * (430.0 + 71.0 * row_there) / (17.0 * ops));
}

// A device copy of `img`, made on a stream of its own in relaxed capture mode: the first
// small batch may be stepped inside a capture of the caller's, or while another thread
// captures.
int upload(const std::vector<double>& img, double** out) {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  SB_CUDA(cudaThreadExchangeStreamCaptureMode(&mode));
  double* d = nullptr;
  cudaStream_t s = nullptr;
  const size_t bytes = img.size() * sizeof(double);
  cudaError_t e = cudaMalloc(&d, bytes);
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
  if (e == cudaSuccess) e = cudaMemcpyAsync(d, img.data(), bytes, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (s != nullptr) cudaStreamDestroy(s);
  if (e != cudaSuccess && d != nullptr) cudaFree(d);
  cudaThreadExchangeStreamCaptureMode(&mode);
  SB_TRY(cuda_check(e, "image of the on-chip steps"));
  *out = d;
  return SB_OK;
}

// The image, made by the first small batch that is stepped (most steppers never see one).
int build_resident(sb_stepper* st) {
  const std::vector<double>& erows = st->e_rows;
  const sb_factor* f = st->fac;
  const int PB = f->P, N = (int)f->N, L = chunk_rows(f->N), Q = 2 * PB;
  Partition p;
  if (!build_partition(PB, N, f->h_diag.data(), L, kLanes, p)) return SB_OK;
  const int K = p.K();
  // levels left off: every coupling from there on is below 2^-100 of the unknown it
  // would be added to, 2^-47 of that unknown's own rounding
  int NL = p.NL;
  auto decayed = [&](int lv) {
    const size_t b = (size_t)lv * K * Q * PB, n = (size_t)K * Q * PB;
    for (size_t t = b; t < b + n; ++t)
      if (std::fabs(p.M1[t]) > 0x1p-100 || std::fabs(p.M2[t]) > 0x1p-100) return false;
    return true;
  };
  while (NL > 0 && decayed(NL - 1)) --NL;
  const int rank = f->periodic ? f->periodic_rank : 0;
  const ResidentLayout lay = resident_layout(PB, L, rank, st->has_e, NL);
  if ((size_t)lay.total * sizeof(double) > (size_t)kMaxDynSmem) return SB_OK;
  std::vector<double> img(lay.total, 0.0);
  auto at = [&](int sec, int width, int i, int k) -> double& {  // value k of row i
    return img[sec + ((i % L) * width + k) * kLanes + i / L];
  };
  for (int i = 0; i < L * kLanes; ++i) {
    for (int k = 0; k <= PB; ++k) at(lay.fwd, PB + 1, i, k) = p.fw[(size_t)(PB + 1) * i + k];
    for (int k = 0; k < PB; ++k) {
      at(lay.bwd, PB, i, k) = p.bw[(size_t)PB * i + k];
      at(lay.cor, Q, i, k) = p.W[(size_t)PB * i + k];
      at(lay.cor, Q, i, PB + k) = p.V[(size_t)PB * i + k];
      if (rank > 0 && i < N) at(lay.cyc, rank, i, k) = f->h_cyc[(size_t)2 * rank * i + rank + k];
    }
    if (st->has_e && i < N)
      for (int k = 0; k < 3; ++k) at(lay.e, 3, i, k) = erows[(size_t)3 * i + k];
  }
  for (int k = 0; k < K; ++k) {
    for (int e = 0; e < Q * Q; ++e) img[lay.T0 + e * kLanes + k] = p.T0[(size_t)k * Q * Q + e];
    for (int lv = 0; lv < NL; ++lv) {
      double* m = img.data() + lay.M + (size_t)lv * (Q * Q + 2 * Q * PB) * kLanes + k;
      const size_t b0 = ((size_t)lv * K + k) * Q * Q, b1 = ((size_t)lv * K + k) * Q * PB;
      for (int e = 0; e < Q * Q; ++e) m[e * kLanes] = p.M0[b0 + e];
      for (int e = 0; e < Q * PB; ++e) {
        m[(Q * Q + e) * kLanes] = p.M1[b1 + e];
        m[(Q * Q + Q * PB + e) * kLanes] = p.M2[b1 + e];
      }
    }
  }
  SB_TRY(upload(img, &st->res_img));
  st->res_L = L;
  st->res_NL = NL;
  st->res_max_M = batch_limit(st, L, NL);
  return SB_OK;
}

}  // namespace

int resident_applies(sb_stepper* st, int64_t M, sb_arith arith, bool* applies) {
  *applies = false;
  const sb_factor* f = st->fac;
  const int L = chunk_rows(f->N);
  if (arith != SB_ARITH_NATIVE || f->N < kLanes || L == 0 || !f->any_order || M > batch_limit(st, L, 0)) return SB_OK;
  std::lock_guard<std::mutex> lk(st->mu);
  if (!st->res_built) {
    SB_TRY(build_resident(st));
    st->res_built = true;
  }
  *applies = st->res_img != nullptr && M <= st->res_max_M;
  return SB_OK;
}

int resident_run(const sb_stepper* st, double* state, int64_t M, int64_t ld, int64_t nsteps, cudaStream_t s) {
  if (st->fac->P == 1) {
    switch (st->res_L) {
      case 4: return dispatch<1, 4>(st, state, M, ld, nsteps, s);
      case 8: return dispatch<1, 8>(st, state, M, ld, nsteps, s);
      case 16: return dispatch<1, 16>(st, state, M, ld, nsteps, s);
      default: return dispatch<1, 32>(st, state, M, ld, nsteps, s);
    }
  }
  switch (st->res_L) {
    case 4: return dispatch<2, 4>(st, state, M, ld, nsteps, s);
    case 8: return dispatch<2, 8>(st, state, M, ld, nsteps, s);
    case 16: return dispatch<2, 16>(st, state, M, ld, nsteps, s);
    default: return dispatch<2, 32>(st, state, M, ld, nsteps, s);
  }
}

}  // namespace sb
