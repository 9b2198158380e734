// The fused time step in native FP64: one thread per simulation builds the right-hand
// side, sweeps forward and back in place, one launch per step (stepper.cu holds the
// schemes, the double-float step and the public calls).
//
// What bounds it: the SM's FP64 unit, which takes one warp operation every 16 cycles and
// one from the same warp every 64.  So the step is written to spend FP64 operations only
// where nothing else will do:
//   * products off the recurrence's chain run on the integer pipes, a batch of rows at a
//     time with one test for the batch (mulc_fast, dmul_fast; bit-identical);
//   * Crank-Nicolson: B = 2 I - A, so C^{n+1} = 2 A^{-1} C - C needs no stencil.  The sweep
//     keeps v of the unscaled factorisation (C_i = v_i + l1_i v_{i-1} + l2_i v_{i-2}), from
//     which the backward sweep has C_i back for P operations: 2P + 1 operations a row
//     instead of 2P + 2P + 1;
//   * periodic ends: the rows of the correction decay away from the ends, and rows whose
//     coefficient is below 2^-100 of the largest take no part; where the rows that do are
//     more than half of a rank-2 correction, its two dot products give way to a third
//     sweep that adds the correction once y_0, y_1 are known (memory is idle, the FP64
//     unit is not);
//   * the WENO term shares differences between rows and divides once, by Newton's
//     iteration from a single-precision reciprocal (see Weno).
// FP64 operations a row (counted on the device), before and now, and a step (of the cycles
// of an SM that has work, those its FP64 unit is busy, now):
//   Crank-Nicolson diffusion, periodic, N = 1024, M = 65536:  7, 4.8 (4 without periodic
//     ends; the correction's rows are 0.2 of the rest, and the dot product of every other
//     batch of the others is issued under a false predicate, 0.5);  0.996 -> 0.624 ms (87 %)
//   Cahn-Hilliard without flux, N = 256, M = 2^20:  9, 8;  4.06 -> 3.58 ms (94 %)
//   periodic, with the coarsening length, N = 256, M = 65536:  14, 11.1;  0.428 -> 0.343 ms (94 %)
//   forced, N = 512, M = 98304:  86, 40.4;  9.18 -> 4.18 ms (80 %; 8 to 40 bytes of its
//     registers spill, 0.03 loads a row)
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "arith.cuh"
#include "narrow.cuh"
#include "sb_internal.h"

namespace sb {
namespace {

enum StepKind { KBE = 0, KCN = 1, KCH = 2 };  // B = I; B = 2 I - A; B = I and E phi(C)

constexpr int kRowsPerBatch = 8;
constexpr int kStepThreads = 256;

template <int n>
struct alignas(n == 3 ? 8 : 8 * n) Vals {
  double v[n];
};

// The rows a step reads, in shared memory or (large N) straight from the device image.
// Offsets in doubles.
struct StepLayout {
  int scale, f, b, e, cyc, total;
};
__host__ __device__ inline StepLayout step_layout(int P, bool ch, int rank, int N) {
  StepLayout l;
  int o = 0;
  l.scale = o, o += 2 * N;              // MulCoef: 1 / pivot
  l.cyc = o, o += rank == 1 ? 2 * N : rank == 2 ? 4 * N + 12 : 0;  // as in sb_factor
  l.f = o, o += P * N;
  l.b = o, o += P * N;
  l.e = o, o += ch ? 3 * N : 0;
  l.total = o;
  return l;
}

__device__ __forceinline__ double max_bits(double a, double b) {  // of non-negative values
  return __longlong_as_double(max(__double_as_longlong(a), __double_as_longlong(b)));
}
__device__ __forceinline__ double abs_bits(double a) {
  return __longlong_as_double(__double_as_longlong(a) & 0x7fffffffffffffffLL);
}
// 2^(k) a for a positive normal a whose result is normal too
__device__ __forceinline__ double scale2(double a, int k) {
  return __hiloint2double(__double2hiint(a) + (k << 20), __double2loint(a));
}
// a * b of positive normal values whose product is normal
__device__ __forceinline__ double dmul_pos(double a, double b) { return mulc_fast(a, mulc_prepare(b)); }
// a * a of any value
__device__ __forceinline__ double dsquare(double a) {
  if (SB_LIKELY(dsq_ok(a))) return mulc_fast(a, mulc_prepare(a));
  return dmul_slow(a, a);
}

// Fifth-order Hamilton-Jacobi WENO derivative (Jiang and Peng's scheme, section 6.1) on a
// grid of spacing 1, biased toward lower rows (SIDE < 0) or higher rows, in a form that
// shares work between neighbouring rows.  With the five one-sided differences q_1..q_5 of
// the scheme, h_k = q_{k+1} - q_k and d_k = h_{k+1} - h_k move along by one place a row, so
// a row adds one q, one h, one d and one square d^2.  Then
//   4 (S_k + eps) = 13/3 d_k^2 + e_k^2 + 4 eps,  e = (3 h2 - h1, h2 + h3, h4 - 3 h3)
//   p_k = q_3 + m_k / 6,  m = (2 e1 - h2, h2 + 2 h3, 4 h3 - h4)
//   W = q_3 + (sum_k a_k m_k) / (6 sum_k a_k),  a = (1, 6, 3) / (S + eps)^2
// The a_k are formed without a division, as products of the other two t = 4 (S + eps)
// scaled by the power of two that brings the largest into [1, 2) (every ratio is then
// above 1e-8, so no product leaves the normal range); those products, the squares and the
// maxima are integer work.  1 / sum a_k: Newton's iteration of third order,
// y (1 + e + e^2) with e = 1 - D y, from a single-precision reciprocal (error 2^-66 before
// rounding).  28 FP64 operations a row, 8 integer products; the form that evaluated the
// candidates and normalised weights row by row took 73.
template <int SIDE>
struct Weno {
  double q[5], h[4], s[3];  // s_k = d_k^2

  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int k = 0; k < 5; ++k) q[k] = 0.0;
#pragma unroll
    for (int k = 0; k < 4; ++k) h[k] = 0.0;
#pragma unroll
    for (int k = 0; k < 3; ++k) s[k] = 0.0;
  }
  // one row on: qn is the difference that enters (q_5 going with SIDE < 0, else q_1)
  __device__ __forceinline__ void advance(double qn) {
    if constexpr (SIDE < 0) {
#pragma unroll
      for (int k = 0; k < 4; ++k) q[k] = q[k + 1];
      q[4] = qn;
#pragma unroll
      for (int k = 0; k < 3; ++k) h[k] = h[k + 1];
      h[3] = q[4] - q[3];
      s[0] = s[1];
      s[1] = s[2];
      s[2] = dsquare(h[3] - h[2]);
    } else {
#pragma unroll
      for (int k = 4; k > 0; --k) q[k] = q[k - 1];
      q[0] = qn;
#pragma unroll
      for (int k = 3; k > 0; --k) h[k] = h[k - 1];
      h[0] = q[1] - q[0];
      s[2] = s[1];
      s[1] = s[0];
      s[0] = dsquare(h[1] - h[0]);
    }
  }
  // r + adv W, adv6 = adv / 6
  __device__ __forceinline__ double add(double r, double adv, double adv6) const {
    const double e1 = fma(3.0, h[1], -h[0]), e2 = h[1] + h[2], e3 = fma(-3.0, h[2], h[3]);
    double qa = max_bits(abs_bits(q[0]), abs_bits(q[1]));
    qa = max_bits(qa, max_bits(abs_bits(q[2]), abs_bits(q[3])));
    qa = max_bits(qa, abs_bits(q[4]));
    const double eps = fma(4e-6, dsquare(qa), 4e-99);
    const double t1 = fma(e1, e1, fma(13.0 / 3.0, s[0], eps));
    const double t2 = fma(e2, e2, fma(13.0 / 3.0, s[1], eps));
    const double t3 = fma(e3, e3, fma(13.0 / 3.0, s[2], eps));
    // t are positive (>= 4e-99): their high words order like their exponents
    // (infinite only where a difference exceeds 1e153: phi of such a C has overflowed too and
    // takes the whole simulation with it, whatever W comes to)
    const int top = max(max(__double2hiint(t1), __double2hiint(t2)), __double2hiint(t3));
    const int k = 1023 - (top >> 20);
    const double r1 = scale2(t1, k), r2 = scale2(t2, k), r3 = scale2(t3, k);
    const double r12 = dmul_pos(r1, r2), r13 = dmul_pos(r1, r3), r23 = dmul_pos(r2, r3);
    const double a = dmul_pos(r23, r23), b2 = scale2(dmul_pos(r13, r13), 1), c = dmul_pos(r12, r12);
    const double m1 = fma(2.0, e1, -h[1]), m2 = fma(2.0, h[2], h[1]), m3 = fma(4.0, h[2], -h[3]);
    const double den = fma(3.0, b2 + c, a);
    const double num = fma(3.0, fma(b2, m2, c * m3), a * m1);
    float y32;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y32) : "f"(f64_to_f32_trunc(den)));
    const double y0 = widen_f32(y32);
    const double e = fma(-den, y0, 1.0);
    const double y = fma(fma(e, e, e), y0, y0);
    return fma(adv6, num * y, fma(adv, q[2], r));
  }
};

struct StepArgs {
  const double* image;
  int N, fast;       // fast: every 1 / pivot suits mulc_fast
  int ka, kb;        // rows outside [ka, kb) take part in the periodic correction
  int64_t M, ld, ntiles;
  const double* src;
  double* state;
  double alpha, beta;  // rank 1
  double* ellm;        // STATS
  const double *gprof, *amp;  // ADV
  double adv;
};

// KIND: the scheme; CYC: rank of the periodic correction (0: none); THIRD: the rank-2
// correction by a third sweep.  STATS: ellm[m] = 1 / (1 - <C^2>) of the new state.  GC: the
// rows are read from the device image (they exceed one CTA's shared memory).  ADV (with
// KCH, CYC = 2): the travelling-wave terms, biased toward lower (-1) or higher (+1) rows.
template <int P, StepKind KIND, int CYC, bool THIRD, bool STATS, bool GC, int ADV>
__global__ void __launch_bounds__(kStepThreads, 2) step64_kernel(const __grid_constant__ StepArgs a) {
  constexpr int R = kRowsPerBatch;
  constexpr bool CH = KIND == KCH;
  constexpr int LA = ADV != 0 ? 3 : CH ? 1 : 0;  // rows of look-ahead
  static_assert(ADV == 0 || (CH && CYC == 2), "the forced scheme is periodic Cahn-Hilliard");
  static_assert(!THIRD || CYC == 2, "the third sweep belongs to the rank-2 correction");
  using RP = Vals<P>;
  const int N = a.N;
  const int64_t ld = a.ld;
  const StepLayout lay = step_layout(P, CH, CYC, N);
  const double* rows = a.image;
  const double* gp = a.gprof;
  if constexpr (!GC) {
    extern __shared__ __align__(16) double step_smem[];
    for (int k = threadIdx.x; k < lay.total; k += blockDim.x) step_smem[k] = a.image[k];
    if constexpr (ADV != 0)
      for (int k = threadIdx.x; k < N; k += blockDim.x) step_smem[lay.total + k] = a.gprof[k];
    __syncthreads();
    rows = step_smem;
    gp = step_smem + lay.total;
  }
  const MulCoef* pc = reinterpret_cast<const MulCoef*>(rows + lay.scale);
  const RP* fr = reinterpret_cast<const RP*>(rows + lay.f);
  const RP* br = reinterpret_cast<const RP*>(rows + lay.b);
  const Vals<3>* er = reinterpret_cast<const Vals<3>*>(rows + lay.e);
  const double* cy = rows + lay.cyc;
  const double adv6 = a.adv * (1.0 / 6.0);

  const int nw = blockDim.x >> 5;
  for (int64_t tile = blockIdx.x + (int64_t)gridDim.x * (threadIdx.x >> 5); tile < a.ntiles;
       tile += (int64_t)gridDim.x * nw) {
    const int64_t m = tile * 32 + (threadIdx.x & 31);
    if (m >= a.M) continue;
    double* const y = a.state + m;
    const double* const c = a.src + m;  // the old state (may be the same array as y)

    // s[j] = v[j] / pivot of row i(j), the batch at once
    auto scaled = [&](double (&s)[R], const double (&v)[R], auto row, auto in) {
      bool ok = a.fast != 0;
#pragma unroll
      for (int j = 0; j < R; ++j) {
        const double t = in(j) ? v[j] : 1.0;
        ok = ok && mulc_ok(t);
        s[j] = mulc_fast(t, pc[in(j) ? row(j) : 0]);
      }
      if (!ok) {
#pragma unroll
        for (int j = 0; j < R; ++j)
          if (in(j)) {
            const MulCoef w = pc[row(j)];
            s[j] = mulc_slow(v[j], w.lo, w.hi, w.ck);
          }
      }
    };

    // ---- forward sweep
    double wrap[LA > 0 ? LA : 1];  // rows 0 .. LA-1, which follow row N-1 when periodic
    double cw[2 * LA + 1] = {};    // rows i-LA .. i+LA (ADV)
    double pm = 0.0, p0 = 0.0;     // phi(C_{i-1}), phi(C_i)
    Weno<ADV < 0 ? -1 : 1> weno;
    double fm = 0.0;
    if constexpr (ADV != 0) fm = a.amp[m];
    auto phi = [](double v) { return fma(dsquare(v), v, -v); };
    double va[R], vb[R];
    auto load = [&](double (&b)[R], int i0, auto guard) {
#pragma unroll
      for (int j = 0; j < R; ++j)
        if (!decltype(guard)::value || i0 + j < N) b[j] = c[(int64_t)(i0 + j) * ld];
    };
    load(va, 0, std::true_type{});
    load(vb, R, std::true_type{});
    if constexpr (CH) {
#pragma unroll
      for (int k = 0; k < LA; ++k) wrap[k] = CYC != 0 ? va[k] : 0.0;
      p0 = phi(va[0]);
      if constexpr (CYC != 0) pm = phi(c[(int64_t)(N - 1) * ld]);
    }
    if constexpr (ADV != 0) {
      auto qn = [&]() { return ADV < 0 ? cw[2 * LA - 1] - cw[2 * LA - 2] : cw[2 * LA] - cw[2 * LA - 1]; };
#pragma unroll
      for (int k = 0; k < 2 * LA + 1; ++k) cw[k] = 0.0;
#pragma unroll
      for (int k = 0; k < LA; ++k) cw[LA + 1 + k] = c[(int64_t)(N - LA + k) * ld];
      weno.clear();
      weno.advance(qn());
#pragma unroll
      for (int k = 0; k < LA; ++k) {  // rows 0 .. LA-1 enter
#pragma unroll
        for (int t = 0; t < 2 * LA; ++t) cw[t] = cw[t + 1];
        cw[2 * LA] = va[k];
        weno.advance(qn());
      }
    }
    double u1 = 0.0, u2 = 0.0, dot = 0.0, dot1 = 0.0;
    // rows i0 .. i0+R-1, raw in b; bn: the R rows after them.  GUARD: test rows against N
    auto forward = [&](double (&b)[R], const double (&bn)[R], int i0, auto guard) {
      constexpr bool GUARD = decltype(guard)::value;
      auto in = [&](int j) { return !GUARD || i0 + j < N; };
      // b[j] becomes the right-hand side of row i0 + j (b[j] itself is not read after that)
      if constexpr (CH) {
#pragma unroll
        for (int j = 0; j < R; ++j) {
          const int i = i0 + j;
          double nx = j + LA < R ? b[j + LA < R ? j + LA : 0] : bn[j + LA < R ? 0 : j + LA - R];
          if (GUARD && i + LA >= N) {
            nx = 0.0;
#pragma unroll
            for (int k = 0; k < LA; ++k)
              if (i + LA - N == k) nx = wrap[k];
          }
          double c0 = b[j], c1 = nx;  // C_i, C_{i+1}
          if constexpr (ADV != 0) {
#pragma unroll
            for (int t = 0; t < 2 * LA; ++t) cw[t] = cw[t + 1];
            cw[2 * LA] = nx;
            weno.advance(ADV < 0 ? cw[2 * LA - 1] - cw[2 * LA - 2] : cw[2 * LA] - cw[2 * LA - 1]);
            c0 = cw[LA];
            c1 = cw[LA + 1];
          }
          const double pp = phi(c1);
          if (in(j)) {
            const Vals<3> e = er[i];
            double r = fma(e.v[0], pm, c0);
            r = fma(e.v[1], p0, r);
            r = fma(e.v[2], pp, r);
            if constexpr (ADV != 0) {
              r = weno.add(r, a.adv, adv6);
              r = fma(fm, gp[i], r);
            }
            b[j] = r;
          }
          pm = p0;
          p0 = pp;
        }
      }
      if constexpr (CYC != 0 && !THIRD) {
        if (i0 < a.ka || i0 + R > a.kb) {
#pragma unroll
          for (int j = 0; j < R; ++j)
            if (in(j)) {
              const int i = i0 + j;
              if constexpr (CYC == 1) dot = fma(cy[2 * i], b[j], dot);
              if constexpr (CYC == 2) {
                dot = fma(cy[4 * i], b[j], dot);
                dot1 = fma(cy[4 * i + 1], b[j], dot1);
              }
            }
        }
      }
      double s[R];
      if constexpr (KIND == KCN) {
#pragma unroll
        for (int j = 0; j < R; ++j) s[j] = b[j];
      } else {
        scaled(s, b, [&](int j) { return i0 + j; }, in);
      }
#pragma unroll
      for (int j = 0; j < R; ++j)
        if (in(j)) {
          const RP w = fr[i0 + j];
          double u = fma(-w.v[0], u1, s[j]);
          if constexpr (P == 2) u = fma(-w.v[P - 1], u2, u);
          y[(int64_t)(i0 + j) * ld] = u;
          u2 = u1;
          u1 = u;
        }
    };
    int i0 = 0;
    for (; i0 + 4 * R <= N; i0 += 2 * R) {
      forward(va, vb, i0, std::false_type{});
      load(va, i0 + 2 * R, std::false_type{});
      forward(vb, va, i0 + R, std::false_type{});
      load(vb, i0 + 3 * R, std::false_type{});
    }
    for (; i0 < N; i0 += 2 * R) {
      forward(va, vb, i0, std::true_type{});
      load(va, i0 + 2 * R, std::true_type{});
      forward(vb, va, i0 + R, std::true_type{});
      load(vb, i0 + 3 * R, std::true_type{});
    }

    // ---- backward sweep: x_i from the stored u (or v, KCN); x1, x2 uncorrected
    double x1 = 0.0, x2 = 0.0, g0 = 0.0, g1 = 0.0, sq = 0.0;
    double yl = 0.0, yl2 = 0.0;  // y_{N-1}, y_{N-2}
    double held = 0.0;           // KCN: C_{N-1} while row N-1 waits for the rank-2 correction
    auto emit = [&](int i, double v) {
      y[(int64_t)i * ld] = v;
      if constexpr (STATS && !THIRD) sq = fma(v, v, sq);
    };
    auto finish = [&](double x, double old) { return KIND == KCN ? fma(2.0, x, -old) : x; };
    // g of the rank-2 correction from (y_0, y_1) and (y_{N-2}, y_{N-1})
    auto rank2 = [&](double ya, double yb) {
      const double* sc = cy + 4 * N;
      const double t0 = fma(sc[0], ya, fma(sc[1], yb, fma(sc[4], yl2, sc[5] * yl)));
      const double t1 = fma(sc[2], ya, fma(sc[3], yb, fma(sc[6], yl2, sc[7] * yl)));
      g0 = fma(sc[8], t0, sc[9] * t1);
      g1 = fma(sc[10], t0, sc[11] * t1);
    };
    auto loadb = [&](double (&b)[R], int ib, auto guard) {
#pragma unroll
      for (int j = 0; j < R; ++j) {
        if (!decltype(guard)::value || ib - j >= 0) b[j] = y[(int64_t)(ib - j) * ld];
        else b[j] = 0.0;
      }
    };
    // rows ib, ib-1, .. ib-R+1, stored values in b; bn: the R rows after them
    auto backward = [&](double (&b)[R], const double (&bn)[R], int ib, auto guard) {
      constexpr bool GUARD = decltype(guard)::value;
      auto in = [&](int j) { return !GUARD || ib - j >= 0; };
      double s[R], old[R];
      if constexpr (KIND == KCN) {
        scaled(s, b, [&](int j) { return ib - j; }, in);
#pragma unroll
        for (int j = 0; j < R; ++j)
          if (in(j)) {
            const RP w = fr[ib - j];
            double t = fma(w.v[0], j + 1 < R ? b[j + 1 < R ? j + 1 : 0] : bn[0], b[j]);
            if constexpr (P == 2) t = fma(w.v[P - 1], j + 2 < R ? b[j + 2 < R ? j + 2 : 0] : bn[j + 2 < R ? 0 : j + 2 - R], t);
            old[j] = t;
          }
      } else {
#pragma unroll
        for (int j = 0; j < R; ++j) s[j] = b[j];
      }
      const bool edge = CYC != 0 && !THIRD && (ib - R + 1 < a.ka || ib >= a.kb);
      auto each = [&](auto with) {
        constexpr bool WITH = decltype(with)::value;  // the correction takes part in this batch
#pragma unroll
        for (int j = 0; j < R; ++j)
          if (in(j)) {
            const int i = ib - j;
            const RP w = br[i];
            double x = fma(-w.v[0], x1, s[j]);
            if constexpr (P == 2) x = fma(-w.v[P - 1], x2, x);
            const double o = KIND == KCN ? old[j] : 0.0;
            if constexpr (CYC == 1 && WITH) {
              if (i == N - 1) g0 = a.beta * fma(a.alpha, x, dot);
              emit(i, finish(fma(cy[2 * i + 1], g0, x), o));
            } else if constexpr (CYC == 2 && WITH) {
              if (i == N - 1) {
                yl = x;  // waits for y_{N-2}
                held = o;
              } else {
                if (i == N - 2) {
                  yl2 = x;
                  rank2(dot, dot1);
                  emit(N - 1, finish(fma(cy[4 * N - 1], g1, fma(cy[4 * N - 2], g0, yl)), held));
                }
                emit(i, finish(fma(cy[4 * i + 3], g1, fma(cy[4 * i + 2], g0, x)), o));
              }
            } else {
              if constexpr (THIRD) {
                if (i == N - 1) yl = x;
                if (i == N - 2) yl2 = x;
              }
              emit(i, finish(x, o));
            }
            x2 = x1;
            x1 = x;
          }
      };
      if (edge) each(std::true_type{});
      else each(std::false_type{});
    };
    loadb(va, N - 1, std::true_type{});
    loadb(vb, N - 1 - R, std::true_type{});
    int ib = N - 1;
    for (; ib - 4 * R + 1 >= 0; ib -= 2 * R) {
      backward(va, vb, ib, std::false_type{});
      loadb(va, ib - 2 * R, std::false_type{});
      backward(vb, va, ib - R, std::false_type{});
      loadb(vb, ib - 3 * R, std::false_type{});
    }
    for (; ib >= 0; ib -= 2 * R) {
      backward(va, vb, ib, std::true_type{});
      loadb(va, ib - 2 * R, std::true_type{});
      backward(vb, va, ib - R, std::true_type{});
      loadb(vb, ib - 3 * R, std::true_type{});
    }

    // ---- third sweep: x = y - z0 g0 - z1 g1 once y_0 (x1) and y_1 (x2) are known
    if constexpr (THIRD) {
      rank2(x1, x2);
      if constexpr (KIND == KCN) {  // the rows hold 2 y - C
        g0 *= 2.0;
        g1 *= 2.0;
      }
      auto loadu = [&](double (&b)[R], int i0) {
#pragma unroll
        for (int j = 0; j < R; ++j)
          if (i0 + j < N) b[j] = y[(int64_t)(i0 + j) * ld];
      };
      auto add = [&](const double (&b)[R], int i0) {
#pragma unroll
        for (int j = 0; j < R; ++j)
          if (i0 + j < N) {
            const int i = i0 + j;
            const double v = fma(cy[4 * i + 3], g1, fma(cy[4 * i + 2], g0, b[j]));
            y[(int64_t)i * ld] = v;
            if constexpr (STATS) sq = fma(v, v, sq);
          }
      };
      loadu(va, 0);
      for (int k = 0; k < N; k += 2 * R) {
        loadu(vb, k + R);
        add(va, k);
        loadu(va, k + 2 * R);
        add(vb, k + R);
      }
    }
    if constexpr (STATS) a.ellm[m] = 1.0 / (1.0 - sq / (double)N);
  }
}

// ------------------------------------------------------------------ host side

template <int P, StepKind KIND, int CYC, bool THIRD, bool STATS, int ADV>
int launch(const sb_stepper* st, const double* src, double* state, int64_t M, int64_t ld, cudaStream_t stream,
           double* ellm, const double* amp) {
  const sb_factor* f = st->fac;
  const int N = (int)f->N;
  size_t smem = ((size_t)step_layout(P, KIND == KCH, CYC, N).total + (ADV != 0 ? N : 0)) * sizeof(double);
  auto k = step64_kernel<P, KIND, CYC, THIRD, STATS, false, ADV>;
  if (smem > (size_t)kMaxDynSmem) {  // large N: rows read from device memory
    k = step64_kernel<P, KIND, CYC, THIRD, STATS, true, ADV>;
    smem = 0;
  }
  int nb = 0;
  SB_TRY(kernel_occupancy(reinterpret_cast<const void*>(k), f->device, kStepThreads, smem, &nb));
  StepArgs a{};
  a.image = st->s64;
  a.N = N;
  a.fast = st->s64_fast;
  a.ka = st->s64_ka;
  a.kb = st->s64_kb;
  a.M = M;
  a.ld = ld;
  a.ntiles = (M + 31) / 32;
  a.src = src;
  a.state = state;
  a.alpha = f->cyc_alpha[0];
  a.beta = f->cyc_beta[0];
  a.ellm = ellm;
  a.gprof = st->g64;
  a.amp = amp;
  a.adv = st->adv;
  const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(a.ntiles, (int64_t)nb * sm_count(f->device)));
  k<<<(unsigned)grid, kStepThreads, smem, stream>>>(a);
  return cuda_check(cudaGetLastError(), "fused step launch");
}

template <int P, StepKind KIND>
int dispatch(const sb_stepper* st, const double* src, double* state, int64_t M, int64_t ld, cudaStream_t s,
             double* ellm) {
  const bool third = st->s64_third;
  if constexpr (KIND == KCH) {
    if (ellm != nullptr) {
      if (!st->fac->periodic) return launch<P, KIND, 0, false, true, 0>(st, src, state, M, ld, s, ellm, nullptr);
      return third ? launch<P, KIND, 2, true, true, 0>(st, src, state, M, ld, s, ellm, nullptr)
                   : launch<P, KIND, 2, false, true, 0>(st, src, state, M, ld, s, ellm, nullptr);
    }
  }
  if (!st->fac->periodic) return launch<P, KIND, 0, false, false, 0>(st, src, state, M, ld, s, nullptr, nullptr);
  if constexpr (P == 2)
    if (third) return launch<P, KIND, 2, true, false, 0>(st, src, state, M, ld, s, nullptr, nullptr);
  return launch<P, KIND, P, false, false, 0>(st, src, state, M, ld, s, nullptr, nullptr);
}

// Unevaluated sum of two doubles, for the host arithmetic below.
struct Two {
  double h, l;
};
Two two_add(Two a, Two b) {
  const double s = a.h + b.h, t = s - a.h;
  const double e = ((a.h - (s - t)) + (b.h - t)) + (a.l + b.l);
  return {s + e, e - ((s + e) - s)};
}
Two two_mul(Two a, double b) {
  const double p = a.h * b;
  const double e = std::fma(a.h, b, -p) + a.l * b;
  return {p + e, e - ((p + e) - p)};
}

// Rounds the reciprocal pivots of the unscaled factorisation (forward rows fw, backward
// rows bw of W = P + 1 values, the first unused in fw) so that constants stay constant: a
// step forms 2 A^{-1} C - C, in which a relative error of A^{-1} on the mean, the one mode
// that never decays, counts twice and the same way every step.  Row i's reciprocal is the
// one that takes v = L^{-1} (A 1) to 1 given the rounded rows, in double-double, with the
// rounding error carried into the next row, so that the errors of a run of rows cancel.
// Left alone where that is not the pivot's reciprocal up to rounding.
void balance_pivots(int P, int N, const double* diag, const double* fw, const double* bw,
                    std::vector<double>& scale) {
  const int W = P + 1;
  Two v1{0, 0}, v2{0, 0}, carry{0, 0};
  for (int i = 0; i < N; ++i) {
    Two v{0, 0};
    for (int o = 0; o <= 2 * P; ++o) v = two_add(v, {diag[(size_t)o * N + i], 0});
    v = two_add(v, two_mul(v1, -fw[(size_t)W * i + 1]));
    if (P == 2) v = two_add(v, two_mul(v2, -fw[(size_t)W * i + 2]));
    Two num{1.0, 0};
    for (int k = 1; k <= P; ++k) num = two_add(num, {bw[(size_t)W * i + k], 0});
    const double q = num.h / v.h;  // num / v
    const Two r = two_add(num, two_mul(v, -q));
    Two g = two_add({q, 0}, {r.h / v.h, 0});
    const Two t = two_add(g, carry);
    if (std::isfinite(t.h) && std::fabs(t.h - scale[i]) <= 0x1p-48 * std::fabs(scale[i])) {
      scale[i] = t.h;
      carry = {t.l, 0};
    } else {
      carry = {0, 0};
    }
    v2 = v1;
    v1 = v;
  }
}

}  // namespace

int build_step64(sb_stepper* st, const std::vector<double>& erows) {
  const sb_factor* f = st->fac;
  const int P = f->P, W = P + 1, N = (int)f->N;
  const int rank = f->periodic ? f->periodic_rank : 0;
  const StepLayout l = step_layout(P, st->has_e, rank, N);
  std::vector<double> img(l.total, 0.0);
  // Crank-Nicolson keeps v of the unscaled factorisation: the adjoint block's rows, which
  // are those of A because every stepper matrix is symmetric
  const bool cn = st->NB > 0;
  const double* fw = f->h_coef.data() + (cn ? op_block_len(P, N) : 0);
  const double* bw = fw + (size_t)W * N;
  std::vector<double> scale(N);
  for (int i = 0; i < N; ++i) scale[i] = (cn ? bw : fw)[(size_t)W * i];
  if (cn) balance_pivots(P, N, f->h_diag.data(), fw, bw, scale);
  st->s64_fast = 1;
  for (int i = 0; i < N; ++i) {
    const double sc = scale[i];
    if (!mulc_usable(sc)) st->s64_fast = 0;
    const MulCoef m = mulc_prepare(sc);
    std::memcpy(&img[l.scale + 2 * (size_t)i], &m, sizeof(m));
    for (int k = 0; k < P; ++k) {
      img[l.f + (size_t)P * i + k] = fw[(size_t)W * i + 1 + k];
      img[l.b + (size_t)P * i + k] = bw[(size_t)W * i + 1 + k];
    }
    if (st->has_e)
      for (int k = 0; k < 3; ++k) img[l.e + (size_t)3 * i + k] = erows[(size_t)3 * i + k];
  }
  st->s64_ka = st->s64_kb = 0;
  if (rank > 0) {
    const size_t n = rank == 1 ? 2 * (size_t)N : 4 * (size_t)N + 12;
    std::copy_n(f->h_cyc.begin(), n, img.begin() + l.cyc);
    // rows whose coefficients (w and z of each rank, against that rank's largest) are
    // below 2^-100 change no digit of a solution in the 2-norm: 2^-47 of its rounding
    const int w = 2 * rank;
    std::vector<double> big(w, 0.0);
    for (int i = 0; i < N; ++i)
      for (int k = 0; k < w; ++k) big[k] = std::max(big[k], std::fabs(f->h_cyc[(size_t)w * i + k]));
    auto small = [&](int i) {
      for (int k = 0; k < w; ++k)
        if (std::fabs(f->h_cyc[(size_t)w * i + k]) > 0x1p-100 * big[k]) return false;
      return true;
    };
    // the widest run of small rows around the middle
    int ka = N / 2, kb = N / 2;
    while (ka > 0 && small(ka - 1)) --ka;
    while (kb < N && small(kb)) ++kb;
    // the end rows themselves always do: the correction is formed there
    st->s64_ka = ka = std::max(ka, rank);
    st->s64_kb = kb = std::min(kb, N - rank);
    st->s64_third = rank == 2 && kb - ka < N / 2;
  }
  DeviceGuard g(f->device);
  SB_TRY(g.rc);
  SB_CUDA(cudaMalloc(&st->s64, img.size() * sizeof(double)));
  return cuda_check(cudaMemcpy(st->s64, img.data(), img.size() * sizeof(double), cudaMemcpyHostToDevice),
                    "cudaMemcpy");
}

int step64(const sb_stepper* st, const double* src, double* state, int64_t M, int64_t ld, cudaStream_t s,
           double* ellm) {
  if (st->has_e) return dispatch<2, KCH>(st, src, state, M, ld, s, ellm);
  if (st->NB > 0)
    return st->fac->P == 1 ? dispatch<1, KCN>(st, src, state, M, ld, s, ellm)
                           : dispatch<2, KCN>(st, src, state, M, ld, s, ellm);
  return st->fac->P == 1 ? dispatch<1, KBE>(st, src, state, M, ld, s, ellm)
                         : dispatch<2, KBE>(st, src, state, M, ld, s, ellm);
}

int step64_forced(const sb_stepper* st, double* state, const double* amp, int64_t M, int64_t ld, cudaStream_t s) {
  if (st->s64_third)
    return st->adv >= 0.0 ? launch<2, KCH, 2, true, false, -1>(st, state, state, M, ld, s, nullptr, amp)
                          : launch<2, KCH, 2, true, false, +1>(st, state, state, M, ld, s, nullptr, amp);
  return st->adv >= 0.0 ? launch<2, KCH, 2, false, false, -1>(st, state, state, M, ld, s, nullptr, amp)
                        : launch<2, KCH, 2, false, false, +1>(st, state, state, M, ld, s, nullptr, amp);
}

}  // namespace sb
