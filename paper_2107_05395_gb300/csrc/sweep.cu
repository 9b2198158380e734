// Batched forward/backward sweeps with one shared factor (Algorithms 2 and 4, and
// the transposed solve), for every arithmetic policy of arith.cuh.
//
// Mapping.  One thread owns one system m; a warp owns 32 consecutive systems (a
// "tile"), so every row access i*ld + m is one coalesced transaction per warp.
// CTAs are persistent: each stages the shared coefficients into shared memory
// once (the single device copy of section 2, broadcast from shared memory instead
// of the caches) and its warps then take tiles round-robin over the grid.
//
// Per system: the forward sweep reads the right-hand side and writes its
// intermediate (A::S, at most the size of an output element) in place into x; the
// backward sweep reads it back (the same thread, so no synchronisation) and
// writes the solution over it.  Rows are fetched R at a time into registers with
// double buffering: the next batch is in flight while the current one is swept.
#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>
#include <type_traits>

#include "sb_internal.h"
#include "sweep_tile.cuh"

namespace sb {
namespace {

// Per-op length of a periodic factor's correction data (rank 1 or 2).
__host__ __device__ constexpr int cyc_len(int rank, int N) { return rank == 1 ? 2 * N : rank == 2 ? 4 * N + 12 : 0; }

// Single-factor kernel: persistent CTAs stage the coefficients once, then their
// warps take tiles round-robin over the grid.  CYC: periodic matrices (rank-1
// tridiagonal of section 3.3, rank-2 cyclic pentadiagonal); the correction data is
// staged after the coefficients.  GC: the factors do not fit in shared memory
// (large N), so the sweeps read the single device copy directly (warp-uniform
// loads, served by L1/L2) instead of a staged one.
template <class A, int P, bool F_ONE, bool B_ONE, typename TI, typename TO, int SPT, int R,
          int CYC, bool GC = false>
__global__ void __launch_bounds__(512)
sweep_kernel(const typename A::C* __restrict__ coef, int N, int64_t M, int64_t ld,
             const TI* rhs, TO* x, int64_t ntiles, const typename A::C* __restrict__ cyc,
             typename A::C alpha, typename A::C beta) {
  using C = typename A::C;
  constexpr int W = P + 1;
  const C* fw;
  const C* cy;
  if constexpr (GC) {
    fw = coef;
    cy = cyc;
  } else {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* cs = reinterpret_cast<C*>(smem_raw);
    stage(cs, coef, 2 * W * N);
    if constexpr (CYC) stage(cs + 2 * W * N, cyc, cyc_len(CYC, N));
    __syncthreads();
    fw = cs;
    cy = cs + 2 * W * N;
  }
  const int nw = blockDim.x >> 5;
  for (int64_t tile = blockIdx.x + (int64_t)gridDim.x * (threadIdx.x >> 5); tile < ntiles;
       tile += (int64_t)gridDim.x * nw)
    sweep_tile<A, P, F_ONE, B_ONE, TI, TO, SPT, R, CYC>(fw, fw + W * N, N, M, ld, rhs, x, tile,
                                                         cy, alpha, beta);
}

// Staged single-factor kernel (SB_ALGO_STAGED): the coefficients as above, then a
// ring of kStagedRows slots per thread for the rows in flight (sweep_tile_staged),
// so that up to 1024 threads per CTA fit in the registers (512 in double-float
// arithmetic, whose values take two registers).
constexpr int kStagedRows = 8;
constexpr int kStagedBatch = 4;

template <class A>
__host__ __device__ constexpr int staged_max_threads() {
  return std::is_same_v<A, DFArith> ? 512 : 1024;
}

template <class A, int P, bool F_ONE, bool B_ONE, typename TI, typename TO>
__global__ void __launch_bounds__(staged_max_threads<A>())
sweep_staged_kernel(const typename A::C* __restrict__ coef, int N, int64_t M, int64_t ld, const TI* rhs,
                    TO* x, int64_t ntiles, unsigned ring_off) {
  using C = typename A::C;
  constexpr int W = P + 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* cs = reinterpret_cast<C*>(smem_raw);
  stage(cs, coef, 2 * W * N);
  __syncthreads();
  const int nw = blockDim.x >> 5;
  for (int64_t tile = blockIdx.x + (int64_t)gridDim.x * (threadIdx.x >> 5); tile < ntiles;
       tile += (int64_t)gridDim.x * nw)
    sweep_tile_staged<A, P, F_ONE, B_ONE, TI, TO, kStagedRows, kStagedBatch>(cs, cs + W * N, N, M, ld, rhs, x,
                                                                            tile, smem_raw + ring_off);
}

// Two-ended kernel (SB_ALGO_TWO_ENDED; FP64 rhs and x, native or double-float): every
// system is eliminated from both ends at once (two_ended.h).  A warp takes 16
// systems: lane l < 16 runs the top half of system l (rows 0 .. s-1 down, then back
// up from the interface) and lane l + 16 its bottom half (rows N-1 .. s up, then back
// down), so a batch gives twice as many warps, each with all 32 lanes busy.  That is
// what the FP64 unit wants: one warp issues at most one FP64 operation every 64 cycles
// however many independent ones it has, and an SM's unit takes one every 16, so it is
// the warps per SM that fill it.  The two halves of a system meet in the 2P x 2P
// interface system through one warp shuffle.  Each lane's rows go through a ring of
// kTwoRows slots in shared memory, as in the staged sweeps.
//
// The forward scaling F0 b is off the recurrence's chain and runs on the integer pipes
// (mulc_fast): the four products of a batch have one test between them, so they overlap
// each other and the FP64 unit; with a test and a branch in each product a warp took
// 500 cycles a row for one FP64 operation of 64.  Bound: the FP64 unit for pentadiagonal
// systems (N = 1024, M = 65536: 480 -> 457 us of a 428 us bound, the unit busy 95 % of the
// time; 4 and 12 bytes of the 64 registers spill, 0.002 loads a row), DRAM for tridiagonal
// ones whose intermediate leaves L2 (the same size: 399 -> 318 us, 2.1 GB), the latency of
// the rows for small batches (tridiagonal, N = 511, M = 30011: 125 -> 92 us; M = 1024:
// 77 -> 44 us).
// Shared memory: prepared F0 (N MulCoef) | F1[, F2] (P N) | B1[, B2] (P N) | the (2P)^2
// interface inverse | ring.
constexpr int kTwoRows = 8;
constexpr int kTwoBatch = 4;

// Arithmetic of the two-ended sweeps: what a row's coefficients are, how a batch of K
// right-hand sides enters (in(j): row j exists), the two recurrences, and how a batch of
// solutions leaves.
template <int P>
struct alignas(8 * P) TwoRow {
  double v[P];
};
template <int P>
struct alignas(8 * P) TwoRowDf {
  df v[P];
};

template <int P>
struct Ends64 {
  static constexpr int kMaxThreads = 1024, kMinCtas = 1;
  using V = double;
  using Pre = MulCoef;  // F0
  using Row = TwoRow<P>;
  static __device__ __forceinline__ V zero() { return 0.0; }
  static __device__ __forceinline__ bool prepare(Pre& p, const double* img) {
    p = mulc_prepare(*img);
    return mulc_usable(*img);
  }
  // F0 b on the integer pipes, one test for the batch
  template <int K, class In>
  static __device__ __forceinline__ void enter(V (&s)[K], const double (&b)[K], const Pre* c, int step,
                                               const Pre* any, bool fast, In in) {
    bool ok = fast;
#pragma unroll
    for (int j = 0; j < K; ++j) {
      ok = ok && mulc_ok(b[j]);
      s[j] = mulc_fast(b[j], *(in(j) ? c + j * step : any));
    }
    if (!ok) {
#pragma unroll
      for (int j = 0; j < K; ++j)
        if (in(j)) {
          const Pre w = c[j * step];
          s[j] = mulc_slow(b[j], w.lo, w.hi, w.ck);
        }
    }
  }
  static __device__ __forceinline__ V forward(const Pre*, const Row& c, V s, V v1, V v2) {
    V u = fma(-c.v[0], v1, s);
    if constexpr (P == 2) u = fma(-c.v[P - 1], v2, u);
    return u;
  }
  static __device__ __forceinline__ V backward(const Row& c, V u, V x1, V x2) {
    V x = fma(-c.v[0], x1, u);
    if constexpr (P == 2) x = fma(-c.v[P - 1], x2, x);
    return x;
  }
  static __device__ __forceinline__ V fmac(V c, V v, V acc) { return fma(c, v, acc); }
  template <int K>
  static __device__ __forceinline__ void leave(double (&o)[K], const V (&x)[K]) {
#pragma unroll
    for (int j = 0; j < K; ++j) o[j] = x[j];
  }
};

// Double-float: the image after the FP64 one holds the same values as (hi, lo) pairs.
// Both conversions test a batch at once, like the products above: a conversion with its
// own branch is a scheduling barrier between rows, and the sweep is bound by issue (66 %
// of the slots at N = 512, M = 65536, pentadiagonal: 174 us, 259 with one-ended sweeps;
// 127 instructions an element, where DRAM would take 79 us for its 16 bytes).  At 72
// registers 20 bytes (tridiagonal) and 40 spill, 0.05 loads an element; 64 spill more.
struct DfBatch {
  df v[kTwoBatch];
};
// A batch with a value that the branchless split does not take, out of line as a whole: one
// call for the batch, and its zeros (point sources, padded states) need no FP64 unit.  N =
// 512, M = 65536, tridiagonal, point sources: 405 -> 225 us with four calls -> this (dense
// 168); a test for zeros in every conversion cost dense double-float steps 2 %.
__device__ __noinline__ DfBatch double_to_df_batch(double b0, double b1, double b2, double b3) {
  static_assert(kTwoBatch == 4);
  const double b[kTwoBatch] = {b0, b1, b2, b3};
  DfBatch r;
#pragma unroll
  for (int j = 0; j < kTwoBatch; ++j) {
    r.v[j] = double_to_df_fast(b[j]);
    if (((d_hi(b[j]) & 0x7FFFFFFFu) | d_lo(b[j])) == 0u)
      r.v[j] = df{u2f(d_hi(b[j])), 0.f};
    else if (!double_to_df_ok(b[j]))
      r.v[j] = double_to_df_slow(b[j]);  // a call, or its FP64 operations would run for all
  }
  return r;
}

template <int P>
struct EndsDf {
  static constexpr int kMaxThreads = 448, kMinCtas = 2;  // 72 registers
  using V = df;
  using Pre = df;  // F0
  using Row = TwoRowDf<P>;
  static __device__ __forceinline__ V zero() { return df{0.f, 0.f}; }
  static __device__ __forceinline__ bool prepare(Pre& p, const double* img) {
    p = *reinterpret_cast<const df*>(img);
    return true;
  }
  template <int K, class In>
  static __device__ __forceinline__ void enter(V (&s)[K], const double (&b)[K], const Pre*, int, const Pre*, bool,
                                               In) {
    bool ok = true;
#pragma unroll
    for (int j = 0; j < K; ++j) {
      ok = ok && double_to_df_ok(b[j]);
      s[j] = double_to_df_fast(b[j]);
    }
    if (!ok) {
      static_assert(K == kTwoBatch);
      const DfBatch r = double_to_df_batch(b[0], b[1], b[2], b[3]);
#pragma unroll
      for (int j = 0; j < K; ++j) s[j] = r.v[j];
    }
  }
  static __device__ __forceinline__ V forward(const Pre* p, const Row& c, V s, V v1, V v2) {
    const df w[3] = {*p, c.v[0], c.v[P - 1]};
    return DFArith::step<P, false>(w, s, v1, v2);
  }
  static __device__ __forceinline__ V backward(const Row& c, V u, V x1, V x2) {
    const df w[3] = {df{0.f, 0.f}, c.v[0], c.v[P - 1]};
    return DFArith::step<P, true>(w, u, x1, x2);
  }
  static __device__ __forceinline__ V fmac(V c, V v, V acc) { return DFArith::fmac(c, v, acc); }
  template <int K>
  static __device__ __forceinline__ void leave(double (&o)[K], const V (&x)[K]) {
    bool ok = true;
#pragma unroll
    for (int j = 0; j < K; ++j) {
      ok = ok && widen_f32_ok(x[j].h) && widen_f32_ok(x[j].l);
      o[j] = widen_f32_fast(x[j].h) + widen_f32_fast(x[j].l);
    }
    if (!ok) {
#pragma unroll
      for (int j = 0; j < K; ++j) o[j] = df_to_double(x[j]);
    }
  }
};

template <int P>
constexpr size_t two_ended_smem(int N, int threads, bool dfl) {
  return ((size_t)N * (dfl ? sizeof(df) : sizeof(MulCoef)) + 15) / 16 * 16 + 2 * N * sizeof(TwoRow<P>) +
         4 * P * P * sizeof(double) +
         (size_t)kTwoRows * threads * sizeof(double);
}

template <int P, class E>
__device__ __forceinline__ void two_ended_tile(const typename E::Pre* pc, const typename E::Row* fw,
                                               const typename E::Row* bw, const typename E::V* minv, bool fast, int N, int s, int64_t M,
                                               int64_t ld, const double* rhs, double* x, int64_t tile,
                                               double* ring) {
  constexpr int D = kTwoRows;
  constexpr int K = kTwoBatch;
  constexpr int NZ = 2 * P;
  using V = typename E::V;
  using Row = typename E::Row;
  static_assert(sizeof(V) == sizeof(double), "an intermediate takes a solution's place");
  static_assert(D == 2 * K, "the ring is two batches");
  const int lane = threadIdx.x & 31;
  const bool top = lane < 16;
  const int64_t m = tile * 16 + (lane & 15);
  // lanes l and l + 16 hold the same system, so both are in the mask or neither
  const unsigned mask = __ballot_sync(0xffffffffu, m < M);
  if (m >= M) return;
  double* y = x + m;
  const int T = blockDim.x;
  // slots of an even batch and of an odd one
  double* slot[2][K];
#pragma unroll
  for (int k = 0; k < D; ++k) slot[k / K][k % K] = ring + threadIdx.x + k * T;
  __threadfence_block();  // this thread's stores of the previous tile before the copies below

  // ---- forward: step t is row t (top) or row N-1-t (bottom); u in place in x
  const int nf = top ? s : N - s;
  const int TF = s, NF = N - s;  // s = ceil(N / 2): every lane has rows up to NF
  const int64_t step = top ? ld : -ld;
  const int cstep = top ? 1 : -1;
  const double* src = rhs + m + (top ? 0 : (int64_t)(N - 1) * ld);  // row the next copy reads
  double* dst = y + (top ? 0 : (int64_t)(N - 1) * ld);              // row the next u goes to
  const int i0 = top ? 0 : N - 1;
  const typename E::Pre* cp = pc + i0;
  const Row* cf = fw + i0;
  auto issue_f = [&](double* to, int t) {
    if (t < nf) cp_async<8>(to, src);
    src += step;
    cp_commit();
  };
#pragma unroll
  for (int t = 0; t < D; ++t) issue_f(slot[t / K][t % K], t);
  V v1 = E::zero(), v2 = E::zero();
  // rows t0 .. t0+K-1; GUARD: only those below nf
  auto batch_f = [&](int t0, double* (&sl)[K], auto guard) {
    constexpr bool GUARD = decltype(guard)::value;
    cp_wait<D - K>();
    auto in = [&](int j) { return !GUARD || t0 + j < nf; };
    double b[K];
    V sc[K];
#pragma unroll
    for (int j = 0; j < K; ++j) b[j] = in(j) ? *sl[j] : 1.0;
    E::template enter<K>(sc, b, cp, cstep, pc, fast, in);
#pragma unroll
    for (int j = 0; j < K; ++j)
      if (in(j)) {
        const V u = E::forward(cp + j * cstep, cf[j * cstep], sc[j], v1, v2);
        *reinterpret_cast<V*>(dst) = u;
        dst += step;
        v2 = v1;
        v1 = u;
      }
    cp += K * cstep;
    cf += K * cstep;
#pragma unroll
    for (int j = 0; j < K; ++j) issue_f(sl[j], t0 + D + j);  // refills the slots used above
  };
  int t0 = 0;
  for (; t0 + D <= NF; t0 += D) {
    batch_f(t0, slot[0], std::false_type{});
    batch_f(t0 + K, slot[1], std::false_type{});
  }
  for (; t0 < TF; t0 += D) {
    batch_f(t0, slot[0], std::true_type{});
    batch_f(t0 + K, slot[1], std::true_type{});
  }
  cp_wait<0>();
  __threadfence_block();  // the stores of u before the copies that read them back

  // ---- interface: z = (x_{s-P} .. x_{s+P-1}) = Minv (u_{s-P} .. u_{s+P-1}); the top
  // lane ends at u_{s-1} (v1), u_{s-2} (v2), the bottom lane at u_s (v1), u_{s+1} (v2)
  auto other = [&](V v) {
    double t = __shfl_xor_sync(mask, *reinterpret_cast<double*>(&v), 16);
    return *reinterpret_cast<V*>(&t);
  };
  const V o1 = other(v1), o2 = other(v2);
  V uz[NZ];
  if constexpr (P == 2) {
    uz[0] = top ? v2 : o2;
    uz[1] = top ? v1 : o1;
    uz[2] = top ? o1 : v1;
    uz[3] = top ? o2 : v2;
  } else {
    uz[0] = top ? v1 : o1;
    uz[1] = top ? o1 : v1;
  }
  const int j0 = top ? 0 : P;  // this lane's interface rows: s-P .. s-1 (top), s .. s+P-1
  V z[P];
#pragma unroll
  for (int jj = 0; jj < P; ++jj) {
    const int j = j0 + jj;
    V v = E::zero();
#pragma unroll
    for (int q = 0; q < NZ; ++q) v = E::fmac(minv[j * NZ + q], uz[q], v);
    z[jj] = v;
  }
  double zo[P];
  E::template leave<P>(zo, z);
#pragma unroll
  for (int jj = 0; jj < P; ++jj) st_stream(y + (int64_t)(s - P + j0 + jj) * ld, zo[jj]);

  // ---- backward: rows s-P-1 .. 0 (top) or s+P .. N-1 (bottom)
  const int nbk = top ? s - P : N - s - P;
  const int TB = s - P, NBK = N - s - P;
  const int b0 = top ? s - P - 1 : s + P;
  const double* bsrc = y + (int64_t)b0 * ld;
  double* bdst = y + (int64_t)b0 * ld;
  const Row* cb = bw + b0;
  auto issue_b = [&](double* to, int t) {
    if (t < nbk) cp_async<8>(to, bsrc);
    bsrc -= step;
    cp_commit();
  };
#pragma unroll
  for (int t = 0; t < D; ++t) issue_b(slot[t / K][t % K], t);
  // the two nearest solved rows: x_{i+1}, x_{i+2} (top) or x_{i-1}, x_{i-2} (bottom)
  V x1 = top ? z[0] : z[P - 1];
  V x2 = P == 2 ? (top ? z[P - 1] : z[0]) : E::zero();
  auto batch_b = [&](int t0b, double* (&sl)[K], auto guard) {
    constexpr bool GUARD = decltype(guard)::value;
    cp_wait<D - K>();
    V xs[K];
#pragma unroll
    for (int j = 0; j < K; ++j) {
      xs[j] = x1;
      if (!GUARD || t0b + j < nbk) {
        xs[j] = E::backward(cb[-j * cstep], *reinterpret_cast<const V*>(sl[j]), x1, x2);
        x2 = x1;
        x1 = xs[j];
      }
    }
    double o[K];
    E::template leave<K>(o, xs);
#pragma unroll
    for (int j = 0; j < K; ++j)
      if (!GUARD || t0b + j < nbk) {
        st_stream(bdst, o[j]);
        bdst -= step;
      }
    cb -= K * cstep;
#pragma unroll
    for (int j = 0; j < K; ++j) issue_b(sl[j], t0b + D + j);
  };
  int tb = 0;
  for (; tb + D <= NBK; tb += D) {
    batch_b(tb, slot[0], std::false_type{});
    batch_b(tb + K, slot[1], std::false_type{});
  }
  for (; tb < TB; tb += D) {
    batch_b(tb, slot[0], std::true_type{});
    batch_b(tb + K, slot[1], std::true_type{});
  }
  cp_wait<0>();
}

template <int P, class E>
__global__ void __launch_bounds__(E::kMaxThreads, E::kMinCtas)
sweep_two_ended_kernel(const double* __restrict__ img, int N, int s, int64_t M, int64_t ld, const double* rhs,
                       double* x, int64_t ntiles) {
  constexpr int W = P + 1;
  using Row = typename E::Row;
  using V = typename E::V;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  typename E::Pre* pc = reinterpret_cast<typename E::Pre*>(smem_raw);
  Row* fw = reinterpret_cast<Row*>(smem_raw + ((size_t)N * sizeof(*pc) + 15) / 16 * 16);
  Row* bw = fw + N;
  V* minv = reinterpret_cast<V*>(bw + N);
  double* ring = reinterpret_cast<double*>(minv + 4 * P * P);
  const V* vi = reinterpret_cast<const V*>(img);
  bool usable = true;
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    usable = E::prepare(pc[i], img + W * i) && usable;
#pragma unroll
    for (int k = 0; k < P; ++k) {
      fw[i].v[k] = vi[W * i + 1 + k];
      bw[i].v[k] = vi[W * N + W * i + 1 + k];
    }
  }
  for (int k = threadIdx.x; k < 4 * P * P; k += blockDim.x) minv[k] = vi[2 * W * N + k];
  const bool fast = __syncthreads_and(usable);
  const int nw = blockDim.x >> 5;
  for (int64_t tile = blockIdx.x + (int64_t)gridDim.x * (threadIdx.x >> 5); tile < ntiles;
       tile += (int64_t)gridDim.x * nw)
    two_ended_tile<P, E>(pc, fw, bw, minv, fast, N, s, M, ld, rhs, x, tile, ring);
}

// The periodic correction data of a factor for an arithmetic policy: (w_i, -z_i)
// rows of op `o` and the scalars alpha, beta as coefficients.
template <class A>
struct CycData;
template <>
struct CycData<NativeArith<double>> {
  static const double* rows(const sb_factor* f, int o) {
    return f->cyc64 ? f->cyc64 + cyc_len(f->periodic_rank, (int)f->N) * o : nullptr;
  }
  static double coef(double v) { return v; }
};
template <>
struct CycData<NativeArith<float>> {
  static const float* rows(const sb_factor* f, int o) {
    return f->cyc32 ? f->cyc32 + cyc_len(f->periodic_rank, (int)f->N) * o : nullptr;
  }
  static float coef(double v) { return (float)v; }
};
template <>
struct CycData<DFArith> {
  static const df* rows(const sb_factor* f, int o) {
    return f->cycdf ? reinterpret_cast<const df*>(f->cycdf) + cyc_len(f->periodic_rank, (int)f->N) * o
                    : nullptr;
  }
  static df coef(double v) {
    const float h = (float)v;
    return df{h, (float)(v - (double)h)};
  }
};

// ----------------------------------------------------------------- launching

template <class A, int P, bool F_ONE, bool B_ONE, typename TI, typename TO, int SPT, int R,
          int CYC>
int launch(const sb_factor* f, const typename A::C* coef, const void* rhs, void* x, int64_t M,
           int64_t ld, const SweepShape& shape, cudaStream_t stream, int op) {
  using C = typename A::C;
  const int N = (int)f->N;
  size_t smem = ((size_t)2 * (P + 1) * N + (size_t)cyc_len(CYC, N)) * sizeof(C);
  auto k = sweep_kernel<A, P, F_ONE, B_ONE, TI, TO, SPT, R, CYC>;
  if (smem > (size_t)kMaxDynSmem) {
    // FP64 factors of a large N are read from device memory; the other policies
    // keep the staged form only
    if constexpr (std::is_same_v<A, NativeArith<double>> && std::is_same_v<TI, double> &&
                  std::is_same_v<TO, double>) {
      k = sweep_kernel<A, P, F_ONE, B_ONE, TI, TO, SPT, R, CYC, true>;
      smem = 0;
    } else {
      return fail(SB_ERR_UNSUPPORTED,
                  "N=%d: the shared factors (%zu B) exceed the shared memory of one CTA "
                  "(only FP64 solves read them from device memory)", N, smem);
    }
  }
  const int threads = shape.threads;
  if (threads < 32 || threads > 512 || threads % 32 != 0)
    return fail(SB_ERR_INVALID_ARG, "threads per CTA must be a multiple of 32 in [32, 512]");
  int nb = 0;
  SB_TRY(kernel_occupancy(reinterpret_cast<const void*>(k), f->device, threads, smem, &nb));
  if (shape.ctas_per_sm > 0) nb = std::min(nb, shape.ctas_per_sm);
  const int64_t ntiles = (M + 32 * SPT - 1) / (32 * SPT);
  // one CTA per resident slot at most, tiles dealt round-robin over the CTAs first
  // (tile = block + grid * warp) so that every SM gets an equal share
  const int64_t grid =
      std::max<int64_t>(1, std::min<int64_t>(ntiles, (int64_t)nb * sm_count(f->device)));
  const C* cyc = CYC ? CycData<A>::rows(f, op) : nullptr;
  const C alpha = CycData<A>::coef(CYC ? f->cyc_alpha[op] : 0.0);
  const C beta = CycData<A>::coef(CYC ? f->cyc_beta[op] : 0.0);
  k<<<(unsigned)grid, threads, smem, stream>>>(coef, N, M, ld, static_cast<const TI*>(rhs),
                                              static_cast<TO*>(x), ntiles, cyc, alpha, beta);
  return cuda_check(cudaGetLastError(), "sweep kernel launch");
}

// The staged sweeps; *applied = false (nothing launched, SB_OK) where they do not
// apply: periodic factors, or coefficients and ring beyond one CTA's shared memory.
template <class A, int P, bool F_ONE, bool B_ONE, typename TI, typename TO, int CYC>
int launch_staged(const sb_factor* f, const typename A::C* coef, const void* rhs, void* x, int64_t M,
                  int64_t ld, const SweepShape& shape, cudaStream_t stream, bool* applied) {
  using C = typename A::C;
  *applied = false;
  if constexpr (CYC != 0) {
    return SB_OK;
  } else {
    const int N = (int)f->N;
    const int threads = shape.threads;
    if (threads < 32 || threads > staged_max_threads<A>() || threads % 32 != 0)
      return fail(SB_ERR_INVALID_ARG, "threads per CTA must be a multiple of 32 in [32, %d] for the staged sweeps",
                  staged_max_threads<A>());
    const size_t ring_off = ((size_t)2 * (P + 1) * N * sizeof(C) + 15) / 16 * 16;
    const size_t smem =
        ring_off + (size_t)kStagedRows * threads * staged_slot_bytes<TI, typename A::S>();
    if (smem > (size_t)kMaxDynSmem) return SB_OK;
    *applied = true;
    auto k = sweep_staged_kernel<A, P, F_ONE, B_ONE, TI, TO>;
    int nb = 0;
    SB_TRY(kernel_occupancy(reinterpret_cast<const void*>(k), f->device, threads, smem, &nb));
    if (shape.ctas_per_sm > 0) nb = std::min(nb, shape.ctas_per_sm);
    const int64_t ntiles = (M + 31) / 32;
    const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(ntiles, (int64_t)nb * sm_count(f->device)));
    k<<<(unsigned)grid, threads, smem, stream>>>(coef, N, M, ld, static_cast<const TI*>(rhs),
                                                static_cast<TO*>(x), ntiles, (unsigned)ring_off);
    return cuda_check(cudaGetLastError(), "staged sweep kernel launch");
  }
}

// The two-ended sweeps of op (A or A^T); *applied = false (nothing launched, SB_OK)
// where they do not apply: no image (periodic factor, N < 4P, a zero pivot or a
// singular interface), or image and ring beyond one CTA's shared memory.
int launch_two_ended(const sb_factor* f, Op op, bool dfl, const void* rhs, void* x, int64_t M, int64_t ld,
                     const SweepShape& shape, cudaStream_t stream, bool* applied) {
  *applied = false;
  const double* img = f->two_img[op == OP_PRIMAL ? 0 : 1];
  if (img == nullptr) return SB_OK;
  const int N = (int)f->N, P = f->P, threads = shape.threads;
  if (threads < 32 || threads > 1024 || threads % 32 != 0)
    return fail(SB_ERR_INVALID_ARG, "threads per CTA must be a multiple of 32 in [32, 1024] for the two-ended sweeps");
  const size_t smem = P == 1 ? two_ended_smem<1>(N, threads, dfl) : two_ended_smem<2>(N, threads, dfl);
  if (smem > (size_t)kMaxDynSmem || (dfl && threads > EndsDf<1>::kMaxThreads)) return SB_OK;
  *applied = true;
  if (dfl) img += 2 * (P + 1) * N + 4 * P * P;  // the (hi, lo) image follows
  auto k = dfl ? (P == 1 ? sweep_two_ended_kernel<1, EndsDf<1>> : sweep_two_ended_kernel<2, EndsDf<2>>)
               : (P == 1 ? sweep_two_ended_kernel<1, Ends64<1>> : sweep_two_ended_kernel<2, Ends64<2>>);
  int nb = 0;
  SB_TRY(kernel_occupancy(reinterpret_cast<const void*>(k), f->device, threads, smem, &nb));
  if (shape.ctas_per_sm > 0) nb = std::min(nb, shape.ctas_per_sm);
  const int64_t ntiles = (M + 15) / 16;  // 16 systems per warp
  const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(ntiles, (int64_t)nb * sm_count(f->device)));
  k<<<(unsigned)grid, threads, smem, stream>>>(img, N, f->two_s, M, ld, static_cast<const double*>(rhs),
                                              static_cast<double*>(x), ntiles);
  return cuda_check(cudaGetLastError(), "two-ended sweep kernel launch");
}

template <class A, int P, bool F_ONE, bool B_ONE, typename TI, typename TO, int CYC>
int launch_spt(const sb_factor* f, const typename A::C* coef, const void* rhs, void* x, int64_t M,
               int64_t ld, const SweepShape& shape, cudaStream_t stream, int op) {
  if (shape.algo == SB_ALGO_STAGED) {
    bool applied = false;
    const int rc = launch_staged<A, P, F_ONE, B_ONE, TI, TO, CYC>(f, coef, rhs, x, M, ld, shape, stream, &applied);
    if (rc != SB_OK || applied) return rc;
    // where the staged sweeps do not apply, the sequential ones with the default shape
    const sb_arith arith = std::is_same_v<A, DFArith> ? SB_ARITH_DF32 : SB_ARITH_NATIVE;
    return launch_spt<A, P, F_ONE, B_ONE, TI, TO, CYC>(f, coef, rhs, x, M, ld, default_shape(f, arith), stream, op);
  }
  if (shape.spt == 2)
    return launch<A, P, F_ONE, B_ONE, TI, TO, 2, 4, CYC>(f, coef, rhs, x, M, ld, shape, stream, op);
  if (shape.spt != 1) return fail(SB_ERR_INVALID_ARG, "systems per thread must be 1 or 2");
  return launch<A, P, F_ONE, B_ONE, TI, TO, 1, kRows, CYC>(f, coef, rhs, x, M, ld, shape, stream, op);
}

template <class A, typename TI, typename TO>
int dispatch_pb(const sb_factor* f, Op op, const typename A::C* base, const void* rhs, void* x,
                int64_t M, int64_t ld, const SweepShape& shape, cudaStream_t stream) {
  const typename A::C* c = base + (op == OP_PRIMAL ? 0 : op_block_len(f->P, f->N));
  const int o = op == OP_PRIMAL ? 0 : 1;
  if (f->P == 1) {
    if (f->periodic)
      return op == OP_PRIMAL
                 ? launch_spt<A, 1, false, true, TI, TO, 1>(f, c, rhs, x, M, ld, shape, stream, o)
                 : launch_spt<A, 1, true, false, TI, TO, 1>(f, c, rhs, x, M, ld, shape, stream, o);
    return op == OP_PRIMAL
               ? launch_spt<A, 1, false, true, TI, TO, 0>(f, c, rhs, x, M, ld, shape, stream, o)
               : launch_spt<A, 1, true, false, TI, TO, 0>(f, c, rhs, x, M, ld, shape, stream, o);
  }
  if (f->periodic)
    return op == OP_PRIMAL
               ? launch_spt<A, 2, false, true, TI, TO, 2>(f, c, rhs, x, M, ld, shape, stream, o)
               : launch_spt<A, 2, true, false, TI, TO, 2>(f, c, rhs, x, M, ld, shape, stream, o);
  return op == OP_PRIMAL
             ? launch_spt<A, 2, false, true, TI, TO, 0>(f, c, rhs, x, M, ld, shape, stream, o)
             : launch_spt<A, 2, true, false, TI, TO, 0>(f, c, rhs, x, M, ld, shape, stream, o);
}

}  // namespace

namespace {
std::mutex g_occ_mu;
std::map<std::tuple<const void*, int, int, size_t>, int> g_occ;
}  // namespace

// The shared-memory attribute below belongs to (kernel, device), so the device is part of
// the key: a kernel's first launch on another device has to set it there too.
int kernel_occupancy(const void* kernel, int device, int threads, size_t smem, int* blocks_per_sm) {
  const auto key = std::make_tuple(kernel, device, threads, smem);
  {
    std::lock_guard<std::mutex> lk(g_occ_mu);
    auto it = g_occ.find(key);
    if (it != g_occ.end()) {
      *blocks_per_sm = it->second;
      return SB_OK;
    }
  }
  SB_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynSmem));
  int nb = 0;
  SB_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel, threads, smem));
  if (nb < 1)
    return fail(SB_ERR_UNSUPPORTED, "kernel cannot be resident (%d threads, %zu B smem)", threads, smem);
  std::lock_guard<std::mutex> lk(g_occ_mu);
  g_occ[key] = nb;
  *blocks_per_sm = nb;
  return SB_OK;
}

bool two_ended_applies(const sb_factor* f, Op op, sb_arith arith, int threads) {
  const int N = (int)f->N;
  const bool dfl = arith == SB_ARITH_DF32;
  const size_t smem = f->P == 1 ? two_ended_smem<1>(N, threads, dfl) : two_ended_smem<2>(N, threads, dfl);
  return f->two_img[op == OP_PRIMAL ? 0 : 1] != nullptr && smem <= (size_t)kMaxDynSmem &&
         (!dfl || threads <= EndsDf<1>::kMaxThreads);
}

SweepShape default_shape(const sb_factor* f, sb_arith arith) {
  SweepShape s;
  s.threads = (arith == SB_ARITH_DF32) ? 128 : 256;
  s.ctas_per_sm = 0;  // occupancy limit
  s.spt = 1;
  (void)f;
  return s;
}

int launch_sweep(const sb_factor* f, Op op, const void* rhs, sb_dtype rhs_dtype, void* x,
                 sb_dtype x_dtype, int64_t M, int64_t ld, sb_arith arith, const SweepShape& shape,
                 cudaStream_t stream) {
  // beyond 64 rows a batch of up to two 32-system tiles an SM is faster partitioned, where
  // its rows allow TMA (microseconds, registers | partitioned, N = 128: tridiagonal M =
  // 2000 5.5 | 3.7, M = 20000 6.2 | 9.3; pentadiagonal M = 1000 6.7 | 4.8, M = 8000 9.2 | 8.3)
  if (shape.reg && reg_sweep_applies(f, rhs_dtype, x_dtype, arith) &&
      !(f->N > 64 && M <= 2 * 32 * (int64_t)sm_count(f->device) && shape.algo == SB_ALGO_PARTITIONED &&
        partitioned_applies(f, op, rhs, rhs_dtype, x_dtype, M, ld, arith, shape.threads)))
    return launch_reg_sweep(f, op, rhs, x, x_dtype, M, ld, stream);
  if (shape.chip && chip_sweep_fits(f, rhs_dtype, x_dtype, arith))
    return launch_chip_sweep(f, op, rhs, x, x_dtype, M, ld, stream);
  if (shape.algo == SB_ALGO_PARTITIONED && shape.threads == kPart64Threads) {
    if (partitioned64_applies(f, op, rhs_dtype, x_dtype, M, arith))
      return launch_partitioned64(f, op, rhs, x, M, ld, shape, stream);
    return launch_sweep(f, op, rhs, rhs_dtype, x, x_dtype, M, ld, arith, default_shape(f, arith),
                        stream);
  }
  if (shape.algo == SB_ALGO_PARTITIONED) {
    if (partitioned_applies(f, op, rhs, rhs_dtype, x_dtype, M, ld, arith, shape.threads))
      return launch_partitioned(f, op, rhs, rhs_dtype, x, x_dtype, M, ld, arith, shape, stream);
    // where the partition does not apply (sizes, dtypes, alignment) the sequential sweeps
    // run, of systems held on chip where that is faster (the same bits), else with their
    // default shape
    if (chip_sweep_applies(f, rhs_dtype, x_dtype, M, arith))
      return launch_chip_sweep(f, op, rhs, x, x_dtype, M, ld, stream);
    return launch_sweep(f, op, rhs, rhs_dtype, x, x_dtype, M, ld, arith, default_shape(f, arith),
                        stream);
  }
  if (shape.algo == SB_ALGO_TWO_ENDED) {
    if (rhs_dtype == SB_F64 && x_dtype == SB_F64) {
      bool applied = false;
      const int rc = launch_two_ended(f, op, arith == SB_ARITH_DF32, rhs, x, M, ld, shape, stream, &applied);
      if (rc != SB_OK || applied) return rc;
    }
    // where the two-ended sweeps do not apply, the sequential ones with the default shape
    return launch_sweep(f, op, rhs, rhs_dtype, x, x_dtype, M, ld, arith, default_shape(f, arith), stream);
  }
  if (shape.algo != SB_ALGO_SEQUENTIAL && shape.algo != SB_ALGO_STAGED)
    return fail(SB_ERR_INVALID_ARG, "unknown algorithm %d", shape.algo);
  if (arith == SB_ARITH_NATIVE) {
    if (rhs_dtype == SB_F64 && x_dtype == SB_F64)
      return dispatch_pb<NativeArith<double>, double, double>(f, op, f->coef64, rhs, x, M, ld,
                                                              shape, stream);
    if (rhs_dtype == SB_F32 && x_dtype == SB_F32)
      return dispatch_pb<NativeArith<float>, float, float>(f, op, f->coef32, rhs, x, M, ld, shape,
                                                           stream);
    if (rhs_dtype == SB_F32 && x_dtype == SB_F64)
      return dispatch_pb<NativeArith<float>, float, double>(f, op, f->coef32, rhs, x, M, ld,
                                                            shape, stream);
  } else if (arith == SB_ARITH_DF32) {
    const df* c = reinterpret_cast<const df*>(f->coefdf);
    if (rhs_dtype == SB_F64 && x_dtype == SB_F64)
      return dispatch_pb<DFArith, double, double>(f, op, c, rhs, x, M, ld, shape, stream);
    if (rhs_dtype == SB_F32 && x_dtype == SB_F64)
      return dispatch_pb<DFArith, float, double>(f, op, c, rhs, x, M, ld, shape, stream);
  }
  return fail(SB_ERR_UNSUPPORTED, "unsupported combination: rhs dtype %d, x dtype %d, arith %d",
              (int)rhs_dtype, (int)x_dtype, (int)arith);
}

}  // namespace sb
