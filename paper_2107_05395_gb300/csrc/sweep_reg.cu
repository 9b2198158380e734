// FP32 solves of short systems, each held whole in its thread's registers.
//
// A system of up to 128 rows fits in a thread: its rows are loaded once (every load of a
// tile in flight before the first is used), swept forward and back in place and stored
// once, 8 bytes an element (12 with an FP64 solution), with no intermediate in memory,
// no barrier and no partition.  The arithmetic and its order are those of the sequential
// sweeps, so the results are the same bits.
//
// Bound: DRAM.  A warp's rows are 128 bytes, which this memory moves at 5.4 TB/s; with
// two adjacent systems per lane they are 256 bytes (6.9 TB/s), taken for N <= 64 where
// the addresses are even and the batch still gives every SM eight warps.
// Microseconds, partitioned or sequential sweeps | this form: tridiagonal N = 64,
// M = 262144 80.6 | 27.1 (5.0 TB/s), M = 100000 33.4 | 10.6; N = 128, M = 262144
// 84.6 | 58.0; pentadiagonal N = 128, M = 100000 58.0 | 25.7; with an FP64 solution N = 100,
// M = 100001 39.1 | 33.3.  More rows do not fit the registers.
#include <algorithm>
#include <cstdint>

#include "sb_internal.h"
#include "sweep_tile.cuh"

namespace sb {
namespace {

template <typename T, int n>
struct alignas(sizeof(T) * n) RegVec {
  T v[n];
};

// Coefficient record of a row in shared memory: forward (P + 1), backward (P + 1), each
// padded to a power of two floats.
template <int P>
struct RegRow {
  static constexpr int W = P == 1 ? 2 : 4;
};

// NMAX rows in registers (NMAX / 2 < N <= NMAX, or N <= NMAX for the smallest), H adjacent
// systems per lane.
template <int P, bool F_ONE, bool B_ONE, typename TO, int NMAX, int H>
__global__ void __launch_bounds__(kRegThreads)
sweep_reg_kernel(const float* __restrict__ coef, int N, int64_t M, int64_t ld, const float* rhs, TO* x,
                 int64_t ntiles) {
  using F = NativeArith<float>;
  constexpr int W = RegRow<P>::W;
  constexpr int kSure = NMAX == 32 ? 0 : NMAX / 2;  // rows that every N of this form has
  using Rec = RegVec<float, W>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Rec* cs = reinterpret_cast<Rec*>(smem_raw);
  for (int k = threadIdx.x; k < 2 * N; k += kRegThreads)
#pragma unroll
    for (int e = 0; e < W; ++e) cs[k].v[e] = e <= P ? coef[k * (P + 1) + e] : 0.f;
  __syncthreads();
  const int64_t warps = (int64_t)gridDim.x * (kRegThreads / 32);
  for (int64_t tile = blockIdx.x + (int64_t)gridDim.x * (threadIdx.x >> 5); tile < ntiles; tile += warps) {
    const int64_t m = (tile * 32 + (threadIdx.x & 31)) * H;
    if (m >= M) return;  // H == 2: M is even
    RegVec<float, H> y[NMAX];
    const float* src = rhs + m;
#pragma unroll
    for (int j = 0; j < NMAX; ++j)
      if (j < kSure || j < N) {
        if constexpr (H == 2) {
          const float2 t = __ldcs(reinterpret_cast<const float2*>(src));
          y[j].v[0] = t.x;
          y[j].v[H - 1] = t.y;
        } else {
          y[j].v[0] = __ldcs(src);
        }
        src += ld;
      }
    float a1[H] = {}, a2[H] = {};
#pragma unroll
    for (int j = 0; j < NMAX; ++j)
      if (j < kSure || j < N) {
        const Rec c = cs[j];
#pragma unroll
        for (int h = 0; h < H; ++h) {
          const float u = F::step<P, F_ONE>(c.v, y[j].v[h], a1[h], a2[h]);
          y[j].v[h] = u;
          a2[h] = a1[h];
          a1[h] = u;
        }
      }
#pragma unroll
    for (int h = 0; h < H; ++h) a1[h] = a2[h] = 0.f;
    const Rec* cb = cs + N;
    TO* dst = x + m + (int64_t)(N - 1) * ld;
#pragma unroll
    for (int j = NMAX - 1; j >= 0; --j)
      if (j < kSure || j < N) {
        const Rec c = cb[j];
        RegVec<TO, H> o;
#pragma unroll
        for (int h = 0; h < H; ++h) {
          const float v = F::step<P, B_ONE>(c.v, y[j].v[h], a1[h], a2[h]);
          a2[h] = a1[h];
          a1[h] = v;
          if constexpr (sizeof(TO) == 8)
            o.v[h] = widen_f32(v);
          else
            o.v[h] = v;
        }
        if constexpr (H == 1)
          st_stream(dst, o.v[0]);
        else if constexpr (sizeof(TO) == 8)
          st_stream(reinterpret_cast<double2*>(dst), make_double2(o.v[0], o.v[H - 1]));
        else
          st_stream(reinterpret_cast<float2*>(dst), make_float2(o.v[0], o.v[H - 1]));
        dst -= ld;
      }
  }
}

template <int P, bool F_ONE, bool B_ONE, typename TO, int NMAX, int H>
int launch(const sb_factor* f, const float* coef, const float* rhs, TO* x, int64_t M, int64_t ld,
           cudaStream_t stream) {
  auto k = sweep_reg_kernel<P, F_ONE, B_ONE, TO, NMAX, H>;
  const size_t smem = (size_t)2 * f->N * RegRow<P>::W * sizeof(float);
  int nb = 0;
  SB_TRY(kernel_occupancy(reinterpret_cast<const void*>(k), f->device, kRegThreads, smem, &nb));
  const int64_t ntiles = (M + 32 * H - 1) / (32 * H);
  const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(ntiles, (int64_t)nb * sm_count(f->device)));
  k<<<(unsigned)grid, kRegThreads, smem, stream>>>(coef, (int)f->N, M, ld, rhs, x, ntiles);
  return cuda_check(cudaGetLastError(), "register-resident sweep launch");
}

template <int P, bool F_ONE, bool B_ONE, typename TO>
int dispatch(const sb_factor* f, const float* coef, const float* rhs, TO* x, int64_t M, int64_t ld,
             cudaStream_t stream) {
  const bool two = M % 2 == 0 && ld % 2 == 0 && (uintptr_t)rhs % 8 == 0 && (uintptr_t)x % (2 * sizeof(TO)) == 0 &&
                   M >= (int64_t)64 * 8 * sm_count(f->device);
  if (f->N <= 32)
    return two ? launch<P, F_ONE, B_ONE, TO, 32, 2>(f, coef, rhs, x, M, ld, stream)
               : launch<P, F_ONE, B_ONE, TO, 32, 1>(f, coef, rhs, x, M, ld, stream);
  if (f->N <= 64)
    return two ? launch<P, F_ONE, B_ONE, TO, 64, 2>(f, coef, rhs, x, M, ld, stream)
               : launch<P, F_ONE, B_ONE, TO, 64, 1>(f, coef, rhs, x, M, ld, stream);
  return launch<P, F_ONE, B_ONE, TO, 128, 1>(f, coef, rhs, x, M, ld, stream);
}

}  // namespace

bool reg_sweep_applies(const sb_factor* f, sb_dtype rt, sb_dtype xt, sb_arith arith) {
  return arith == SB_ARITH_NATIVE && rt == SB_F32 && (xt == SB_F32 || xt == SB_F64) && !f->periodic &&
         f->N <= kRegMaxRows;
}

int launch_reg_sweep(const sb_factor* f, Op op, const void* rhs, void* x, sb_dtype xt, int64_t M, int64_t ld,
                     cudaStream_t stream) {
  const float* c = f->coef32 + (op == OP_PRIMAL ? 0 : op_block_len(f->P, f->N));
  const float* b = static_cast<const float*>(rhs);
  auto go = [&](auto* xp) {
    using TO = std::remove_pointer_t<decltype(xp)>;
    if (f->P == 1)
      return op == OP_PRIMAL ? dispatch<1, false, true, TO>(f, c, b, xp, M, ld, stream)
                             : dispatch<1, true, false, TO>(f, c, b, xp, M, ld, stream);
    return op == OP_PRIMAL ? dispatch<2, false, true, TO>(f, c, b, xp, M, ld, stream)
                           : dispatch<2, true, false, TO>(f, c, b, xp, M, ld, stream);
  };
  return xt == SB_F32 ? go(static_cast<float*>(x)) : go(static_cast<double*>(x));
}

}  // namespace sb
