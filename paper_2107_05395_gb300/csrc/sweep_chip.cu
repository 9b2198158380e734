// FP32 solves whose rows TMA cannot copy (a right-hand side or leading dimension that is
// not a multiple of 16 bytes): 32 systems at a time held whole in shared memory.
//
// The partitioned solve of partition.cu, which aligned rows take, joins its chunks with
// extra FP32 operations; these calls took the sequential sweeps, and here they get the
// arithmetic and the order of those, hence the same bits, without their trips to memory.
// (The partitioned solve with cp.async copies had 1.06 times the sequential sweeps' error
// against FP64 in the median of 195 matrices, 1.32 times at most.)
//
// One warp of a CTA sweeps; its time is the chain of 2 N rows, so it does nothing else: the
// other three copy the tile in and the solution out, a quarter of the rows behind or ahead
// of it, and refill the rows of a stored quarter with the next tile's.  Every element is
// copied, stored and replaced by the same thread, and the four quarters change hands at
// barriers of the CTA.  A system's rows lie in fours, so that the sweeping warp reads and
// writes 16 bytes at a time: with 4-byte accesses it took 25 ns a row, now 12 (17 a
// pentadiagonal one).
//
// Microseconds, sequential | partitioned with cp.async | this form (chip_sweep_applies
// draws the line): tridiagonal N = 1000: M = 501 134 | 13.3 | 19.9, M = 60001 217 | 138 |
// 213; N = 256: M = 6001 37.5 | 11.6 | 13.2, M = 60001 52 | 51 | 41; pentadiagonal N = 512:
// M = 6001 77 | 19 | 21, M = 20001 88 | 36 | 43; with an FP64 solution, tridiagonal N = 130,
// M = 240001 184 | 123 | 98, pentadiagonal N = 256, M = 60001 76 | 66 | 49.
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "sb_internal.h"
#include "sweep_tile.cuh"

namespace sb {
namespace {

constexpr int kChipThreads = 128;
constexpr int kChipBatch = 8;  // rows the sweeping warp reads at once
constexpr int kChipParts = 4;

// Coefficients of a row of one sweep (P + 1), padded to a power of two.
template <int P>
struct alignas(P == 1 ? 8 : 16) ChipRec {
  static constexpr int W = P == 1 ? 2 : 4;
  float v[W];
};

__device__ __forceinline__ void cp_row4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global.L2::256B [%0], [%1], 4;\n" ::"r"(shared_addr(dst)),
               "l"(__cvta_generic_to_global(src))
               : "memory");
}

template <int P, bool F_ONE, bool B_ONE, typename TO>
__global__ void __launch_bounds__(kChipThreads)
sweep_chip_kernel(const float* __restrict__ coef, int N, int64_t M, int64_t ld, const float* rhs, TO* x,
                  int64_t ntiles, int sms) {
  using F = NativeArith<float>;
  constexpr int R = kChipBatch;
  using Rec = ChipRec<P>;
  constexpr int CV = R * Rec::W / 4;  // 16-byte reads of a batch's coefficients
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int NP = (N + 3) / 4 * 4;
  Rec* cs = reinterpret_cast<Rec*>(smem_raw);  // forward rows, then (NP rows on) backward rows
  const int lane = threadIdx.x & 31;
  float4* const col = reinterpret_cast<float4*>(cs + 2 * NP) + lane;  // four rows of this lane's system each
  auto at = [&](int i) -> float* { return reinterpret_cast<float*>(col + (i >> 2) * 32) + (i & 3); };
  // CTAs of one SM have block indices about `sms` apart: their sweeping warps go to
  // different schedulers.  role 0 sweeps, 1 to 3 copy.
  const int role = ((threadIdx.x >> 5) + (int)(blockIdx.x / sms)) & 3;
  const int part = ((N + kChipParts - 1) / kChipParts + R - 1) / R * R;  // rows of a quarter, whole batches
  const int last = (N + part - 1) / part - 1;                            // quarters that have rows: 0 .. last
  auto end = [&](int q) { return min(N, (q + 1) * part); };
  auto fill = [&](int64_t m, int first, int q, int step) {  // this warp's rows of a quarter
    if (m < M) {
      const float* src = rhs + m + (int64_t)(q * part + first) * ld;
#pragma unroll 4
      for (int i = q * part + first; i < end(q); i += step, src += step * ld) cp_row4(at(i), src);
    }
  };

  int64_t m = (int64_t)blockIdx.x * 32 + lane;
  for (int q = 0; q < kChipParts; ++q) {  // the first tile: every warp copies
    if (q <= last) fill(m, role, q, 4);
    cp_commit();
  }
  for (int k = threadIdx.x; k < 2 * N; k += kChipThreads) {
    Rec* c = cs + (k < N ? k : NP - N + k);
#pragma unroll
    for (int e = 0; e < Rec::W; ++e) c->v[e] = e <= P ? coef[k * (P + 1) + e] : 0.f;
  }

  struct Batch {
    float4 b[R / 4], c[CV];
  } A, B;
  auto get = [&](Batch& t, const Rec* rec, int i0) {  // rows i0 .. i0+R-1
#pragma unroll
    for (int k = 0; k < R / 4; ++k) t.b[k] = col[((i0 >> 2) + k) * 32];
    const float4* c = reinterpret_cast<const float4*>(rec + i0);
#pragma unroll
    for (int k = 0; k < CV; ++k) t.c[k] = c[k];
  };
  // one batch of a sweep upwards (D = 1) or downwards (-1), in place in the tile
  auto sweep = [&](const Batch& t, int i0, float& v1, float& v2, auto dir) {
    constexpr int D = decltype(dir)::value;
    Batch w = t;
    float* bv = reinterpret_cast<float*>(w.b);
    const Rec* cv = reinterpret_cast<const Rec*>(w.c);
#pragma unroll
    for (int n = 0; n < R; ++n) {
      const int j = D > 0 ? n : R - 1 - n;
      const float v = F::step<P, (D > 0 ? F_ONE : B_ONE)>(cv[j].v, bv[j], v1, v2);
      bv[j] = v;
      v2 = v1;
      v1 = v;
    }
#pragma unroll
    for (int k = 0; k < R / 4; ++k) col[((i0 >> 2) + k) * 32] = w.b[k];
  };
  auto row = [&](const Rec* rec, int i, float& v1, float& v2, auto dir) {
    const float v = F::step<P, (decltype(dir)::value > 0 ? F_ONE : B_ONE)>(rec[i].v, *at(i), v1, v2);
    *at(i) = v;
    v2 = v1;
    v1 = v;
  };
  auto sweep_part = [&](int q, const Rec* rec, float& v1, float& v2, auto dir) {
    constexpr int D = decltype(dir)::value;
    const int lo = q * part, hi = end(q), nb = (hi - lo) / R, whole = lo + nb * R;
    if constexpr (D < 0)
      for (int i = hi - 1; i >= whole; --i) row(rec, i, v1, v2, dir);
    auto first = [&](int k) { return lo + (D > 0 ? k : nb - 1 - k) * R; };  // of batch k
    if (nb > 0) get(A, rec, first(0));
    int k = 0;
    for (; k + 2 < nb; k += 2) {
      get(B, rec, first(k + 1));
      sweep(A, first(k), v1, v2, dir);
      get(A, rec, first(k + 2));
      sweep(B, first(k + 1), v1, v2, dir);
    }
    if (k + 1 < nb) get(B, rec, first(k + 1));
    if (k < nb) sweep(A, first(k), v1, v2, dir);
    if (k + 1 < nb) sweep(B, first(k + 1), v1, v2, dir);
    if constexpr (D > 0)
      for (int i = whole; i < hi; ++i) row(rec, i, v1, v2, dir);
  };
  using Up = std::integral_constant<int, 1>;
  using Down = std::integral_constant<int, -1>;

  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x, m += (int64_t)gridDim.x * 32) {
    // ---- forward, each quarter as it arrives
    float u1 = 0.f, u2 = 0.f;
    for (int q = 0; q <= last; ++q) {
      if (tile != blockIdx.x || q == 3)
        cp_wait<0>();
      else if (q == 0)
        cp_wait<3>();
      else if (q == 1)
        cp_wait<2>();
      else
        cp_wait<1>();
      __syncthreads();
      if (role == 0) sweep_part(q, cs, u1, u2, Up{});
    }
    // ---- backward; a finished quarter is stored and refilled while the next one is swept
    float x1 = 0.f, x2 = 0.f;
    const int64_t mn = m + (int64_t)gridDim.x * 32;
    for (int q = last; q >= 0; --q) {
      if (role == 0) sweep_part(q, cs + NP, x1, x2, Down{});
      __syncthreads();
      if (role != 0) {
        if (m < M) {
          TO* dst = x + m + (int64_t)(q * part + role - 1) * ld;
#pragma unroll 4
          for (int i = q * part + role - 1; i < end(q); i += 3, dst += 3 * ld)
            st_stream(dst, Conv<F, TO>::out(*at(i)));
        }
        if (tile + gridDim.x < ntiles) fill(mn, role - 1, q, 3);
        cp_commit();
      }
    }
  }
}

size_t chip_bytes(const sb_factor* f) {
  const size_t rows = (f->N + 3) / 4 * 4;
  return rows * (2 * (f->P == 1 ? sizeof(ChipRec<1>) : sizeof(ChipRec<2>)) + 32 * sizeof(float));
}

template <int P, bool F_ONE, bool B_ONE, typename TO>
int launch(const sb_factor* f, const float* coef, const float* rhs, TO* x, int64_t M, int64_t ld,
           cudaStream_t stream) {
  const size_t smem = chip_bytes(f);
  auto k = sweep_chip_kernel<P, F_ONE, B_ONE, TO>;
  int nb = 0;
  SB_TRY(kernel_occupancy(reinterpret_cast<const void*>(k), f->device, kChipThreads, smem, &nb));
  const int64_t ntiles = (M + 31) / 32;
  const int sms = std::max(1, sm_count(f->device));
  const int64_t grid = std::min<int64_t>(ntiles, (int64_t)nb * sms);
  k<<<(unsigned)grid, kChipThreads, smem, stream>>>(coef, (int)f->N, M, ld, rhs, x, ntiles, sms);
  return cuda_check(cudaGetLastError(), "on-chip sweep launch");
}

}  // namespace

bool chip_sweep_fits(const sb_factor* f, sb_dtype rt, sb_dtype xt, sb_arith arith) {
  return arith == SB_ARITH_NATIVE && rt == SB_F32 && (xt == SB_F32 || xt == SB_F64) && !f->periodic &&
         chip_bytes(f) <= (size_t)kMaxDynSmem;
}

// Against the sequential sweeps: always faster with an FP64 solution, whose FP32
// intermediate takes 8-byte places there.  With an FP32 solution those sweeps catch up once
// they have enough warps to hide their latency and the intermediate still finds place in
// L2: up to 16 warps an SM, or 10 where only one tile fits an SM (microseconds, sequential |
// here: N = 256 M = 60001 52 | 41, M = 120001 77 | 82; N = 130 pentadiagonal M = 60001
// 30 | 29, M = 120001 41 | 50; N = 1000 M = 20001 167 | 86, M = 60001 217 | 213,
// pentadiagonal 225 | 242).
bool chip_sweep_applies(const sb_factor* f, sb_dtype rt, sb_dtype xt, int64_t M, sb_arith arith) {
  const int64_t warps = 2 * chip_bytes(f) <= (size_t)kMaxDynSmem ? 16 : 10;
  return chip_sweep_fits(f, rt, xt, arith) && M >= 1 &&
         (xt == SB_F64 || M <= 32 * warps * sm_count(f->device));
}

int launch_chip_sweep(const sb_factor* f, Op op, const void* rhs, void* x, sb_dtype xt, int64_t M, int64_t ld,
                      cudaStream_t stream) {
  const float* c = f->coef32 + (op == OP_PRIMAL ? 0 : op_block_len(f->P, f->N));
  const float* b = static_cast<const float*>(rhs);
  auto go = [&](auto* xp) {
    using TO = std::remove_pointer_t<decltype(xp)>;
    if (f->P == 1)
      return op == OP_PRIMAL ? launch<1, false, true, TO>(f, c, b, xp, M, ld, stream)
                             : launch<1, true, false, TO>(f, c, b, xp, M, ld, stream);
    return op == OP_PRIMAL ? launch<2, false, true, TO>(f, c, b, xp, M, ld, stream)
                           : launch<2, true, false, TO>(f, c, b, xp, M, ld, stream);
  };
  return xt == SB_F32 ? go(static_cast<float*>(x)) : go(static_cast<double*>(x));
}

}  // namespace sb
