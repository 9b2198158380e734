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
// others copy the tile in and the solution out, a quarter of the rows behind or ahead
// of it.  The backward sweep is done with the last quarter first, and the next tile needs
// its first quarter first: it goes into the place of the last, so quarters lie in turn
// upwards and downwards.  A quarter changes hands at a barrier of the CTA, and a place is
// stored and refilled by the same warp.  A system's rows lie in fours, so that the sweeping
// warp reads and writes 16 bytes at a time: with 4-byte accesses it took 25 ns a row, now
// 10 (12 a pentadiagonal one).
//
// Microseconds, sequential | partitioned with cp.async | this form (chip_sweep_applies
// draws the line): tridiagonal N = 1000: M = 501 134 | 13.3 | 21, M = 20001 167 | 55 | 80;
// N = 256: M = 6001 38 | 11.6 | 12.4, M = 60001 52 | 51 | 41; pentadiagonal N = 512: M = 6001
// 77 | 19 | 20, M = 20001 88 | 36 | 41; with an FP64 solution, tridiagonal N = 130, M =
// 240001 184 | 123 | 90, pentadiagonal N = 256, M = 60001 76 | 66 | 51.
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "sb_internal.h"
#include "sweep_tile.cuh"

namespace sb {
namespace {

constexpr int kChipBatch = 8;  // rows the sweeping warp reads at once
constexpr int kChipParts = 4;

// Coefficients of a row of one sweep (P + 1), padded to a power of two.
template <int P>
struct alignas(P == 1 ? 8 : 16) ChipRec {
  static constexpr int W = P == 1 ? 2 : 4;
  float v[W];
};

// Rows of a quarter.
__host__ __device__ inline int chip_part(int N) {
  return ((N + kChipParts - 1) / kChipParts + kChipBatch - 1) / kChipBatch * kChipBatch;
}

__device__ __forceinline__ void cp_row4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global.L2::256B [%0], [%1], 4;\n" ::"r"(shared_addr(dst)),
               "l"(__cvta_generic_to_global(src))
               : "memory");
}

template <int P, bool F_ONE, bool B_ONE, typename TO, int T>
__global__ void __launch_bounds__(T)
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
  // CTAs of one SM have block indices about `sms` apart: their sweeping warps go to
  // different schedulers.  role 0 sweeps, 1 to nw - 1 copy.
  constexpr int nw = T / 32;  // 4 or 8
  const int role = ((threadIdx.x >> 5) + (int)(blockIdx.x / sms)) & (nw - 1);
  const int part = chip_part(N);               // rows of a quarter, whole batches
  const int last = (N + part - 1) / part - 1;  // quarters that have rows: 0 .. last
  auto end = [&](int q) { return min(N, (q + 1) * part); };
  // how far a quarter's rows lie from their own places: none, or (down) in reverse order
  auto shift = [&](int q, bool down) { return down ? (last - 2 * q) * part : 0; };
  auto at = [&](int i) -> float* { return reinterpret_cast<float*>(col + (i >> 2) * 32) + (i & 3); };
  auto fill = [&](int64_t m, int first, int q, int step, bool down) {  // this warp's rows of a quarter
    if (m < M) {
      const int off = shift(q, down);
      const float* src = rhs + m + (int64_t)(q * part + first) * ld;
#pragma unroll 4
      for (int i = q * part + first; i < end(q); i += step, src += step * ld) cp_row4(at(i + off), src);
    }
  };

  int64_t m = (int64_t)blockIdx.x * 32 + lane;
  for (int q = 0; q < kChipParts; ++q) {  // the first tile: every warp copies
    if (q <= last) fill(m, role, q, nw, false);
    cp_commit();
  }
  for (int k = threadIdx.x; k < 2 * N; k += T) {
    Rec* c = cs + (k < N ? k : NP - N + k);
#pragma unroll
    for (int e = 0; e < Rec::W; ++e) c->v[e] = e <= P ? coef[k * (P + 1) + e] : 0.f;
  }

  struct Batch {
    float4 b[R / 4], c[CV];
  } A, B;
  auto get = [&](Batch& t, const float4* p, const float4* c) {  // a batch's rows and coefficients
#pragma unroll
    for (int k = 0; k < R / 4; ++k) t.b[k] = p[k * 32];
#pragma unroll
    for (int k = 0; k < CV; ++k) t.c[k] = c[k];
  };
  // one batch of a sweep upwards (D = 1) or downwards (-1), in place in the tile
  auto sweep = [&](const Batch& t, float4* p, float& v1, float& v2, auto dir) {
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
    for (int k = 0; k < R / 4; ++k) p[k * 32] = w.b[k];
  };
  auto row = [&](const Rec& c, float* p, float& v1, float& v2, auto dir) {
    const float v = F::step<P, (decltype(dir)::value > 0 ? F_ONE : B_ONE)>(c.v, *p, v1, v2);
    *p = v;
    v2 = v1;
    v1 = v;
  };
  // quarter q, whose rows lie `off` rows from their own places: whole batches, one read ahead,
  // and the rows that are left over at its upper end
  auto sweep_part = [&](int q, int off, const Rec* rec, float& v1, float& v2, auto dir) {
    constexpr int D = decltype(dir)::value;
    constexpr int ps = D * (R / 4) * 32, ks = D * CV;  // from a batch to the next one swept
    const int lo = q * part, hi = end(q), whole = lo + (hi - lo) / R * R;
    int nb = (hi - lo) / R;
    if constexpr (D < 0)
      for (int i = hi - 1; i >= whole; --i) row(rec[i], at(i + off), v1, v2, dir);
    if (nb > 0) {
      const int first = D > 0 ? lo : whole - R;
      float4* p = col + ((first + off) >> 2) * 32;
      const float4* c = reinterpret_cast<const float4*>(rec + first);
      get(A, p, c);
      for (; nb > 2; nb -= 2, p += 2 * ps, c += 2 * ks) {
        get(B, p + ps, c + ks);
        sweep(A, p, v1, v2, dir);
        get(A, p + 2 * ps, c + 2 * ks);
        sweep(B, p + ps, v1, v2, dir);
      }
      if (nb > 1) get(B, p + ps, c + ks);
      sweep(A, p, v1, v2, dir);
      if (nb > 1) sweep(B, p + ps, v1, v2, dir);
    }
    if constexpr (D > 0)
      for (int i = whole; i < hi; ++i) row(rec[i], at(i + off), v1, v2, dir);
  };
  using Up = std::integral_constant<int, 1>;
  using Down = std::integral_constant<int, -1>;

  bool down = false;  // how this tile's quarters lie
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x, m += (int64_t)gridDim.x * 32, down = !down) {
    // ---- forward, each quarter as it arrives (one group each, in order)
    float u1 = 0.f, u2 = 0.f;
    for (int q = 0; q <= last; ++q) {
      if (q == 3 || last != 3)
        cp_wait<0>();
      else if (q == 0)
        cp_wait<3>();
      else if (q == 1)
        cp_wait<2>();
      else
        cp_wait<1>();
      __syncthreads();
      if (role == 0) sweep_part(q, shift(q, down), cs, u1, u2, Up{});
    }
    // ---- backward; a finished quarter is stored while the next one is swept, and its place
    // takes quarter last - q of the next tile
    float x1 = 0.f, x2 = 0.f;
    const int64_t mn = m + (int64_t)gridDim.x * 32;
    for (int q = last; q >= 0; --q) {
      if (role == 0) sweep_part(q, shift(q, down), cs + NP, x1, x2, Down{});
      __syncthreads();
      if (role != 0) {
        if (m < M) {
          const int off = shift(q, down);
          TO* dst = x + m + (int64_t)(q * part + role - 1) * ld;
#pragma unroll 4
          for (int i = q * part + role - 1; i < end(q); i += nw - 1, dst += (nw - 1) * ld)
            st_stream(dst, Conv<F, TO>::out(*at(i + off)));
        }
        if (tile + gridDim.x < ntiles) fill(mn, role - 1, last - q, nw - 1, !down);
        cp_commit();
      }
    }
  }
}

size_t chip_bytes(const sb_factor* f) {
  const size_t N = (size_t)f->N, part = (size_t)chip_part((int)f->N);
  return (N + 3) / 4 * 4 * 2 * (f->P == 1 ? sizeof(ChipRec<1>) : sizeof(ChipRec<2>)) +
         (N + part - 1) / part * part * 32 * sizeof(float);
}

template <int P, bool F_ONE, bool B_ONE, typename TO>
int launch(const sb_factor* f, const float* coef, const float* rhs, TO* x, int64_t M, int64_t ld,
           cudaStream_t stream) {
  const size_t smem = chip_bytes(f);
  // Seven copying warps where at most two tiles fit an SM: with an FP64 solution three take
  // longer over a quarter than its sweep (N = 1000, M = 20001: 105 -> 92 us, FP32 86 -> 81).
  const int threads = 3 * smem > (size_t)kMaxDynSmem ? 256 : 128;
  auto k = threads == 256 ? sweep_chip_kernel<P, F_ONE, B_ONE, TO, 256> : sweep_chip_kernel<P, F_ONE, B_ONE, TO, 128>;
  int nb = 0;
  SB_TRY(kernel_occupancy(reinterpret_cast<const void*>(k), f->device, threads, smem, &nb));
  const int64_t ntiles = (M + 31) / 32;
  const int sms = std::max(1, sm_count(f->device));
  const int64_t grid = std::min<int64_t>(ntiles, (int64_t)nb * sms);
  k<<<(unsigned)grid, threads, smem, stream>>>(coef, (int)f->N, M, ld, rhs, x, ntiles, sms);
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
// here with three copying warps: N = 256 M = 60001 52 | 41, M = 120001 77 | 82; N = 130
// pentadiagonal M = 60001 30 | 29, M = 120001 41 | 50; N = 1000 M = 20001 167 | 86, M =
// 60001 217 | 213, pentadiagonal 225 | 242).
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
