// Launch-shape table and autotuner for the batched solves.
//
// A shape (threads per CTA, resident CTAs per SM, systems per thread, algorithm) is looked up
// per (device, half bandwidth, N, arithmetic, rhs dtype, x dtype).  Entries come
// from sb_shape_set (e.g. a persisted tuning cache) or from sb_autotune, which
// times every candidate shape on the caller's buffers with CUDA events and keeps
// the fastest.  Without an entry, FP32 right-hand sides in native arithmetic use the
// register-resident sweeps up to 128 rows and the partitioned solve where it applies,
// FP64 ones the two-ended sweeps or, for a small batch, the FP64 partitioned solve, and
// everything else the default of sweep.cu.
//
// That default is a rule on M and alignment, and some of its forms no shape names, so it
// cannot be an entry: the shape that stands for it (default_route of a large batch) is
// never stored, and storing it drops the entry instead.  Where an explicit request for the
// same kernel is possible, the two differ in ctas_per_sm: 1 in the default, 0 in a
// request, which run alike because one such CTA fills an SM.
#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>
#include <vector>

#include "sb_internal.h"

namespace sb {
namespace {

using Key = std::tuple<int, int, int64_t, int, int, int>;
std::mutex g_mu;
std::map<Key, SweepShape> g_table;

Key make_key(const sb_factor* f, sb_arith arith, sb_dtype rt, sb_dtype xt) {
  return Key(f->device, f->P, f->N, (int)arith, (int)rt, (int)xt);
}

// The FP64 solve of a batch of M systems without a stored entry.  Both forms eliminate
// in another order than the plain sweeps, so the matrix has to allow any (any_order).
//
// Up to which M the partitioned form is taken: its time grows with the tiles of 8 systems
// an SM gets, each costing c + d L microseconds (L rows per chunk), while the two-ended
// sweeps of a batch that does not fill the chip take a latency of about a N whatever M
// is.  Microseconds, partitioned | two-ended (the line's M):
//   tridiagonal   N = 64:  M = 1024 5.8 | 7.9, 4096 12.3 | 8.1 (1700);
//                 N = 256: M = 1024 8.1 | 23.3, 4096 19 | 23, 16384 55 | 28 (5000)
//   pentadiagonal N = 64:  M = 64 12.2 | 10.0 (60);
//                 N = 256: M = 1024 15 | 32, 4096 42 | 32, 16384 148 | 39 (2200)
// Above it the two-ended sweeps are the fastest form at every size measured (N = 64 to
// 2000, M to 65536), with the widest CTA whose ring fits beside the coefficients.
bool fp64_shape(const sb_factor* f, Op op, int64_t M, SweepShape* s) {
  const int o = op == OP_PRIMAL ? 0 : 1;
  if (!f->any_order) return false;
  const double a = f->P == 1 ? 0.082 : 0.115, b = f->P == 1 ? 1.0 : 7.0;
  const double c = f->P == 1 ? 1.0 : 3.5, d = f->P == 1 ? 0.21 : 0.47;
  if (f->part64_img[o] != nullptr &&
      (double)M <= 0.9 * 8 * sm_count(f->device) * (a * (double)f->N - b) / (c + d * f->part64_L)) {
    s->threads = kPart64Threads;
    s->algo = SB_ALGO_PARTITIONED;
    return true;
  }
  for (int threads : {1024, 512, 256})
    if (two_ended_applies(f, op, SB_ARITH_NATIVE, threads)) {
      s->threads = threads;
      s->ctas_per_sm = 1;  // all that fit
      s->algo = SB_ALGO_TWO_ENDED;
      return true;
    }
  return false;
}

// The shape a solve of M systems takes without a stored entry.
SweepShape default_route(const sb_factor* f, Op op, sb_arith arith, sb_dtype rt, sb_dtype xt, int64_t M) {
  SweepShape s;
  const bool reg = reg_sweep_applies(f, rt, xt, arith);
  // FP32 right-hand sides in native arithmetic default to the partitioned solve where
  // the factor has its data (the launcher falls back to the sweeps per call where it
  // does not apply)
  if (arith == SB_ARITH_NATIVE && rt == SB_F32 && (f->part_img[0][0] || f->part_img[1][0])) {
    // two systems per thread (variant 2) where the factor has its image
    s.threads = (f->part_img[0][2] || f->part_img[1][2]) ? 256 : 512;
    s.ctas_per_sm = 1;  // all that fit
    s.algo = SB_ALGO_PARTITIONED;
    s.reg = reg;
    return s;
  }
  if (reg) {
    s = default_shape(f, arith);
    s.threads = kRegThreads;
    s.reg = true;
    return s;
  }
  if (arith == SB_ARITH_NATIVE && rt == SB_F64 && xt == SB_F64 && fp64_shape(f, op, M, &s)) return s;
  // double-float: the two-ended sweeps at every size (two CTAs of 448 threads an SM, 72
  // registers a thread).  Microseconds, sequential | two-ended: tridiagonal N = 256, M = 64
  // 66 | 18, M = 131072 218 | 158; pentadiagonal N = 64, M = 65536 32 | 23; N = 1024,
  // M = 30011 378 | 200, M = 65536 512 | 343; N = 2000, M = 65536 1443 | 846
  if (arith == SB_ARITH_DF32 && rt == SB_F64 && xt == SB_F64 && f->any_order &&
      two_ended_applies(f, op, arith, 448)) {
    s.threads = 448;
    s.algo = SB_ALGO_TWO_ENDED;
    return s;
  }
  return default_shape(f, arith);
}

bool same_shape(const SweepShape& a, const SweepShape& b) {
  return a.threads == b.threads && a.ctas_per_sm == b.ctas_per_sm && a.spt == b.spt && a.algo == b.algo;
}

void copy_shape(const SweepShape& s, sb_shape* out) {
  out->threads = s.threads;
  out->ctas_per_sm = s.ctas_per_sm;
  out->systems_per_thread = s.spt;
  out->algorithm = s.algo;
}

}  // namespace

SweepShape shape_for(const sb_factor* f, Op op, sb_arith arith, sb_dtype rt, sb_dtype xt, int64_t M) {
  {
    std::lock_guard<std::mutex> lk(g_mu);
    auto it = g_table.find(make_key(f, arith, rt, xt));
    if (it != g_table.end()) return it->second;
  }
  return default_route(f, op, arith, rt, xt, M);
}

SweepShape shape_for_pieces(const sb_factor* f, Op op, sb_arith arith, sb_dtype rt, sb_dtype xt) {
  SweepShape s = shape_for(f, op, arith, rt, xt, kLargeBatch);
  // FP32: registers or partition by a piece's M, TMA or not by its width.  The sequential
  // sweeps on chip are one form for all (the copies to and from the host take several times
  // as long as any of them).
  if (rt == SB_F32 && same_shape(s, default_route(f, op, arith, rt, xt, kLargeBatch))) {
    const bool reg = s.reg;
    s = default_shape(f, arith);
    s.reg = reg;
    s.chip = !reg;
  }
  return s;
}

}  // namespace sb

using namespace sb;

extern "C" {

int sb_shape_get(const sb_factor* f, sb_arith arith, sb_dtype rhs_dtype, sb_dtype x_dtype,
                 sb_shape* out) {
  clear_error();
  if (!f || !out) return fail(SB_ERR_INVALID_ARG, "NULL argument");
  copy_shape(shape_for(f, OP_PRIMAL, arith, rhs_dtype, x_dtype, kLargeBatch), out);
  return SB_OK;
}

int sb_shape_set(const sb_factor* f, sb_arith arith, sb_dtype rhs_dtype, sb_dtype x_dtype,
                 const sb_shape* shape) {
  clear_error();
  if (!f || !shape) return fail(SB_ERR_INVALID_ARG, "NULL argument");
  if (shape->algorithm != SB_ALGO_SEQUENTIAL && shape->algorithm != SB_ALGO_PARTITIONED &&
      shape->algorithm != SB_ALGO_STAGED && shape->algorithm != SB_ALGO_TWO_ENDED)
    return fail(SB_ERR_INVALID_ARG, "unknown algorithm %d", shape->algorithm);
  if (shape->ctas_per_sm < 0 || shape->ctas_per_sm > 32)
    return fail(SB_ERR_INVALID_ARG, "ctas_per_sm must be in [0, 32]");
  if (shape->algorithm == SB_ALGO_SEQUENTIAL) {
    if (shape->threads < 32 || shape->threads > 512 || shape->threads % 32 != 0)
      return fail(SB_ERR_INVALID_ARG, "threads must be a multiple of 32 in [32, 512]");
    if (shape->systems_per_thread != 1 && shape->systems_per_thread != 2)
      return fail(SB_ERR_INVALID_ARG, "systems_per_thread must be 1 or 2");
  } else if (shape->algorithm == SB_ALGO_STAGED || shape->algorithm == SB_ALGO_TWO_ENDED) {
    const int cap = (arith == SB_ARITH_DF32 && shape->algorithm == SB_ALGO_STAGED) ? 512 : 1024;
    if (shape->threads < 32 || shape->threads > cap || shape->threads % 32 != 0)
      return fail(SB_ERR_INVALID_ARG, "threads must be a multiple of 32 in [32, %d] for this algorithm", cap);
    if (shape->systems_per_thread != 1)
      return fail(SB_ERR_INVALID_ARG, "the staged and two-ended sweeps take systems_per_thread = 1");
  } else {
    if (part_variant(shape->threads) < 0 && shape->threads != kPart64Threads)
      return fail(SB_ERR_INVALID_ARG, "the partitioned solve runs 128, 256, 512 or 1024 threads per CTA");
    if (shape->systems_per_thread != 1 || shape->ctas_per_sm > 1)
      return fail(SB_ERR_INVALID_ARG,
                  "the partitioned solve takes systems_per_thread = 1 and ctas_per_sm 0 or 1");
  }
  SweepShape s;
  s.threads = shape->threads;
  s.ctas_per_sm = shape->ctas_per_sm;
  s.spt = shape->systems_per_thread;
  s.algo = shape->algorithm;
  const bool is_default = same_shape(s, default_route(f, OP_PRIMAL, arith, rhs_dtype, x_dtype, kLargeBatch));
  std::lock_guard<std::mutex> lk(g_mu);
  if (is_default)
    g_table.erase(make_key(f, arith, rhs_dtype, x_dtype));
  else
    g_table[make_key(f, arith, rhs_dtype, x_dtype)] = s;
  return SB_OK;
}

int sb_autotune(const sb_factor* f, int transpose, const void* rhs, sb_dtype rhs_dtype, void* x,
                sb_dtype x_dtype, int64_t M, int64_t ld, sb_arith arith, void* stream,
                sb_shape* best, float* best_ms) {
  clear_error();
  if (!f) return fail(SB_ERR_INVALID_ARG, "factor handle is NULL");
  if (M < 1) return fail(SB_ERR_INVALID_ARG, "autotuning needs M >= 1");
  if (rhs == x) return fail(SB_ERR_INVALID_ARG, "autotuning needs rhs and x to be different arrays");
  // Validate once through the normal path (also rejects unsupported combinations).
  SB_TRY(sb_solve_batched_ex(f, transpose, rhs, rhs_dtype, x, x_dtype, M, ld, arith, stream));
  DeviceGuard g(f->device);
  SB_TRY(g.rc);
  cudaStream_t st = (cudaStream_t)stream;
  const Op op = transpose ? OP_ADJOINT : OP_PRIMAL;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  SB_CUDA(cudaEventCreate(&e0));
  int rc = cuda_check(cudaEventCreate(&e1), "cudaEventCreate");
  if (rc != SB_OK) {
    cudaEventDestroy(e0);
    return rc;
  }
  // The default route first.  It adapts to every batch and a stored entry does not, so a
  // shape has to beat it by 2 % (above the spread of three launches) to be stored.
  const SweepShape route = default_route(f, op, arith, rhs_dtype, x_dtype, M);
  SweepShape winner = route;
  float winner_ms = 1e30f;
  bool route_wins = true;
  std::vector<SweepShape> cands{route};
  for (int spt : {1, 2})
    for (int threads : {64, 128, 256, 512})
      for (int cps : {0, 1, 2}) {
        SweepShape s;
        s.threads = threads;
        s.ctas_per_sm = cps;
        s.spt = spt;
        cands.push_back(s);
      }
  for (int threads : {256, 512, 768, 1024})
    if (threads <= 512 || arith != SB_ARITH_DF32) {
      SweepShape s;
      s.threads = threads;
      s.ctas_per_sm = 0;
      s.algo = SB_ALGO_STAGED;
      cands.push_back(s);
    }
  if (rhs_dtype == SB_F64 && x_dtype == SB_F64)
    for (int threads : {256, 448, 512, 768, 1024}) {
      if (!two_ended_applies(f, op, arith, threads)) continue;
      SweepShape s;
      s.threads = threads;
      s.ctas_per_sm = 0;
      s.algo = SB_ALGO_TWO_ENDED;
      cands.push_back(s);
    }
  if (partitioned64_applies(f, op, rhs_dtype, x_dtype, M, arith)) {
    SweepShape s;
    s.threads = kPart64Threads;
    s.ctas_per_sm = 0;
    s.algo = SB_ALGO_PARTITIONED;
    cands.push_back(s);
  }
  for (int threads : {256, 512, 1024})
    if (partitioned_applies(f, op, rhs, rhs_dtype, x_dtype, M, ld, arith, threads)) {
      SweepShape s;
      s.threads = threads;
      s.ctas_per_sm = 0;
      s.algo = SB_ALGO_PARTITIONED;
      cands.push_back(s);
    }
  for (const SweepShape& s : cands) {
    // one warm-up launch, then the best of three timed launches
    if (launch_sweep(f, op, rhs, rhs_dtype, x, x_dtype, M, ld, arith, s, st) != SB_OK) {
      clear_error();
      continue;
    }
    float ms_best = 1e30f;
    bool good = true;
    for (int rep = 0; rep < 3 && good; ++rep) {
      good = cudaEventRecord(e0, st) == cudaSuccess &&
             launch_sweep(f, op, rhs, rhs_dtype, x, x_dtype, M, ld, arith, s, st) == SB_OK &&
             cudaEventRecord(e1, st) == cudaSuccess && cudaEventSynchronize(e1) == cudaSuccess;
      float ms = 0.f;
      if (good && cudaEventElapsedTime(&ms, e0, e1) == cudaSuccess) ms_best = std::min(ms_best, ms);
    }
    if (!good) {
      cudaGetLastError();
      clear_error();
      continue;
    }
    const bool is_route = &s == cands.data();
    if (is_route || ms_best < (route_wins ? 0.98f : 1.0f) * winner_ms) {
      winner_ms = ms_best;
      winner = s;
      route_wins = is_route;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (winner_ms >= 1e30f) return fail(SB_ERR_CUDA, "no candidate shape could be launched");
  if (route_wins) winner = default_route(f, OP_PRIMAL, arith, rhs_dtype, x_dtype, kLargeBatch);
  {
    std::lock_guard<std::mutex> lk(g_mu);
    if (route_wins)
      g_table.erase(make_key(f, arith, rhs_dtype, x_dtype));
    else
      g_table[make_key(f, arith, rhs_dtype, x_dtype)] = winner;
  }
  if (best) copy_shape(winner, best);
  if (best_ms) *best_ms = winner_ms;
  return SB_OK;
}

}  // extern "C"
