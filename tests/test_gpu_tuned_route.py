"""GPU tests that storing what the library reports, or tuning, never gives a slower solve
than storing nothing: the default adapts to the batch and has forms that no shape names,
so its shape put back, or found fastest by the autotuner, has to mean the default.

Routes are told apart by their bits (each eliminates in its own order) and, after tuning,
by time: the forms in question are 3 to 13 times as fast as the best stored shape, so the
bound of 1.5 leaves room for the spread of short launches.  The N are used by no other
test: entries are process-wide."""
import numpy as np
import pytest

import synth
from tests.gpu_util import lib_or_skip, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    return lib_or_skip()


def batch(torch, sb, kind, N, M, pad, dtype):
    diags = (synth.random_tri_diagonals if kind == "tri" else synth.random_penta_diagonals)(seed=N, N=N)
    fac = (sb.sb_factor_shared_tri if kind == "tri" else sb.sb_factor_shared_penta)(*diags)
    return fac, to_dev(synth.rhs_normal(seed=M, N=N, M=M, ld=M + pad, pad_value=0.0).astype(dtype), torch)


@pytest.mark.parametrize("kind", ["tri", "penta"])
@pytest.mark.parametrize("N,M,dtype", [
    (94, 12000, np.float32),   # registers; the shape reported is the partitioned solve's
    (187, 70, np.float64),     # partitioned; the shape reported is the two-ended sweeps'
])
def test_the_reported_shape_put_back_changes_nothing(env, kind, N, M, dtype):
    sb, torch = env
    fac, b = batch(torch, sb, kind, N, M, 0, dtype)
    code = sb.SB_F32 if dtype == np.float32 else sb.SB_F64
    x, y, z = torch.empty_like(b), torch.empty_like(b), torch.empty_like(b)
    sb.sb_solve_batched(fac, b, x)
    named = sb.sb_shape_get(fac, rhs_dtype=code, x_dtype=code)
    # a request for the named kernel itself holds, and gives other bits
    sb.sb_shape_set(fac, (named[0], 0, named[2], named[3]), rhs_dtype=code, x_dtype=code)
    sb.sb_solve_batched(fac, b, y)
    assert sb.sb_shape_get(fac, rhs_dtype=code, x_dtype=code) == (named[0], 0, named[2], named[3])
    sb.sb_shape_set(fac, named, rhs_dtype=code, x_dtype=code)
    sb.sb_solve_batched(fac, b, z)
    assert sb.sb_shape_get(fac, rhs_dtype=code, x_dtype=code) == named
    assert torch.equal(x, z) and not torch.equal(x, y)


def best_ms(torch, run):
    run()
    ts = []
    for _ in range(7):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(10):
            run()
        e1.record()
        e1.synchronize()
        ts.append(e0.elapsed_time(e1) / 10)
    return min(ts)


@pytest.mark.parametrize("N,M,pad,dtype", [
    (62, 262144, 0, np.float32),   # registers
    (997, 501, 2, np.float32),     # rows that TMA cannot copy
    (253, 1024, 0, np.float64),    # small batch, partitioned
])
def test_tuning_is_not_slower_than_the_default(env, N, M, pad, dtype):
    sb, torch = env
    fac, b = batch(torch, sb, "tri", N, M, pad, dtype)
    x = torch.empty_like(b)
    run = lambda: sb.sb_solve_batched(fac, b, x, M=M)
    before = best_ms(torch, run)
    best, ms = sb.sb_autotune(fac, b, x, M=M)
    code = sb.SB_F32 if dtype == np.float32 else sb.SB_F64
    assert sb.sb_shape_get(fac, rhs_dtype=code, x_dtype=code) == best and ms > 0
    assert best_ms(torch, run) <= 1.5 * before
