"""GPU tests that the default routes are taken, which agreement with the oracle cannot show
(every fallback agrees too): bit for bit the form asked for by an explicit shape, and other
bits than the sequential sweeps.  The N are used by no other test: entries are process-wide."""
import numpy as np
import pytest

import synth
from tests.gpu_util import lib_or_skip, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    return lib_or_skip()


def solve(sb, torch, fac, b, arith, transpose):
    x = torch.empty_like(b)
    sb.sb_solve_batched_ex(fac, b, x, transpose=transpose, arith=arith)
    return x


@pytest.mark.parametrize("transpose", [False, True])
@pytest.mark.parametrize("kind,N,M,arith,shape", [
    ("tri", 243, 900, "native", (128, 0, 1, 1)),     # small FP64 batch: partitioned
    ("penta", 243, 500, "native", (128, 0, 1, 1)),
    ("tri", 245, 40000, "native", (512, 0, 1, 3)),   # large: two-ended (of any width)
    ("penta", 245, 40000, "native", (512, 0, 1, 3)),
    ("penta", 1501, 700, "native", (256, 0, 1, 3)),  # image and ring beside each other
    ("tri", 247, 300, "df32", (256, 0, 1, 3)),       # double-float: two-ended at every size
    ("penta", 247, 40000, "df32", (256, 0, 1, 3)),
])
def test_fp64_route(env, kind, N, M, arith, shape, transpose):
    sb, torch = env
    d = (synth.random_tri_diagonals if kind == "tri" else synth.random_penta_diagonals)(seed=N, N=N)
    fac = (sb.sb_factor_shared_tri if kind == "tri" else sb.sb_factor_shared_penta)(*d)
    b = to_dev(synth.rhs_normal(seed=M, N=N, M=M), torch)
    default = sb.sb_shape_get(fac, arith=arith)
    x = solve(sb, torch, fac, b, arith, transpose)
    sb.sb_shape_set(fac, shape, arith=arith)
    y = solve(sb, torch, fac, b, arith, transpose)
    sb.sb_shape_set(fac, (256, 0, 1, sb.SB_ALGO_SEQUENTIAL), arith=arith)
    z = solve(sb, torch, fac, b, arith, transpose)
    sb.sb_shape_set(fac, default, arith=arith)
    assert torch.equal(x, y) and not torch.equal(x, z)
    assert torch.equal(x, solve(sb, torch, fac, b, arith, transpose))  # put back: the default again


@pytest.mark.parametrize("kind", ["tri", "penta"])
def test_aligned_fp32_rows_are_partitioned(env, kind):
    """Beyond 128 rows TMA-aligned rows take the partitioned solve (16 chunks: 256 and 512
    threads give the same bits), the same systems in rows of odd length the sequential
    sweeps' bits."""
    sb, torch = env
    N, M = 391, 2000
    d = (synth.random_tri_diagonals if kind == "tri" else synth.random_penta_diagonals)(seed=N, N=N)
    fac = (sb.sb_factor_shared_tri if kind == "tri" else sb.sb_factor_shared_penta)(*d)
    b = to_dev(synth.rhs_normal(seed=M, N=N, M=M).astype(np.float32), torch)
    odd = torch.zeros((N, M + 1), dtype=torch.float32, device="cuda")
    odd[:, :M] = b
    x, xo, y, z = (torch.empty_like(b), torch.zeros_like(odd), torch.empty_like(b), torch.empty_like(b))
    sb.sb_solve_batched(fac, b, x)
    sb.sb_solve_batched(fac, odd, xo, M=M)
    key = dict(rhs_dtype=sb.SB_F32, x_dtype=sb.SB_F32)
    default = sb.sb_shape_get(fac, **key)
    sb.sb_shape_set(fac, (512, 0, 1, sb.SB_ALGO_PARTITIONED), **key)
    sb.sb_solve_batched(fac, b, y)
    sb.sb_shape_set(fac, (256, 0, 1, sb.SB_ALGO_SEQUENTIAL), **key)
    sb.sb_solve_batched(fac, b, z)
    sb.sb_shape_set(fac, default, **key)
    assert torch.equal(x, y) and not torch.equal(x, z)
    assert torch.equal(xo[:, :M], z)
