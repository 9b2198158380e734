"""GPU tests of FP32 solves of more than 128 rows that TMA cannot copy (odd leading
dimensions, right-hand sides off a 16-byte boundary): 32 systems at a time in shared
memory.  Bit for bit the sequential sweeps, which a grouped solve of one group runs, at the
edges of the quarters and batches the rows are cut into, with ragged tiles, one and several
tiles a CTA, both solution types, systems of zeros, infinities and NaNs among the others;
the adjoint against the oracle (2e-5, the bound of an FP32 solve in the other tests)."""
import os
import subprocess
import sys

import numpy as np
import pytest

import synth
from oracle import banded
from tests.gpu_util import lib_or_skip, relerr_per_system, to_host

pytestmark = pytest.mark.gpu


def bits(torch, t):
    return t.view(torch.int32 if t.dtype == torch.float32 else torch.int64)


def check(kind, xt):
    sb, torch = lib_or_skip()
    tx = torch.float32 if xt == "f32" else torch.float64
    for N in (129, 130, 131, 136, 159, 160, 161, 255, 289, 512, 801, 1023, 1024):
        d = (synth.random_tri_diagonals if kind == "tri" else synth.random_penta_diagonals)(seed=N, N=N)
        fac = (sb.sb_factor_shared_tri if kind == "tri" else sb.sb_factor_shared_penta)(*d)
        for M, pad, off in ((1, 0, 1), (33, 0, 0), (64, 0, 2), (100, 1, 0), (9001, 2, 0), (40003, 0, 0)):
            ld = M + pad
            h = synth.rhs_uniform(seed=M, N=N, M=M, ld=ld, dtype=np.float32, pad_value=9.0)
            if M > 8:
                h[:, 3] = 0.0
                h[N // 2, 4], h[0, 5], h[N - 1, 6] = np.inf, np.nan, -np.inf
            b = torch.from_numpy(np.pad(h.ravel(), (off, 0))).cuda()[off:].view(N, ld)
            x = torch.full((N, ld), 7.0, dtype=tx, device="cuda")
            y = torch.full((N, ld), 7.0, dtype=tx, device="cuda")
            sb.sb_solve_batched_ex(fac, b, x, M=M)
            sb.sb_solve_batched_groups([fac], [b], [y], Ms=[M])
            torch.cuda.synchronize()
            assert torch.equal(bits(torch, x), bits(torch, y)), (N, M, pad, off)
            if xt == "f32":
                sb.sb_solve_batched_ex(fac, b, b, M=M)  # in place
                assert torch.equal(bits(torch, x)[:, :M], bits(torch, b)[:, :M]), (N, M, pad, off)
        h = synth.rhs_uniform(seed=N, N=N, M=501, dtype=np.float32)
        z = torch.full((N, 501), 7.0, dtype=tx, device="cuda")
        sb.sb_solve_batched_ex(fac, torch.from_numpy(h).cuda(), z, transpose=True)
        h = h.astype(np.float64)
        if kind == "tri":
            bh, ch = banded.tri_factor(*d)
            ref = banded.tri_solve_adjoint(d[0], bh, ch, h)
        else:
            ref = banded.penta_solve_adjoint(*banded.penta_factor(*d), h)
        assert np.max(relerr_per_system(to_host(z).astype(np.float64), ref)) <= 2e-5, N


def check_asked(kind, xt):
    """The partitioned solve asked for where it does not apply: fewer rows than four quarters,
    and more than it takes, aligned or not."""
    sb, torch = lib_or_skip()
    tx, code = (torch.float32, sb.SB_F32) if xt == "f32" else (torch.float64, sb.SB_F64)
    for N in (1, 2, 7, 8, 9, 16, 25, 32, 40, 63, 1025, 1400):
        d = (synth.random_tri_diagonals if kind == "tri" else synth.random_penta_diagonals)(seed=N, N=N)
        fac = (sb.sb_factor_shared_tri if kind == "tri" else sb.sb_factor_shared_penta)(*d)
        sb.sb_shape_set(fac, (512, 0, 1, sb.SB_ALGO_PARTITIONED), rhs_dtype=sb.SB_F32, x_dtype=code)
        for M in (1, 33, 5000, 40000):
            b = torch.from_numpy(synth.rhs_uniform(seed=M, N=N, M=M, dtype=np.float32)).cuda()
            x, y = torch.empty((N, M), dtype=tx, device="cuda"), torch.empty((N, M), dtype=tx, device="cuda")
            sb.sb_solve_batched_ex(fac, b, x)
            sb.sb_solve_batched_groups([fac], [b], [y])
            torch.cuda.synchronize()
            assert torch.equal(bits(torch, x), bits(torch, y)), (N, M)


@pytest.mark.parametrize("what", ["check", "check_asked"])
@pytest.mark.parametrize("kind", ["tri", "penta"])
@pytest.mark.parametrize("xt", ["f32", "f64"])
def test_bits_of_the_sequential_sweeps(what, kind, xt):
    """In a process of its own: a launch shape stored by another test would be taken instead."""
    lib_or_skip()
    code = f"import tests.test_gpu_chip_sweep as t; t.{what}({kind!r}, {xt!r})"
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
