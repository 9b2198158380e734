"""GPU test that the chunk size of a host-memory solve does not show in the bits of an FP32
solve: rows of up to 128 (registers) and more (shared memory), odd and even chunk widths,
one chunk and many, both solution types, A and A^T.  The bits are those of the sequential
sweeps, which a grouped solve of one group runs.

In a process of its own: a launch shape stored by another test would be taken instead."""
import os
import subprocess
import sys

import numpy as np
import pytest

import synth
from tests.gpu_util import lib_or_skip

pytestmark = pytest.mark.gpu


def check(kind, N):
    sb, torch = lib_or_skip()
    d = (synth.random_tri_diagonals if kind == "tri" else synth.random_penta_diagonals)(seed=N, N=N)
    fac = (sb.sb_factor_shared_tri if kind == "tri" else sb.sb_factor_shared_penta)(*d)
    M, ld = 21000, 21002
    h = torch.from_numpy(synth.rhs_normal(seed=N + 1, N=N, M=M, ld=ld, pad_value=-1.5).astype(np.float32)).pin_memory()
    for tx, code in ((torch.float32, sb.SB_F32), (torch.float64, sb.SB_F64)):
        y = torch.full((N, ld), -1.5, dtype=tx, device="cuda")
        sb.sb_solve_batched_groups([fac], [h.cuda()], [y], Ms=[M])
        for transpose in (False, True):
            first = None
            for chunk in (0, 20000, 3000, 1001, 10502):
                x = torch.full((N, ld), -1.5, dtype=tx).pin_memory()
                work = torch.empty(sb.sb_host_workspace_bytes(fac, M, chunk, rhs_dtype=sb.SB_F32, x_dtype=code),
                                   dtype=torch.uint8, device="cuda")
                sb.sb_solve_batched_host(fac, h, x, work, transpose=transpose, chunk_systems=chunk, M=M)
                torch.cuda.synchronize()
                first = x if first is None else first
                assert torch.equal(x, first), (tx, transpose, chunk)
            if not transpose:
                assert torch.equal(first, y.cpu()), tx


@pytest.mark.parametrize("kind,N", [("tri", 100), ("penta", 100), ("tri", 300), ("penta", 300)])
def test_chunking_does_not_change_the_bits_of_fp32(kind, N):
    lib_or_skip()
    code = f"import tests.test_gpu_host_chunks_f32 as t; t.check({kind!r}, {N})"
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
