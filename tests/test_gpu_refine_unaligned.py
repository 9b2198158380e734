"""GPU tests of refined solves of large batches whose rows are aligned to nothing and whose
coefficients nearly fill shared memory (a group of N = 1700 to 2659, tridiagonal): sampled
systems against the oracle (1e-10, the bound of the other refinement tests), and the time
against the same batches with one system less, whose rows are aligned.  Bound: 1.25, since a
row of 128 bytes touches 5 sectors of 32 instead of 4."""
import numpy as np
import pytest

from oracle import matrices, steppers
from tests.gpu_util import lib_or_skip, relerr_per_system, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    return lib_or_skip()


def test_unaligned_rows(env):
    sb, torch = env
    groups = ((128, 1498240, 0.1), (512, 748800, 0.5), (2048, 374400, 2.0))
    facs = [sb.sb_factor_shared_tri(*sb.sb_build_matrix("diffusion", N, r)) for N, _, r in groups]
    ms = []
    for more in (0, 1):
        g = torch.Generator(device="cuda").manual_seed(more)
        b = [torch.rand((N, M + more), generator=g, device="cuda").mul_(2.0).sub_(1.0) for N, M, _ in groups]
        x = [torch.empty(t.shape, dtype=torch.float64, device="cuda") for t in b]
        work = [torch.empty(sb.sb_refine_workspace_bytes(f, t.shape[1]), dtype=torch.uint8, device="cuda")
                for f, t in zip(facs, b)]
        ts = []
        for _ in range(6):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            sb.sb_solve_batched_groups(facs, b, x, n_refine=2, work=work)
            e1.record()
            e1.synchronize()
            ts.append(e0.elapsed_time(e1))
        ms.append(min(ts))
        for (N, M, r), bg, xg in zip(groups, b, x):
            idx = torch.from_numpy(np.unique(np.linspace(0, M + more - 1, 60).astype(int))).cuda()
            ref = steppers.SharedTri(*matrices.diffusion_matrix(N, r)).solve(to_host(bg[:, idx]).astype(np.float64))
            assert np.max(relerr_per_system(to_host(xg[:, idx]), ref)) <= 1e-10
        del b, x, work
    assert ms[1] <= 1.25 * ms[0], ms
