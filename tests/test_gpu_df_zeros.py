"""GPU test that zeros among the right-hand sides of a double-float solve do not send their
rows through the out-of-line conversion: a batch of point sources took 2.3 times as long as
a dense one, 1.6 times with the sequential sweeps that were the default before the two-ended
ones.  Bound: that 1.6."""
import pytest

from tests.gpu_util import lib_or_skip

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    return lib_or_skip()


@pytest.mark.parametrize("kind", ["diffusion", "hinged"])
def test_zeros_are_not_slow(env, kind):
    sb, torch = env
    N, M = 505, 65536
    d = sb.sb_build_matrix(kind, N, 0.25)
    fac = (sb.sb_factor_shared_tri if len(d) == 3 else sb.sb_factor_shared_penta)(*d)
    dense = torch.randn((N, M), dtype=torch.float64, device="cuda")
    zero = torch.zeros_like(dense)
    x = torch.empty_like(dense)

    def ms(b):
        ts = []
        for _ in range(6):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            for _ in range(4):
                sb.sb_solve_batched_ex(fac, b, x, arith="df32")
            e1.record()
            e1.synchronize()
            ts.append(e0.elapsed_time(e1))
        return min(ts)

    t = ms(dense)
    assert ms(zero) <= 1.6 * t
    assert not torch.any(x)
    zero[N // 3] = 1.0
    assert ms(zero) <= 1.6 * t
