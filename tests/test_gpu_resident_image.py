"""GPU tests of when the image of the on-chip time steps is made: by the first small batch
that is stepped and not with the stepper (a forced or coarsening run, a rollout and a large
batch never use it); and that this first batch may come inside a stream capture."""
import pytest

import synth
from tests.gpu_util import lib_or_skip, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    return lib_or_skip()


def test_image_is_made_by_the_first_small_batch(env):
    """200 steppers whose images take 14 doubles a row each (no flux, N = 1024, 32 rows a
    lane): the device memory they take appears with the first small batch, half of it at
    least whatever the allocator's granularity."""
    sb, torch = env
    N, count = 1024, 200
    sts = [sb.sb_stepper_create("cahn_hilliard", "be", "noflux", N, 1.0, 0.05) for _ in range(count)]
    C = to_dev(synth.rhs_uniform(seed=1, N=N, M=32), torch).mul_(0.1)
    big = torch.zeros((N, 40000), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    for st in sts[:2]:
        sb.sb_stepper_run(st, C.clone(), 1, arith="df32")
        sb.sb_stepper_run(st, big, 1)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    for st in sts:
        sb.sb_stepper_run(st, C, 1)
    torch.cuda.synchronize()
    taken = before - torch.cuda.mem_get_info()[0]
    assert taken >= count * 14 * N * 8 // 2, taken


@pytest.mark.parametrize("mode", ["direct", "graph"])
def test_first_small_batch_inside_a_capture(env, mode):
    sb, torch = env
    N, M, nsteps = 131, 50, 30
    args = ("hyperdiffusion", "cn", "periodic", N, 0.4, 0.0)
    C0 = to_dev(synth.rhs_uniform(seed=2, N=N, M=M), torch)
    ref = sb.sb_stepper_run(sb.sb_stepper_create(*args), C0.clone(), nsteps, mode=mode)
    st = sb.sb_stepper_create(*args)
    C = C0.clone()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        sb.sb_stepper_run(st, C, nsteps, mode=mode)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(C, ref)
