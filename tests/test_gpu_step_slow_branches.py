"""GPU tests of the time steps and the rollout where their batch tests fail: exact zeros,
magnitudes whose squares leave the range of the integer products, and infinities and NaNs,
which have to stay in their own simulation.  Fused steps (large batches), on-chip steps
(small ones), the coarsening and forced runs and the adjoint step.

Bounds: 1e-12 relative per simulation and 1e-10 for the adjoint, as for these paths
elsewhere; simulations beside a non-finite one keep their bits."""
import numpy as np
import pytest

import synth
from oracle import matrices, rollout, steppers
from tests.gpu_util import lib_or_skip, relerr_per_system, to_dev, to_host
from tests.test_gpu_resident import CASES, oracle_run

pytestmark = pytest.mark.gpu

BIG = 1.0e150  # its square is 1e300; 2^480 = 3.1e144 ends the range of the integer square


@pytest.fixture(scope="module")
def env():
    return lib_or_skip()


def special_state(N, M, amp, ch):
    """Simulations 0 to 9: zeros everywhere, one non-zero row, zeros in a half, in every third
    row, tiny and huge magnitudes (small enough for their cubes, where there are any)."""
    C = synth.rhs_uniform(seed=N + M, N=N, M=M, lo=-amp, hi=amp)
    C[:, 0] = 0.0
    C[:, 1] = 0.0
    C[N // 3, 1] = amp
    C[N // 2:, 2] = 0.0
    C[::3, 3] = 0.0
    C[:, 4] *= 1e-160   # squares below 2^-480
    C[:, 5] *= 1e-300
    C[:, 6] = -0.0
    C[0, 6] = amp
    if not ch:
        C[:, 7] *= BIG
        C[:, 8] *= 1e290
    return C


@pytest.mark.parametrize("kind,scheme,bc,coef,dt,amp", CASES)
@pytest.mark.parametrize("N,M", [(64, 40), (100, 33000)])
def test_zeros_and_magnitudes(env, kind, scheme, bc, coef, dt, amp, N, M):
    sb, torch = env
    nsteps = 3
    C = special_state(N, M, amp, kind == "cahn_hilliard")
    d = to_dev(C, torch)
    sb.sb_stepper_run(sb.sb_stepper_create(kind, scheme, bc, N, coef, dt), d, nsteps)
    cols = np.arange(12)
    out = to_host(d[:, :12])
    ref = oracle_run(kind, scheme, bc, N, coef, dt, C[:, cols], nsteps)
    assert np.all(out[:, 0] == 0.0)
    big = np.maximum(np.abs(ref).max(axis=0), 1e-305)  # into the range whose squares can be summed
    assert np.max(relerr_per_system(out / big, ref / big)) <= 1e-12


@pytest.mark.parametrize("kind,scheme,bc,coef,dt,amp", CASES)
@pytest.mark.parametrize("N,M", [(64, 40), (100, 33000)])
def test_non_finite_values_stay_in_their_simulation(env, kind, scheme, bc, coef, dt, amp, N, M):
    sb, torch = env
    st = sb.sb_stepper_create(kind, scheme, bc, N, coef, dt)
    C = to_dev(synth.rhs_uniform(seed=7, N=N, M=M, lo=-amp, hi=amp), torch)
    D = C.clone()
    sb.sb_stepper_run(st, C, 3)
    D[N // 2, 3], D[0, 8], D[N - 1, 20], D[5, M - 1] = float("nan"), float("inf"), -float("inf"), float("nan")
    sb.sb_stepper_run(st, D, 3)
    hit = [3, 8, 20, M - 1]
    keep = [m for m in range(M) if m not in hit]
    assert torch.equal(C[:, keep], D[:, keep])
    assert torch.all(torch.any(~torch.isfinite(D[:, hit]), dim=0))


@pytest.mark.parametrize("adv", [0.05, -0.05])
def test_forced_steps(env, adv):
    sb, torch = env
    N, M, gamma, dt = 64, 50, 1.0, 0.02
    st = sb.sb_stepper_create("cahn_hilliard", "be", "periodic", N, gamma, dt)
    g = dt * np.cos(2 * np.pi * np.arange(N) / N)
    sb.sb_stepper_set_forcing(st, adv, g)
    C = special_state(N, M, 0.5, True)
    amp = np.linspace(0.0, 1.0, M)
    amp[:10] = 0.0
    d = to_dev(C, torch)
    sb.sb_stepper_run_forced(st, d, to_dev(amp, torch), 3)
    ref, A = C, steppers.SharedPentaPeriodic(*matrices.ch_matrix_periodic(N, dt * gamma))
    for _ in range(3):
        ref = steppers.forced_ch_step_periodic(A, ref, dt, adv, amp, g)
    out = to_host(d)
    big = np.maximum(np.abs(ref).max(axis=0), 1e-305)
    # (the squared differences of simulations 4 and 5 vanish under the scheme's 1e-99: both
    # sides take the linear weights there)
    assert np.max(relerr_per_system(out / big, ref / big)) <= 1e-12
    assert np.all(out[:, 0] == 0.0)
    e = to_dev(C, torch)
    e[9, 11] = float("nan")
    sb.sb_stepper_run_forced(st, e, to_dev(amp, torch), 3)
    keep = [m for m in range(M) if m != 11]
    assert torch.equal(e[:, keep], d[:, keep]) and not torch.all(torch.isfinite(e[:, 11]))


@pytest.mark.parametrize("bc", ["noflux", "periodic"])
def test_coarsening_run(env, bc):
    """The state agrees with the plain steps, and the last length with the state."""
    sb, torch = env
    N, M = 100, 33000
    st = sb.sb_stepper_create("cahn_hilliard", "be", bc, N, 1.0, 0.05)
    state = special_state(N, M, 0.5, True)
    state[:, 4:6] = 0.25  # (squares of the tiny ones cannot be summed)
    C = to_dev(state, torch)
    D, ell = C.clone(), torch.empty(3, dtype=torch.float64, device="cuda")
    work = torch.empty(M + 256, dtype=torch.float64, device="cuda")
    sb.sb_stepper_run_coarsening(st, D, 3, ell, work)
    sb.sb_stepper_run(st, C, 3)
    assert np.max(relerr_per_system(to_host(D)[:, :12] , to_host(C)[:, :12] )) <= 1e-12
    assert float((C - D).norm() / C.norm()) <= 1e-12
    mean = (1.0 / (1.0 - (C * C).mean(dim=0))).mean()
    assert abs(float(ell[2] - mean)) <= 1e-12 * float(mean)


@pytest.mark.parametrize("kind", ["diffusion", "hyperdiffusion", "cahn_hilliard"])
def test_adjoint_step(env, kind):
    sb, torch = env
    N, M, T, k = 40, 45, 5, 2
    p, dt = (1.0, 0.05) if kind == "cahn_hilliard" else (0.3, 0.0)
    bc = {"diffusion": "dirichlet", "hyperdiffusion": "hinged", "cahn_hilliard": "noflux"}[kind]
    prob = {"diffusion": lambda: rollout.diffusion_problem(N, p),
            "hyperdiffusion": lambda: rollout.hyperdiffusion_problem(N, p),
            "cahn_hilliard": lambda: rollout.ch_problem(N, p, dt)}[kind]()
    x0, y = special_state(N, M, 0.5, True), synth.rhs_uniform(seed=2, N=N, M=M)
    y[:, 0] = 0.0  # state and gradient are zero
    y[::2, 2] = 0.0
    st = sb.sb_stepper_create(kind, "be", bc, N, p, dt)

    def grads(x0, scale=1.0):
        d0 = to_dev(x0, torch)
        work = torch.empty(sb.sb_rollout_workspace_bytes(st, M, T, k) // 8, dtype=torch.float64, device="cuda")
        CT, g = torch.empty_like(d0), torch.empty_like(d0)
        sb.sb_rollout_forward(st, d0, CT, T, k, work)
        dp = torch.empty(M, dtype=torch.float64, device="cuda")
        sb.sb_rollout_backward(st, scale * 2.0 * (CT - to_dev(y, torch)) / (N * M), g, T, k, work,
                               grad_param_per_system=dp)
        torch.cuda.synchronize()
        return to_host(g), to_host(dp)

    g, dp = grads(x0)
    _, gr, dpr = rollout.adjoint(prob, x0, y, T)
    assert np.max(np.abs(g - gr)) <= 1e-10 * np.max(np.abs(gr))
    assert np.max(np.abs(dp - dpr)) <= 1e-10 * np.max(np.abs(dpr))
    assert np.all(g[:, 0] == 0.0) and dp[0] == 0.0
    tiny = 2.0 ** -960  # the adjoint is linear: scaled by a power of two, out of the products' range
    gs, dps = grads(x0, tiny)
    assert np.max(np.abs(gs / tiny - gr)) <= 1e-10 * np.max(np.abs(gr))
    assert np.max(np.abs(dps / tiny - dpr)) <= 1e-10 * np.max(np.abs(dpr))
    x0[7, 11] = np.nan
    gn, dpn = grads(x0)
    keep = [m for m in range(M) if m != 11]
    assert np.array_equal(gn[:, keep], g[:, keep]) and np.array_equal(dpn[keep], dp[keep])
    assert not np.all(np.isfinite(gn[:, 11]))
