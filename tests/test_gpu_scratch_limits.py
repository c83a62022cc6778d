"""Calls near the device's memory limit: what is only a shortcut falls back when its memory cannot be had."""
import numpy as np
import pytest

from paper_2109_00857_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mdp():
    from paper_2109_00857_gb300 import mdp as m
    m.load()
    return m


@pytest.mark.parametrize("n_obj", [1, 2, 3])
@pytest.mark.parametrize("speeds", [1, 2])
def test_a_cold_solve_without_memory_for_the_chains(mdp, n_obj, speeds):
    env = inputs.energy(nx=17, ny=13, nt=9, N=40, K=2, sigma=(0.2, 0.1), n_speeds=speeds, square=3, objectives=(0, 1, 2))
    m = mdp.mdp_build(mdp.DeviceEnv(env), objs=env.objectives)
    slots = tuple(range(n_obj))
    want = mdp.mdp_solve_multi(m, slots, method=mdp.MDP_SOLVE_JACOBI_FULL)
    assert mdp.load().mdp_test_inject(3, 1) == 0   # the first allocation of the solve: the chains' table
    try:
        V, p, s = mdp.mdp_solve_multi(m, slots)
    finally:
        mdp.load().mdp_test_inject(3, 0)
    for i in range(n_obj):
        assert np.array_equal(V[i].cpu().numpy(), want[0][i].cpu().numpy())
        assert np.array_equal(p[i].cpu().numpy(), want[1][i].cpu().numpy())
        assert (s[i].sweeps, s[i].residual) == (want[2][i].sweeps, want[2][i].residual)
    assert s[0].backups != 2 * env.nS * env.A   # (the sweeps')


def test_allocations_that_are_needed_still_fail_the_call(mdp):
    env = inputs.tiny(nx=9, ny=9, nt=4, N=30)
    d = mdp.DeviceEnv(env)
    m = mdp.mdp_build(d)
    lib = mdp.load()
    for call in (lambda: mdp.mdp_build(d), lambda: mdp.mdp_solve(m, 0, method=mdp.MDP_SOLVE_JACOBI_FULL)):
        assert lib.mdp_test_inject(3, 1) == 0
        try:
            with pytest.raises(mdp.MdpError) as ei:
                call()
            assert ei.value.code in (-2, -6)
        finally:
            lib.mdp_test_inject(3, 0)
        call()
