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


@pytest.mark.parametrize("nx, ny, nt, headings, speeds", [(60, 50, 20, 16, 1), (60, 50, 20, 16, 2), (7, 5, 3, 3, 1),
                                                          (1, 1, 1, 16, 1), (9, 7, 3, 31, 1), (40, 40, 300, 1, 1)])
def test_an_export_without_memory_for_its_sums(mdp, nx, ny, nt, headings, speeds):
    env = inputs.make_env(nx=nx, ny=max(ny, 2), nt=nt, K=2, N=30, L=11, sigma=(0.2, 0.1), seed=5, amplitude=1.0,
                          n_headings=headings, n_speeds=speeds, with_gbar=True, objectives=(0, 2))
    m = mdp.mdp_build(mdp.DeviceEnv(env), objs=env.objectives)
    for entries in (True, False):
        want = mdp.mdp_export_csr(m, 1, with_entries=entries)
        assert mdp.load().mdp_test_inject(3, 1) == 0
        try:
            got = mdp.mdp_export_csr(m, 1, with_entries=entries)
        finally:
            mdp.load().mdp_test_inject(3, 0)
        for x, y in zip(got, want):
            assert (x is None and y is None) or np.array_equal(x.cpu().numpy(), y.cpu().numpy())
