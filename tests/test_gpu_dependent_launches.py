"""Layers whose kernels overlap, when a wait runs out: the error word may be set at any moment of the
next layer's start, so every CTA has to take one decision for all its threads, and the calls that
follow have to find every layer ended.  The limit of the wait (about 50 us to 1 ms, far above a copy's
latency) puts the word's arrival at different points of the next layer's start."""
import numpy as np
import pytest

from paper_2109_00857_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mdp():
    from paper_2109_00857_gb300 import mdp as m
    m.load()
    return m


@pytest.mark.parametrize("side, headings, speeds", [(24, 8, 1), (60, 16, 1), (60, 16, 2), (200, 16, 2)])
@pytest.mark.parametrize("method", ["jacobi", "layered"])
def test_a_wait_that_runs_out_while_the_next_layer_starts(mdp, side, headings, speeds, method):
    method = {"jacobi": mdp.MDP_SOLVE_JACOBI, "layered": mdp.MDP_SOLVE_LAYERED}[method]
    env = inputs.energy(nx=side, ny=side, nt=8, N=24, K=2, sigma=(0.2, 0.1), amplitude=1.0, n_headings=headings,
                        n_speeds=speeds, square=4, objectives=(0, 1, 2))
    m = mdp.mdp_build(mdp.DeviceEnv(env), objs=env.objectives)
    lib = mdp.load()
    want = [v.cpu().numpy() for v in mdp.mdp_solve_multi(m, (0, 1, 2), method=method, tol=0.0)[0]]
    for i, cycles in enumerate(np.geomspace(100_000, 2_000_000, 12).astype(int)):
        slots = (0,) if i % 2 else (0, 1, 2)
        assert lib.mdp_test_inject(2, int(cycles)) == 0
        assert lib.mdp_test_inject(1, 1024) == 0
        try:
            with pytest.raises(mdp.MdpError) as ei:
                mdp.mdp_solve_multi(m, slots, method=method, tol=0.0)
            assert ei.value.code == -5
        finally:
            lib.mdp_test_inject(2, 0)
        V = mdp.mdp_solve_multi(m, slots, method=method, tol=0.0)[0]   # (on the memory just given back)
        for o, v in zip(slots, V):
            assert np.array_equal(v.cpu().numpy(), want[o])
