"""The backward passes' launch shapes: layers of one slice per warp, layers on both
sides of the size where one-state-per-slice models change from the warp-per-slice
to the warp-specialized kernel (7 slices per resident warp for one or two value
components a state, 3 for more; 152 SMs x 32 warps: 34,048 and 14,592 slices), and a
wait that runs out in either.  Values and policies equal the full sweeps' bit for bit."""
import numpy as np
import pytest

from paper_2109_00857_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mdp():
    from paper_2109_00857_gb300 import mdp as m
    m.load()
    return m


def model_of(mdp, side_x, side_y, headings, speeds, nt=3):
    env = inputs.energy(nx=side_x, ny=side_y, nt=nt, N=24, K=2, sigma=(0.2, 0.1), amplitude=1.0, n_headings=headings,
                        n_speeds=speeds, square=max(2, min(side_x, side_y) // 10), objectives=(0, 1, 2))
    return mdp.mdp_build(mdp.DeviceEnv(env), objs=env.objectives)


@pytest.mark.parametrize("side_x, side_y, headings, speeds", [
    (3, 2, 16, 2), (31, 33, 16, 2), (120, 121, 16, 2), (125, 125, 16, 2), (184, 185, 16, 2), (190, 181, 16, 2),
    (5, 3, 16, 1), (41, 39, 16, 1), (111, 113, 8, 1), (20, 19, 1, 1)])
def test_layers_equal_full_sweeps(mdp, side_x, side_y, headings, speeds):
    m = model_of(mdp, side_x, side_y, headings, speeds)
    full = [mdp.mdp_solve(m, o, method=mdp.MDP_SOLVE_JACOBI_FULL, tol=0.0) for o in range(3)]
    for slots in ((0,), (1, 2), (0, 1, 2)):
        for method in (mdp.MDP_SOLVE_JACOBI, mdp.MDP_SOLVE_LAYERED):
            V, pi, _ = mdp.mdp_solve_multi(m, slots, method=method, tol=0.0)
            for i, o in enumerate(slots):
                assert np.array_equal(V[i].cpu().numpy(), full[o][0].cpu().numpy()), (slots, method)
                assert np.array_equal(pi[i].cpu().numpy(), full[o][1].cpu().numpy()), (slots, method)


@pytest.mark.parametrize("side, headings, speeds", [(40, 16, 1), (40, 16, 2), (200, 16, 2)])
def test_a_wait_that_runs_out_in_a_layer(mdp, side, headings, speeds):
    """A completion that nothing delivers, with a short limit: the kernel gives up, drains and
    returns; the call reports the timeout and the next solve is right."""
    m = model_of(mdp, side, side, headings, speeds)
    lib = mdp.load()
    for method in (mdp.MDP_SOLVE_JACOBI, mdp.MDP_SOLVE_LAYERED):
        before = mdp.mdp_solve(m, 0, method=method, tol=0.0)[0].cpu().numpy()
        assert lib.mdp_test_inject(2, 2_000_000) == 0   # about 1 ms
        assert lib.mdp_test_inject(1, 1024) == 0
        try:
            with pytest.raises(mdp.MdpError) as ei:
                mdp.mdp_solve(m, 0, method=method, tol=0.0)
            assert ei.value.code == -5
        finally:
            lib.mdp_test_inject(2, 0)
        assert np.array_equal(mdp.mdp_solve(m, 0, method=method, tol=0.0)[0].cpu().numpy(), before)
