"""A layered batch's CTAs work out their shares of a step themselves: over fewer
and more models than a warp's lanes, uneven in layers, cells and actions (one to
four states per slice), every member has its solo layered solve's values and policy."""
import numpy as np
import pytest

from paper_2109_00857_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mdp():
    from paper_2109_00857_gb300 import mdp as m
    m.load()
    return m


@pytest.mark.parametrize("n", [1, 31, 33, 70])
def test_layer_shares_over_many_models(mdp, n):
    shapes = ((5, 4, 1, 16, 2), (9, 7, 3, 16, 1), (21, 13, 6, 8, 1), (41, 39, 2, 16, 2), (3, 2, 9, 3, 1))
    denvs = []
    for i in range(n):
        nx, ny, nt, headings, speeds = shapes[i % len(shapes)]
        env = inputs.energy(nx=nx + i % 3, ny=ny, nt=nt + i % 2, N=30 + i, K=2, sigma=(0.2, 0.1), amplitude=1.0,
                            n_headings=headings, n_speeds=speeds, square=2, objectives=(0,), seed=50 + i)
        denvs.append(mdp.DeviceEnv(env))
    b = mdp.Batch(denvs, tol=0.0)
    b.run()
    for i, d in enumerate(denvs):
        V, pi, _ = mdp.mdp_solve(mdp.mdp_build(d, objs=(0,)), 0, method=mdp.MDP_SOLVE_LAYERED, tol=0.0)
        assert np.array_equal(b.V[i].cpu().numpy(), V.cpu().numpy()), i
        assert np.array_equal(b.policy[i].cpu().numpy(), pi.cpu().numpy()), i
    b.close()
