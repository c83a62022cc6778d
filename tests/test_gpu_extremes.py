"""The automatic sub-grid from the fields' component-wise extremes: the largest
magnitude is found wherever it stands, at the edges of the pieces that a block
reads (16 x 256 values, or the multiple of the components below) included."""
import math

import numpy as np
import pytest

from conftest import custom_env

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mdp():
    from paper_2109_00857_gb300 import mdp as m
    m.load()
    return m


def subgrid(env):
    """Side for offsets up to ceil(1/2 + max|v| + max|a|), one cell of buffer (dt = dx);
    the extremes are kept in 32 bits."""
    top = lambda x, ax: np.abs(x.astype(np.float32)).max(axis=ax).astype(np.float64)
    vb, ph, y = top(env.vbar, (0, 1, 2)), top(env.modes, (0, 2, 3)), top(env.Y, (0, 1))
    h = 0
    for c in range(2):
        w = vb[c]
        for k in range(env.K):
            w += y[k] * ph[k, c]
        amax = np.abs(env.actions[:, c]).max()
        h = max(h, math.ceil(0.5 + (w + amax) * (1 + 1e-6)) + 1)
    return 2 * h + 1


@pytest.mark.parametrize("nx, ny, nt, K, N", [(1, 1, 1, 1, 1), (7, 5, 3, 2, 9), (64, 32, 2, 1, 4096),
                                              (241, 17, 2, 5, 816), (33, 31, 3, 16, 300)])
@pytest.mark.parametrize("field", ["vbar", "modes", "Y"])
@pytest.mark.parametrize("place", [0.0, 0.37, 1.0])
def test_automatic_subgrid_of_a_single_extreme(mdp, nx, ny, nt, K, N, field, place):
    rng = np.random.default_rng(nx * 7 + K)
    arr = dict(vbar=rng.uniform(-.5, .5, (nt, ny, nx, 2)), modes=rng.uniform(-.5, .5, (nt, K, ny, nx, 2)),
               Y=rng.uniform(-.5, .5, (nt, N, K)))
    x = arr[field].reshape(-1)
    at = int(place * (x.size - 1))
    x[at] = -9.3 if at % 2 else 9.3
    env = custom_env(nx=nx, ny=ny, nt=nt, K=K, N=N, L=0, sigma=np.full(K, 0.1), **arr)
    for precision in (mdp.MDP_FP32, mdp.MDP_FP64_CHECK):
        m = mdp.mdp_build(mdp.DeviceEnv(env, precision), subgrid_L=0, objs=(0,))
        assert m.info().L == subgrid(env), (precision, at)
        m.free()
