"""The two-comparison rank lookup with a crowded first bucket (action sets whose zero
displacements differ by rounding at three and more speeds, beside thresholds that
share a bucket): fractions below, at and above the tiny thresholds, exact zeros
included, give the full-window kernel's model bit for bit."""
import numpy as np
import pytest

from conftest import custom_env
from paper_2109_00857_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mdp():
    from paper_2109_00857_gb300 import mdp as m
    m.load()
    return m


@pytest.mark.parametrize("headings, speeds, K", [(8, 3, 1), (8, 3, 4), (8, 3, 8), (8, 3, 9), (4, 3, 3), (10, 3, 2)])
@pytest.mark.parametrize("tiny", [False, True])
def test_crowded_first_bucket(mdp, headings, speeds, K, tiny):
    rng = np.random.default_rng(headings * 10 + K)
    nx, ny, nt, N = 13, 9, 3, 190
    vbar = rng.uniform(-.6, .6, (nt, ny, nx, 2))
    modes = rng.uniform(-.5, .5, (nt, K, ny, nx, 2))
    if tiny:   # u = 1/2 + w an integer, or within rounding of one, on a third of the cells
        vbar[:, ::3] = rng.choice([-0.5, 0.5, np.float32(-0.5) + 2.0 ** -25, -0.5 + 2.0 ** -24], vbar[:, ::3].shape)
        modes[:, :, ::3] = 0.0
        vbar[:, 1::3, ::2] = -0.5
        modes[:, :, 1::3, ::2] *= 2.0 ** -22
    actions = inputs.action_table(headings, speeds, 1.0)
    env = custom_env(nx=nx, ny=ny, nt=nt, K=K, N=N, L=13, vbar=vbar, modes=modes, sigma=np.full(K, 0.5),
                     Y=np.clip(rng.normal(0, 0.5, (nt, N, K)), -1.2, 1.2), actions=actions, r_outbound=-3.0)
    d = mdp.DeviceEnv(env)
    outs = []
    for cap in (0, 1):
        o = mdp.MdpBuildOpts()
        o.hist_cap = cap
        m = mdp.mdp_build(d, objs=(0,), opts=o)
        outs.append([x.cpu().numpy() for x in mdp.mdp_export_csr(m, 0)])
    for x, y in zip(*outs):
        assert np.array_equal(x, y)
