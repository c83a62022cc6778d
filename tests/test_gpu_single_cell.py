"""States whose realizations all land in one fine cell (no spread at all, whole or half cells a step, one
realization) and rows of 13 and more successors: the shortcuts of the group build kernel's counts give the
full-window kernel's model bit for bit."""
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


def same_model(mdp, env, hist_cap=0):
    d, outs = mdp.DeviceEnv(env), []
    for cap in (1, hist_cap):
        o = mdp.MdpBuildOpts()
        o.hist_cap = cap
        m = mdp.mdp_build(d, objs=(0, 2), opts=o)
        outs.append((m.info(), [x.cpu().numpy() for k in (0, 1) for x in mdp.mdp_export_csr(m, k)]))
    assert outs[1][0].wide_slices < outs[0][0].wide_slices   # the group kernel built slices
    for x, y in zip(outs[0][1], outs[1][1]):
        assert np.array_equal(x, y)
    return outs[1][0]


@pytest.mark.parametrize("headings, speeds", [(16, 2), (16, 1), (8, 3), (8, 1), (3, 1), (1, 1)])
@pytest.mark.parametrize("K, N, shift", [(2, 100, 0.5), (2, 100, 0.0), (0, 70, 0.5), (0, 1, 0.25), (3, 1, 0.5), (9, 40, -0.5)])
def test_every_realization_in_one_cell(mdp, headings, speeds, K, N, shift):
    rng = np.random.default_rng(K + N)
    nx, ny, nt = 13, 9, 3
    vbar = np.full((nt, ny, nx, 2), shift)
    vbar[:, ::2] += rng.integers(-1, 2, vbar[:, ::2].shape)
    env = custom_env(nx=nx, ny=ny, nt=nt, K=K, N=N, L=9, vbar=vbar, modes=rng.uniform(-1, 1, (nt, K, ny, nx, 2)),
                     sigma=np.zeros(K), Y=np.zeros((nt, N, K)), actions=inputs.action_table(headings, speeds, 1.0),
                     gbar=rng.random((nt, ny, nx)), r_outbound=-5.0)
    same_model(mdp, env)


@pytest.mark.parametrize("headings, speeds, hist_cap", [(16, 2, 6144), (16, 1, 6144), (8, 1, 0), (4, 1, 0)])
def test_rows_longer_than_are_staged(mdp, headings, speeds, hist_cap):
    rng = np.random.default_rng(headings)
    nx, ny, nt, N, K = 15, 12, 3, 400, 2
    obstacle = (rng.random((nt, ny, nx)) < 0.1).astype(np.uint8)
    target = np.zeros((ny, nx), np.uint8)
    target[5, 6] = 1
    env = custom_env(nx=nx, ny=ny, nt=nt, K=K, N=N, L=21, vbar=rng.uniform(-.5, .5, (nt, ny, nx, 2)),
                     modes=rng.uniform(0.5, 0.9, (nt, K, ny, nx, 2)) * np.array([[1, 1], [1, -1]])[None, :, None, None],
                     sigma=np.full(K, 0.6), seed=4, actions=inputs.action_table(headings, speeds, 1.0), obstacle=obstacle,
                     target=target, gbar=rng.random((nt, ny, nx)), r_term=2.0, r_outbound=-5.0)
    assert same_model(mdp, env, hist_cap).max_row_nnz > 14


def test_batched_models_without_modes(mdp):
    rng = np.random.default_rng(3)
    envs = []
    for i, headings in enumerate((16, 16, 8, 1)):
        nx, ny, nt = 9 + i, 8, 4
        envs.append(custom_env(nx=nx, ny=ny, nt=nt, K=0, N=60 + i, L=9, vbar=rng.uniform(-1, 1, (nt, ny, nx, 2)),
                               modes=np.zeros((nt, 0, ny, nx, 2)), sigma=np.zeros(0), gbar=rng.random((nt, ny, nx)),
                               actions=inputs.action_table(headings, 1 + i % 2, 1.0), r_outbound=-5.0))
    b = mdp.Batch([mdp.DeviceEnv(e) for e in envs])
    b.run()
    for e, V, pi in zip(envs, b.V, b.policy):
        same_model(mdp, e)
        m = mdp.mdp_build(mdp.DeviceEnv(e))
        V1, p1, _ = mdp.mdp_solve(m, 0, method=mdp.MDP_SOLVE_LAYERED)
        assert np.array_equal(V.cpu().numpy(), V1.cpu().numpy()) and np.array_equal(pi.cpu().numpy(), p1.cpu().numpy())
