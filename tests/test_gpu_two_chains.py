"""MDP_SOLVE_JACOBI from two backward chains: a cold-started run gives the values,
policy, sweep count and residual of MDP_SOLVE_JACOBI_FULL (every state in every
sweep) bit for bit, whether the chains prove that it ends in sweep nt + 1 or
leave it (or some of its objectives) to the sweeps."""
import numpy as np
import pytest

from conftest import custom_env
from paper_2109_00857_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mdp():
    import torch
    torch.cuda.set_device(0)
    from paper_2109_00857_gb300 import build_native, mdp as m
    build_native.build()
    m.load()
    return m


def same(mdp, model, slots, tol, max_sweeps=0):
    got = mdp.mdp_solve_multi(model, slots, method=mdp.MDP_SOLVE_JACOBI, tol=tol, max_sweeps=max_sweeps)
    for i, o in enumerate(slots):
        V, pi, st = mdp.mdp_solve(model, o, method=mdp.MDP_SOLVE_JACOBI_FULL, tol=tol, max_sweeps=max_sweeps)
        assert np.array_equal(got[0][i].cpu().numpy(), V.cpu().numpy())
        assert np.array_equal(got[1][i].cpu().numpy(), pi.cpu().numpy())
        assert (got[2][i].sweeps, got[2][i].residual) == (st.sweeps, st.residual)
    return got[2]


@pytest.mark.parametrize("headings,speeds", [(1, 1), (3, 1), (8, 1), (16, 1), (16, 2)])
@pytest.mark.parametrize("nx,ny,nt", [(7, 5, 1), (9, 7, 2), (33, 21, 9)])
def test_two_chains_equal_full_sweeps(mdp, headings, speeds, nx, ny, nt):
    env = inputs.energy(nx=nx, ny=ny, nt=nt, N=70, K=2, sigma=(0.2, 0.1), amplitude=1.0, n_headings=headings,
                        n_speeds=speeds, square=3, objectives=(0, 1, 2))
    m = mdp.mdp_build(mdp.DeviceEnv(env), objs=env.objectives)
    for slots in ((0,), (2, 0), (0, 1, 2)):
        for tol in (0.0, 1e-6, 0.5, 40.0, 1e9):
            same(mdp, m, slots, tol)
    same(mdp, m, (0, 2), 0.0, max_sweeps=nt + 5)
    same(mdp, m, (0, 2), 0.0, max_sweeps=max(1, nt // 2))


def test_runs_that_converge_early_are_swept(mdp):
    # zero flow, every cell reaches the target in three steps: converged after a few of 13 sweeps
    target = np.zeros((5, 5), np.uint8)
    target[2, 2] = 1
    env = custom_env(nx=5, ny=5, nt=12, K=1, N=4, target=target, objectives=(0, 1, 2), gbar=np.ones((12, 5, 5)),
                     r_outbound=-100.0, c_r=0.5)
    m = mdp.mdp_build(mdp.DeviceEnv(env), objs=env.objectives)
    st = same(mdp, m, (0,), 0.0)
    assert st[0].sweeps < env.nt + 1
    # net energy: staying afloat pays, the horizon's penalty reaches every layer
    st = same(mdp, m, (2, 0), 0.0)
    assert st[1].sweeps < env.nt + 1


def test_two_chains_with_spill_rows(mdp):
    env = inputs.energy(nx=24, ny=20, nt=5, N=200, K=2, sigma=(0.6, 0.4), objectives=(0, 2), L=41)
    for n_headings, n_speeds in ((16, 2), (16, 1)):
        env.actions = inputs.action_table(n_headings, n_speeds, 1.0)
        m = mdp.mdp_build(mdp.DeviceEnv(env), objs=(0, 2), opts=mdp.MdpBuildOpts(row_cap=5))
        assert m.info().spill_rows > 0
        same(mdp, m, (0, 1), 0.0)
