"""The paper-layout export over its forms: blocks of 32 states that the model
does not fill, one to 32 states per slice, rows too long for the staged
entries and slices too wide for the staged columns, prefix sums over one tile
and several.  FP64 check models equal the oracle's arrays; an export without
entries gives the same row pointers and R."""
import numpy as np
import pytest

import oracle
from conftest import custom_env
from paper_2109_00857_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mdp():
    from paper_2109_00857_gb300 import mdp as m
    m.load()
    return m


def env_of(nx, ny, nt, A, N, spread, L, seed=3):
    """A random flow; `spread` sets how many successors a row has."""
    rng = np.random.default_rng(seed)
    K = 2
    obst = (rng.random((nt, ny, nx)) < 0.05).astype(np.uint8)
    target = np.zeros((ny, nx), np.uint8)
    target[ny // 2, nx // 2] = 1
    return custom_env(nx=nx, ny=ny, nt=nt, K=K, N=N, L=L, vbar=rng.uniform(-.5, .5, (nt, ny, nx, 2)),
                      modes=rng.uniform(-1, 1, (nt, K, ny, nx, 2)), sigma=np.full(K, 0.1),
                      Y=np.clip(rng.normal(0, spread, (nt, N, K)), -3.5 * spread, 3.5 * spread),
                      obstacle=obst, target=target, actions=inputs.action_table(A, 1, 1.0), r_outbound=-3.0)


CASES = {
    "one_cell": (1, 1, 1, 16, 3, 0.2, 5),
    "one_action": (5, 3, 4, 1, 20, 0.3, 9),
    "three_actions": (7, 5, 3, 3, 33, 0.3, 9),
    "a16": (13, 7, 4, 16, 60, 0.3, 9),
    "a31": (9, 8, 3, 31, 50, 0.3, 9),
    "a32_one_more_state": (11, 3, 3, 32, 40, 0.3, 9),
    "long_rows": (12, 11, 3, 16, 400, 0.9, 21),
    "wide_slices": (12, 11, 3, 32, 400, 1.2, 25),
}
# an action's 32 rows exceed their 384 staged entries; (True) so do the block's 320 columns
BEYOND = {"long_rows": False, "wide_slices": True}


@pytest.mark.parametrize("case", sorted(CASES))
def test_export_equals_the_oracle(mdp, case):
    env = env_of(*CASES[case])
    ref = oracle.build(env, objs=(0, 1))
    assert ref.overflow == 0
    if case in BEYOND:
        length = np.diff(ref.rowptr).reshape(env.A, env.nS)
        rows = [length[:, b:b + 32].sum(axis=1).max() for b in range(0, env.nS, 32)]
        spw = 32 // (1 << (env.A - 1).bit_length())
        width = length.max(axis=0)[:env.nS // spw * spw].reshape(-1, spw).max(axis=1)
        cols = [width[b:b + 32 // spw].sum() for b in range(0, len(width), 32 // spw)]
        assert max(rows) > 384 + 64 and (max(cols) > 320 + 32) == BEYOND[case]
    m = mdp.mdp_build(mdp.DeviceEnv(env, mdp.MDP_FP64_CHECK), objs=(0, 1))
    for o in range(2):
        rp, col, cnt, R = (x.cpu().numpy() for x in mdp.mdp_export_csr(m, o))
        assert np.array_equal(rp, ref.rowptr) and np.array_equal(col, ref.col) and np.array_equal(cnt, ref.cnt)
        np.testing.assert_allclose(R, ref.R[o], rtol=1e-12, atol=1e-12)
        rp2, c2, n2, R2 = mdp.mdp_export_csr(m, o, with_entries=False)
        assert c2 is None and n2 is None
        assert np.array_equal(rp2.cpu().numpy(), rp) and np.array_equal(R2.cpu().numpy(), R)


def test_prefix_sums_over_several_tiles(mdp):
    """More than 4096 blocks of rows and slices: the scans take several tiles."""
    env = inputs.energy(nx=90, ny=80, nt=12, N=40, L=15, objectives=(0,))
    d = mdp.DeviceEnv(env, mdp.MDP_FP32)
    m = mdp.mdp_build(d, objs=(0,))
    assert env.nS // 32 * env.A > 2 * 4096 and env.nS > 2 * 4096
    rp, col, cnt, R = (x.cpu().numpy() for x in mdp.mdp_export_csr(m, 0))
    assert rp[0] == 0 and rp[-1] == m.info().nnz == len(col)
    assert (np.diff(rp) >= 0).all()
    # every sampled or sink row's counts sum to N, terminal rows are empty
    sums = np.add.reduceat(np.concatenate([cnt, [0]]), np.minimum(rp[:-1], len(cnt)))
    sums[np.diff(rp) == 0] = 0
    fixed = np.tile(np.broadcast_to(env.target.reshape(1, -1) != 0, (env.nt, env.Nc)).reshape(-1), env.A)
    assert (sums[~fixed] == env.N).all() and (sums[fixed] == 0).all()
    inner = np.ones(len(col), bool)
    inner[rp[1:-1][rp[1:-1] < len(col)]] = False
    assert (np.diff(col)[inner[1:]] > 0).all()   # ascending within a row
