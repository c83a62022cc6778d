"""Slices with a state whose fine table is larger than the state's share of the slice's table memory: the
states' tables are packed into the whole, so a slice goes to the full-window kernel only when they do not fit
hist_cap together -- and a model with a sub-grid too large for that kernel is built.  The reference is the
full-window kernel on a 41 x 41 sub-grid that holds the same landings: the models are the same bit for bit."""
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


def field(A, K, N, L, wide, narrow, every, seed=4, nx=13, ny=11, nt=3):
    """Every `every`-th cell spreads its realizations `wide` standard deviations, the others `narrow`."""
    rng = np.random.default_rng(seed)
    modes = np.zeros((nt, K, ny, nx, 2))
    scale = np.full(nx * ny, narrow)
    scale[::every] = wide
    modes[:] = (rng.uniform(0.7, 1.0, (nt, K, ny, nx, 2)) * scale.reshape(ny, nx, 1)) / np.sqrt(K)
    actions = inputs.action_table(16, 2, 1.0) if A == 32 else inputs.action_table(A, 1, 1.0)
    target = np.zeros((ny, nx), np.uint8)
    target[4, 5] = 1
    return custom_env(nx=nx, ny=ny, nt=nt, K=K, N=N, L=L, vbar=rng.uniform(-.5, .5, (nt, ny, nx, 2)), modes=modes,
                      sigma=np.ones(K), seed=seed, target=target, actions=actions, gbar=rng.random((nt, ny, nx)),
                      objectives=(0, 2), r_term=2.0, r_outbound=-9.0)


def build(mdp, env, cap):
    o = mdp.MdpBuildOpts()
    o.hist_cap = cap
    m = mdp.mdp_build(mdp.DeviceEnv(env), objs=env.objectives, opts=o)
    return m.info(), [x.cpu().numpy() for k in (0, 1) for x in mdp.mdp_export_csr(m, k)]


# (actions, modes, draws, wide, narrow, every, capacities: each holds every slice's tables together, but no
# power of two below holds the widest state's in its equal share)
CASES = {
    "one_state_6144": (32, 4, 400, 0.70, 0.5, 2, (6144,)),
    "four_states_uneven": (8, 3, 300, 1.1, 0.05, 4, (2048, 3000, 6144)),
    "eight_states_uneven": (4, 9, 200, 1.3, 0.02, 8, (2048, 1537)),
    "lone_action": (1, 2, 250, 2.0, 0.02, 32, (2048,)),
    "no_share_at_all": (1, 2, 60, 0.02, 0.02, 32, (500,)),   # 15 words a state
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_uneven_tables_share_the_slices_memory(mdp, name):
    A, K, N, wide, narrow, every, caps = CASES[name]
    want_info, want = build(mdp, field(A, K, N, 41, wide, narrow, every), 1)
    assert want_info.wide_slices > 0   # the full-window kernel
    for cap in caps:
        for L in (41, 43):   # (43: no full-window kernel, so the build is refused if a slice needs it)
            info, got = build(mdp, field(A, K, N, L, wide, narrow, every), cap)
            assert info.wide_slices == 0, (cap, L)
            for x, y in zip(got, want):
                assert np.array_equal(x, y), (cap, L)


@pytest.mark.parametrize("A", [2, 16, 32])
def test_far_velocities_are_tabled(mdp, A):
    """A flow of 20,000 cells a step against an equal own displacement."""
    env = field(A, 2, 100, 41, 0.2, 0.2, 3)
    env.vbar[:] += 20000.0
    env.actions[:, 0] -= 20000.0
    env.actions[:, 1] -= 20000.0
    want = build(mdp, env, 1)[1]
    env.L = 43
    info, got = build(mdp, env, 2048)
    assert info.wide_slices == 0
    for x, y in zip(got, want):
        assert np.array_equal(x, y)


def test_batch_with_packed_tables(mdp):
    envs = [field(8, 3, 300, 41, 1.1, 0.05, 4, seed=s) for s in (4, 5)]
    b = mdp.Batch([mdp.DeviceEnv(e) for e in envs])
    b.run()
    for e, V, pi in zip(envs, b.V, b.policy):
        m = mdp.mdp_build(mdp.DeviceEnv(e))
        V1, p1, _ = mdp.mdp_solve(m, 0, method=mdp.MDP_SOLVE_LAYERED)
        assert np.array_equal(V.cpu().numpy(), V1.cpu().numpy()) and np.array_equal(pi.cpu().numpy(), p1.cpu().numpy())
