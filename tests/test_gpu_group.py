"""The FP32 group build kernel at the sizes where it can go wrong: every number
of states per slice (1..32 actions), mode counts of each instantiation, N
around the realizations a CTA counts per trip, grids whose last group of
slices is partial, count windows that are predicted badly (heavy-tailed,
correlated or constant coefficient tables, integer displacements of the flow),
action tables with crowded step thresholds, single-model and batched.  The
reference is the full-window kernel, which counts one increment per
(realization, action): the model must be the same bit for bit."""
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


def field(nx, ny, nt, K, N, A, seed, Y=None, L=15, amp=0.8, actions=None, n_obj=3, sigma=0.25):
    rng = np.random.default_rng(seed)
    vbar = rng.uniform(-amp, amp, (nt, ny, nx, 2))
    modes = rng.standard_normal((nt, K, ny, nx, 2)).clip(-2, 2)
    obstacle = (rng.random((nt, ny, nx)) < 0.08).astype(np.uint8)
    target = np.zeros((ny, nx), np.uint8)
    target[ny // 2, nx // 2] = 1
    if actions is None:
        actions = inputs.action_table(A, 1, 1.0) if A != 32 else inputs.action_table(16, 2, 1.0)
    gbar = rng.random((nt, ny, nx))
    return custom_env(nx=nx, ny=ny, nt=nt, K=K, N=N, L=L, vbar=vbar, modes=modes,
                      sigma=sigma / np.sqrt(max(K, 1)) * np.ones(K), seed=seed, obstacle=obstacle, target=target,
                      actions=actions, gbar=gbar, Y=Y, objectives=(0, 1, 2)[:n_obj], r_term=3.0, r_outbound=-50.0)


def check(mdp, env):
    d = mdp.DeviceEnv(env)
    o = mdp.MdpBuildOpts()
    o.hist_cap = 1   # every sampled slice through the full-window kernel
    m0, m1 = mdp.mdp_build(d, objs=env.objectives, opts=o), mdp.mdp_build(d, objs=env.objectives)
    assert m1.info().wide_slices < m0.info().wide_slices   # the group kernel built slices
    for k in range(len(env.objectives)):
        for x, y in zip(mdp.mdp_export_csr(m0, k), mdp.mdp_export_csr(m1, k)):
            assert np.array_equal(x.cpu().numpy(), y.cpu().numpy())
    return m1


@pytest.mark.parametrize("A", [1, 2, 3, 5, 8, 12, 16, 31, 32])
@pytest.mark.parametrize("K,N", [(0, 7), (1, 1), (2, 33), (3, 64), (4, 257), (5, 31), (6, 100), (7, 65), (8, 513), (9, 50)])
def test_group_kernel_equals_the_full_window_kernel(mdp, A, K, N):
    # 9 x 7 cells: 63 states a layer, so groups straddle layers and the last one is partial
    check(mdp, field(9, 7, 3, K, N, A, seed=100 * A + K))


@pytest.mark.parametrize("kind", ["heavy_tail", "correlated", "constant", "offset", "integer"])
@pytest.mark.parametrize("A,K", [(32, 4), (16, 3), (8, 2)])
def test_badly_predicted_windows(mdp, kind, A, K):
    rng = np.random.default_rng(5)
    nt, N = 3, 300
    Y = rng.standard_normal((nt, N, K)) * 0.1
    amp = 0.8
    if kind == "heavy_tail":
        Y[:, ::97] *= 4.0
    elif kind == "correlated":
        Y = np.repeat(Y[:, :, :1] * 2.0, K, axis=2)
    elif kind == "constant":
        Y[:] = 0.2
    elif kind == "offset":
        Y += 0.7
    else:   # every u an exact integer or half: fractions 0, steps at equality
        Y[:] = 0.0
    env = field(10, 9, nt, K, N, A, seed=11, Y=Y, amp=amp, L=31)
    if kind == "integer":
        env.vbar[:] = np.round(env.vbar * 2) / 2 + 0.5
    check(mdp, env)


@pytest.mark.parametrize("A,spread", [(32, 1.0), (32, 1e-3), (16, 1e-6), (7, 1e-2)])
def test_crowded_step_thresholds(mdp, A, spread):
    """Random displacements, and clusters of displacements within `spread`."""
    rng = np.random.default_rng(int(1e7 * spread) + A)
    act = np.zeros((A, 3))
    act[:, :2] = 0.3 + spread * rng.uniform(-0.5, 0.5, (A, 2))
    act[:, 2] = rng.uniform(0.1, 1.0, A)
    act[0, :2] = (0.0, 1.0)
    check(mdp, field(8, 9, 3, 3, 200, A, seed=3, actions=act))


def test_wide_tables_go_to_the_full_window_kernel(mdp):
    env = field(8, 8, 3, 4, 400, 32, seed=2, L=31, sigma=0.4)
    assert check(mdp, env).info().wide_slices > 0


@pytest.mark.parametrize("A", [3, 16, 32])
def test_batched_group_kernel_equals_single_builds(mdp, A):
    rng = np.random.default_rng(8)
    envs = []
    for i, (K, N) in enumerate([(3, 100), (4, 77), (3, 210), (9, 40)]):
        Y = rng.standard_normal((4, N, K)) * 0.2 if i == 2 else None
        envs.append(field(7 + 2 * i, 9, 4, K, N, A, seed=40 + i, n_obj=1, Y=Y))
    b = mdp.Batch([mdp.DeviceEnv(e) for e in envs])
    for _ in range(2):
        b.run()
        for e, V, pi in zip(envs, b.V, b.policy):
            m = mdp.mdp_build(mdp.DeviceEnv(e))
            V1, p1, _ = mdp.mdp_solve(m, 0, method=mdp.MDP_SOLVE_LAYERED)
            assert np.array_equal(V.cpu().numpy(), V1.cpu().numpy())
            assert np.array_equal(pi.cpu().numpy(), p1.cpu().numpy())
