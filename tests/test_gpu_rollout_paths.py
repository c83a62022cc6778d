"""Rollouts by mode count and alignment: fields and coefficients at addresses
that allow vector loads and fixed mode counts give the paths of the general
kernel, which the same arrays one element further take; both end where a walk
through the velocities on the host ends."""
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


def shifted(x):
    """The same values one element further into an allocation."""
    import torch
    buf = torch.empty(x.numel() + 1, dtype=x.dtype, device=x.device)
    buf[1:] = x.reshape(-1)
    assert buf[1:].data_ptr() % 8 == 4
    return buf[1:].view(x.shape)


def walk(env, policy, start):
    """(steps, status) of every realization in float32, as the moves are defined."""
    f = np.float32
    ph, vb, Y = env.modes.astype(f), env.vbar.astype(f), env.Y.astype(f)
    steps, status = np.zeros(env.N, np.int32), np.ones(env.N, np.int8)
    for w in range(env.N):
        i, j = start
        for t in range(env.nt):
            if env.target[j, i]:
                status[w] = 0
                break
            steps[w] += 1
            a = policy[t, j, i]
            if env.obstacle[t, j, i] or t == env.nt - 1 or a < 0:
                break
            v = [float(vb[t, j, i, c]) + sum(float(Y[t, w, k]) * float(ph[t, k, j, i, c]) for k in range(env.K))
                 for c in range(2)]
            i += int(np.floor(0.5 + v[0] + env.actions[a, 0]))
            j += int(np.floor(0.5 + v[1] + env.actions[a, 1]))
            if not (0 <= i < env.nx and 0 <= j < env.ny) or env.obstacle[t + 1, j, i]:
                break
    return steps, status


@pytest.mark.parametrize("K, N, nt", [(0, 5, 4), (1, 129, 6), (2, 130, 6), (3, 127, 6), (4, 200, 7), (5, 64, 6),
                                      (6, 65, 6), (7, 33, 6), (8, 257, 8), (9, 70, 6), (16, 31, 5), (8, 1, 1)])
def test_vector_loads_and_fixed_mode_counts_give_the_general_paths(mdp, K, N, nt):
    import torch
    rng = np.random.default_rng(100 * K + N)
    nx, ny = 23, 17
    obst = (rng.random((nt, ny, nx)) < 0.04).astype(np.uint8)
    target = np.zeros((ny, nx), np.uint8)
    target[8:10, 11:13] = 1
    # exact in float32 and in the sums: the walk's double arithmetic takes the same floors
    q = lambda shape, n: rng.integers(-n, n + 1, shape) / 64.0
    env = custom_env(nx=nx, ny=ny, nt=nt, K=K, N=N, L=31, vbar=q((nt, ny, nx, 2), 48),
                     modes=q((nt, K, ny, nx, 2), 32), sigma=np.full(K, 0.1), Y=q((nt, N, K), 64),
                     obstacle=obst, target=target, gbar=rng.random((nt, ny, nx)),
                     actions=np.concatenate([q((16, 2), 64), np.ones((16, 1))], axis=1))
    pol = rng.integers(-1, 16, (nt, ny, nx)).astype(np.int16)
    pol[rng.random(pol.shape) < 0.9] = 3
    starts = [(3, 4), (12, 8), (22, 16), (0, 0), (11, 11)]
    d = mdp.DeviceEnv(env, mdp.MDP_FP32)
    dpol = torch.as_tensor(pol.reshape(-1)).cuda()
    got = [x.cpu().numpy() for x in mdp.mdp_rollout(d, dpol, starts, objs=(0, 1, 2))[:3]]
    d.vbar = shifted(d.vbar)
    if K:
        d.modes, d.coeffs = shifted(d.modes), shifted(d.coeffs)
    gen = [x.cpu().numpy() for x in mdp.mdp_rollout(d, dpol, starts, objs=(0, 1, 2))[:3]]
    for x, y in zip(got, gen):
        assert np.array_equal(x, y)
    for n, start in enumerate(starts):
        steps, status = walk(env, pol, start)
        assert np.array_equal(got[1][n], steps) and np.array_equal(got[2][n], status), start
