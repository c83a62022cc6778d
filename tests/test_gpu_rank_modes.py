"""That the rank lookup's modes are reached: the step thresholds of the crowded action sets, worked out here,
rule out the one-comparison lookup and allow the two-comparison one with a trap in its first bucket, fractions
below the trap occur, and the group kernel (not the full-window kernel on both sides) builds the model."""
import numpy as np
import pytest

from conftest import custom_env
from paper_2109_00857_gb300 import inputs


def thresholds(d):
    """Distinct step thresholds of float32 displacements: the smallest float >= 1 - frac(d), integers excluded."""
    out = set()
    for x in np.asarray(d, dtype=np.float32).astype(np.float64):
        t1 = np.floor(x) + 1.0 - x
        if x == np.floor(x):
            continue
        f = np.float32(t1)
        if float(f) < t1:
            f = np.nextafter(f, np.float32(2))
        out.add(float(f))
    return np.array(sorted(out))


def crowds(T, B):
    return np.bincount(np.floor(T * B).astype(int), minlength=B + 1)


def plan(actions):
    """(mode, trap) by the rule stated at ActionTable."""
    axes = [thresholds(actions[:, 0]), thresholds(actions[:, 1])]
    for B in (128, 256, 512):
        traps = [T[crowds(T, B)[0] - 2] if len(T) and crowds(T, B)[0] >= 2 else 0.0 for T in axes]
        if all(crowds(T, B)[1:].max() <= 1 for T in axes if len(T)) and max(traps) <= 2.0 ** -24:
            return 1, max(traps)
    traps = [T[crowds(T, 128)[0] - 3] if len(T) and crowds(T, 128)[0] > 2 else 0.0 for T in axes]
    if all(crowds(T, 128)[1:].max() <= 2 for T in axes if len(T)) and max(traps) <= 2.0 ** -24:
        return 2, max(traps)
    return 3, 0.0


def test_the_action_sets_reach_the_modes():
    modes = {hs: plan(inputs.action_table(*hs, 1.0)) for hs in ((16, 1), (16, 2), (8, 1), (8, 3), (10, 3), (4, 3))}
    assert modes[(16, 1)][0] == 1 and modes[(16, 2)][0] == 1 and modes[(16, 2)][1] > 0.0
    assert modes[(8, 3)][0] == 2 and modes[(8, 3)][1] > 0.0
    assert modes[(10, 3)][0] == 2


@pytest.mark.gpu
@pytest.mark.parametrize("headings, speeds", [(16, 2), (8, 3), (10, 3), (4, 3)])
@pytest.mark.parametrize("K", [1, 3, 9])
def test_trapped_fractions_through_the_group_kernel(headings, speeds, K):
    from paper_2109_00857_gb300 import mdp
    mdp.load()
    actions = inputs.action_table(headings, speeds, 1.0)
    mode, trap = plan(actions)
    rng = np.random.default_rng(headings + K)
    nx, ny, nt, N = 13, 9, 3, 150
    vbar = rng.uniform(-.6, .6, (nt, ny, nx, 2))
    modes = rng.uniform(-.4, .4, (nt, K, ny, nx, 2))
    vbar[:, ::3] = rng.choice([-0.5, 0.5, -0.5 + 2.0 ** -24], vbar[:, ::3].shape)
    modes[:, :, ::3] *= 2.0 ** -24   # beside an integer: fractions of a few 2^-24, and 0
    Y = np.clip(rng.normal(0, 0.5, (nt, N, K)), -1.2, 1.2)
    u = np.float32(0.5) + np.float32(vbar[0, ::3].reshape(-1, 1, 2) + np.einsum("wk,kcd->cwd", Y[0], modes[0][:, ::3].reshape(K, -1, 2)))
    frac = u - np.floor(u)
    if trap > 0.0:
        assert (frac < trap).any() and (frac > trap).any()
    env = custom_env(nx=nx, ny=ny, nt=nt, K=K, N=N, L=13, vbar=vbar, modes=modes, sigma=np.full(K, 0.5), Y=Y,
                     actions=actions, r_outbound=-3.0)
    d, outs = mdp.DeviceEnv(env), []
    for cap in (1, 0):
        o = mdp.MdpBuildOpts()
        o.hist_cap = cap
        m = mdp.mdp_build(d, objs=(0,), opts=o)
        outs.append((m.info().wide_slices, [x.cpu().numpy() for x in mdp.mdp_export_csr(m, 0)]))
    assert outs[1][0] < outs[0][0]
    for x, y in zip(outs[0][1], outs[1][1]):
        assert np.array_equal(x, y)
