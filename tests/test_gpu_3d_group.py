"""The 3-D warp kernel over its forms: mode counts (registers, or the general
loop from nine modes on and where the coefficients' address does not allow
vector loads), numbers of realizations around a warp's trips, groups of four
slices that end inside a group, rows of more than the staged entries, one, two
and four states per slice, thresholds from none to eight per axis.  Every
model equals the one counted per action, bit for bit."""
import dataclasses
import math

import numpy as np
import pytest

from paper_2109_00857_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mdp():
    from paper_2109_00857_gb300 import mdp as m
    m.load()
    return m


def same_models(mdp, d, objs, L=None):
    kw = dict(objs=objs) if L is None else dict(objs=objs, subgrid_L=L)
    fast, ref = mdp.mdp_build3d(d, **kw), mdp.mdp_build3d(d, per_action=True, **kw)
    assert fast.info().nnz == ref.info().nnz
    assert fast.info().max_row_nnz == ref.info().max_row_nnz and fast.info().samples == ref.info().samples
    for o in range(len(objs)):
        a = [x.cpu().numpy() for x in mdp.mdp_export_csr(fast, o)]
        b = [x.cpu().numpy() for x in mdp.mdp_export_csr(ref, o)]
        assert all(np.array_equal(x, y) for x, y in zip(a[:3], b[:3])), o
        assert np.array_equal(a[3].view(np.uint32), b[3].view(np.uint32)), o
    return fast.info()


def env3(K, N, nx=9, ny=7, nz=5, nt=3, n_headings=8, elevations=(-math.pi / 4, 0.0, math.pi / 4), sigma=0.2,
         amplitude=0.6, L=9, **kw):
    k8 = min(K, 8)
    env = inputs.make_env3d(nx=nx, ny=ny, nz=nz, nt=nt, K=k8, N=N, L=L, sigma=[sigma * 0.8 ** k for k in range(k8)],
                            seed=11 + K, amplitude=amplitude, n_headings=n_headings, elevations=elevations,
                            with_gbar=True, objectives=(0, 1, 2), **kw)
    if K > 8:   # the first modes again, weaker
        env = dataclasses.replace(env, K=K, modes=np.concatenate([env.modes, 0.3 * env.modes], axis=1)[:, :K],
                                  sigma=np.concatenate([env.sigma, env.sigma])[:K])
    return env


@pytest.mark.parametrize("K, N", [(1, 1), (1, 31), (2, 32), (2, 33), (3, 63), (4, 64), (4, 65), (4, 300), (5, 97),
                                  (6, 128), (7, 127), (8, 200), (9, 90), (16, 40)])
def test_mode_counts_and_realizations(mdp, K, N):
    same_models(mdp, mdp.DeviceEnv3D(env3(K, N), mdp.MDP_FP32), (0, 1, 2))


@pytest.mark.parametrize("K", [2, 4, 6])
def test_coefficients_at_an_odd_address(mdp, K):
    import torch
    env = env3(K, 150)
    sampled = mdp.mdp_sample_coeffs(env.nt, env.N, K, list(env.sigma), seed=3, mdp_id=0, precision=mdp.MDP_FP32)
    d = mdp.DeviceEnv3D(env, mdp.MDP_FP32)
    buf = torch.empty(sampled.numel() + 1, device="cuda")
    buf[1:] = sampled.reshape(-1)
    d.coeffs = buf[1:].view(sampled.shape)
    assert d.coeffs.data_ptr() % 8 == 4
    same_models(mdp, d, (0, 2))


@pytest.mark.parametrize("kw", [
    dict(n_headings=5, elevations=(0.0, 0.7), speeds=(0.9,)),             # two states per slice
    dict(n_headings=3, elevations=(-0.5, 0.5)),                           # four
    dict(n_headings=4, elevations=(-math.pi / 2, 0.0, math.pi / 2)),      # integer displacements: no step thresholds
    dict(n_headings=8, elevations=(-0.6, 0.0, 0.6), speeds=(1.0,), nx=1, ny=1, nz=1, nt=2),   # fewer slices than a group
    dict(n_headings=1, elevations=(0.3,), speeds=(1.3,), nx=6, ny=5, nz=3),
], ids=["spw2", "spw4", "integer", "one_cell", "one_action"])
def test_states_per_slice_and_thresholds(mdp, kw):
    same_models(mdp, mdp.DeviceEnv3D(env3(3, 140, **kw), mdp.MDP_FP32), (0, 1, 2))


def test_rows_beyond_the_staged_entries(mdp):
    env = env3(2, 600, n_headings=2, elevations=(-0.4, 0.0, 0.4), sigma=0.42, amplitude=0.5, L=11, nx=12, ny=11, nz=6)
    env.actions = env.actions[:5] * 0.0
    info = same_models(mdp, mdp.DeviceEnv3D(env, mdp.MDP_FP32), (0, 1, 2))
    assert info.max_row_nnz > 17 and info.wide_slices < env.nS


def test_a_landing_outside_the_subgrid_is_refused(mdp):
    d = mdp.DeviceEnv3D(env3(4, 200, sigma=0.9, amplitude=2.5), mdp.MDP_FP32)
    for L in (1, 3):
        with pytest.raises(mdp.MdpError) as ei:
            mdp.mdp_build3d(d, subgrid_L=L, objs=(0,))
        assert ei.value.code == -3
