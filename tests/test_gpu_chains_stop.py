"""Runs whose tolerance is met before the last sweeps: the two chains of a cold Jacobi solve are given up at the
first layer that proves nothing for any objective, and the sweeps give the result; a run that ends in sweep nt
or nt + 1 comes from the chains.  Values, policy, sweeps and residual are those of the full sweeps bit for bit."""
import numpy as np
import pytest

from paper_2109_00857_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mdp():
    from paper_2109_00857_gb300 import mdp as m
    m.load()
    return m


def model_of(mdp, nx, ny, nt, speeds, headings=16):
    env = inputs.make_env(nx=nx, ny=ny, nt=nt, K=2, N=60, L=11, sigma=(0.3, 0.2), seed=3, amplitude=1.0,
                          n_headings=headings, n_speeds=speeds, obstacle="none", with_gbar=True, objectives=(0, 1, 2))
    return env, mdp.mdp_build(mdp.DeviceEnv(env), objs=env.objectives)


def bits(x):
    return x.cpu().numpy().view(np.uint8)


@pytest.mark.parametrize("nx, ny, nt, speeds", [(9, 8, 40, 1), (9, 8, 40, 2), (21, 27, 103, 1), (130, 130, 30, 2),
                                                (12, 11, 3, 1), (7, 5, 1, 2), (6, 6, 2, 1)])
def test_every_ending_equals_the_full_sweeps(mdp, nx, ny, nt, speeds):
    env, m = model_of(mdp, nx, ny, nt, speeds)
    # tolerances at, just below and above every residual of the run, so that it ends in every sweep it can
    res = []
    for k in range(1, nt + 2):
        s = mdp.mdp_solve(m, 0, method=mdp.MDP_SOLVE_JACOBI_FULL, tol=0.0, max_sweeps=k)[2]
        if s.sweeps < k:
            break
        res.append(s.residual)
    picked = sorted({0, 1, len(res) // 2, len(res) - 3, len(res) - 2, len(res) - 1} & set(range(len(res))))
    tols = {0.0, 1e-6, 1.0, 1e4}
    for i in picked:
        tols |= {res[i], np.nextafter(res[i], 0.0), np.nextafter(res[i], np.inf)}
    for tol in sorted(tols):
        for slots in ((0,), (2, 0), (0, 1, 2)):
            V, p, s = mdp.mdp_solve_multi(m, slots, tol=tol)
            Vf, pf, sf = mdp.mdp_solve_multi(m, slots, method=mdp.MDP_SOLVE_JACOBI_FULL, tol=tol)
            for i in range(len(slots)):
                assert (s[i].sweeps, s[i].residual) == (sf[i].sweeps, sf[i].residual), (tol, slots, i)
                assert np.array_equal(bits(V[i]), bits(Vf[i])) and np.array_equal(bits(p[i]), bits(pf[i]))
                if sf[i].sweeps >= nt:   # from the chains
                    assert s[i].backups == 2 * env.nS * env.A


def test_a_run_that_ends_early_is_given_up_early(mdp):
    """The layers that run after the first that proves nothing are those already launched."""
    env, m = model_of(mdp, 12, 12, 400, 1)
    V = mdp.mdp_solve(m, 0, tol=0.0)[0]
    best = {}
    for what, kw in (("cold", {}), ("full", dict(method=mdp.MDP_SOLVE_JACOBI_FULL))):
        for _ in range(6):
            s = mdp.mdp_solve(m, 0, tol=1.0, V=V, **kw)[2]
            assert s.sweeps < 60
            best[what] = min(best.get(what, 1e9), s.solve_ms)
    layers = min(mdp.mdp_solve(m, 0, method=mdp.MDP_SOLVE_LAYERED)[2].solve_ms for _ in range(6))
    # active-layer sweeps cost no more than full ones; all the chains' layers would add a layered pass
    assert best["cold"] < best["full"] + 0.5 * layers
