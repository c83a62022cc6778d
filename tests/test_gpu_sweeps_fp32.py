"""The FP32 Jacobi sweeps themselves.  A cold solve that the two chains prove runs none, so these are reached
the ways that always sweep: a warm start from V = 0 is the cold run, sweep by sweep; a tolerance that every
objective of a fused solve meets early leaves all of them open; and the full sweeps.  Bounded waits that run out
in a sweep, with its residual's reduction behind it.  The backward passes' kernels on both sides of the size
where three objectives with two chains change kernels (3 slices per resident warp of 3 CTAs an SM: 152 x 3 x 8 x 3
= 10,944 slices)."""
import numpy as np
import pytest

from paper_2109_00857_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mdp():
    from paper_2109_00857_gb300 import mdp as m
    m.load()
    return m


def bits(x):
    return x.cpu().numpy().view(np.uint8)


CASES = {
    "three_objectives": lambda: inputs.large(nx=22, ny=22, nt=9, N=300, L=15, square=5),
    "A12_straddling_slices": lambda: inputs.make_env(nx=9, ny=7, nt=8, K=3, N=250, L=9, sigma=(0.3, 0.2, 0.1), seed=5,
                                                     amplitude=0.8, n_headings=12, n_speeds=1, obstacle="squares",
                                                     square=3, with_gbar=True, objectives=(0, 2)),
    "tiny_rterm": lambda: inputs.tiny(nx=13, ny=11, nt=12, N=77, r_term=4.0),
    "rounds": lambda: inputs.energy(nx=70, ny=61, nt=5, N=30, K=2, sigma=(0.2, 0.1), objectives=(0, 1, 2)),
}


@pytest.mark.parametrize("case", sorted(CASES))
def test_active_layer_sweeps_equal_full_sweeps(mdp, case):
    import torch
    env = CASES[case]()
    m = mdp.mdp_build(mdp.DeviceEnv(env), objs=env.objectives)
    for tol, ms in ((0.0, 0), (0.0, 3), (0.0, env.nt), (1e-3, 0), (0.5, 0), (-1.0, 0)):
        for o in range(len(env.objectives)):
            V0 = torch.zeros(env.nS + 1, device="cuda")
            Va, pa, sa = mdp.mdp_solve(m, o, tol=tol, max_sweeps=ms, V=V0, warm=True)
            Vf, pf, sf = mdp.mdp_solve(m, o, method=mdp.MDP_SOLVE_JACOBI_FULL, tol=tol, max_sweeps=ms)
            assert np.array_equal(bits(Va), bits(Vf)) and np.array_equal(bits(pa), bits(pf)), (tol, ms, o)
            assert (sa.sweeps, sa.residual) == (sf.sweeps, sf.residual), (tol, ms, o)
            assert sa.backups < sf.backups if sf.sweeps > 2 else sa.backups <= sf.backups
            assert sf.backups == sf.sweeps * env.nS * env.A


@pytest.mark.parametrize("case", ["three_objectives", "A12_straddling_slices", "rounds"])
def test_fused_sweeps_of_open_objectives(mdp, case):
    env = CASES[case]()
    m = mdp.mdp_build(mdp.DeviceEnv(env), objs=env.objectives)
    n = len(env.objectives)
    res = [mdp.mdp_solve(m, o, method=mdp.MDP_SOLVE_JACOBI_FULL, max_sweeps=3)[2].residual for o in range(n)]
    for tol in (max(res), 2.0 * max(res)):   # met by sweep 3 by every objective, so none is the chains'
        V, p, s = mdp.mdp_solve_multi(m, tuple(range(n)), tol=tol)
        Vf, pf, sf = mdp.mdp_solve_multi(m, tuple(range(n)), method=mdp.MDP_SOLVE_JACOBI_FULL, tol=tol)
        for o in range(n):
            assert sf[o].sweeps <= 3 < env.nt
            assert (s[o].sweeps, s[o].residual) == (sf[o].sweeps, sf[o].residual)
            assert np.array_equal(bits(V[o]), bits(Vf[o])) and np.array_equal(bits(p[o]), bits(pf[o]))


@pytest.mark.parametrize("side, headings, speeds", [(40, 16, 1), (40, 16, 2), (200, 16, 2)])
@pytest.mark.parametrize("kind", ["full", "warm", "fused"])
def test_a_wait_that_runs_out_in_a_sweep(mdp, side, headings, speeds, kind):
    import torch
    env = inputs.energy(nx=side, ny=side, nt=3, N=24, K=2, sigma=(0.2, 0.1), amplitude=1.0, n_headings=headings,
                        n_speeds=speeds, square=side // 10, objectives=(0, 1, 2))
    m = mdp.mdp_build(mdp.DeviceEnv(env), objs=env.objectives)
    lib = mdp.load()

    def solve():
        if kind == "fused":
            return mdp.mdp_solve_multi(m, (0, 1, 2), method=mdp.MDP_SOLVE_JACOBI_FULL)[0]
        if kind == "warm":
            return [mdp.mdp_solve(m, 0, V=torch.zeros(env.nS + 1, device="cuda"), warm=True)[0]]
        return [mdp.mdp_solve(m, 0, method=mdp.MDP_SOLVE_JACOBI_FULL)[0]]

    before = [bits(v) for v in solve()]
    assert lib.mdp_test_inject(2, 2_000_000) == 0   # about 1 ms
    assert lib.mdp_test_inject(1, 1024) == 0
    try:
        with pytest.raises(mdp.MdpError) as ei:
            solve()
        assert ei.value.code == -5
    finally:
        lib.mdp_test_inject(2, 0)
    assert all(np.array_equal(bits(v), b) for v, b in zip(solve(), before))


@pytest.mark.parametrize("nx, ny", [(104, 105), (105, 105)])
def test_both_sides_of_the_kernel_change_for_six_components(mdp, nx, ny):
    env = inputs.energy(nx=nx, ny=ny, nt=3, N=24, K=2, sigma=(0.2, 0.1), amplitude=1.0, square=10, objectives=(0, 1, 2))
    m = mdp.mdp_build(mdp.DeviceEnv(env), objs=env.objectives)
    V, p, s = mdp.mdp_solve_multi(m, (0, 1, 2))
    assert s[0].backups == 2 * env.nS * env.A   # the chains
    for o in range(3):
        Vf, pf, sf = mdp.mdp_solve(m, o, method=mdp.MDP_SOLVE_JACOBI_FULL)
        assert np.array_equal(bits(V[o]), bits(Vf)) and np.array_equal(bits(p[o]), bits(pf))
        assert (s[o].sweeps, s[o].residual) == (sf.sweeps, sf.residual)
