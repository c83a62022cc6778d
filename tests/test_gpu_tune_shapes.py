"""The autotuner times every launch shape once: six capacities of the count tables, the CTA sizes of the
full-window kernel where slices are deferred to it, three sizes of the sweep's slots."""
import pytest

from paper_2109_00857_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K, sigma0, deferring", [(3, 0.3, False), (2, 0.9, True)])
def test_candidates_are_distinct(tmp_path, K, sigma0, deferring):
    from paper_2109_00857_gb300 import mdp
    mdp.load()
    env = inputs.large(nx=24, ny=23, nt=5, K=K, N=300, L=31, square=4, sigma=tuple(sigma0 * 2.0 ** (-k / 2.0) for k in range(K)),
                       name="a class of its own")
    d = mdp.DeviceEnv(env)
    assert (mdp.mdp_build(d, objs=env.objectives).info().wide_slices > 0) == deferring
    t = mdp.mdp_autotune(d, objs=env.objectives, json_path=str(tmp_path / "t.json"))
    assert t.candidates == (12 if deferring else 9) and t.build_warps == 4
