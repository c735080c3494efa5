"""Chain kernels with a team of four warps per chain, known to have run: the same
chains, bit for bit, as with one warp per chain, in each instance (lean and general
physics, with and without gradients), for step counts that end inside a round or
a batch of 32, at the smallest cap and when a run is aborted."""
import dataclasses

import numpy as np
import pytest

from paper_1811_04156_gb300 import scenes as S

pytestmark = pytest.mark.gpu

SCENES = {
    "lean": lambda: S.plain(n_chains=37, cap=41),
    "lean_gradients": lambda: S.plain(n_chains=12, cap=64),
    "lean_cap_2": lambda: S.plain(n_chains=3, cap=2),
    "general": lambda: S.general_small(n_chains=5),
    "mala_gradients": lambda: S.gradients(n_chains=9, cap=30),
}


def _scene(name):
    sc = SCENES[name]()
    sc.run = dataclasses.replace(sc.run, burn_in=20, layout=S.LAYOUT_WARP, gradients="gradients" in name)
    return sc


def _chains(sc, **shape):
    from paper_1811_04156_gb300 import api
    ctx = api.Context(0)
    return api.Chains(ctx, api.Medium(ctx, sc.medium), api.Geometry(ctx, sc.sources, sc.sensors, sc.pairs), sc.run,
                      **shape)


def _teams(sc):
    """Tuned chains that run in teams (a block of four warps per chain), in which a few
    chains are a fifth faster; a disturbed probe may choose otherwise, so in a few contexts."""
    for _ in range(8):
        ch = _chains(sc)
        row = ch.launch_info()[0]
        chains = row["hi"] - row["lo"]
        if row["warps_per_block"] == 4 and row["grid"] > (chains + 3) // 4:
            return ch
    pytest.fail(f"no team was chosen: {row}")


def _state(ch):
    return [*ch.read_states(), ch.read_accumulators(), ch.status()]


def _same(a, b):
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("name", list(SCENES))
def test_teams_step_as_one_warp_per_chain_does(name):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    sc = _scene(name)
    team, one = _teams(sc), _chains(sc, warps_per_block=2)
    for steps in (1, 2, 3, 31, 33, 700, 255, 1):
        team.run_steps(steps)
        one.run_steps(steps)
        _same(_state(team), _state(one))
    assert (one.read_accumulators()[:, 0] > 0).any()
    for ch in (team, one):
        ch.request_abort(True)
        ch.run_steps(500)
    _same(_state(team), _state(one))
    assert team.status() != 0
