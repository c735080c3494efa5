"""Scenes of very small lengths: a scene with every length scaled by 2^-40 (metres
to 1e-12 m) has the same path distribution, so the mean vertex count over the
recorded states agrees with the unscaled scene's.  Tolerance: five standard
errors of the difference of two independent samples, from the spread of the
chains' means."""
import dataclasses

import numpy as np
import pytest

from paper_1811_04156_gb300 import scenes as S

pytestmark = pytest.mark.gpu


def _scaled(sc, f):
    m = sc.medium
    layers = {k: None if getattr(m, k) is None else getattr(m, k) * f for k in ("lambda_s_layers", "lambda_a_layers")}
    sc.medium = dataclasses.replace(m, lambda_s=m.lambda_s * f, lambda_a=m.lambda_a * f, z0=m.z0 * f, dz=m.dz * f, **layers)
    sc.sources = [dataclasses.replace(s, pos=tuple(x * f for x in s.pos)) for s in sc.sources]
    sc.sensors = [dataclasses.replace(s, centre=tuple(x * f for x in s.centre), radius=s.radius * f) for s in sc.sensors]
    if sc.run.within != S.WITHIN_TREE:  # (tree moves: a step in dimensionless coordinates)
        sc.run.sigma *= f
    sc.run.mala_step *= f
    return sc


def _scene(name, n_sm):
    run = dict(burn_in=200)
    if name.endswith("lane"):
        run["layout"] = S.LAYOUT_LANE
    elif name != "groups":
        run["layout"] = S.LAYOUT_WARP
    if "tree" in name:
        run.update(within=S.WITHIN_TREE, sigma=0.3)
    if "hmc" in name:
        run.update(within=S.WITHIN_HMC, mala_step=0.01, hmc_steps=4)
    if name == "groups":
        sc = S.general_small(n_chains=24 * n_sm)
    elif name == "few":
        sc = S.plain(n_chains=256)
    elif name == "wavelength":
        sc = S.wavelength(n_chains=2048)
    else:
        make = S.general_small if "general" in name else (S.gradients if "mala" in name else S.plain)
        sc = make(n_chains=1024)
    sc.run = dataclasses.replace(sc.run, **run)
    return sc


@pytest.mark.parametrize("name", ["plain_lane", "plain_warp", "mala_lane", "tree_lane", "tree_warp", "hmc_warp",
                                  "general_warp", "general_tree_warp", "groups", "few", "wavelength"])
def test_a_scene_scaled_to_tiny_lengths_has_the_same_path_lengths(name):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1811_04156_gb300 import api
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    means = []
    for f in (1.0, 2.0 ** -40):
        sc = _scaled(_scene(name, n_sm), f)
        ctx = api.Context(0)
        # (steps of a caller's launch shape; groups and teams need the tuner's choice)
        shape = {} if name in ("groups", "few") else {"warps_per_block": 2}
        ch = api.Chains(ctx, api.Medium(ctx, sc.medium), api.Geometry(ctx, sc.sources, sc.sensors, sc.pairs), sc.run,
                        **shape)
        ch.run_steps(2000)
        acc = ch.read_accumulators()
        assert ch.status() == 0
        means.append(acc[:, 2] / acc[:, 0])
    a, b = means
    tolerance = 5.0 * np.sqrt(a.var() / len(a) + b.var() / len(b))
    assert abs(a.mean() - b.mean()) <= tolerance, (a.mean(), b.mean(), tolerance)
