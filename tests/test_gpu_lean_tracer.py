"""The tracer's lean instance (quotients by shared divisors) against the general one,
which pmc_trace_noalloc runs: the same photons, so the same sums up to the order of the
FP64 additions, over scattering lengths and mean cosines whose quotients are not
exact; and the seeding, whose two passes run one instance each, finds every
photon again."""
import numpy as np
import pytest

from paper_1811_04156_gb300 import scenes as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale,g", [(0.37, 0.9), (3.3, -0.57), (0.0123, 0.0031), (777.7, 0.99), (1.0 / 3.0, -1.7e-6),
                                     (1.1e6, 0.3)])
def test_lean_photons_are_the_general_ones(scale, g):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1811_04156_gb300 import api
    ctx = api.Context(0)
    medium = api.Medium(ctx, S.Medium(lambda_s=scale, lambda_a=7.1 * scale, g=g))
    sensor = S.Sensor((0.2 * scale, -0.3 * scale, 1.1 * scale), 0.4 * scale)
    geom = api.Geometry(ctx, [S.Source()], [sensor], [S.Pair(0, 0, 500, 34)])
    lean = api.trace(ctx, medium, geom, 0, 77, 1_000_003, max_scatter=32)
    (general,) = api.trace_noalloc(ctx, medium, geom, [0], 77, 1_000_003, max_scatter=32)
    assert lean["detected"] == general["detected"] > 1000
    for k in ("sum_w", "sum_w2", "sum_wl"):
        assert np.isclose(lean[k], general[k], rtol=1e-9, atol=0), k
    run = S.Run(sigma=0.05 * scale)
    chains = api.Chains(ctx, medium, geom, run, warps_per_block=1)
    api.seed_from_tracer(chains, photons_per_round=1 << 18)
    assert chains.status() == 0
    n = chains.read_states()[1]
    assert n.min() >= 2 and n.max() > 3
