"""pmc_score writes every row: paths with an invalid vertex count score zero in
either kind of medium and leave their neighbours alone."""
import numpy as np
import pytest

from paper_1811_04156_gb300 import scenes as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["homogeneous", "layered"])
def test_invalid_counts_score_zero(kind):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1811_04156_gb300 import api
    sc = S.plain() if kind == "homogeneous" else S.general_small()
    ctx = api.Context(0)
    medium = api.Medium(ctx, sc.medium)
    geom = api.Geometry(ctx, sc.sources, sc.sensors, sc.pairs)
    cap, batch = 12, 70
    sen = sc.sensors[0]
    xyz, n = S.random_paths(sc.sources[0].pos, sen.centre, sen.radius, batch, cap, 2, cap, 5)
    x, k = torch.from_numpy(xyz).cuda(), torch.from_numpy(n).cuda()
    ref = api.score(ctx, medium, geom, 0, x, k).cpu().numpy()
    bad = [0, 3, 31, 32, 69]
    k[bad] = torch.tensor([0, 1, cap + 1, -5, 2**31 - 1], dtype=torch.int32, device="cuda")
    for _ in range(3):  # (the output's memory held other values before)
        filler = torch.full((batch, medium.n_theta), 7.0, device="cuda")
        del filler
        out = api.score(ctx, medium, geom, 0, x, k).cpu().numpy()
        assert (out[bad] == 0.0).all()
        ok = np.delete(np.arange(batch), bad)
        assert np.allclose(out[ok], ref[ok], rtol=1e-5, atol=1e-4)  # (layered sums in any order)
