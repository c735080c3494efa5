"""log p of batches at the edges of the density kernel's tiles (32 or 4 paths,
1,024 vertices held at once), against the FP64 oracle: |delta log p| <= 1e-5 +
2e-6 n; invalid vertex counts give NaN and leave their neighbours alone."""
import numpy as np
import pytest

from paper_1811_04156_gb300 import scenes as S

pytestmark = pytest.mark.gpu

LEAN = (S.Medium(lambda_s=0.5, lambda_a=5.0, g=0.9), S.Source(), S.Sensor((0.0, 0.0, 1.0), 0.1), 0.3)
MIXED = (S.Medium(lambda_s=0.8, lambda_a=6.0, g=0.95, f_sl=0.45),
         S.Source((0.3, -0.2, 0.1), S.EMIT_VMF, 38.0, (0.0, 0.0, 1.0)),
         S.Sensor((0.5, 0.4, 3.0), 0.15, S.RHO_PAPER, (0.0, -1.0, 0.0)), 0.4)


# tiles of 32 paths with a ragged last tile (more than 32 per SM); the same
# with every path at the cap (several chunks per tile); tiles of 4 in a small
# batch, with long paths (several chunks), and a single shortest path
@pytest.mark.parametrize("scene,batch,cap,n_lo", [(LEAN, 4867, 40, 2), (MIXED, 4867, 64, 2), (LEAN, 4864, 50, 50),
                                                  (MIXED, 7, 40, 2), (LEAN, 5, 700, 650), (LEAN, 1, 2, 2)])
def test_logp_tile_edges(oracle_lib, scene, batch, cap, n_lo):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1811_04156_gb300 import api
    O = oracle_lib
    med, src, sen, lateral = scene
    ctx = api.Context(0)
    geom = api.Geometry(ctx, [src], [sen], [S.Pair(0, 0, 1, max(2, min(cap, 1024)))])
    xyz, n = S.random_paths(src.pos, sen.centre, sen.radius, batch, cap, n_lo, cap, 41, lateral=lateral)
    given = n.copy()
    bad = [b for b in (1, 31, 32, 4863) if b < batch - 1 and n_lo == 2]
    for k, b in enumerate(bad):
        given[b] = (0, 1, cap + 1, -3)[k]
    lp = api.logp(ctx, api.Medium(ctx, med), geom, 0, torch.from_numpy(xyz).cuda(),
                  torch.from_numpy(given).cuda()).cpu().numpy()
    assert np.isnan(lp[bad]).all()
    m, s, d = O.medium(med), O.source(src), O.sensor(sen)
    picks = sorted({b for b in [0, 2, 3, 4, 30, 33, 63, 64, batch // 2, batch - 3, batch - 2, batch - 1]
                    + list(range(0, batch, 97)) if 0 <= b < batch and b not in bad})
    for b in picks:
        k = int(n[b])
        ref = O.logp(m, s, d, xyz[:, b, :k].T.astype(np.float64))
        if np.isfinite(ref):
            assert abs(lp[b] - ref) <= 1e-5 + 2e-6 * k, (b, k, lp[b], ref)
        else:
            assert lp[b] == -np.inf, (b, k, lp[b])
