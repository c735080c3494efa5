"""log p of batches large enough for the density kernel's tiles of 32 paths, with a
ragged last tile and invalid vertex counts at the tiles' edges: the same
paths in small batches (tiles of 4) have the same log p, bit for bit where a
tile's vertices are held at once (1,024: caps up to 32), else within twice the
tolerance to the FP64 oracle, |delta log p| <= 1e-5 + 2e-6 n, which a sample of
the paths meets; invalid counts give NaN and leave their neighbours alone."""
import numpy as np
import pytest

from paper_1811_04156_gb300 import scenes as S
from test_gpu_tiles import LEAN, MIXED

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cap", [32, 64, 100])
@pytest.mark.parametrize("scene", [LEAN, MIXED], ids=["lean", "mixed"])
def test_large_batches_agree_with_small_ones(oracle_lib, scene, cap):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1811_04156_gb300 import api
    O = oracle_lib
    med, src, sen, lateral = scene
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    batch = (8 if cap > 64 else 3) * 32 * n_sm + 3
    ctx = api.Context(0)
    medium, geom = api.Medium(ctx, med), api.Geometry(ctx, [src], [sen], [S.Pair(0, 0, 1, cap)])
    xyz, n = S.random_paths(src.pos, sen.centre, sen.radius, batch, cap, 2, cap, 43, lateral=lateral)
    given = n.copy()
    bad = [1, 31, 32, batch - 4]
    given[bad] = (0, 1, cap + 1, -3)
    x, k = torch.from_numpy(xyz).cuda(), torch.from_numpy(given).cuda()
    large = api.logp(ctx, medium, geom, 0, x, k).cpu().numpy()
    small = np.concatenate([api.logp(ctx, medium, geom, 0, x[:, i:i + 999].contiguous(),
                                     k[i:i + 999].contiguous()).cpu().numpy() for i in range(0, batch, 999)])
    assert np.array_equal(np.flatnonzero(np.isnan(large)), bad) and np.isnan(small[bad]).all()
    ok = np.delete(np.arange(batch), bad)
    if cap <= 32:
        assert np.array_equal(large[ok], small[ok])
    finite = ok[np.isfinite(large[ok])]
    assert len(finite) > 100 and np.array_equal(large[ok] == -np.inf, small[ok] == -np.inf)
    assert (np.abs(large[finite] - small[finite]) <= 2e-5 + 4e-6 * n[finite]).all()
    m, s, d = O.medium(med), O.source(src), O.sensor(sen)
    for b in sorted({0, 2, 30, 33, 63, 64, batch - 5, batch - 3, batch - 2, batch - 1, *range(0, batch, 997)} - set(bad)):
        c = int(n[b])
        ref = O.logp(m, s, d, xyz[:, b, :c].T.astype(np.float64))
        if np.isfinite(ref):
            assert abs(large[b] - ref) <= 1e-5 + 2e-6 * c, (b, c, large[b], ref)
        else:
            assert large[b] == -np.inf, (b, c, large[b])
