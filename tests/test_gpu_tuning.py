"""Launch shapes that the library picks: what a chain set computes and which
kernel it gets depend on the set, not on the chain window or on what the
context ran before."""
import dataclasses

import numpy as np
import pytest

from paper_1811_04156_gb300 import scenes as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def n_sm():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1811_04156_gb300 import build
    build.build()
    return torch.cuda.get_device_properties(0).multi_processor_count


def _chains(ctx, sc, **kw):
    from paper_1811_04156_gb300 import api
    return api.Chains(ctx, api.Medium(ctx, sc.medium), api.Geometry(ctx, sc.sources, sc.sensors, sc.pairs), sc.run, **kw)


def _run(ctx, sc, steps, **kw):
    ch = _chains(ctx, sc, **kw)
    ch.run_steps(steps)
    return (*ch.read_states(), ch.read_accumulators())


def _same(a, b):
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


def _long_caps(chains):
    sc = S.plain(n_chains=chains, n_steps=1500, cap=512)
    sc.run.layout = S.LAYOUT_WARP
    return sc


@pytest.mark.parametrize("per_sm", [(14, 18), (18, 14)])
def test_rounding_does_not_depend_on_earlier_sets(n_sm, per_sm):
    """Chain counts of one power of two, on both sides of the count (16 warps of
    512 vertices per SM) from which a window of 128 needs fewer waves of warps."""
    from paper_1811_04156_gb300 import api
    ctx = api.Context(0)
    for k in per_sm:
        sc = _long_caps(k * n_sm)
        own = _run(ctx, sc, 1500)
        _same(own, _run(api.Context(0), sc, 1500, warps_per_block=2, smem_window=128 if k > 16 else 0))


def test_windows_of_a_tuned_set_replay_it(n_sm):
    from paper_1811_04156_gb300 import api
    sc = _long_caps(18 * n_sm)
    whole = _run(api.Context(0), sc, 1500)
    for r in range(3):
        lo, hi = api.shard_range(sc.pairs, r, 3)
        _same(_run(api.Context(0), sc, 1500, chain_window=(lo, hi)), [x[lo:hi] for x in whole])


def test_windows_with_a_caller_set_window_replay_the_whole_set(n_sm):
    """Two pairs of one cap class, one of them with the whole cap in the shared window."""
    from paper_1811_04156_gb300 import api
    sc = _long_caps(256)
    sc.pairs = [S.Pair(0, 0, 256, 300), S.Pair(0, 0, 256, 512)]
    shape = dict(warps_per_block=2, smem_window=320)
    whole = _run(api.Context(0), sc, 1500, **shape)
    for lo in (0, 256):
        part = _run(api.Context(0), sc, 1500, chain_window=(lo, lo + 256), **shape)
        _same(part, [x[lo:lo + 256] for x in whole])


def _is_team(row):
    """A team of four warps per chain has a block per chain, one warp per chain a block per four."""
    chains = row["hi"] - row["lo"]
    return row["warps_per_block"] == 4 and row["grid"] > (chains + 3) // 4


@pytest.mark.parametrize("per_sm", [(21, 15), (15, 21)])
def test_groups_do_not_depend_on_earlier_sets(n_sm, per_sm):
    """Chain counts of one power of two on both sides of the groups' 20 chains per SM."""
    from paper_1811_04156_gb300 import api
    ctx = api.Context(0)
    for k in per_sm:
        sc = S.general_small(n_chains=k * n_sm)
        sc.pairs = [dataclasses.replace(sc.pairs[0], cap=200)]
        assert _chains(ctx, sc).launch_info()[0]["smem_cap"] == (128 if k > 20 else 224)


def test_no_team_for_many_chains_after_a_team_for_few(n_sm):
    """The teams' limit, four chains per SM, lies between powers of two as well.  Near
    it a probe may choose either, so in a few contexts."""
    from paper_1811_04156_gb300 import api
    for _ in range(8):
        ctx = api.Context(0)
        for chains in (7 * n_sm // 2, 5 * n_sm):
            sc = S.plain(n_chains=chains)
            sc.run.layout = S.LAYOUT_WARP
            row = _chains(ctx, sc).launch_info()[0]
        assert not _is_team(row), row


def test_the_window_follows_the_number_of_chains(n_sm):
    """Eight warps per SM hold whole caps of 1,024 vertices, twelve do not; the counts are
    of one power of two."""
    from paper_1811_04156_gb300 import api
    ctx = api.Context(0)
    for per_sm in (12, 8, 12):
        sc = S.plain(n_chains=per_sm * n_sm, cap=1024)
        sc.run.layout = S.LAYOUT_WARP
        window = _chains(ctx, sc).launch_info()[0]["smem_cap"]
        assert window == 1024 if per_sm == 8 else 320 <= window < 1024, (per_sm, window)
