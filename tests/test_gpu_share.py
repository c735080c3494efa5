"""Chain kernels in which several chains share a warp or several warps a chain:
the same chains, bit for bit, as the kernel with one warp per chain (which a request for warps per
block selects), at ragged chain counts, paths on both sides of the shared
window, step counts that end inside a batch, and split runs."""
import dataclasses

import numpy as np
import pytest

from paper_1811_04156_gb300 import scenes as S

pytestmark = pytest.mark.gpu


def _run(scene, steps, **shape):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1811_04156_gb300 import api
    ctx = api.Context(0)
    medium = api.Medium(ctx, scene.medium)
    geom = api.Geometry(ctx, scene.sources, scene.sensors, scene.pairs)
    ch = api.Chains(ctx, medium, geom, scene.run, **shape)
    for k in steps:
        ch.run_steps(k)
    return ch.launch_info()[0], ch.read_states(), ch.read_accumulators(), ch.status()


def _same(a, b, ran=100):
    for x, y in zip(a[1], b[1]):
        assert np.array_equal(x, y)
    assert np.array_equal(a[2], b[2])
    assert a[3] == b[3]  # (jittered straight starts that touch the sensor do not run)
    assert (a[2][:, 0] > 0).sum() >= ran


@pytest.mark.parametrize("grad", [False, True])
@pytest.mark.parametrize("init_k,cap", [(0, 40), (125, 200)])
def test_lane_groups_match_one_warp_per_chain(grad, init_k, cap):
    """General physics (layers, vMF emission, detection probability, phase
    mixture), 8 lanes per chain; straight starts of 127 vertices grow and shrink
    across the groups' window of 128."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    sc = S.general_small(n_chains=24 * n_sm + 3)
    sc.pairs = [dataclasses.replace(sc.pairs[0], cap=cap)]
    sc.run = dataclasses.replace(sc.run, gradients=grad, burn_in=50, p_birth=0.25, p_death=0.15, init_jitter=0.05,
                                 init=S.INIT_STRAIGHT, init_k=init_k)
    steps = (733, 35)
    a = _run(sc, steps)
    assert a[0]["general"] == 1 and a[0]["smem_cap"] == (128 if cap > 128 else 64)
    _same(a, _run(sc, steps, warps_per_block=2))
    if cap > 128:
        assert a[1][1].max() > 128
        _same(a, _run(sc, steps, warps_per_block=4, smem_window=64))


@pytest.mark.parametrize("name", ["plain", "general", "mala_gradients"])
def test_teams_match_one_warp_per_chain(name):
    """Few chains: the autotuner may give each chain a team of four warps."""
    if name == "plain":
        sc = S.plain(n_chains=37, cap=41)
    elif name == "general":
        sc = S.general_small(n_chains=5)
    else:
        sc = S.gradients(n_chains=9, cap=30)
    sc.run = dataclasses.replace(sc.run, burn_in=50, layout=S.LAYOUT_WARP)
    steps = (1500, 33, 1)
    _same(_run(sc, steps), _run(sc, steps, warps_per_block=2), 1)


@pytest.mark.parametrize("chains,window", [(90, 0), (13, 0), (17, 128)])
def test_tuned_long_caps_match_a_caller_set_shape(chains, window):
    """Long vertex caps of lean runs: tuned chains are those of the whole cap in
    shared memory while as many waves of warps hold them as with a window of
    128, else those of the window (per SM: 16 warps of 512 vertices, 24 of 128)."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    sc = S.plain(n_chains=chains if chains > 64 else chains * n_sm, n_steps=1500, cap=512)
    sc.run.layout = S.LAYOUT_WARP
    a = _run(sc, (1500,))
    _same(a, _run(sc, (1500,), warps_per_block=2, smem_window=window), ran=80)
