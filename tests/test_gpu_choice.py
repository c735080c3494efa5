"""Kernels that a launch chooses by the lengths of the paths: the same chains, bit for
bit, whichever ran, with paths inside the shared window, beyond it, and on both
sides of it."""
import dataclasses

import numpy as np
import pytest

from paper_1811_04156_gb300 import scenes as S

pytestmark = pytest.mark.gpu


def _scene(name, chains, cap, init_k):
    sc = S.general_small(n_chains=chains) if name == "general" else S.plain(n_chains=chains)
    within = S.WITHIN_MALA if name == "mala" else S.WITHIN_PERTURB
    sc.pairs = [dataclasses.replace(sc.pairs[0], cap=cap)]
    sc.run = dataclasses.replace(sc.run, burn_in=100, layout=S.LAYOUT_WARP, within=within, mala_step=0.02,
                                 gradients=name in ("gradients", "general"), init=S.INIT_STRAIGHT, init_k=init_k,
                                 init_jitter=0.01, p_birth=0.25, p_death=0.15)
    return sc


def _run(sc, steps, **shape):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1811_04156_gb300 import api
    ctx = api.Context(0)
    ch = api.Chains(ctx, api.Medium(ctx, sc.medium), api.Geometry(ctx, sc.sources, sc.sensors, sc.pairs), sc.run,
                    **shape)
    out = []
    for k in steps:
        ch.run_steps(k)
        out.append([*ch.read_states(), ch.read_accumulators(), ch.status()])
    return out


def _same(a, b):
    for x, y in zip(a, b):
        for u, v in zip(x, y):
            assert np.array_equal(u, v)


@pytest.mark.parametrize("name", ["lean", "gradients", "general", "mala"])
@pytest.mark.parametrize("init_k", [0, 28, 60])
def test_windows_of_any_size_step_alike(name, init_k):
    """Windows that hold no path, some paths and every path of a cap of 128: one copy of
    the step code, either copy, and the copy without tests; paths grow and shrink
    between the launches."""
    sc = _scene(name, 70, 128, init_k)
    steps = (1, 31, 300, 700, 33)
    ref = _run(sc, steps, warps_per_block=2, smem_window=96)
    longest = max(r[1].max() for r in ref)
    assert longest > (3 if init_k == 0 else init_k) and (ref[-1][3][:, 0] > 0).mean() > 0.9
    for window in (32, 64):
        _same(_run(sc, steps, warps_per_block=4, smem_window=window), ref)


def test_long_paths_in_whole_caps():
    """Few lean chains with caps above 320 in shared memory: short paths and paths of
    more than 320 vertices, against the warp layout set by the caller."""
    for init_k in (5, 400):
        sc = _scene("lean", 700, 512, init_k)
        sc.run.init_jitter = 2e-4  # (400 vertices stand 2 mm apart: none may touch the sensor)
        a = _run(sc, (1, 200, 257))
        _same(a, _run(sc, (1, 200, 257), warps_per_block=1))
        assert (a[-1][3][:, 0] > 0).mean() > 0.9 and a[-1][1].mean() > init_k / 2


def test_long_runs_are_cut_without_a_trace():
    """A geometry whose paths grow past 112 vertices: runs of more than 4,096 steps are cut
    for a new choice; the chains are those of short runs and of other windows."""
    sc = _scene("general", 40, 256, 5)
    sc.medium = S.Medium(lambda_s=0.2, lambda_a=100.0, g=0.2)
    sc.run = dataclasses.replace(sc.run, gradients=False, p_birth=0.2, p_death=0.2)
    (whole,) = _run(sc, (9000,), warps_per_block=2, smem_window=32)
    parts = _run(sc, (1000,) * 9, warps_per_block=4, smem_window=64)[-1]
    for u, v in zip(whole[:3], parts[:3]):
        assert np.array_equal(u, v)
    assert np.allclose(whole[3], parts[3], rtol=1e-5) and whole[1].max() > 64
    (other,) = _run(sc, (9000,), warps_per_block=4, smem_window=96)
    _same([whole], [other])


@pytest.mark.parametrize("cap,init_k", [(200, 118), (700, 20), (700, 118), (700, 200), (700, 400)])
def test_groups_give_way_to_warps(cap, init_k):
    """Enough general chains for groups of 8 lanes: paths inside the groups' window of 128,
    paths that grow across it within a launch, and paths that start beyond it or
    beyond the warp layout's window, against the warp layout set by the caller."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    sc = _scene("general", 21 * n_sm + 3, cap, init_k)
    sc.run.init_jitter = 2e-4
    if init_k == 118:  # (a dense medium: 101 scatterings on the straight line, paths grow)
        sc.medium = S.Medium(lambda_s=0.0125, lambda_a=100.0, g=0.2)
        sc.run.sigma = 0.005
    steps = (733, 35, 300)
    a = _run(sc, steps)
    _same(a, _run(sc, steps, warps_per_block=2))
    assert (a[-1][3][:, 0] > 0).mean() > 0.9
    if init_k == 118:
        assert a[0][1].max() > 128
