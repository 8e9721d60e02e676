"""Launches over arrays where the hits kernel's bound may cost more than it
saves ask some of the steps first and take one of two kernels: the crossings,
values, counters and profile of the launch that never asks (no persistent
grid), for arrays and steps on both sides of the choice, around the number of
steps from which a launch asks and past one wave of warps.  The same arithmetic
per bunch, so bit-equal; a profile's sums to the order of their additions."""
import ctypes

import numpy as np
import pytest

import paper_2006_14927_gb300 as P
import workloads
from parity import FP32
from test_reach_gpu import H_OBS

pytestmark = pytest.mark.gpu


def _grid(n, half, r, rng):
    m = int(np.ceil(np.sqrt(n)))
    g = (np.arange(m) + 0.5) / m * 2 * half - half
    xy = np.stack(np.meshgrid(g, g), -1).reshape(-1, 2)[rng.permutation(m * m)[:n]]
    return np.column_stack([xy + rng.uniform(-2.0, 2.0, xy.shape), np.zeros(n), np.full(n, r)])


@pytest.mark.parametrize("array,zenith,n,option", [
    ("dense", 0.0, 10_000, "none"), ("dense", 0.0, 200_003, "profile"),
    ("dense", 0.3, 160_001, "both"), ("thousand", 1.05, 10_003, "none"),
    ("thousand", 1.05, 200_003, "dispersion"), ("thousand", 0.0, 200_003, "transmission"),
    ("thousand", 0.3, 9_999, "none"), ("km100", 1.2, 160_001, "fallback"),
    ("km100", 0.3, 200_003, "none"), ("wide4096", 0.5, 60_001, "transmission"),
    ("wide4096", 1.0, 160_001, "none")])
def test_both_choices_give_the_same(array, zenith, n, option):
    import torch
    rng = np.random.Generator(np.random.PCG64(n))
    tel = dict(dense=lambda: _grid(64, 150.0, 8.0, rng),
               thousand=lambda: _grid(1000, 1000.0, 6.0, rng),
               wide4096=lambda: _grid(4096, 4000.0, 6.0, rng),
               km100=lambda: workloads.scattered_telescopes(rng))[array]()
    seg, t_ref = workloads.shower_segments(rng, n, 1.0e6, zenith, 0.7, 0.0, 0.0, H_OBS)
    ctx = P.Context(workloads.us_standard_atmosphere(), H_OBS, tel)
    ctx.build_refraction_tables(400, 64, 70.0, 60000.0)
    if option in ("transmission", "both"):
        ctx.set_transmission(workloads.synthetic_transmission())
    if option in ("dispersion", "both"):
        ctx.set_dispersion(workloads.synthetic_dispersion())
    if option == "fallback":
        ctx.set_fallback(84.0)
    dev = P.device_tracks(seg, FP32, t_ref=t_ref)
    cap = 600_000_000 // (40 * len(tel))
    got = []
    for launch in ((128, 0), (128, 8), (256, 2)):
        ctx.set_launch(*launch)
        out = ctx.alloc_hits(cap, FP32)
        prof = torch.zeros((1, 150), dtype=torch.float64, device="cuda")
        ctx.generate_propagate(dev, 11, FP32, out, profile=prof if option == "profile" else None)
        code, st = ctx.sync_status(out)
        assert code == 0, st
        got.append((np.asarray(st), out.records(), prof.cpu().numpy()))
        del out
    assert got[0][0][9] > 100
    for st, rec, prof in got[1:]:
        assert np.array_equal(st, got[0][0])
        for k in rec:
            assert np.array_equal(rec[k], got[0][1][k]), k
        assert (np.abs(prof - got[0][2]) <= n * 2.0 ** -52 * got[0][2]).all()
    if option in ("none", "transmission"):
        ctx.set_launch(128, 8)
        out = ctx.alloc_hits(cap, FP32)
        t, o = ctx.tracks_struct(dev), out.struct()
        assert P.lib().cher_generate_propagate_noalloc(ctx._h, ctypes.byref(t), 11, FP32,
                                                       ctypes.byref(o), None) == 0
        _, st = ctx.sync_status(out)
        assert np.array_equal(np.asarray(st), got[0][0])
        graph = ctx.graph(dev, 11, FP32, out)
        for _ in range(2):
            graph.launch()
            _, st = ctx.sync_status(out)
            assert np.array_equal(np.asarray(st), got[0][0])
        for k, v in out.records().items():
            assert np.array_equal(v, got[0][1][k]), k
