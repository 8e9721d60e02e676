"""The hits kernel's bound of the azimuths that can reach a sphere, for arrays
and cores far from the origin of the coordinates (map coordinates reach 1e7 m):
the crossings, counters and values of the trace kernel, which propagates every
bunch with the same arithmetic, so nothing is left out and no tolerance is
needed; and in FP64, where the ground points keep nanometres there, the
oracle's crossings."""
import numpy as np
import pytest

import oracle
import paper_2006_14927_gb300 as P
import workloads
from parity import FP32, FP64, context, gpu_hits, host_tracks, oracle_model
from test_reach_gpu import H_OBS, KINDS, _arrays, _steps

pytestmark = pytest.mark.gpu


def all_bunches(ctx, dev, n, seed, prec):
    """The trace of every bunch, and where each step's bunches start."""
    import torch
    nb, _ = ctx.segment_yield(dev, prec)
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.cumsum(nb.to(torch.int64), 0)
    return ctx.trace_bunches(dev, seed, prec, off), off


def crossings_match(ctx, dev, n, seed, prec):
    """Records and counters of the hits kernel against the trace's; returns
    the number of crossings."""
    tr, off = all_bunches(ctx, dev, n, seed, prec)
    tr, off = {k: v.cpu().numpy() for k, v in tr.items()}, off.cpu().numpy()
    nhit = tr["nhit"].astype(np.int64)
    assert nhit.max(initial=0) < 32
    out = ctx.alloc_hits(max(int(nhit.sum()), 1), prec)
    ctx.generate_propagate(dev, seed, prec, out)
    code, st = ctx.sync_status(out)
    assert code == 0 and st[3] == off[-1] and st[10] == 0
    for s, idx in ((1, 4), (2, 5), (3, 6), (4, 7), (5, 11), (0, 8)):
        assert st[idx] == (tr["status"] == s).sum(), P.STAT_NAMES[idx]
    assert st[9] == nhit.sum()
    rec = out.records()
    at = off[(rec["key"] >> np.uint64(32)).astype(np.int64)] + \
        (rec["key"] & np.uint64(0xffffffff)).astype(np.int64)
    assert np.array_equal(np.bincount(at, minlength=off[-1]), nhit)
    for name, col in (("cx", tr["pos"][:, 2]), ("zem", tr["tim"][:, 1]), ("w", tr["tim"][:, 2])):
        assert np.array_equal(rec[name], col[at]), name
    return int(nhit.sum())


@pytest.mark.parametrize("prec", [FP64, FP32])
@pytest.mark.parametrize("far", [1e5, 1e6, 5e6, 2e7])
@pytest.mark.parametrize("kind,array", [("steep", "hex19"), ("grazing", "km100")])
def test_crossings_far_from_the_origin(kind, array, far, prec):
    rng = np.random.Generator(np.random.PCG64(KINDS.index(kind) * 10 + len(array)))
    tel = _arrays(rng)[array]
    n = 60000
    seg, t_ref = _steps(kind, n, rng)
    dx, dy = -0.11 * far, far
    tel[:, 0] += dx
    tel[:, 1] += dy
    seg["x0"] += dx
    seg["y0"] += dy
    ctx = P.Context(workloads.us_standard_atmosphere(), H_OBS, tel)
    ctx.build_refraction_tables(400, 64, 84.0 if kind == "grazing" else 70.0, 60000.0)
    dev = P.device_tracks(seg, prec, t_ref=t_ref)
    hits = crossings_match(ctx, dev, n, 99, prec)
    assert hits > 1000 or kind != "steep"


def test_oracle_crossings_far_from_the_origin():
    sc = workloads.vertical_1tev(n=20_011)
    tel = np.array(sc["telescopes"], dtype=float)
    tel[:, :2] += (5.0e5, 5.0e6)
    sc["telescopes"] = tel
    sc["tracks"] = dict(sc["tracks"], x0=sc["tracks"]["x0"] + 5.0e5, y0=sc["tracks"]["y0"] + 5.0e6)
    tr = host_tracks(sc, FP64)
    o = oracle_model(sc).bunches(tr, 7)
    code, stats, out = gpu_hits(context(sc), tr, sc["t_ref"], 7, FP64, 200_000)
    assert code == 0
    orec, grec = oracle.hit_records(o, 0), out.records()
    assert len(orec["key"]) > 5000
    # (a crossing within 1 um of a sphere's surface could fall either way)
    same = np.isin(orec["key"], grec["key"])
    assert abs(len(grec["key"]) - len(orec["key"])) <= 1 and (~same).sum() <= 1


def test_readout_far_from_the_origin():
    """Places off by some nanometres (2.4e-10 m a rounding) change a bunch's
    Gaussian weight by less than 6 sigma x 4e-9 m / sigma^2 = 2.4e-8, and its
    presence at the 6 sigma cut a sum by e^-18."""
    sc = workloads.vertical_1tev(n=20_011)
    tr = host_tracks(sc, FP64)
    D = []
    for dx, dy in ((0.0, 0.0), (5.0e5, 5.0e6)):
        tel = np.array(sc["telescopes"], dtype=float)
        tel[:, :2] += (dx, dy)
        ctx = context(dict(sc, telescopes=tel))
        dev = P.device_tracks(dict(tr, x0=tr["x0"] + dx, y0=tr["y0"] + dy), FP64,
                              t_ref=sc["t_ref"])
        D.append([v.cpu().numpy() for v in ctx.density(dev, 7, FP64, 1.0)])
    assert (D[0][0] > 0).all()
    np.testing.assert_allclose(D[1][0], D[0][0], rtol=1e-7, atol=1e-7 * D[0][0].max())
