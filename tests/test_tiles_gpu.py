"""Tiles of fewer steps than a CTA has threads (launches that would leave SMs
idle otherwise) give every bunch and crossing of tiles of one step per thread:
a trace of n steps against the same steps traced a few at a time, and the
curved atmosphere's crossings with few CTAs (whole blocks) against many (tiles
of a few steps), at sizes around the smallest tile, uneven last tiles and more
waves than one.  The same arithmetic per bunch, so bit-equal."""
import numpy as np
import pytest

import paper_2006_14927_gb300 as P
import workloads
from parity import FP32, FP64, context, gpu_hits, gpu_trace, host_tracks

pytestmark = pytest.mark.gpu


def _part(tr, lo, hi):
    return {k: v[lo:hi] for k, v in tr.items()}


@pytest.mark.parametrize("prec,n", [(FP32, 1), (FP32, 5), (FP32, 129), (FP32, 4865), (FP32, 6083),
                                    (FP32, 90001), (FP64, 3), (FP64, 457 * 4 + 1), (FP64, 30001)])
def test_trace_of_small_tiles(prec, n):
    sc = workloads.vertical_1tev(n=n)
    ctx = context(sc)
    tr = host_tracks(sc, prec)
    whole = gpu_trace(ctx, tr, sc["t_ref"], 7, prec)
    piece = -(-n // 3) if n < 10_000 else 2000
    parts = [gpu_trace(ctx, _part(tr, lo, min(lo + piece, n)), sc["t_ref"], 7, prec, track_base=lo)
             for lo in range(0, n, piece)
             if whole["nb"][lo:lo + piece].any()]          # (a trace of no bunches is refused)
    for k in set(whole) - {"nb", "w"}:                     # per bunch
        assert np.array_equal(whole[k], np.concatenate([p[k] for p in parts])), k


@pytest.mark.parametrize("prec,n", [(FP32, 3), (FP32, 1300), (FP32, 20011), (FP64, 1300)])
def test_curved_crossings_of_small_tiles(prec, n):
    sc = workloads.vertical_1tev(n=n)
    ctx = context(sc)
    ctx.set_curved(6.371e6)
    tr = host_tracks(sc, prec)
    got = []
    for launch in ((128, 1), (128, 8), (128, 0)):
        code, stats, out = gpu_hits(ctx, tr, sc["t_ref"], 7, prec, 40 * n, launch=launch)
        assert code == 0
        r = out.records()
        at = np.lexsort((r["tel"], r["key"]))
        got.append((stats, {k: v[at] for k, v in r.items()}))
    for stats, r in got[1:]:
        assert np.array_equal(stats, got[0][0])
        for k in r:
            assert np.array_equal(r[k], got[0][1][k]), k
    assert n < 1000 or len(got[0][1]["key"]) > 100


@pytest.mark.parametrize("prec,n", [(FP32, 24_321), (FP32, 70_001), (FP64, 25_003)])
def test_profile_of_showers_taken_in_turn(prec, n):
    """A production profile of several showers, whose groups the warps take in
    turn from parts of the list, against each shower in a launch of its own
    (in order, equal bins combined): the same crossings and counters, and sums
    that differ by the order of at most n FP64 additions of positive terms."""
    import torch
    sc = workloads.vertical_1tev(n=n)
    ctx, tr = context(sc), host_tracks(sc, prec)
    rows, edges = 3, [0, n // 5, n // 5 + 7, n]
    t_ref = np.repeat(sc["t_ref"][:1], rows)

    def run(lo, hi, shower, prof):
        t = dict(_part(tr, lo, hi), shower=shower[lo:hi])
        dev = P.device_tracks(t, prec, t_ref=t_ref)
        out = ctx.alloc_hits(n, prec)
        ctx.generate_propagate(dev, 7, prec, out, track_base=lo, profile=prof, bin_gcm2=10.0)
        code, stats = ctx.sync_status(out)
        assert code == 0
        return np.asarray(stats), out.records()

    shower = np.repeat(np.arange(rows), np.diff(edges)).astype(tr["shower"].dtype)
    prof = torch.zeros((rows, 120), dtype=torch.float64, device="cuda")
    stats, rec = run(0, n, shower, prof)
    alone, total, recs = torch.zeros_like(prof), 0, []
    for k in range(rows):
        one = torch.zeros((rows, 120), dtype=torch.float64, device="cuda")
        ctx.set_launch(128, 1 if k == 0 else 8)          # fewer warps: full groups, no parts
        st, r = run(edges[k], edges[k + 1], shower, one)
        alone += one
        total = total + st
        recs.append(r)
    assert np.array_equal(stats, total)
    both = {k: np.concatenate([r[k] for r in recs]) for k in rec}
    at = np.lexsort((both["key"], both["tel"]))
    for k in rec:
        assert np.array_equal(rec[k], both[k][at]), k
    assert prof.sum() > 0
    bound = n * 2.0 ** -52 * alone
    assert bool(((prof - alone).abs() <= bound).all())
