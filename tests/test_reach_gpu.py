"""The hits kernel's bound of the azimuths that can reach a sphere, against the
trace kernel, which propagates every bunch: the same crossings (telescope and
bunch), the same counters and bit-equal values, for steps and arrays at the
edges of what the bound covers -- steep and grazing steps, steps whose bunches
drop out at the tables' edges, long steps, steps close to the observation
level, directions that are not unit vectors, vertical and nearly vertical
steps (the azimuth basis switches there), energies at the Cherenkov threshold;
spheres small, large, overlapping, raised and sunk, arrays of more than 32
telescopes.  Both kernels run the same arithmetic per bunch, so nothing is
left out and no tolerance is needed."""
import numpy as np
import pytest

import paper_2006_14927_gb300 as P
import workloads
from parity import FP32, FP64

pytestmark = pytest.mark.gpu

H_OBS = 2200.0


def _arrays(rng):
    hexa = workloads.hex_telescopes(rng)
    wide = workloads.scattered_telescopes(rng)
    many = np.column_stack([rng.uniform(-1500, 1500, 300), rng.uniform(-1500, 1500, 300),
                            rng.uniform(-40, 60, 300), rng.uniform(1.0, 30.0, 300)])
    dense = np.column_stack([rng.uniform(-60, 60, 24), rng.uniform(-60, 60, 24),
                             rng.uniform(-5, 5, 24), rng.uniform(10.0, 40.0, 24)])
    return dict(single=np.array([[0.0, 0.0, 0.0, 12.0]]), hex19=hexa, km100=wide, many300=many,
                dense24=dense)


def _steps(kind, n, rng):
    """Shower-like steps, a third of them turned into the case's odd ones."""
    zen = dict(steep=0.0, inclined=1.05, grazing=1.4).get(kind, 0.3)
    seg, t_ref = workloads.shower_segments(rng, n, 1.0e6, zen, 0.7, 0.0, 0.0, H_OBS)
    d = np.stack([seg["ux"], seg["uy"], seg["uz"]], 1)
    odd = rng.random(n) < 0.33
    m = int(odd.sum())
    if kind == "low":                 # close above and around the observation level
        seg["z0"][odd] = H_OBS + rng.uniform(-20.0, 300.0, m)
        seg["x0"][odd] = rng.uniform(-200.0, 200.0, m)
        seg["y0"][odd] = rng.uniform(-200.0, 200.0, m)
    elif kind == "long":
        seg["len"][odd] = np.exp(rng.uniform(np.log(20.0), np.log(4000.0), m))
    elif kind == "odd_directions":
        d[odd] = rng.normal(size=(m, 3))
        d[odd] /= np.linalg.norm(d[odd], axis=1)[:, None]
        scale = np.exp(rng.uniform(np.log(0.9), np.log(1.1), m))
        d[odd] *= np.where(rng.random(m) < 0.5, scale, 1.0 + rng.uniform(-3e-6, 3e-6, m))[:, None]
    elif kind == "vertical":
        eps = np.where(rng.random(m) < 0.3, 0.0, 10.0 ** rng.uniform(-11.5, -8.0, m))
        phi = rng.uniform(0, 2 * np.pi, m)
        d[odd] = np.stack([eps * np.cos(phi), eps * np.sin(phi), -np.ones(m)], 1)
    elif kind == "threshold":
        eta = 2.83e-4 * np.exp(-seg["z0"][odd] / 8400.0)
        seg["ekin"][odd] = 0.511 * (1.0 / np.sqrt(2.0 * eta) - 1.0) * rng.uniform(0.98, 1.1, m)
    elif kind == "high":
        seg["z0"][odd] = rng.uniform(2.9e4, 6.2e4, m)
    seg["ux"], seg["uy"], seg["uz"] = d.T.copy()
    return seg, t_ref


KINDS = ["steep", "inclined", "grazing", "low", "long", "odd_directions", "vertical", "threshold",
         "high"]
CASES = [(k, a, FP32, "none") for k in KINDS
         for a in ("hex19", "km100" if k == "grazing" else "many300")]
CASES += [(k, a, FP64, "none") for k in ("steep", "grazing", "low", "vertical")
          for a in ("single", "km100")]
CASES += [(k, "dense24", FP32, "none") for k in ("low", "steep", "odd_directions")]
CASES += [(k, "km100", FP32, o) for k in ("steep", "grazing", "long", "odd_directions")
          for o in ("transmission", "dispersion", "both")]
CASES += [("grazing", "km100", FP64, "both")]


@pytest.mark.parametrize("kind,array,prec,option", CASES)
def test_crossings_are_those_of_all_bunches(kind, array, prec, option):
    import torch
    rng = np.random.Generator(np.random.PCG64(KINDS.index(kind) * 10 + len(array)))
    tel = _arrays(rng)[array]
    n = 4000 if prec == FP64 else 12000
    seg, t_ref = _steps(kind, n, rng)
    ctx = P.Context(workloads.us_standard_atmosphere(), H_OBS, tel)
    ctx.build_refraction_tables(400, 64, 84.0 if kind == "grazing" else 70.0, 60000.0)
    if option in ("transmission", "both"):
        ctx.set_transmission(workloads.synthetic_transmission())
    if option in ("dispersion", "both"):
        ctx.set_dispersion(workloads.synthetic_dispersion())
    dev = P.device_tracks(seg, prec, t_ref=t_ref)
    nb, _ = ctx.segment_yield(dev, prec)
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.cumsum(nb.to(torch.int64), 0)
    tr = {k: v.cpu().numpy() for k, v in ctx.trace_bunches(dev, 99, prec, off).items()}
    off = off.cpu().numpy()
    status, nhit = tr["status"], tr["nhit"].astype(np.int64)
    assert nhit.max(initial=0) < 32
    out = ctx.alloc_hits(max(int(nhit.sum()), 1), prec)
    for block, ctas in ((128, 8), (256, 0)):
        ctx.set_launch(block, ctas)
        ctx.generate_propagate(dev, 99, prec, out)
        code, st = ctx.sync_status(out)
        assert code == 0
        assert st[0] == n and st[1] == (nb > 0).sum().item() and st[3] == off[-1]
        for s, idx in ((1, 4), (2, 5), (3, 6), (4, 7), (5, 11), (0, 8)):
            assert st[idx] == (status == s).sum(), P.STAT_NAMES[idx]
        assert st[9] == nhit.sum() and st[10] == 0
        rec = out.records()
        key = rec["key"]
        at = off[(key >> np.uint64(32)).astype(np.int64)] + (key & np.uint64(0xffffffff)).astype(np.int64)
        assert np.array_equal(np.bincount(at, minlength=off[-1]), nhit)
        first = np.full(off[-1], 1 << 30)
        np.minimum.at(first, at, rec["tel"])
        assert np.array_equal(np.where(nhit > 0, first, -1), tr["first_hit"])
        for name, col in (("cx", tr["pos"][:, 2]), ("cy", tr["pos"][:, 3]), ("zem", tr["tim"][:, 1]),
                          ("w", tr["tim"][:, 2]), ("lam", tr["tim"][:, 3])):
            assert np.array_equal(rec[name], col[at]), name
    if kind in ("steep", "low") and array != "single":
        assert nhit.sum() > 50
