"""The transmission draw that the hits kernel decides before a bunch is
propagated, from bounds of its step's arrival zenith, against the draw of the
trace kernel, which propagates every bunch: the same bunches absorbed."""
import numpy as np
import pytest

import paper_2006_14927_gb300 as P
import workloads
from parity import FP32, FP64
from test_reach_far_gpu import all_bunches
from test_reach_gpu import H_OBS

pytestmark = pytest.mark.gpu


def _constant_tau(tau):
    return dict(lambda_nm=(250.0, 700.0), height_m=(0.0, 60000.0), tau=np.full((2, 2), tau))


@pytest.mark.parametrize("prec", [FP32, FP64])
@pytest.mark.parametrize("zenith", [80.0, 83.0])
def test_draw_at_the_cone_s_smallest_zenith(zenith, prec):
    """At large zenith 1 / cos changes by 4 - 8 times the sine's error times
    its tangent, and a bound that is too tight there loses bunches at the side
    of the cone nearest the vertical whose deviate is just below the survival
    probability: about one in 1e7.  1e8 bunches on narrow cones (energies
    just above the threshold, small bunches), tau sec = 1.2 at the axis."""
    import torch
    rng = np.random.Generator(np.random.PCG64(int(zenith)))
    atm = workloads.us_standard_atmosphere()
    n, h = 300_000, 3200.0
    z = np.radians(zenith)
    rho = [b / c * np.exp(-x / c) for b, c, x in
           ((atm["b"][0], atm["c"][0], h), (atm["b"][0], atm["c"][0], 0.0))]
    eta = 2.83e-4 * rho[0] / rho[1]
    gamma = (1.0 + 1.2e-3) / np.sqrt(2.0 * eta)
    phi = rng.uniform(0, 2 * np.pi, n)
    seg = dict(x0=rng.uniform(-500, 500, n), y0=rng.uniform(-500, 500, n),
               z0=h + rng.uniform(-1, 1, n), t0=np.zeros(n), len=rng.uniform(1.0, 2.0, n),
               ekin=np.full(n, 0.51099895 * (gamma - 1.0)), ux=np.sin(z) * np.cos(phi),
               uy=np.sin(z) * np.sin(phi), uz=np.full(n, -np.cos(z)))
    ctx = P.Context(atm, H_OBS, [[0.0, 0.0, 0.0, 5.0]], bunch_size=4e-4)
    ctx.build_refraction_tables(400, 64, 84.5, 60000.0)
    ctx.set_transmission(_constant_tau(1.2 * np.cos(z)))
    dev = P.device_tracks(seg, prec)
    out = ctx.alloc_hits(200_000, prec)
    bunches = 0
    for seed in range(2):
        tr, _ = all_bunches(ctx, dev, n, seed, prec)
        status = tr["status"]
        want = [int((status == s).sum()) for s in range(6)]
        bunches += status.numel()
        del tr, status
        ctx.generate_propagate(dev, seed, prec, out)
        code, st = ctx.sync_status(out)
        assert code == 0
        got = [int(st[i]) for i in (8, 4, 5, 6, 7, 11)]
        assert got == want
        assert want[0] > 0 and want[5] > 0 and want[0] + want[5] == sum(want)
    assert bunches > 8e7
    torch.cuda.empty_cache()


@pytest.mark.parametrize("prec", [FP32, FP64])
def test_draw_with_opaque_nodes(prec):
    """Optical depths beyond FP32's range (opaque air): upward bunches and
    those past the tables' edges are counted as such, the rest absorbed."""
    rng = np.random.Generator(np.random.PCG64(5))
    n = 4000
    seg, t_ref = workloads.shower_segments(rng, n, 1.0e6, 0.3, 0.7, 0.0, 0.0, H_OBS)
    d = rng.normal(size=(n, 3))
    d /= np.linalg.norm(d, axis=1)[:, None]
    seg["ux"], seg["uy"], seg["uz"] = d.T.copy()
    ctx = P.Context(workloads.us_standard_atmosphere(), H_OBS, [[0.0, 0.0, 0.0, 5.0]])
    ctx.build_refraction_tables(400, 64, 70.0, 60000.0)
    ctx.set_transmission(_constant_tau(1e39))
    dev = P.device_tracks(seg, prec, t_ref=t_ref)
    tr, _ = all_bunches(ctx, dev, n, 3, prec)
    status = tr["status"].cpu().numpy()
    out = ctx.alloc_hits(1000, prec)
    ctx.generate_propagate(dev, 3, prec, out)
    _, st = ctx.sync_status(out)
    want = [int((status == s).sum()) for s in range(6)]
    assert [int(st[i]) for i in (8, 4, 5, 6, 7, 11)] == want
    assert want[1] > 1000 and want[4] > 1000 and want[5] > 1000 and want[0] == 0
