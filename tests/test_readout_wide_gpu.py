"""The read-out's sums of a long list (a wide Gaussian), which the warps keep to
themselves until their end, against the sums of short lists, which go out pair
by pair: the same bunches in calls of a few steps each.  Sums of up to 4e6
terms, so within 4e6 x 2^-53 of the sums of their magnitudes."""
import numpy as np
import pytest

import paper_2006_14927_gb300 as P
import workloads
from parity import FP32, FP64, context, host_tracks

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,n,sigma,n_tel", [(FP32, 6001, 50.0, 19), (FP64, 4003, 50.0, 19),
                                                (FP32, 40_001, 8.0, 19), (FP32, 6001, 60.0, 128),
                                                (FP32, 6001, 60.0, 129)])
def test_long_lists(prec, n, sigma, n_tel):
    sc = workloads.vertical_1tev(n=n)
    if n_tel > 19:
        rng = np.random.Generator(np.random.PCG64(n_tel))
        sc["telescopes"] = np.column_stack([rng.uniform(-900, 900, (n_tel, 2)), np.zeros(n_tel),
                                            np.full(n_tel, 1.0)])
    ctx, tr = context(sc), host_tracks(sc, prec)

    def sums(lo, hi):
        dev = P.device_tracks({k: v[lo:hi] for k, v in tr.items()}, prec, t_ref=sc["t_ref"])
        D, T = (v.cpu().numpy() for v in ctx.density(dev, 7, prec, sigma, track_base=lo))
        return D, D * T

    S, U = sums(0, n)
    parts = [sums(lo, min(lo + 200, n)) for lo in range(0, n, 200)]
    S0, U0 = sum(p[0] for p in parts), sum(p[1] for p in parts)
    size = sum(np.abs(p[1]) for p in parts)
    assert (S0 > 0).all()
    np.testing.assert_allclose(S, S0, rtol=5e-10)
    assert (np.abs(U - U0) <= 5e-10 * (size + S0)).all()
