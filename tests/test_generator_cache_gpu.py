"""The step generator's kept depth tables: calls with more showers than it keeps
(4096), with showers that it kept or dropped before among them, give the steps
of a new context."""
import numpy as np
import pytest

import paper_2006_14927_gb300 as P
import workloads
from parity import FP32

pytestmark = pytest.mark.gpu


def test_more_showers_than_are_kept():
    import torch
    rng = np.random.Generator(np.random.PCG64(9))
    showers = [dict(e0_mev=float(e), zenith=float(z), azimuth=0.3, core_x=0.0, core_y=0.0, n=40)
               for e, z in zip(np.exp(rng.uniform(9, 16, 4200)), rng.uniform(0, 1, 4200))]
    lists = [showers[:100] * 2, showers + showers[:100], showers[4000:] + showers[:300]]

    def context():
        ctx = P.Context(workloads.us_standard_atmosphere(), 2200.0, [[0.0, 0.0, 0.0, 5.0]])
        ctx.build_refraction_tables(100, 16, 70.0, 60000.0)
        return ctx

    kept = context()
    for some in lists:
        a, b = (c.generate_steps(some, 5, FP32) for c in (kept, context()))
        for k in a:
            assert torch.equal(a[k], b[k]), k
    z = a["z0"].reshape(-1, 40).mean(1).cpu().numpy()
    assert np.isfinite(z).all() and (z > 2200.0).all()
