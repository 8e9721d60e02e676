"""The autotuner's cache: a shape found for this library's kernels is taken
from it, one that an earlier library wrote (whose lines name no revision of the
kernels) is measured again."""
import pytest

import paper_2006_14927_gb300 as P
import workloads
from parity import FP32, context, host_tracks

pytestmark = pytest.mark.gpu


def test_cached_shapes_are_those_of_these_kernels(tmp_path):
    import torch
    sc = workloads.vertical_1tev(n=3000)
    dev = P.device_tracks(host_tracks(sc, FP32), FP32, t_ref=sc["t_ref"])
    ctx = context(sc)
    out = ctx.alloc_hits(10_000, FP32)
    cache = tmp_path / "shapes"
    name = torch.cuda.get_device_properties(0).name.replace(" ", "_")
    cache.write_text(f"{name}|{FP32}|11|{len(sc['telescopes'])}|{sc['Z']} 512 9\n")
    found = ctx.autotune(dev, 5, FP32, out, cache_path=str(cache))
    assert found != (512, 9)                    # (nothing that it would try)
    lines = cache.read_text().splitlines()
    assert len(lines) == 2
    cache.write_text(lines[1].rsplit(" ", 2)[0] + " 512 9\n")
    again = context(sc)
    assert again.autotune(dev, 5, FP32, again.alloc_hits(10_000, FP32),
                          cache_path=str(cache)) == (512, 9)
