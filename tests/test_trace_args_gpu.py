"""Trace arrays that 16-byte stores cannot write are refused before any launch,
by the trace as by the call that clears its arrays."""
import ctypes

import numpy as np
import pytest

import paper_2006_14927_gb300 as P
import workloads
from paper_2006_14927_gb300 import _binding as B
from parity import FP32, FP64, context, host_tracks

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [FP32, FP64])
@pytest.mark.parametrize("which", ["pos", "tim"])
def test_misaligned_trace_arrays(which, prec):
    import torch
    sc = workloads.plain_fp64()
    ctx = context(sc)
    dev = P.device_tracks(host_tracks(sc, prec), prec, t_ref=sc["t_ref"])
    nb, _ = ctx.segment_yield(dev, prec)
    off = torch.zeros(len(nb) + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.cumsum(nb.to(torch.int64), 0)
    n = int(off[-1])
    arr = {k: torch.full((32 * n + 64,), 7, dtype=torch.uint8, device="cuda")
           for k in ("pos", "tim", "status", "nhit", "first")}
    at = {k: v.data_ptr() for k, v in arr.items()}
    at[which] += 8
    tr = B.Trace(at["pos"], at["tim"], at["status"], at["nhit"], at["first"], n)
    t = ctx.tracks_struct(dev)
    assert B.lib().cher_clear_trace(ctx._h, prec, ctypes.byref(tr), None) == 1
    assert B.lib().cher_trace_bunches(ctx._h, ctypes.byref(t), ctypes.c_uint64(3), prec,
                                      off.data_ptr(), ctypes.byref(tr), None) == 1
    torch.cuda.synchronize()
    assert all(bool((v == 7).all()) for v in arr.values())
    at[which] -= 8
    tr = B.Trace(at["pos"], at["tim"], at["status"], at["nhit"], at["first"], n)
    assert B.lib().cher_clear_trace(ctx._h, prec, ctypes.byref(tr), None) == 0
    assert B.lib().cher_trace_bunches(ctx._h, ctypes.byref(t), ctypes.c_uint64(3), prec,
                                      off.data_ptr(), ctypes.byref(tr), None) == 0
    torch.cuda.synchronize()
    assert set(np.unique(arr["status"].cpu().numpy().view(np.int32)[:n])) <= {0, 1, 2, 3, 4}


@pytest.mark.parametrize("prec", [FP32, FP64])
@pytest.mark.parametrize("n,shift", [(1, 0), (3, 4), (1023, 12), (4097, 8), (300_001, 0),
                                     (300_001, 4)])
def test_cleared_arrays(n, shift, prec):
    """Every entry and nothing behind it, at any address of the integers."""
    import torch
    ctx = context(workloads.plain_fp64())
    size = 16 if prec == FP32 else 32
    arr = {k: torch.full((b * n + 48,), 7, dtype=torch.uint8, device="cuda")
           for k, b in (("pos", size), ("tim", size), ("status", 4), ("nhit", 4), ("first", 4))}
    at = {k: v.data_ptr() + (0 if k in ("pos", "tim") else shift) for k, v in arr.items()}
    tr = B.Trace(at["pos"], at["tim"], at["status"], at["nhit"], at["first"], n)
    assert B.lib().cher_clear_trace(ctx._h, prec, ctypes.byref(tr), None) == 0
    torch.cuda.synchronize()
    for k, v in arr.items():
        v, lo = v.cpu().numpy(), at[k] - v.data_ptr()
        hi = lo + (size if k in ("pos", "tim") else 4) * n
        assert (v[:lo] == 7).all() and (v[hi:] == 7).all()
        assert (v[lo:hi] == (255 if k == "status" else 0)).all(), k
