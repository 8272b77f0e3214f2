"""One handle whose cache pointers change from tick to tick. The handle's tensor maps of the caches are rewritten at
the same device address on every change, so each tick must load whole 64-key chunks through the maps of its own caches:
ticks alternate between two caches of different contents and lengths (300 to 2000 rows a vehicle), on the single-launch
tick (B = 1), with key splits (B = 2) and with several items a CTA (B = 6), and every one is compared with the oracle.
A tick over caches that no map can be made for (not 16-byte aligned) is refused, and refused again."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_2607_15621_gb300 import fsx, synth

import fsx_cases as fc

pytestmark = pytest.mark.gpu
DIMS = synth.Dims(n_layers=2)


@pytest.mark.parametrize("lengths_a,lengths_b", [
    ([2000], [300]), ([704, 300], [512, 1100]), ([300, 641, 320, 512, 449, 384], [576, 300, 450, 333, 640, 321]),
])
def test_ticks_that_alternate_between_two_caches(lengths_a, lengths_b):
    cases = [fc.Case(DIMS, lengths_a, "bf16", seed=21), fc.Case(DIMS, lengths_b, "bf16", seed=22)]
    B = len(lengths_a)
    cases[1].w = cases[0].w  # one handle, one set of weights
    ref = [[c.oracle_vehicle(b, capture=False)[0] for b in range(B)] for c in cases]
    ex = fsx.Expert(DIMS, cases[0].w, B, max(c.total for c in cases), "bf16", "bf16")
    outs = [torch.empty(B, DIMS.n_waypoints, 2, device="cuda") for _ in range(8)]
    try:
        for i, out in enumerate(outs):  # no waiting in between: the copy of the next maps follows the tick
            c = cases[i & 1]
            ex.tick(c.k, c.v, c.offsets, c.frames, out)
        assert ex.status() == fsx.FSX_OK
    finally:
        ex.close()
    for i, out in enumerate(outs):
        got = out.cpu().double().numpy()
        for b in range(B):
            r = ref[i & 1][b]
            assert np.linalg.norm(got[b] - r) <= fc.WAYPOINT_TOL * np.linalg.norm(r), (i, b)


@pytest.mark.parametrize("B", [1, 6])
def test_misaligned_caches_are_refused_every_time(B):
    case = fc.Case(DIMS, [130] * B, "bf16", seed=23)
    shifted = [torch.empty(t.numel() + 8, dtype=t.dtype, device="cuda")[4:4 + t.numel()] for t in case.k]
    assert shifted[1].data_ptr() % 16 == 8
    ex = case.expert()
    try:
        first = fc.run_tick(ex, case)
        out = torch.full((B, DIMS.n_waypoints, 2), 123.0, device="cuda")
        for k in ([case.k[0], shifted[1]], [case.k[0], shifted[1]], shifted, shifted):
            with pytest.raises(fsx.FsxError) as e:
                ex.tick(k, case.v, case.offsets, case.frames, out)
            assert e.value.status == fsx.FSX_ERR_INVALID_ARG
        assert ex.status() == fsx.FSX_OK and torch.all(out == 123.0)
        again = fc.run_tick(ex, case)
    finally:
        ex.close()
    for b in range(B):
        ref = case.oracle_vehicle(b, capture=False)[0]
        for got in (first[b], again[b]):
            assert np.linalg.norm(got - ref) <= fc.WAYPOINT_TOL * np.linalg.norm(ref)
