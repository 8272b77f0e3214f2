"""One handle whose cache pointers change from tick to tick. The handle's tensor maps of the caches are rewritten at
the same device address on every change, so each tick must load whole 64-key chunks through the maps of its own caches:
ticks alternate between two caches of different contents and lengths (300 to 2000 rows a vehicle), on the single-launch
tick (B = 1), with key splits (B = 2) and with several items a CTA (B = 6), and every one is compared with the oracle."""
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
