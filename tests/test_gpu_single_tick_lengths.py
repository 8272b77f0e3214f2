"""The single-launch tick at the edges of its cache staging: no chunk, one key, whole and ragged last chunks, one to
many chunks per CTA (three staging buffers of 64 keys, 36 for fp32, on each of a head's four CTAs), so that every buffer
is refilled and the layers start at every buffer; with the first rows of the cache at an offset.

Tolerance: attention rows within the method's 2e-2 of a row's largest entry; waypoints (relative L2, two layers): operand
roundings to fp16 (2^-11) at seven points a layer, P among them, add up to sqrt(14) 2^-11 = 1.8e-3 for 10 to 84 values;
5e-3 is asked."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from oracle import fsx_oracle
from paper_2607_15621_gb300 import fsx, synth

import fsx_cases as fc

pytestmark = pytest.mark.gpu
DIMS = synth.Dims(n_layers=2, n_waypoints=42)


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("L", [0, 1, 36, 63, 65, 145, 256, 257, 577, 768, 1025, 1793])
def test_single_tick_lengths(L, dtype):
    w = fc.weights(DIMS, 2, dtype)
    start = 5
    k, v, _ = synth.make_cache(DIMS, [L + start + 3], L, dtype)
    frames = synth.make_frames(DIMS, 1, L, dtype)
    ex = fsx.Expert(DIMS, w, 1, L + start + 3, dtype, dtype)
    try:
        off = torch.tensor([start, start + L], device="cuda")
        out = torch.full((1, 42, 2), float("nan"), device="cuda")
        attn = torch.empty(2, 42, 4096, dtype=torch.float16, device="cuda")
        kg, vg, fg = [t.cuda() for t in k], [t.cuda() for t in v], frames.cuda()
        for _ in range(2):  # the second tick starts from used barriers and buffers
            ex.tick_debug(kg, vg, off, fg, out, attn)
        assert ex.status() == fsx.FSX_OK
    finally:
        ex.close()
    ref, cap = fsx_oracle.expert_tick(w, [synth.as_f64(t[start:start + L]) for t in k],
                                      [synth.as_f64(t[start:start + L]) for t in v], np.array([0, L]),
                                      synth.as_f64(frames), DIMS.n_heads, DIMS.head_dim, 42, capture_attention=True)
    got = out.cpu().double().numpy()
    assert np.linalg.norm(got - ref) <= 5e-3 * np.linalg.norm(ref)
    cap = np.asarray(cap).reshape(2, 42, 4096)
    a = attn.cpu().double().numpy()
    assert (np.abs(a - cap).max(-1) / np.abs(cap).max(-1)).max() <= fc.ATTN_ROW_TOL
