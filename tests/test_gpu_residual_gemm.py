"""The residual projections with K cut over a cluster, at the edges of their token tiles (48, 64, 96, 128, 144 and
160 tokens; the 16-token tile runs in the append's tests), with ragged 4-token groups, two to eight splits and K too
short or tokens too many to cut, through one-layer ticks against the fp64 oracle. Every token
is decoded as a waypoint, so every updated row is compared.

Tolerance (relative L2 per vehicle): operands are rounded to fp16 (2^-11 each) at six points of a layer (x, q/k/v, P V,
the SwiGLU product and the two weight-side products), which add up like independent errors to sqrt(12) 2^-11 = 1.7e-3;
4e-3 is asked."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from oracle import fsx_oracle
from paper_2607_15621_gb300 import fsx, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,tokens,d_ff", [
    (2, 24, 1408), (7, 7, 1408), (3, 43, 64), (3, 48, 1408), (5, 29, 192), (9, 41, 1408), (16, 42, 1408),
    (29, 47, 1408), (60, 45, 320), (96, 42, 1408),
])
def test_residual_projections(B, tokens, d_ff):
    dims = synth.Dims(n_layers=1, d_ff=d_ff, n_action=4, n_frame=tokens - 4, n_waypoints=tokens)
    w = synth.make_weights(dims, 3, "bf16")
    lengths = [b % 3 for b in range(B)]
    k, v, off = synth.make_cache(dims, lengths, 4, "bf16")
    frames = synth.make_frames(dims, B, 5, "bf16")
    ex = fsx.Expert(dims, w, B, int(off[-1]) + 1)
    try:
        out = torch.full((B, tokens, 2), float("nan"), device="cuda")
        ex.tick([t.cuda() for t in k], [t.cuda() for t in v], torch.as_tensor(off).cuda(), frames.cuda(), out)
        assert ex.status() == fsx.FSX_OK
        got = out.cpu().double().numpy()
        again = torch.empty_like(out)
        ex.tick([t.cuda() for t in k], [t.cuda() for t in v], torch.as_tensor(off).cuda(), frames.cuda(), again)
        torch.cuda.synchronize()
        assert torch.equal(out, again)  # sums in a fixed order
    finally:
        ex.close()
    ref = fsx_oracle.expert_tick(w, [synth.as_f64(t) for t in k], [synth.as_f64(t) for t in v], off,
                                 synth.as_f64(frames), dims.n_heads, dims.head_dim, dims.n_waypoints)
    err = np.linalg.norm((got - ref).reshape(B, -1), axis=1) / np.linalg.norm(ref.reshape(B, -1), axis=1)
    assert err.max() <= 4e-3
