"""The append's kernels at the edges of their tiling, against the fp64 append oracle: cached lengths around the 8-key
units and around the 32 keys that one CTA's four warps take in turn, 1 to 8 new tokens (both query-slot variants),
batches whose (vehicle, head) pairs run on 8, 4, 2 and 1 CTAs, and 17 to 256 token rows at a width where the equal
shares of the weight stream cut tiles, whose parts are then summed by one CTA.

Tolerance per row (one token's hidden state or one appended cache row), as a share of the row's largest entry: the
new keys and values are rounded to bf16 (2^-9 = 2.0e-3 of an entry), the GEMM operands to fp16 (2^-11 = 4.9e-4 each,
three GEMMs deep for a hidden state): below 2^-9 + 4 * 2^-11 = 4e-3; 6e-3 is asked."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from oracle import append_oracle
from paper_2607_15621_gb300 import fsx, synth

pytestmark = pytest.mark.gpu
TOL = 6e-3


def row_err(got, ref):
    ref = np.asarray(ref, np.float64)
    ref = ref.reshape(-1, ref.shape[-1])
    got = np.asarray(got, np.float64).reshape(ref.shape)
    return (np.abs(got - ref).max(-1) / np.maximum(np.abs(ref).max(-1), 1e-30)).max()


def check(dims, n_new, lengths, v_offset=0, calls=1):
    H, D, B = dims.n_heads, dims.head_dim, len(lengths)
    w = synth.make_backbone_weights(dims, 5, "bf16")
    off = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    total = int(off[-1])
    dst = np.array([total + n_new * (B - 1 - b) for b in range(B)], dtype=np.int64)  # not in vehicle order
    rows = total + n_new * B + 1
    g = torch.Generator().manual_seed(n_new * 100 + B)
    kc = (torch.randn(rows, H, D, generator=g) * torch.exp(0.5 * torch.randn(H, D, generator=g))).bfloat16()
    vc = torch.randn(rows, H, D, generator=g).bfloat16()
    x = synth.make_append_tokens(dims, B, seed=6)
    kg = kc.cuda()
    vg = torch.empty(vc.numel() + v_offset, dtype=vc.dtype, device="cuda")[v_offset:].view_as(vc)
    vg.copy_(vc)
    assert vg.data_ptr() % 16 == 2 * v_offset
    hidden = [torch.empty(B, n_new, dims.d_model, device="cuda") for _ in range(calls)]
    ap = fsx.Append(dims, w, B, rows)
    try:
        for h in hidden:  # a repeated call reads the same cached rows and writes the same new ones
            ap.append([kg], [vg], torch.as_tensor(off).cuda(), torch.as_tensor(dst).cuda(), x.cuda(), h)
        assert ap.status() == fsx.FSX_OK
    finally:
        ap.close()
    assert all(torch.equal(h, hidden[0]) for h in hidden)  # sums in a fixed order
    h_ref, k_ref, v_ref = append_oracle.backbone_append(w, [kc[:total].float().numpy()], [vc[:total].float().numpy()],
                                                        off, x.float().numpy(), H, D)
    written = np.concatenate([np.arange(d0, d0 + n_new) for d0 in dst])
    assert row_err(hidden[0].cpu().numpy().reshape(B * n_new, -1), np.asarray(h_ref).reshape(B * n_new, -1)) <= TOL
    for got, was, ref in ((kg, kc, k_ref), (vg, vc, v_ref)):
        got = got.cpu()
        assert row_err(got[written].float().numpy().reshape(B * n_new, -1),
                       np.asarray(ref[0]).reshape(B * n_new, -1)) <= TOL
        keep = np.setdiff1d(np.arange(rows), written)
        assert torch.equal(got[keep], was[keep])


@pytest.mark.parametrize("n_new,lengths,v_offset", [(n, l, 0) for n, l in (
    (4, [0]), (4, [31]), (1, [32]), (3, [33]), (8, [128]), (5, [1025]),
    (4, [127, 0]), (8, [129, 32, 257]), (4, [1, 64, 31, 300, 0]), (7, [5, 0, 97, 128, 33]),
)] + [(4, [127, 0, 9], 4), (8, [33, 70], 4)])  # values' cache aligned to 8 bytes only
def test_append_attention_edges(n_new, lengths, v_offset):
    check(synth.BackboneDims(n_layers=1, d_model=256, d_ff=256, n_new=n_new), n_new, lengths, v_offset)


def splits(B, heads, sms):
    """CTAs per (vehicle, head): the largest power of two up to 8 within two waves of four CTAs an SM."""
    s = 8
    while s > 1 and B * heads * s > 8 * sms:
        s //= 2
    return s


@pytest.mark.parametrize("B,n_new,d_ff,ctas", [
    (17, 1, 448, 2), (11, 3, 1408, 2), (16, 4, 448, 2), (13, 5, 1408, 2), (12, 8, 448, 2),   # 17, 33, 64, 65, 96 tokens
    (43, 3, 1408, 1), (25, 8, 448, 1), (64, 4, 1408, 1), (32, 8, 448, 1), (20, 4, 448, 1),   # 129, 200, 256, 256, 80
])
def test_append_of_many_vehicles(B, n_new, d_ff, ctas):
    """At width 1024 no SM's share of QKV (96 tiles of 16 steps) or gate/up (14 or 22 tiles) is whole tiles; W_d is
    cut over clusters at 1408 inputs and streamed, 8 tiles of 7 steps on 14 CTAs, at 448."""
    dims = synth.BackboneDims(n_layers=1, d_model=1024, d_ff=d_ff, n_new=n_new)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if sms == 152:
        assert splits(B, dims.n_heads, sms) == ctas
    check(dims, n_new, [(0, 7, 8, 9, 31, 33, 1, 64)[b % 8] for b in range(B)], calls=2)


def test_misaligned_caches_are_refused_on_the_host():
    dims = synth.BackboneDims(n_layers=1, d_model=256, d_ff=256)
    flat = torch.zeros(24 * dims.n_heads * dims.head_dim + 8, dtype=torch.bfloat16, device="cuda")
    x = synth.make_append_tokens(dims, 1, seed=6).cuda()
    hidden = torch.empty(1, dims.n_new, dims.d_model, device="cuda")
    off, dst = torch.tensor([0, 8]).cuda(), torch.tensor([8]).cuda()
    ap = fsx.Append(dims, synth.make_backbone_weights(dims, 5, "bf16"), 1, 20)
    try:
        for k0, v0 in ((4, 0), (0, 2)):
            with pytest.raises(fsx.FsxError) as e:
                ap.append([flat[k0:]], [flat[v0:]], off, dst, x, hidden)
            assert e.value.status == fsx.FSX_ERR_INVALID_ARG
        assert ap.status() == fsx.FSX_OK
    finally:
        ap.close()
