"""The tensor-core attention's key splits and fp32 caches at the edges of their tiling, through fsx_attention against
the fp64 oracle: cache lengths around the 64-key chunks, splits without any cache key, one to 48 queries, one to 64 own
keys, launches of more than one wave (longest caches first), and the range check of every cache value that split and fp32
launches make.

Tolerance, as a share of a row's largest entry. bf16 caches: q, k and the scores' operands are exact in fp16, P keeps 16
bits, so the fp16 result's own rounding (2^-11 = 4.9e-4) dominates: 1e-3. fp32 caches: K and V are rounded to fp16 (2^-12
relative on average); a score of size s moves by about 2^-12 s, at most ~4e-3 for the largest scores here (|s| < 16) but
averaged over keys, plus 2^-12 of V: 3e-3."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_2607_15621_gb300 import fsx

from test_gpu_attention import D, H, gpu_attention, make, oracle_attention, row_err

pytestmark = pytest.mark.gpu
TOL = {"bf16": 1e-3, "fp32": 3e-3}


@pytest.mark.parametrize("cache_dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("n_splits,lengths,n_q,n_own", [
    (1, [64, 1, 0, 129], 42, 42), (1, [63], 48, 64), (1, [191, 320], 1, 1),
    (2, [64], 42, 42), (2, [65, 0], 48, 48), (3, [128, 63], 33, 1), (4, [191, 192, 193], 10, 64),
    (5, [64, 321], 42, 42), (7, [450], 5, 7), (8, [0], 42, 42), (8, [511, 513], 42, 10), (8, [1100], 48, 48),
])
def test_splits_and_dtypes(cache_dtype, n_splits, lengths, n_q, n_own):
    c = make(lengths, n_q=n_q, n_own=n_own, cache_dtype=cache_dtype, seed=n_splits * 31 + len(lengths))
    out, lse = gpu_attention(c, n_splits)
    ref, ref_lse = oracle_attention(c)
    assert row_err(out, ref).max() <= TOL[cache_dtype]
    assert np.abs(lse - ref_lse).max() <= 2e-3


@pytest.mark.parametrize("cache_dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("n_splits,lengths", [
    (1, [7, 64, 64, 0, 130, 1, 64, 129, 0, 200]),      # 320 CTAs, just over one wave: longest first, ties by index
    (8, [5, 70, 70]), (1, [3 * (i * 37 % 128 // 4) for i in range(128)]), (1, [i % 3 for i in range(129)]),
    (1, [65 * (i % 5 == 0) for i in range(310)]),      # more items than one wave of CTAs takes
])
def test_more_than_one_wave(cache_dtype, n_splits, lengths):
    c = make(lengths, n_q=42 if len(lengths) < 100 else 3, n_own=10, cache_dtype=cache_dtype, seed=len(lengths))
    out, lse = gpu_attention(c, n_splits)
    ref, ref_lse = oracle_attention(c)
    assert row_err(out, ref).max() <= TOL[cache_dtype]
    assert np.abs(lse - ref_lse).max() <= 2e-3


@pytest.mark.parametrize("cache_dtype", ["bf16", "fp32"])
def test_vehicles_without_valid_offsets_are_passed_over(cache_dtype):
    """Two vehicles of negative length among sixteen (512 items): reported, their rows untouched, the rest right."""
    lengths = [70 - 4 * i for i in range(16)]
    c = make(lengths, n_q=10, n_own=10, cache_dtype=cache_dtype, seed=3)
    ref, _ = oracle_attention(c)
    bad = (5, 14)
    off = c["off"].copy()
    off[6] = off[5] - 1     # vehicle 5: length -1; vehicle 6 starts one row early
    off[15] = off[14] - 1   # vehicle 14: length -1; vehicle 15 starts one row early
    dev = lambda t: t.to("cuda").contiguous()
    n_q = n_own = 10
    out = torch.full((16 * n_q, H * D), -7.0, device="cuda", dtype=torch.float16)
    ws = torch.empty(fsx.attention_workspace_bytes(16, H, n_q, 1), device="cuda", dtype=torch.uint8)
    fsx.attention(dev(c["q"]), H * D, dev(c["ko"]), dev(c["vo"]), H * D, n_q, n_own, dev(c["kc"]), dev(c["vc"]),
                  c["dtype"], torch.as_tensor(off, device="cuda"), 16, H, 1, out, None, ws)
    torch.cuda.synchronize()
    out = out.cpu().double().numpy()
    assert int(ws[:4].cpu().view(torch.int32)[0]) != 0
    for b in range(16):
        rows = slice(b * n_q, (b + 1) * n_q)
        if b in bad:
            assert (out[rows] == -7.0).all()
        elif b - 1 not in bad:
            assert row_err(out[rows], ref[rows]).max() <= TOL[cache_dtype]


@pytest.mark.parametrize("cache_dtype,n_splits", [("bf16", 2), ("bf16", 8), ("fp32", 1), ("fp32", 3)])
@pytest.mark.parametrize("which,row,dim", [("kc", 0, 0), ("kc", 200, 127), ("vc", 63, 5), ("vc", 64, 64), ("vc", 200, 127)])
def test_values_beyond_fp16_are_reported(cache_dtype, n_splits, which, row, dim):
    c = make([201], cache_dtype=cache_dtype, seed=9)
    dev = lambda t: t.to("cuda").contiguous()
    off = torch.as_tensor(c["off"], device="cuda")
    ws = torch.empty(fsx.attention_workspace_bytes(1, H, 42, n_splits), device="cuda", dtype=torch.uint8)
    out = torch.empty(42, H * D, device="cuda", dtype=torch.float16)

    def status():
        fsx.attention(dev(c["q"]), H * D, dev(c["ko"]), dev(c["vo"]), H * D, 42, 42, dev(c["kc"]), dev(c["vc"]),
                      cache_dtype, off, 1, H, n_splits, out, None, ws)
        torch.cuda.synchronize()
        return int(ws[:4].view(torch.int32).item())

    c[which][row, 7, dim] = 65280.0  # the largest bf16 value below 65504
    assert status() == fsx.FSX_OK
    for bad in (65536.0, -1e30, float("inf"), float("nan")):
        c[which][row, 7, dim] = bad
        assert status() == fsx.FSX_ERR_RANGE, bad


@pytest.mark.parametrize("cache_dtype,n_splits,n_own", [
    ("bf16", 2, 42), ("bf16", 8, 42), ("fp32", 1, 42), ("fp32", 3, 42), ("bf16", 3, 70), ("fp32", 2, 70)])
@pytest.mark.parametrize("which,bad", [("kc", 1.0e6), ("kc", float("-inf")), ("vc", -3.0e5), ("vc", float("inf"))])
def test_rows_beside_a_range_error_are_those_of_the_clipped_cache(cache_dtype, n_splits, n_own, which, bad):
    """70 own keys: the mma.sync kernel, which rounds P to fp16.

    Tolerance, as a share of a row's largest entry, where a value of 65504 carries nearly the whole row: 2^-11 for the
    fp16 result; bf16 V is clipped to 65536, another 2^-11; together 1e-3 and the usual 1e-3: 2e-3. P in fp16 has units
    of 2^-24 below 2^-14: 2^-25 * 65504 = 2e-3 of an entry, over rows whose largest is at least 0.4, and 3e-3 as usual:
    8e-3. The log-sum-exp of scores up to 3e5 is an fp32 sum: 1e-5 of it."""
    c = make([201], n_own=n_own, cache_dtype=cache_dtype, seed=10)
    clipped = dict(c)
    for row, head, dim in ((3, 5, 7), (130, 5, 70), (200, 17, 127)):
        c[which][row, head, dim] = bad
    clipped[which] = c[which].double().clamp(-65504.0, 65504.0)
    ref, ref_lse = oracle_attention(clipped)
    out, lse = gpu_attention(c, n_splits)
    assert np.isfinite(out).all() and np.isfinite(lse).all()
    assert row_err(out, ref).max() <= (2e-3 if cache_dtype == "bf16" and n_own <= 64 else 8e-3)
    assert (np.abs(lse - ref_lse) <= 2e-3 + 1e-5 * np.abs(ref_lse)).all()


def test_default_stream_of_a_call_is_the_current_one():
    side = torch.cuda.Stream()
    for s in (torch.cuda.default_stream(), side):
        with torch.cuda.stream(s):
            assert fsx._stream(None) == torch.cuda.current_stream().cuda_stream == s.cuda_stream
