"""Infinities in V: a visible key's infinity reaches the output as an infinity of its
sign, in its column alone, through the weight's parts (d_head 64) and the merges
of an item's CTAs (several sequences: the stream-K split; one: clusters, and clusters
that exchange through global memory)."""

import pytest
import torch

from gpu_cases import ensure_lib
from paper_2608_06849_gb300 import aoh
from paper_2608_06849_gb300.workloads import randn_bf16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hq,Hkv,d,n", [(1, 8, 2, 64, 700), (40, 8, 2, 64, 700), (1, 14, 2, 64, 201), (1, 2, 2, 64, 30000),
                                          (1, 8, 2, 128, 700), (40, 8, 2, 128, 700), (1, 2, 2, 128, 30000)])
def test_infinite_value_rows(B, Hq, Hkv, d, n):
    ensure_lib()
    inf = float("inf")
    cache = aoh.Cache(B, Hq, Hkv, d, n + 1, 4, 60, [0] * Hkv)
    k, v = randn_bf16((B, n, Hkv, d), 11, "cuda"), randn_bf16((B, n, Hkv, d), 12, "cuda")
    v[:, n - 3, :, 5] = inf
    v[:, n - 2, :, 9] = -inf
    v[:, 1, :, 20] = inf
    cache.prefill(None, k, v)
    q, kn, vn = (randn_bf16((B, h, d), 13 + h, "cuda") for h in (Hq, Hkv, Hkv))
    vn[:, :, 11] = inf
    out = torch.empty_like(q)
    cache.decode_step(q, kn, vn, out)
    cache.check()
    want = {5: inf, 9: -inf, 11: inf, 20: inf}
    for col, x in want.items():
        assert (out[..., col] == x).all(), (col, out[..., col].unique().tolist()[:4])
    assert torch.isfinite(out[..., [c for c in range(d) if c not in want]]).all()
    cache.close()
