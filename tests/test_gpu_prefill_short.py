"""Prefill calls of many short work items, which one CTA an SM goes through in one
pipeline, against the oracle: ragged lengths around the query tiles, single-tile
items, odd groups, a cached prefix that ends inside a tile, the chunk-eviction
rule, and more items than travel as kernel arguments."""

import numpy as np
import pytest
import torch

from gpu_cases import assert_matches, ensure_lib, f64, run_case
from oracle import attention as oatt
from paper_2608_06849_gb300 import aoh
from paper_2608_06849_gb300.workloads import randn_bf16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hq,Hkv,d,T,S,W,labels,lens", [
    (16, 32, 4, 128, 384, 4, 130, [0, 1, 0, 1], [1 + 383 * b // 15 for b in range(16)]),
    (16, 28, 4, 64, 385, 130, 129, [0, 1, 0, 1], [385, 1, 127, 128, 129, 255, 256, 257] * 2),
    (32, 32, 4, 64, 128, 0, 1, [0, 1, 1, 1], [128, 1, 64, 127] * 8),   # one tile each
    (30, 16, 16, 128, 257, 4, 60, [0, 1] * 8, None),                   # a head a group
])
def test_ragged(B, Hq, Hkv, d, T, S, W, labels, lens):
    run_case(B, Hq, Hkv, d, T, S, W, labels, seq_lens=lens)


@pytest.mark.parametrize("d,B,Hq,Hkv,T,prefix,rule", [
    (128, 12, 32, 4, 300, 200, 0),
    (64, 12, 28, 4, 260, 400, 0),
    (128, 12, 32, 4, 300, 600, 300),
    (128, 113, 32, 4, 257, 0, 0),  # 3,888 items
])
def test_chunks_and_long_lists(d, B, Hq, Hkv, T, prefix, rule):
    ensure_lib()
    labels, S, W = [0, 1] * (Hkv // 2), 5, 130
    n = prefix + T
    q, k, v = (randn_bf16((B, n, h, d), 70 + i, "cuda") for i, h in enumerate((Hq, Hkv, Hkv)))
    lens = [T - b % 7 for b in range(B)]
    cache = aoh.Cache(B, Hq, Hkv, d, n, S, W, labels, chunk=rule)
    if prefix:
        cache.prefill(None, k[:, :prefix].contiguous(), v[:, :prefix].contiguous())
    qc, kc, vc = (x[:, prefix:].contiguous() for x in (q, k, v))
    out = torch.full_like(qc, float("nan"))
    cache.prefill(qc, kc, vc, out, seq_lens=lens)
    cache.check()
    kw = {"chunk": rule} if rule else {}
    for b in sorted({0, 1, 6, B // 2, B - 1}):
        end = prefix + lens[b]
        rows = np.arange(prefix, end)
        qn, kn, vn = (f64(x[b, :end]) for x in (q, k, v))
        want = oatt.prefill(qn, kn, vn, labels, S, W, rows=rows, **kw)
        mag = oatt.prefill(qn, kn, np.abs(vn), labels, S, W, rows=rows, **kw)
        assert_matches(f64(out[b, :lens[b]]), want, f"b={b}", mag)
    cache.close()
