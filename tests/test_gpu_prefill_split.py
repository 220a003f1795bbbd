"""Prefill calls small enough that clusters of two CTAs share each work item,
around the rule's edges (seven visited tiles, 76 items), and larger ones whose last
wave is shared, against the oracle: odd lengths, a cached prefix, streaming heads
whose halves see no key of some rows, the chunk-eviction rule."""

import numpy as np
import pytest
import torch

from gpu_cases import assert_matches, ensure_lib, f64, run_case
from oracle import attention as oatt
from paper_2608_06849_gb300 import aoh
from paper_2608_06849_gb300.workloads import randn_bf16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hq,Hkv,d,T,S,W,labels,lens", [
    (1, 8, 2, 128, 768, 4, 60, [0, 1], None),             # six tiles: not split
    (1, 8, 2, 128, 769, 4, 60, [0, 1], None),             # seven
    (1, 8, 2, 64, 1025, 16, 100, [0, 1], None),           # a last item of one row
    (2, 12, 2, 128, 800, 200, 130, [1, 0], [800, 513]),   # ragged, sinks past a tile
    (1, 4, 4, 128, 2300, 0, 1, [1, 0, 1, 0], None),       # a window of one
    (1, 16, 2, 64, 1100, 4, 60, [0, 1], None),            # 72 items
])
def test_small_calls(B, Hq, Hkv, d, T, S, W, labels, lens):
    run_case(B, Hq, Hkv, d, T, S, W, labels, seq_lens=lens)


@pytest.mark.parametrize("d,rule", [(128, 0), (64, 0), (128, 300)])
def test_after_a_cached_prefix(d, rule):
    """A second chunk reads the first one's rows through the cache tiles."""
    ensure_lib()
    Hq, Hkv, S, W, labels, cut, T = 8, 2, 5, 130, [0, 1], 600, 1111
    q, k, v = (randn_bf16((1, T, h, d), 40 + h, "cuda") for h in (Hq, Hkv, Hkv + 1))
    v = v[:, :, :Hkv].contiguous()
    cache = aoh.Cache(1, Hq, Hkv, d, T, S, W, labels, chunk=rule)
    got = []
    for a, b in ((0, cut), (cut, T)):
        out = torch.full_like(q[:, a:b], float("nan")).contiguous()
        cache.prefill(*(x[:, a:b].contiguous() for x in (q, k, v)), out)
        got.append(f64(out[0]))
    cache.check()
    assert cache.lens() == [T]
    qn, kn, vn = f64(q[0]), f64(k[0]), f64(v[0])
    kw = {"chunk": rule} if rule else {}
    want = oatt.prefill(qn, kn, vn, labels, S, W, **kw)
    mag = oatt.prefill(qn, kn, np.abs(vn), labels, S, W, **kw)
    assert_matches(np.concatenate(got), want, "two chunks", mag)
    cache.close()


@pytest.mark.parametrize("d,B,Hq,Hkv,light,T,prefix", [
    (128, 20, 8, 1, 0, 256, 1280),   # 160 items: the 8 past the first wave are shared
    (64, 33, 7, 1, 1, 200, 2048),    # 231: 76 shared, then three light ones and an entry without work
    (128, 4, 32, 4, 0, 300, 1500),   # 192 items of three tiles a sequence: a wave of whole ones, then 40 shared
    (128, 4, 25, 5, 1, 250, 2999),   # 100: the 75 heavy ones and one light one shared
])
def test_last_wave_shared(d, B, Hq, Hkv, light, T, prefix):
    """Chunks after a long prefix whose last wave of items is shared; `light`
    sequences have a prefix of one token."""
    ensure_lib()
    labels, S, W = [0] * Hkv, 4, 60
    pk, pv, k, v = (randn_bf16((B, n, Hkv, d), 50 + i, "cuda") for i, n in enumerate((prefix, prefix, T, T)))
    q = randn_bf16((B, T, Hq, d), 60, "cuda")
    before = [prefix] * (B - light) + [1] * light
    lens = [T - b % 3 for b in range(B)]
    cache = aoh.Cache(B, Hq, Hkv, d, prefix + T, S, W, labels)
    cache.prefill(None, pk, pv, seq_lens=before)
    out = torch.full_like(q, float("nan"))
    cache.prefill(q, k, v, out, seq_lens=lens)
    cache.check()
    for b in sorted({0, 152 // Hq, 228 // Hq, B - 1} & set(range(B))):
        n = before[b] + lens[b]
        rows = np.arange(before[b], n)
        kn, vn = (np.concatenate([f64(x[b, :before[b]]), f64(y[b, :lens[b]])]) for x, y in ((pk, k), (pv, v)))
        qn = np.concatenate([np.zeros((before[b], Hq, d)), f64(q[b, :lens[b]])])
        want = oatt.prefill(qn, kn, vn, labels, S, W, rows=rows)
        mag = oatt.prefill(qn, kn, np.abs(vn), labels, S, W, rows=rows)
        assert_matches(f64(out[b, :lens[b]]), want, f"b={b}", mag)
    cache.close()


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("group", [1, 2, 7, 8])
def test_items_of_two_heads(d, group):
    """An item is one query tile of two heads, or two tiles of an odd group's last
    head: lengths around both, more items than SMs at the larger groups."""
    run_case(6, 4 * group, 4, d, 641, 130, 129, [0, 1, 0, 1], seq_lens=[641, 1, 127, 128, 129, 385])


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("T", [512, 1024])
def test_a_nan_row_whose_weight_rounds_to_zero(d, T):
    """Keys of the first half of the rows score 300 below the others' for the last
    rows: zero times the NaN in a visible V row is NaN, in items of one CTA (512
    rows) and of two (1024) alike. Columns without a NaN row stay finite."""
    ensure_lib()
    cache = aoh.Cache(1, 8, 8, d, T, 4, 60, [0] * 8)
    u = torch.full((d,), d ** -0.5, device="cuda")
    c = (150 * d ** 0.5) ** 0.5  # the scores are +-150
    sign = torch.where(torch.arange(T, device="cuda") < T // 2, -1.0, 1.0).view(1, T, 1, 1)
    q = (c * u).expand(1, T, 8, d).to(torch.bfloat16).contiguous()
    k = (c * u * sign).expand(1, T, 8, d).to(torch.bfloat16).contiguous()
    v = randn_bf16((1, T, 8, d), 71, "cuda")
    v[0, 5, :, 3] = float("nan")
    out = torch.empty_like(q)
    cache.prefill(q, k, v, out)
    cache.check()
    late = out[0, T // 2 + 128:]
    assert torch.isnan(late[..., 3]).all()
    assert torch.isfinite(late[..., [x for x in range(d) if x != 3]]).all()
    cache.close()
