"""The decode step's two splits at their edges, against the oracle: few items
run on whole clusters of 2, 4, 8 or 16 CTAs each (states added up in distributed
shared memory, items of several clusters through one global exchange), other
steps on the stream-K split. Tolerances are the parity suite's."""

import pytest
import torch

from gpu_cases import assert_matches, ensure_lib, f64, run_case
from paper_2608_06849_gb300 import aoh

pytestmark = pytest.mark.gpu

CASES = {
    # name: (B, Hq, Hkv, T, S, W, labels, seq_lens); head size 128
    "one_cluster_an_item": (1, 28, 4, 1000, 16, 500, [0, 1, 0, 1], None),
    "sixteen_ctas_an_item": (1, 28, 4, 2048, 16, 300, [0, 1, 0, 1], None),
    "several_clusters_an_item": (1, 28, 4, 4095, 128, 2048, [1, 0, 0, 1], None),
    "nine_clusters_an_item": (1, 8, 2, 9300, 4, 127, [0, 1], None),
    "whole_tiles": (1, 16, 2, 3071, 0, 1024, [0, 1], None),
    "a_row_past_whole_tiles": (1, 16, 2, 3073, 0, 1024, [0, 1], None),
    "many_items_lengths_one_to_2k": (8, 16, 4, 2049, 3, 130, [0, 1, 0, 0], [1, 126, 127, 128, 700, 2046, 2047, 2049]),
    "sixteen_heads_a_group": (1, 32, 2, 1500, 8, 100, [0, 1], None),
    "one_head_a_group": (2, 3, 3, 900, 4, 130, [1, 0, 0], [900, 257]),
    "all_streaming": (4, 16, 4, 600, 16, 240, [1, 1, 1, 1], [600, 1, 255, 256]),
    # more than 32 items: the stream-K split
    "stream_k_ragged": (9, 28, 4, 1500, 16, 300, [0, 1, 0, 0], [1500, 1, 2, 127, 128, 129, 700, 1499, 300]),
    "stream_k_group4": (11, 16, 4, 900, 4, 64, [0, 0, 1, 0], None),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_split(name):
    B, Hq, Hkv, T, S, W, labels, lens = CASES[name]
    run_case(B, Hq, Hkv, 128, T, S, W, labels, seq_lens=lens, decode_steps=2, check_prefill_out=False)


@pytest.mark.parametrize("batch", [8, 40])  # clusters, stream-K
def test_last_tile_of_every_warp_edge(batch, monkeypatch):
    """A last tile of 1 to 128 rows: cache rows past it hold NaNs, which a weight
    of zero would not hide."""
    init = aoh.Cache.__init__

    def filled(self, *args, **kw):
        init(self, *args, **kw)
        self.buffer.fill_(0xFF)  # every bf16 a NaN

    monkeypatch.setattr(aoh.Cache, "__init__", filled)
    lens = [(256 + r if i % 2 else r) for i, r in enumerate([30, 31, 32, 62, 63, 94, 126, 127] * (batch // 8))]
    run_case(batch, 7, 1, 128, 400, 4, 60, [0], seq_lens=lens, decode_steps=2, check_prefill_out=False)


def test_stream_k_two_merge_levels():
    """One item of 3.1M rows: past the length where whole clusters fit the rows
    as evenly as the stream-K split, whose 152 parts merge in two levels."""
    ensure_lib()
    T, G, D = 3100000, 7, 128
    g = torch.Generator(device="cuda").manual_seed(1)
    k, v = (torch.randn((1, T + 1, 1, D), generator=g, device="cuda", dtype=torch.bfloat16) for _ in range(2))
    q = torch.randn((1, G, D), generator=g, device="cuda", dtype=torch.bfloat16)
    cache = aoh.Cache(1, G, 1, D, T + 1, 4, 64, [0])
    cache.prefill(None, k[:, :T].contiguous(), v[:, :T].contiguous())
    out = torch.empty_like(q)
    cache.decode_step(q, k[:, T].contiguous(), v[:, T].contiguous(), out)
    cache.check()
    p = torch.softmax(q[0].double() @ k[0, :, 0].double().T / D ** 0.5, -1)
    want, mag = p @ v[0, :, 0].double(), p @ v[0, :, 0].double().abs()
    assert_matches(f64(out[0]), want.cpu().numpy(), "3.1M rows", mag.cpu().numpy())
    cache.close()
