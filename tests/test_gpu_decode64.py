"""Decode at d_head 64 on the tensor cores, where an MMA row holds two
neighbouring keys, against the oracle: odd lengths and capacities (an item's
last pair holds one key), rings of one row, tiles of 256 keys at their edges,
every group size, whole clusters and the stream-K split. The cache starts
filled with NaN, so a key that the item does not hold must not reach a result."""

import numpy as np
import pytest
import torch

from gpu_cases import bf16_round, ensure_lib, f64, run_case
from oracle import attention as oatt
from paper_2608_06849_gb300 import aoh
from paper_2608_06849_gb300.workloads import Workload, decode_inputs, randn_bf16

pytestmark = pytest.mark.gpu

CASES = {
    # name: (B, Hq, Hkv, T, S, W, labels, seq_lens, steps)
    "odd_then_even_lengths": (1, 8, 2, 254, 3, 60, [0, 1], None, 5),
    "tile_edges": (2, 8, 2, 513, 0, 255, [0, 1], [513, 255], 3),
    "one_key_and_two": (3, 4, 2, 3, 0, 1, [0, 1], [1, 2, 3], 3),
    "ring_of_one_row": (1, 7, 1, 5, 0, 1, [1], None, 4),
    "odd_ring_wraps": (1, 16, 2, 40, 2, 5, [1, 0], None, 20),
    "group1_many_items": (5, 8, 8, 700, 4, 129, [0, 1, 0, 0, 1, 0, 1, 0], [700, 1, 255, 256, 257], 2),
    "group2_several_clusters": (1, 4, 2, 9000, 16, 1023, [0, 1], None, 2),
    "group7_stream_k": (9, 28, 4, 1300, 5, 200, [0, 1, 0, 0], [1300, 1, 2, 511, 512, 513, 700, 1299, 300], 2),
    "group8_stream_k_long": (5, 64, 8, 6001, 16, 700, [0, 1, 0, 0, 1, 0, 0, 0], None, 2),
    "group4_whole_tiles": (1, 16, 4, 4095, 16, 1008, [0, 1, 0, 1], None, 2),
}


@pytest.fixture
def nan_cache(monkeypatch):
    init = aoh.Cache.__init__

    def filled(self, *args, **kw):
        init(self, *args, **kw)
        self.buffer.fill_(0xFF)  # every bf16 a NaN

    monkeypatch.setattr(aoh.Cache, "__init__", filled)


@pytest.mark.parametrize("name", sorted(CASES))
def test_decode64(name, nan_cache):
    B, Hq, Hkv, T, S, W, labels, lens, steps = CASES[name]
    run_case(B, Hq, Hkv, 64, T, S, W, labels, seq_lens=lens, decode_steps=steps, check_prefill_out=False)


def test_weights_keep_fp32_precision():
    """Only the bf16 output rounds noticeably: beyond storing the exact value in
    bf16 the error stays within 2^-17 of the weighted |v| (softmax weights are
    carried as three bf16 parts; fp32 sums over 3,000 keys), where weights
    rounded to bf16 would miss by up to 2^-9 of it."""
    ensure_lib()
    B, Hq, Hkv, T, S, W, labels = 1, 16, 2, 3000, 4, 600, [0, 1]
    wl = Workload("p64", B, Hq, Hkv, 64, T, 1, S, W, 1, seed=2)
    cache = aoh.Cache(B, Hq, Hkv, 64, T + 1, S, W, labels)
    k, v = randn_bf16((B, T, Hkv, 64), 5, "cuda"), randn_bf16((B, T, Hkv, 64), 6, "cuda")
    cache.prefill(None, k, v)
    q, kn, vn = decode_inputs(wl, 0, device="cuda")
    out = torch.empty_like(q)
    cache.decode_step(q, kn, vn, out)
    kk, vv = np.concatenate([f64(k[0]), f64(kn)]), np.concatenate([f64(v[0]), f64(vn)])
    want = oatt.decode_step(f64(q[0]), kk, vv, labels, S, W)
    mag = oatt.decode_step(f64(q[0]), kk, np.abs(vv), labels, S, W)
    assert (np.abs(f64(out[0]) - want) <= np.abs(bf16_round(want) - want) + 2.0 ** -17 * mag).all()
    cache.close()
