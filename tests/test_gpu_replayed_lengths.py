"""Prefill chunks after replays of a captured graph: a replay moves the lengths on
the device alone, so the next chunk is placed by those and not by the handle's
copy, at any batch (65 takes the uploaded rows). Outputs against the oracle, the
cache image bit for bit."""

import numpy as np
import pytest
import torch

from gpu_cases import assert_matches, check_cache_image, ensure_lib, f64
from oracle import attention as oatt
from paper_2608_06849_gb300 import aoh
from paper_2608_06849_gb300.workloads import randn_bf16

pytestmark = pytest.mark.gpu


def _capture(call):
    """`call` as a graph; capturing it moves no length on the device."""
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        call()
    return graph


def _check_chunk(out, q, k, v, labels, S, W, start, lens, what):
    for b in range(len(lens)):
        L = start[b] + lens[b]
        rows = np.arange(start[b], L)
        qn, kn, vn = f64(q[b, :L]), f64(k[b, :L]), f64(v[b, :L])
        want = oatt.prefill(qn, kn, vn, labels, S, W, rows=rows)
        mag = oatt.prefill(qn, kn, np.abs(vn), labels, S, W, rows=rows)
        assert_matches(f64(out[b, :lens[b]]), want, f"{what} b={b}", mag)


@pytest.mark.parametrize("B,Hq,Hkv,d,labels", [(2, 8, 2, 128, [0, 1]), (3, 8, 2, 64, [1, 0]), (65, 2, 2, 64, [0, 1])])
def test_chunk_after_replayed_steps(B, Hq, Hkv, d, labels):
    """A prompt, five replays of one captured step, a chunk, two more replays, a
    captured chunk of one row replayed three times."""
    ensure_lib()
    S, W, steps, more, single = 4, 60, 5, 2, 3
    first = [150 - b % 7 for b in range(B)]
    lens = [140 - b % 5 for b in range(B)]
    T = 150 + steps + 140 + more + single
    q, k, v = (randn_bf16((B, T, h, d), 70 + i, "cuda") for i, h in enumerate((Hq, Hkv, Hkv)))
    cache = aoh.Cache(B, Hq, Hkv, d, T, S, W, labels)
    at = torch.zeros(B, dtype=torch.long, device="cuda")
    pick = lambda x, n: torch.stack([x[b, int(at[b]):int(at[b]) + n] for b in range(B)]).contiguous()
    cache.prefill(pick(q, 150), pick(k, 150), pick(v, 150), seq_lens=first)
    at += torch.tensor(first, device="cuda")

    sq, sk, sv = (pick(x, 1)[:, 0].clone() for x in (q, k, v))
    so = torch.empty_like(sq)
    step = _capture(lambda: cache.decode_step(sq, sk, sv, so))

    def replay(graph, n, bufs, out):
        for _ in range(n):
            for buf, x in zip(bufs, (q, k, v)):
                buf.copy_(pick(x, 1).view(buf.shape))
            graph.replay()
            _check_chunk(out.view(B, 1, Hq, d), q, k, v, labels, S, W, at.tolist(), [1] * B, "replay")
            at.add_(1)

    replay(step, steps, (sq, sk, sv), so)
    chunk = [pick(x, 140) for x in (q, k, v)]
    out = torch.full_like(chunk[0], float("nan"))
    cache.prefill(*chunk, out, seq_lens=lens)
    _check_chunk(out, q, k, v, labels, S, W, at.tolist(), lens, "chunk")
    at += torch.tensor(lens, device="cuda")
    replay(step, more, (sq, sk, sv), so)
    if B <= 64:  # more sequences upload their rows, which is not captured
        one = [pick(x, 1) for x in (q, k, v)]
        oo = torch.empty_like(one[0])
        replay(_capture(lambda: cache.prefill(*one, oo)), single, one, oo)
    cache.check()
    check_cache_image(cache, k, v, at.tolist(), labels, S, W)
    cache.close()


@pytest.mark.parametrize("B", [1, 65])
def test_chunk_that_replays_left_no_room_for(B):
    """max_seq 64, 40 tokens, 20 replays (60 on the device, 41 in the handle): a chunk
    of 10 passes the host's check, is left out on the device and reported once."""
    ensure_lib()
    Hq, Hkv, d, S, W, labels = 2, 2, 64, 4, 16, [0, 1]
    q, k, v = (randn_bf16((B, 64, h, d), 90 + i, "cuda") for i, h in enumerate((Hq, Hkv, Hkv)))
    cache = aoh.Cache(B, Hq, Hkv, d, 64, S, W, labels)
    cache.prefill(None, k[:, :40].contiguous(), v[:, :40].contiguous())
    so = torch.empty(B, Hq, d, dtype=torch.bfloat16, device="cuda")
    sq, sk, sv = (x[:, 40].clone() for x in (q, k, v))
    step = _capture(lambda: cache.decode_step(sq, sk, sv, so))
    for i in range(20):
        sk.copy_(k[:, 40 + i])
        sv.copy_(v[:, 40 + i])
        step.replay()
    cache.check()
    part = [x[:, 50:60].contiguous() for x in (q, k, v)]
    cache.prefill(*part, torch.empty_like(part[0]))
    with pytest.raises(aoh.AohError) as e:
        cache.check()
    assert e.value.status == 2
    cache.check()
    check_cache_image(cache, k, v, [60] * B, labels, S, W)
    sk.copy_(k[:, 60])
    sv.copy_(v[:, 60])
    step.replay()  # the lengths stayed
    cache.check()
    check_cache_image(cache, k, v, [61] * B, labels, S, W)
    cache.close()
