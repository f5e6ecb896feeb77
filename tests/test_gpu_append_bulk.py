"""Bulk appends at the sizes where the one-launch kernel can go wrong: runs around a tile, around the ring and around
several rings (a new window token then lands in the slot of a token that leaves the window in the same launch), ragged
starts, every body width, evictions one by one and in groups; and decode steps enqueued back to back, whose attention
launch may start while the append in front of it still runs."""
import numpy as np
import pytest
import torch

from paper_2505_18610_b200 import binding as B
from paper_2505_18610_b200 import synth
from tests.helpers import Mirror, make_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits", [2, 4, 8, 16])
@pytest.mark.parametrize("window,evict_chunk,n_sink,sizes", [
    (32, 1, 1, (1, 2, 15, 16, 17, 31, 47, 48, 49, 64, 97, 200)),
    (32, 8, 5, (3, 33, 16, 40, 2, 130, 63)),
    (0, 1, 0, (5, 16, 27, 2, 32)),
    (128, 16, 1, (100, 45, 143, 144, 145, 161, 7)),
    (200, 1, 17, (217, 1, 16, 208, 15, 33, 400, 31)),
    (64, 16, 0, (64, 16, 80, 5, 96, 11, 64, 160, 48)),
])
def test_append_runs_around_tile_and_ring_edges(bits, window, evict_chunk, n_sink, sizes):
    total = sum(sizes)
    k, v = make_inputs(7, 0, total, 2, 2)
    lam = synth.make_lambda(k[:64]).numpy()[None]
    # a cache whose budget asks for `bits` from the first token on
    m = Mirror(1, 4, 2, 2, total, [bits], lam=lam, window=window, evict_chunk=evict_chunk, n_sink=n_sink)
    m.cache.restore_layer_state(0, 0, bits)
    m.oracles[0].p.cur_bits = bits
    done = 0
    for n in sizes:
        m.append(0, k[done:done + n], v[done:done + n])
        done += n
        m.check_state(0)


def test_append_of_inputs_no_16_byte_load_can_take():
    k, v = make_inputs(9, 0, 300, 1, 2)
    m = Mirror(1, 2, 2, 1, 300, [4], window=32)
    dev = []
    for x in (k, v):
        buf = torch.empty(x.numel() + 4, dtype=torch.bfloat16, device="cuda")
        buf[4:] = x.cuda().view(-1)                 # 8 bytes behind a 256-byte boundary
        dev.append(buf[4:].view(x.shape))
    m.cache.append(0, dev[0], dev[1])
    m.oracles[0].append_bulk(k.float().numpy().reshape(300, 2, 128), v.float().numpy().reshape(300, 2, 128))
    m.check_state(0)


@pytest.mark.parametrize("evict_chunk", [1, 16])
@pytest.mark.parametrize("context,batch", [(20, 1), (300, 2), (2100, 3)])
def test_back_to_back_decode_steps_equal_separate_calls(context, batch, evict_chunk):
    layers, kvh, hq, steps = 3, 2, 8, 24
    mk = lambda: Mirror(layers, hq, kvh, batch, context + steps, [4, 2, 16], window=64, evict_chunk=evict_chunk)  # noqa: E731
    a, b = mk(), mk()
    for l in range(layers):
        k, v = make_inputs(3, l, context, batch, kvh)
        for m in (a, b):
            m.cache.append(l, k.cuda().contiguous(), v.cuda().contiguous())
    kv = [make_inputs(4, l, steps, batch, kvh, pos0=context) for l in range(layers)]
    K = torch.stack([x[0] for x in kv], 1).cuda().contiguous()
    V = torch.stack([x[1] for x in kv], 1).cuda().contiguous()
    Q = torch.randn(steps, layers, batch, hq, 128, generator=torch.Generator().manual_seed(5)).bfloat16().cuda()
    together = [a.cache.decode_step(K[s], V[s], Q[s]) for s in range(steps)]      # nothing waits in between
    torch.cuda.synchronize()
    for s in range(steps):
        for l in range(layers):
            b.cache.append(l, K[s, l], V[s, l])
            torch.cuda.synchronize()
            want = b.cache.decode_attention(l, Q[s, l])
            torch.cuda.synchronize()
            got = together[s][l]
            # two partitions of one sum at the kernels' precision (the bound of the split-invariance test)
            assert float((got - want).abs().max()) <= 1e-3
    for l in range(layers):
        for s in range(batch * kvh):
            for is_v in (False, True):
                for x, y in zip(a.cache.export_slice(l, s // kvh, s % kvh, is_v), b.cache.export_slice(l, s // kvh, s % kvh, is_v)):
                    assert np.array_equal(x, y)


@pytest.mark.parametrize("shift_variant", [0, 1])
@pytest.mark.parametrize("bits", [2, 4, 8, 16])
@pytest.mark.parametrize("batch,sizes", [(1, (37, 250)), (32, (37, 700, 90, 513))])
def test_appends_of_one_and_of_two_warps_per_half_tile(bits, batch, sizes, shift_variant):
    """32 x 4 slices x 700 tokens take one warp per half tile, the rest two; constant tokens and scales outside the plain
    quotient's range, alone and beside ordinary ones in a tile."""
    total, kvh = sum(sizes), 4
    k, v = make_inputs(11, 0, total, batch, kvh)
    for t in (3, 40, 41, 130, 200):
        k[t], v[t] = 0.75, -1.5
    for t, f in ((5, 1e-25), (44, 1e25), (131, 1e-30), (201, 1e-36)):
        k[t], v[t] = k[t] * f, v[t] * f
    m = Mirror(1, kvh, kvh, batch, total, [bits], slices=sorted({0, 1, batch * kvh // 2, batch * kvh - 1}), window=64, evict_chunk=8,
               shift_variant=shift_variant)
    m.cache.restore_layer_state(0, 0, bits)
    m.oracles[0].p.cur_bits = bits
    done = 0
    for n in sizes:
        m.append(0, k[done:done + n], v[done:done + n])
        done += n
        m.check_state(0)


@pytest.mark.parametrize("bits", [2, 4, 8, 16])
@pytest.mark.parametrize("value", [float("inf"), -float("inf"), float("nan")])
def test_bulk_append_of_a_token_without_a_scale(bits, value):
    """A Value vector of infinities or NaNs has no scale: its codes are 0 as in the token-by-token append, and the token it shares
    words with is not touched."""
    n = 40
    k, v = make_inputs(33, 0, n, 1, 1)
    v[5], v[36] = value, value                       # one in the body, one in the window
    v[20], v[21] = value, 0.25                       # beside a constant token
    caches = [B.Cache(1, 1, 1, 1, n, [bits], window=16) for _ in range(2)]
    for c in caches:
        c.restore_layer_state(0, 0, bits)
    k, v = k.cuda(), v.cuda()
    caches[0].append(0, k, v)
    for t in range(n):
        caches[1].append(0, k[t], v[t])
    for is_v in (False, True):
        for x, y in zip(*(c.export_slice(0, 0, 0, is_v) for c in caches)):
            assert np.array_equal(x, y, equal_nan=x.dtype.kind == "f")
