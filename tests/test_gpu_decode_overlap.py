"""Decode steps whose attention launch starts under the step's append: a new Value far larger than every one before it, and
input buffers that are overwritten between the steps."""
import numpy as np
import pytest
import torch

from paper_2505_18610_b200.binding import Cache
from tests.helpers import Mirror, make_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits", [2, 4])
@pytest.mark.parametrize("window", [0, 1])
def test_new_value_far_above_all_earlier_ones(bits, window):
    """window = 0: the new token enters the body in the same append that raises the slice's largest Value scale, in a tile
    that is a late step of its warp (two CTAs on 2000 tokens x 2 slices: 63 tiles and more per warp)."""
    context, steps, kvh, group = 2000, 4, 2, 4
    k, v = make_inputs(21, 0, context + steps, 1, kvh, n_outlier=0)
    v = v.float()
    for s in range(steps):
        v[context + s] *= 64.0 ** (s + 1)
    v = v.to(torch.bfloat16)
    m = Mirror(1, kvh * group, kvh, 1, context + steps, [bits], window=window)
    m.cache.restore_layer_state(0, 0, bits)
    m.oracles[0].p.cur_bits = bits
    m.append(0, k[:context], v[:context])
    m.cache.set_attention_ctas(2)
    # every query head asks for the newest token (its score is |k|^2 / 11.3 = 11, the others' are N(0, 1))
    q = k[context:].repeat_interleave(group, dim=2).contiguous().cuda()         # [steps, 1, heads, 128]
    K, V = k[context:, None].cuda().contiguous(), v[context:, None].cuda().contiguous()
    got = [m.cache.decode_step(K[s], V[s], q[s][None].contiguous()) for s in range(steps)]    # nothing waits in between
    torch.cuda.synchronize()
    for s in range(steps):
        t = context + s
        m.oracles[0].append(k[t:t + 1].float().numpy().reshape(1, kvh, 128), v[t:t + 1].float().numpy().reshape(1, kvh, 128))
        ref = m.oracles[0].decode_attention(q[s].float().cpu().numpy().reshape(kvh, group, 128))
        out = got[s].cpu().numpy().reshape(kvh, group, 128).astype(np.float64)
        assert np.all(np.isfinite(out))
        # the stated tolerance, relative to outputs of the magnitude of the new Value
        assert np.abs(out - ref).max() <= 2e-3 * max(1.0, np.abs(ref).max())
        assert np.linalg.norm(out - ref) <= 1e-3 * np.linalg.norm(ref)
    m.check_state(0)


@pytest.mark.parametrize("evict_chunk", [1, 16])
def test_inputs_rewritten_between_steps(evict_chunk):
    """One buffer each for K, V and Q, overwritten on the stream before every step, and Values that grow by a factor of 8 from step to
    step, so the body's unit, read under the append, and the window's differ in each; several steps of body tiles per warp."""
    layers, batch, kvh, hq, context, steps = 4, 2, 2, 8, 4100, 20
    mk = lambda: Cache(layers, hq, kvh, batch, context + steps, [2, 4, 8, 16], window=64, evict_chunk=evict_chunk)  # noqa: E731
    a, b = mk(), mk()
    for layer in range(layers):
        k, v = make_inputs(22, layer, context, batch, kvh)
        for c in (a, b):
            c.append(layer, k.cuda().contiguous(), v.cuda().contiguous())
    a.set_attention_ctas(8)
    K, V = (torch.stack(x, 1).cuda().contiguous() for x in
            zip(*[make_inputs(23, layer, steps, batch, kvh, pos0=context) for layer in range(layers)]))
    scale = torch.tensor([8.0 ** s for s in range(steps)], device="cuda")
    V = (V.float() * scale.view(-1, 1, 1, 1, 1)).bfloat16()
    Q = torch.randn(steps, layers, batch, hq, 128, generator=torch.Generator().manual_seed(6)).bfloat16().cuda()
    kb, vb, qb = torch.empty_like(K[0]), torch.empty_like(V[0]), torch.empty_like(Q[0])
    got = []
    for s in range(steps):
        kb.copy_(K[s]), vb.copy_(V[s]), qb.copy_(Q[s])
        got.append(a.decode_step(kb, vb, qb))
    torch.cuda.synchronize()
    for s in range(steps):
        for layer in range(layers):
            b.append(layer, K[s, layer], V[s, layer])
            torch.cuda.synchronize()
            want = b.decode_attention(layer, Q[s, layer])
            # two partitions of one sum (the bound of the split-invariance test), relative to outputs of this size
            assert float((got[s][layer] - want).abs().max()) <= 1e-3 * max(1.0, float(want.abs().max()))
