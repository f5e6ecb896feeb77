"""Decode steps whose attention launch starts under the step's append: a new Value far larger than every one before it."""
import numpy as np
import pytest
import torch

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
