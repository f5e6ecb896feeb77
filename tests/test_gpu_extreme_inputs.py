"""Numbers at the ends of their range in decode attention: Values that are not finite, queries near the largest exponent the kernels
carry."""
import pytest
import torch

from tests.helpers import Mirror, make_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits", [2, 4, 8, 16])
def test_rolled_back_token_with_infinite_value(bits, attention_path):
    """The largest Value scale of a slice stays infinite after the token is rolled back; attention over the rest is what it was."""
    n, kvh, group = 300, 2, 4
    k, v = make_inputs(32, 0, n + 1, 1, kvh)
    m = Mirror(1, group * kvh, kvh, 1, n + 1, [bits], window=32, attention_path=attention_path)
    m.cache.restore_layer_state(0, 0, bits)
    m.oracles[0].p.cur_bits = bits
    m.append(0, k[:n], v[:n])
    bad = v[n:].clone()
    bad[..., 17] = float("inf")
    m.cache.append(0, k[n:].cuda(), bad.cuda())
    m.cache.restore_layer_state(0, n, bits)
    q = torch.randn(1, group * kvh, 128, generator=torch.Generator().manual_seed(3)).bfloat16()
    m.check_attention(0, q)
