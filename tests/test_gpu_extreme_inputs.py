"""Numbers at the ends of their range in decode attention: Values that are not finite, queries near the largest exponent the kernels
carry."""
import numpy as np
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


@pytest.mark.parametrize("bits", [2, 4, 8, 16])
@pytest.mark.parametrize("d", [0, 3, 5])
def test_queries_up_to_two_to_the_116(bits, d, attention_path):
    """Tiny Keys and huge queries whose scores are ordinary: Q * lambda * scale * log2(e) reaches 2^(110 + d) and the cache holds
    Keys of 2^-(112 + d), INT16 scales around 2^-(122 + d)."""
    n, kvh, group = 500, 1, 4
    k, v = make_inputs(31, 0, n, 1, kvh)
    q = torch.randn(1, group, 128, generator=torch.Generator().manual_seed(2))
    m = Mirror(1, group, kvh, 1, n, [bits], lam=np.full((1, kvh, 128), 2.0 ** 10, np.float32), window=32, attention_path=attention_path)
    m.append(0, (k.float() * 2.0 ** -(102 + d)).to(torch.bfloat16), v)
    m.check_state(0)
    m.check_attention(0, (q * 2.0 ** (102 + d)).to(torch.bfloat16))
