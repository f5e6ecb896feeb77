"""The alpha grid search around the edges of its attention tiles (64 keys, 128 and 256 queries), with more alphas than one launch
takes, several slices of ragged length, Values far from unit scale, and the two-plane form of 16-bit codes."""
import numpy as np
import pytest
import torch

from oracle import pmkvq_oracle as O

pytestmark = pytest.mark.gpu


def _tensors(n_tokens, n_seq, kv_heads, group, seed, v_scale=1.0):
    g = torch.Generator().manual_seed(seed)
    k = torch.randn(n_tokens, n_seq, kv_heads, 128, generator=g)
    k[..., 9] *= 25.0
    q = torch.randn(n_tokens, n_seq, kv_heads * group, 128, generator=g)
    v = torch.randn(n_tokens, n_seq, kv_heads, 128, generator=g) * v_scale
    return [t.to(torch.bfloat16) for t in (k, q, v)]


@pytest.mark.parametrize("n_tokens,n_seq,kv_heads,group,bits,n_alphas,v_scale", [
    (2, 1, 1, 1, 2, 1, 1.0), (63, 1, 2, 1, 4, 3, 1.0), (64, 2, 1, 2, 2, 5, 1.0), (65, 3, 1, 1, 2, 4, 1.0), (127, 1, 1, 2, 2, 2, 1.0),
    (128, 1, 2, 1, 4, 6, 2.0 ** 9), (129, 2, 2, 1, 2, 3, 2.0 ** -12), (191, 1, 1, 1, 2, 2, 1.0), (256, 1, 1, 2, 2, 9, 1.0),
    (258, 1, 1, 1, 4, 2, 1.0), (385, 1, 2, 1, 2, 2, 1.0), (513, 1, 1, 1, 8, 2, 1.0)])
def test_losses_match_the_oracle_at_tile_edges(n_tokens, n_seq, kv_heads, group, bits, n_alphas, v_scale):
    from paper_2505_18610_b200 import binding as B
    k, q, v = _tensors(n_tokens, n_seq, kv_heads, group, n_tokens, v_scale)
    alphas = np.arange(n_alphas) / max(1, n_alphas)
    want = O.attention_reconstruction_losses(k.float().numpy(), q.float().numpy(), v.float().numpy(), group, bits, alphas, pos_scale=2.0)
    _, got = B.alpha_grid_search(k.cuda(), q.cuda(), v.cuda(), bits, alphas=alphas, pos_scale=2.0)
    # as in test_calibration.py: both outputs are good to about 2^-20, the loss is a square of their difference
    assert np.allclose(got, want, rtol=2e-2 if bits == 8 else 2e-3, atol=0)


@pytest.mark.parametrize("group", [1, 2, 3, 5])
@pytest.mark.parametrize("n_tokens,n_seq,kv_heads,bits", [(1, 2, 1, 2), (17, 2, 3, 4), (64, 1, 2, 2), (127, 1, 1, 8), (128, 2, 2, 2), (129, 1, 2, 4)])
def test_pairs_of_heads_of_a_short_sequence(n_tokens, n_seq, kv_heads, group, bits):
    """Up to 128 tokens a CTA takes two query heads of a KV head, the last one of an odd group alone."""
    from paper_2505_18610_b200 import binding as B
    k, q, v = _tensors(n_tokens, n_seq, kv_heads, group, n_tokens)
    q *= torch.arange(1, kv_heads * group + 1).view(-1, 1) / (kv_heads * group)      # no two heads alike
    alphas = [0.0, 0.3, 0.5, 0.8, 1.0]
    want = O.attention_reconstruction_losses(k.float().numpy(), q.float().numpy(), v.float().numpy(), group, bits, alphas)
    _, got = B.alpha_grid_search(k.cuda(), q.cuda(), v.cuda(), bits, alphas=alphas)
    assert np.allclose(got, want, rtol=2e-2 if bits == 8 else 2e-3, atol=0)           # as above


@pytest.mark.parametrize("n_tokens", [65, 300])
def test_sixteen_bit_codes_lose_next_to_nothing(n_tokens):
    from paper_2505_18610_b200 import binding as B
    k, q, v = (t.cuda() for t in _tensors(n_tokens, 2, 2, 2, 5))
    _, l16 = B.alpha_grid_search(k, q, v, 16, alphas=[0.0, 0.5])
    _, l8 = B.alpha_grid_search(k, q, v, 8, alphas=[0.0, 0.5])
    # the step is 257 times finer; what is left is that and the arithmetic's 2^-20 of unit outputs
    assert np.all(l16 >= 0) and np.all(l16 < l8 / 100.0)


@pytest.mark.parametrize("v_scale", [1.0, 2.0 ** 9])
@pytest.mark.parametrize("n_tokens,n_seq,kv_heads,group", [(2, 1, 1, 1), (63, 2, 1, 2), (64, 1, 2, 2), (65, 2, 2, 2), (128, 1, 2, 1),
                                                           (129, 1, 1, 3), (256, 1, 1, 2), (300, 2, 2, 2)])
def test_sixteen_bit_losses_match_the_oracle_at_tile_edges(n_tokens, n_seq, kv_heads, group, v_scale):
    """The two-plane form.  Both outputs are good to 2^-20 of Values of unit size (root mean square), so the root of the loss is, by
    the triangle inequality; without a second plane a Key is good to 2^-12 and the root of the loss is off by 2^-13 or more."""
    from paper_2505_18610_b200 import binding as B
    k, q, v = _tensors(n_tokens, n_seq, kv_heads, group, 5, v_scale)
    alphas = [0.0, 0.3, 0.5, 1.0]
    want = O.attention_reconstruction_losses(k.float().numpy(), q.float().numpy(), v.float().numpy(), group, 16, alphas)
    _, got = B.alpha_grid_search(k.cuda(), q.cuda(), v.cuda(), 16, alphas=alphas)
    assert np.all(np.abs(np.sqrt(got) - np.sqrt(want)) <= 2.0 ** -20 * v_scale)


@pytest.mark.parametrize("offset", [1, 2, 4])
@pytest.mark.parametrize("bits", [4, 16])
def test_tensors_at_any_bf16_address(offset, bits):
    from paper_2505_18610_b200 import binding as B
    at_0 = [t.cuda() for t in _tensors(70, 2, 2, 2, 3)]
    shifted = []
    for t in at_0:
        buf = torch.zeros(t.numel() + 8, dtype=torch.bfloat16, device="cuda")
        buf[offset:offset + t.numel()] = t.flatten()
        shifted.append(buf[offset:offset + t.numel()].view(t.shape))
    _, want = B.alpha_grid_search(*at_0, bits, alphas=[0.0, 0.5])
    _, got = B.alpha_grid_search(*shifted, bits, alphas=[0.0, 0.5])
    assert np.allclose(got, want, rtol=1e-12, atol=0)     # the same numbers, summed in fp64 in another order
