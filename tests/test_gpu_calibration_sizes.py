"""Abs-max calibration at the edges of its work split: fewer and more tokens than a CTA takes, sequence counts around the
unrolled and the split loop, head counts that do and do not divide the eight vector slots of a CTA, more than eight
heads, and Keys at an address that allows no 16-byte load."""
import numpy as np
import pytest
import torch

from oracle import pmkvq_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_tokens,n_seq,kv_heads,offset", [
    (1, 1, 1, 0), (3, 5, 3, 0), (4, 31, 1, 0), (5, 33, 1, 1), (17, 4, 8, 0), (17, 3, 8, 4), (9, 7, 5, 0), (33, 2, 11, 0),
    (70, 65, 8, 0), (6, 257, 4, 0), (10000, 1, 2, 0)])
def test_absmax_work_split_edges(n_tokens, n_seq, kv_heads, offset):
    from paper_2505_18610_b200 import binding as B
    n = n_tokens * n_seq * kv_heads * 128
    flat = torch.randn(n, generator=torch.Generator().manual_seed(n)).to(torch.bfloat16)
    buf = torch.zeros(n + 8, dtype=torch.bfloat16, device="cuda")
    buf[offset:offset + n] = flat.cuda()
    k = buf[offset:offset + n].view(n_tokens, n_seq, kv_heads, 128)
    want = O.calibrate_lambda(flat.float().numpy().reshape(n_tokens, n_seq, kv_heads, 128), pos_scale=2.0, alpha=1.0)
    got = B.calibrate_lambda(k, pos_scale=2.0, alpha=1.0).cpu().numpy()
    # fp32 rotation from correctly rounded angles: two products and a sum, each within half an ulp, and the power
    assert np.allclose(got, want, rtol=2e-6, atol=0)


def test_calibration_reads_a_nan_as_a_channel_without_a_maximum():
    """A channel that saw a NaN gets the floor, whatever else it saw; the others keep their maxima."""
    from paper_2505_18610_b200 import binding as B
    k = torch.randn(9, 5, 3, 128, generator=torch.Generator().manual_seed(4)).bfloat16()
    clean = B.calibrate_lambda(k.cuda(), alpha=1.0, floor_value=0.125).cpu()
    k[0, 2, 1, 7] = float("nan")                     # channels 7 and 71 are rotated into one another
    k[8, 4, 2, 100] = float("nan")
    got = B.calibrate_lambda(k.cuda(), alpha=1.0, floor_value=0.125).cpu()
    want = clean.clone()
    want[1, 7] = want[1, 71] = want[2, 36] = want[2, 100] = 0.125
    assert torch.equal(got, want)


@pytest.mark.parametrize("t", [1, 5, 100, 1500])
def test_rotation_of_one_token_bit_for_bit(t):
    """Two products, each rounded, and their rounded sum: the Key that pmkvq_append would be given."""
    from paper_2505_18610_b200 import binding as B
    k = torch.zeros(t + 1, 1, 8, 128)
    k[t] = torch.randn(1, 8, 128, generator=torch.Generator().manual_seed(t))
    k = k.bfloat16()
    angle = np.float64(t) * 10000.0 ** (-2.0 * np.arange(64) / 128)
    c, s = np.cos(angle).astype(np.float32), np.sin(angle).astype(np.float32)
    x1, x2 = k[t, 0, :, :64].float().numpy(), k[t, 0, :, 64:].float().numpy()
    want = np.abs(np.concatenate([x1 * c - x2 * s, x1 * s + x2 * c], -1))
    got = B.calibrate_lambda(k.cuda(), alpha=1.0, floor_value=1e-30).cpu().numpy()
    assert np.array_equal(got, want)
