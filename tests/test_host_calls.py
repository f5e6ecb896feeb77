"""The native host path of the token loop: which arguments it refuses and with which exception, the caller's own output and
stream."""
import pytest
import torch

from paper_2505_18610_b200 import binding as B
from paper_2505_18610_b200 import build


def test_the_extension_is_rebuilt_for_another_torch(monkeypatch):
    build.build()
    assert not build.needs_build()
    made = []
    monkeypatch.setattr(build, "_build_library", lambda verbose: made.append("library"))
    monkeypatch.setattr(build, "_build_host_calls", lambda: made.append("extension"))
    monkeypatch.setattr(build, "HOST_FOR", build.HOST_FOR.replace(torch.__version__, "2.0.0+cu118"))
    assert build.needs_build()
    build.build()
    assert made == ["extension"]                  # the CUDA library does not depend on torch


def test_nvcc_may_be_a_name_on_the_path(monkeypatch, tmp_path):
    home = tmp_path / "toolkit"
    (home / "bin").mkdir(parents=True)
    (home / "bin" / "nvcc").write_text("#!/bin/sh\n")
    (home / "bin" / "nvcc").chmod(0o755)
    (tmp_path / "bin").mkdir()
    (tmp_path / "bin" / "nvcc").symlink_to(home / "bin" / "nvcc")
    monkeypatch.setenv("PATH", str(tmp_path / "bin"))
    ran = []
    monkeypatch.setattr(build.subprocess, "run", lambda cmd, **kw: ran.append(cmd) or build.subprocess.CompletedProcess(cmd, 0, "", ""))
    for name in ("nvcc", str(tmp_path / "bin" / "nvcc"), str(home / "bin" / "nvcc")):
        monkeypatch.setenv("NVCC", name)
        build._build_host_calls()
        assert "-I" + str(home / "include") in ran[-1]


def test_refusals_without_a_device():
    B.lib()
    x = torch.zeros(1, 1, 128, dtype=torch.bfloat16)
    with pytest.raises(ValueError, match="k must be a contiguous CUDA tensor of torch.bfloat16"):
        B._calls.append(0, 0, x, x, 128, None)
    with pytest.raises(ValueError, match="q must be a contiguous CUDA tensor"):
        B._calls.decode_attention(0, 0, x, 1, 1, None, None)
    with pytest.raises(TypeError):
        B._calls.append(0, 0, None, x, 128, None)
    with pytest.raises(TypeError):
        B._calls.append(0, 0.5, x, x, 128, None)
    with pytest.raises(TypeError):
        B._calls.append(0, 0, x, x, 128)
    with pytest.raises(B.PmkvqError) as e:
        B._calls.restore_layer_state(0, 0, 1, 16)
    assert e.value.status == B.INVALID_ARG and "pmkvq_restore_layer_state" in str(e.value)


@pytest.mark.gpu
def test_shapes_outputs_and_streams():
    # which warp takes which tile may differ from call to call: the probabilities' 11 significant bits are rounded against another
    # maximum, 2^-11 of Values of magnitude 4 at most
    def same(a, b):
        torch.testing.assert_close(a, b, rtol=0, atol=4 * 2.0 ** -11)

    c = B.Cache(2, 8, 2, 3, 64, [4, 4], window=16)
    g = torch.Generator(device="cuda").manual_seed(1)
    k, v = (torch.randn(20, 3, 2, 128, device="cuda", generator=g).bfloat16() for _ in range(2))
    q = torch.randn(2, 3, 8, 128, device="cuda", generator=g).bfloat16()
    for bad_k, bad_v in ((k[:, :, :1].contiguous(), v), (k, v[:19]), (k[0, 0, 0], v[0, 0, 0])):
        with pytest.raises(ValueError, match="bad K/V shape"):
            c.append(0, bad_k, bad_v)
    for bad in (k.transpose(1, 2), k.float(), k.cpu()):
        with pytest.raises(ValueError, match="k must be"):
            c.append(0, bad, v)
    with pytest.raises(IndexError):
        c.append(0, k[0, 0, 0, 0], v[0, 0, 0, 0])
    with pytest.raises(B.PmkvqError) as e:
        c.append(2, k, v)
    assert e.value.status == B.INVALID_ARG and c.append(2, k, v, check=False) == B.INVALID_ARG
    assert c.append(0, k, v) == B.OK and c.append(1, k, v) == B.OK
    with pytest.raises(ValueError, match="bad Q shape"):
        c.decode_attention(0, q)
    with pytest.raises(ValueError, match="out must be a contiguous CUDA tensor of torch.float32"):
        c.decode_attention(0, q[0], out=q[0])
    with pytest.raises(ValueError, match="bad K/V/Q shape"):
        c.decode_step(k[:1], v[:1], q)
    with pytest.raises(ValueError, match="bad out shape"):
        c.decode_step(k[:2], v[:2], q, out=torch.empty(1, 3, 8, 128, device="cuda"))
    want = c.decode_attention(1, q[1])
    assert want.shape == (3, 8, 128) and want.dtype == torch.float32 and want.device == q.device
    mine = torch.full_like(want, float("nan"))
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    assert c.decode_attention(1, q[1], out=mine, stream=side) is mine
    side.synchronize()
    same(mine, want)
    with torch.cuda.stream(side):       # the current stream is the caller's, not the default one
        step = c.decode_step(k[:2], v[:2], q)
        assert c.layer_state(1)["n_tokens"] == 21
        c.restore_layer_state(0, 20, 16), c.restore_layer_state(1, 20, 16)
        mine = torch.empty_like(step)
        assert c.decode_step(k[:2], v[:2], q, out=mine) is mine
    side.synchronize()
    same(mine, step)
    c.close()
    with pytest.raises(B.PmkvqError):
        c.append(0, k, v)


@pytest.mark.gpu
def test_an_output_too_small_for_the_result_is_refused():
    c = B.Cache(1, 8, 2, 3, 64, [4], window=16)
    k = torch.randn(20, 3, 2, 128, device="cuda").bfloat16()
    q = torch.randn(3, 8, 128, device="cuda").bfloat16()
    c.append(0, k, k)
    launches = c.launch_count()
    for shape in ((3, 8, 127), (2, 8, 128), (0,)):
        with pytest.raises(ValueError, match="bad out shape"):
            c.decode_attention(0, q, out=torch.empty(shape, device="cuda"))
    assert c.launch_count() == launches
    want = c.decode_attention(0, q)
    large = torch.zeros(4 * 8 * 128, device="cuda")
    assert c.decode_attention(0, q, out=large) is large
    torch.testing.assert_close(large[:want.numel()], want.flatten(), rtol=0, atol=4 * 2.0 ** -11)   # as in `same` above
    assert not large[want.numel():].any()


@pytest.mark.gpu
def test_an_output_off_a_16_byte_boundary_is_refused():
    c = B.Cache(2, 2, 1, 1, 64, [4, 4])
    k = torch.randn(20, 1, 1, 128, device="cuda").bfloat16()
    q = torch.randn(2, 1, 2, 128, device="cuda").bfloat16()
    for layer in range(2):
        c.append(layer, k, k)
    launches = c.launch_count()
    buf = torch.zeros(2 * 2 * 128 + 4, device="cuda")
    for off in (1, 2, 3):
        one, two = buf[off:off + 256].view(1, 2, 128), buf[off:off + 512].view(2, 1, 2, 128)
        for call in (lambda: c.decode_attention(0, q[0], out=one), lambda: c.decode_attention_static(0, q[0], one),
                     lambda: c.decode_attention_all(q, out=two), lambda: c.decode_step(k[:2], k[:2], q, out=two)):
            with pytest.raises(B.PmkvqError) as e:
                call()
            assert e.value.status == B.INVALID_ARG
    assert c.launch_count() == launches and c.layer_state(0)["n_tokens"] == c.layer_state(1)["n_tokens"] == 20
    got = c.decode_attention_all(q, out=buf[4:].view(2, 1, 2, 128))
    torch.testing.assert_close(got, c.decode_attention_all(q), rtol=0, atol=4 * 2.0 ** -11)
