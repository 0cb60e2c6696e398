"""The CPython binding and the ctypes path make the same calls: same results, same keys, same errors."""
import pytest
import torch

pytestmark = pytest.mark.gpu


class _Refuses:
    """Stands in for the binding and leaves every call to ctypes."""

    def __getattr__(self, name):
        return lambda *args: None


def both(monkeypatch, call):
    from paper_2502_05003_b200 import _lib
    real = _lib.binding()

    def outcome():
        try:
            return call()
        except Exception as e:                            # the two paths must raise alike
            return type(e), str(e)
    with monkeypatch.context() as m:
        m.setattr(_lib, "_binding", _Refuses())
        slow = outcome()
    assert _lib.binding() is real
    return outcome(), slow


def same(a, b):
    assert type(a) is type(b)
    if isinstance(a, torch.Tensor):
        assert a.dtype == b.dtype and a.shape == b.shape and torch.equal(a, b)
    elif isinstance(a, dict):
        assert list(a) == list(b)
        for k in a:
            if k != "workspace":
                same(a[k], b[k])
    elif isinstance(a, tuple):
        assert len(a) == len(b)
        for u, v in zip(a, b):
            same(u, v)
    else:
        assert a == b


def test_results_and_errors_are_those_of_the_ctypes_path(monkeypatch):
    import paper_2502_05003_b200 as q
    gen = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn((72, 256), generator=gen, device="cuda").bfloat16()
    w = torch.randn((48, 256), generator=gen, device="cuda").bfloat16()
    dy = torch.randn((72, 48), generator=gen, device="cuda").bfloat16()
    fwd = q.quest_linear_fwd(x, w, 4, 128)
    cached = {"wq": fwd["wq"], "sw": fwd["sw"]}
    xs, ws, _ = q.quest_quantize(x, 8, 128)
    calls = [
        lambda: q.quest_quantize(x, 4, 128), lambda: q.quest_quantize(x, 3, 64, 0.5, want_mask=False),
        lambda: q.quest_quantize(x, 4, 128, mask=torch.empty((72, 32), dtype=torch.uint8, device="cuda"), want_mask=False),
        lambda: q.quest_quantize(x[:, ::2], 4, 128), lambda: q.quest_quantize(x.cpu(), 4, 128), lambda: q.quest_quantize(x, 9, 128),
        lambda: q.quest_quantize(x, 4, 100), lambda: q.quest_quantize(x.half(), 4, 128), lambda: q.quest_quantize(x[1:, 4:], 4, 4),
        lambda: q.quest_linear_fwd(x, w, 4, 128, out_dtype=torch.float32), lambda: q.quest_linear_fwd(x, w, 1, 128, 1.3, want_masks=False),
        lambda: q.quest_linear_fwd(x, None, 4, 128, w_cached=cached), lambda: q.quest_linear_fwd(x, None, 4, 128),
        lambda: q.quest_linear_fwd(x, w, 0, 128), lambda: q.quest_linear_fwd(x, w, 4, 96), lambda: q.quest_linear_fwd(x, w, 4, 128, -1.0),
        lambda: q.quest_linear_fwd(x, w, 4, 128, out_dtype=torch.float16), lambda: q.quest_linear_fwd(x[:, :40], w[:, :40], 4, 8),
        lambda: q.quest_linear_fwd(x, w, 4, 128, saved={"xq": fwd["xq"].clone(), "other": 1}),
        lambda: q.quest_linear_fwd(x, w, 4, 128, workspace=torch.empty(256, dtype=torch.uint8, device="cuda")),
        lambda: q.quest_linear_fwd(x[:0], w, 4, 128),
        lambda: q.quest_lowbit_gemm(xs, ws, 8, xs[:8], ws[:8], 8, 256, want_acc=True),
        lambda: q.quest_lowbit_gemm(xs, ws, 8, xs[:8], ws[:8], 8, 256, want_y=False), lambda: q.quest_lowbit_gemm(xs, ws, 8, xs, ws, 8, 250),
        lambda: q.quest_lowbit_gemm(xs, None, 8, xs, None, 8, 256, want_y=False, want_acc=True),
        lambda: q.quest_linear_bwd(dy, fwd, 4, 128, 256), lambda: q.quest_linear_bwd(dy, fwd, 4, 128, 256, torch.bfloat16, want_dx=False),
        lambda: q.quest_linear_bwd(dy, fwd, 4, 128, 256, want_dx=False, want_dw=False), lambda: q.quest_linear_bwd(dy.float(), fwd, 4, 128, 256),
        lambda: q.quest_linear_bwd(dy[:7], fwd, 4, 128, 256), lambda: q.quest_linear_bwd(dy, {"xq": fwd["xq"]}, 4, 128, 256),
        lambda: q.quest_linear_fwd_fp4(x, w, 128), lambda: q.quest_linear_fwd_fp4(x, None, 128, out_dtype=torch.float32, w_cached=cached),
        lambda: q.quest_linear_fwd_weight_only(x, w, 3, 128), lambda: q.quest_linear_fwd_weight_only(x, w.float(), 8, 64, out_dtype=torch.float32),
        lambda: q.quest_linear_fwd_weight_only(x, w[:, :128], 4, 128),
        lambda: q.quest_mlp_fwd(x, w, w.flip(0).contiguous(), torch.cat([w] * 6)[:256, :48].contiguous(), 4, 16),
        lambda: q.quest_mlp_fwd(x, w, w, w, 4, 128),
        lambda: q.quest_mlp_fwd(x[:, :64].contiguous(), x, x, x, 4, 64, buffers={}),
    ]
    for i, call in enumerate(calls):
        fast, slow = both(monkeypatch, call)
        try:
            same(fast, slow)
        except AssertionError as e:
            raise AssertionError(f"call {i}") from e
    torch.cuda.synchronize()


def test_given_outputs_are_used_and_returned():
    import paper_2502_05003_b200 as q
    x = torch.randn((40, 128), device="cuda")
    codes, scales = torch.empty((40, 64), dtype=torch.uint8, device="cuda"), torch.empty(40, device="cuda")
    c, s, m = q.quest_quantize(x, 4, 128, codes=codes, scales=scales, want_mask=False)
    assert c is codes and s is scales and m is None
    saved, y = {"sx": scales}, torch.empty((40, 40), device="cuda")
    r = q.quest_linear_fwd(x, x, 4, 128, y=y, saved=saved)
    assert r["y"] is y and r["sx"] is scales and list(saved) == ["sx"]
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):                         # the current stream is the one the call runs on
        r2 = q.quest_linear_fwd(x, x, 4, 128)
    side.synchronize()
    assert torch.equal(r2["y"], y)
