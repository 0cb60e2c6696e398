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


def test_strided_inputs_are_read_as_what_they_show(monkeypatch):
    """The last position of every sequence, a slice of wider rows, an expanded row, transposed storage: the same as copies."""
    import paper_2502_05003_b200 as q
    gen = torch.Generator(device="cuda").manual_seed(4)
    hidden = torch.randn((24, 3, 256), generator=gen, device="cuda").bfloat16()
    wide = torch.randn((256, 512), generator=gen, device="cuda").bfloat16()
    full = q.quest_linear_fwd(hidden[:, 0].contiguous(), wide[:48, :256].contiguous(), 4, 128)
    cached = {"wq": full["wq"], "sw": full["sw"]}
    xs = [hidden[:, -1], hidden[:, 1, 128:], wide[:24, 128:384], hidden[0, :1].expand(8, 256), wide[:, :256].t()]
    for x in xs:
        K = x.shape[1]
        for w in (wide[:48, :K], wide[:K, :48].t()):
            assert not x.is_contiguous() and not w.is_contiguous()
            for call in (lambda a, b: q.quest_linear_fwd(a, b, 4, 128), lambda a, b: q.quest_linear_fwd_fp4(a, b, 128, out_dtype=torch.float32)):
                fast, slow = both(monkeypatch, lambda: call(x, w))
                same(fast, slow)
                same(fast, call(x.contiguous(), w.contiguous()))
        if K == 256:
            same(q.quest_linear_fwd(x, None, 4, 128, w_cached=cached), q.quest_linear_fwd(x.contiguous(), None, 4, 128, w_cached=cached))
    saved = {k: torch.zeros_like(v) for k, v in full.items() if k != "y"}
    ws = q.alloc_workspace(24, 48, 256, 4, 4)
    q.quest_linear_fwd_quantize(hidden[:, 0], wide[:48, :256], 4, 128, 1.0, saved, ws)
    same(saved, {k: full[k] for k in saved})


def test_arguments_that_do_not_fit_are_refused(monkeypatch):
    import paper_2502_05003_b200 as q
    x, w = torch.randn((16, 256), device="cuda").bfloat16(), torch.randn((48, 256), device="cuda").bfloat16()
    full = q.quest_linear_fwd(x, w, 4, 128)
    e = lambda *shape, dt=torch.uint8, dev="cuda": torch.empty(shape, dtype=dt, device=dev)
    fwd = lambda **kw: lambda: q.quest_linear_fwd(x, w, 4, 128, **kw)
    refused = [
        (TypeError, lambda: q.quest_linear_fwd(x, w.float(), 4, 128)), (TypeError, lambda: q.quest_linear_fwd_fp4(x.float(), w, 128)),
        (ValueError, lambda: q.quest_linear_fwd(x, w[:, :128], 4, 128)), (ValueError, lambda: q.quest_linear_fwd_fp4(x, w[:, :128], 128)),
        (ValueError, fwd(y=e(48, 16, dt=torch.bfloat16).t())), (ValueError, fwd(y=e(16, 40, dt=torch.bfloat16))),
        (ValueError, fwd(saved={"xq": e(16, 64)})), (ValueError, fwd(saved={"sx": e(16, dt=torch.float32, dev="cpu")})),
        (ValueError, fwd(saved={"mx": e(16, 64)[:, ::2]})), (ValueError, fwd(saved={"mw": e(40, 32)})),
        (ValueError, lambda: q.quest_linear_fwd(x, None, 4, 128, w_cached={"wq": full["wq"][:, :64], "sw": full["sw"]})),
        (ValueError, lambda: q.quest_linear_fwd(x, None, 4, 128, w_cached={"wq": full["wq"], "sw": full["sw"][:40]})),
        (ValueError, lambda: q.quest_linear_fwd_fp4(x, None, 128, w_cached={"wq": full["wq"][:, :64], "sw": full["sw"]})),
    ]
    for i, (error, call) in enumerate(refused):
        fast, slow = both(monkeypatch, call)
        assert fast == slow and isinstance(fast, tuple) and fast[0] is error, (i, fast, slow)
    for w_cached in ({"wq": full["wq"]}, {"wq": full["wq"], "sw": None}):
        for call in (lambda: q.quest_linear_fwd(x, None, 4, 128, w_cached=w_cached), lambda: q.quest_linear_fwd_fp4(x, None, 128, w_cached=w_cached)):
            fast, slow = both(monkeypatch, call)
            assert fast == slow and isinstance(fast, tuple), (fast, slow)
    # a pitched y stays welcome where the call takes one
    wide = e(16, 64, dt=torch.bfloat16)
    r, plain = (q.quest_linear_fwd_weight_only(x, w, 4, 128, out=o) for o in ({"y": wide[:, :48]}, None))
    assert torch.equal(wide[:, :48], plain["y"]) and r["y"].data_ptr() == wide.data_ptr()
    # room to spare and other shapes of the same bytes stay welcome
    y, xq = e(20, 48, dt=torch.bfloat16), e(16 * 128, dt=torch.int8)
    r = q.quest_linear_fwd(x, w, 4, 128, y=y, saved={"xq": xq})
    assert torch.equal(r["y"][:16], full["y"]) and torch.equal(xq.view(torch.uint8).view(16, 128), full["xq"])
