"""GPU parity of the inference layer with cached weights and few rows of x: bit for bit what the same rows give in a
call with many rows (the path that the oracle tests cover), and against the oracle directly."""
import numpy as np
import pytest
import torch

from oracle import quest_oracle as qo

pytestmark = pytest.mark.gpu


def layer(M, N, K, dtype, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn((M, K), generator=gen, device="cuda")
    x[:, 0] *= 30.0                                       # clipped elements
    if M > 2:
        x[2] = 0.0                                        # a row whose RMS is zero
    w = torch.randn((N, K), generator=gen, device="cuda") * 0.02
    return x.to(dtype), w.to(dtype)


def check(M, N, K, bits, g, dtype=torch.bfloat16, out=torch.bfloat16, trust=1.0, seed=0):
    import paper_2502_05003_b200 as quest
    big = 40                                              # above the decoding path
    x, w = layer(big, N, K, dtype, seed)
    full = quest.quest_linear_fwd(x, w, bits, g, trust, out_dtype=out)
    cached = {"wq": full["wq"], "sw": full["sw"]}
    ws = quest.alloc_workspace(big, N, K, bits, bits)
    ws.fill_(0x5A)
    for mode in (False, True):                            # packed codes (writes the operand), then the operand
        cached["operand_in_workspace"] = mode
        got = quest.quest_linear_fwd(x[:M], None, bits, g, trust, out_dtype=out, w_cached=cached, workspace=ws)
        torch.cuda.synchronize()
        assert quest.quest_device_status() == 0
        for key in ("xq", "sx", "mx", "y"):
            assert torch.equal(got[key], full[key][:M]), (key, mode)
        bare = quest.quest_linear_fwd(x[:M], None, bits, g, trust, out_dtype=out, w_cached=cached, workspace=ws,
                                      want_masks=False)
        assert torch.equal(bare["y"], full["y"][:M]) and torch.equal(bare["xq"], full["xq"][:M])
    # the operand that the decoding path left in the workspace serves the general path
    again = quest.quest_linear_fwd(x, None, bits, g, trust, out_dtype=out, w_cached=cached, workspace=ws)
    assert torch.equal(again["y"], full["y"])


@pytest.mark.parametrize("bits", [1, 2, 3, 4, 6, 8])
@pytest.mark.parametrize("M", [1, 3, 8, 9, 17, 32])
def test_rows_and_widths(M, bits):
    check(M, 264, 544, bits, 32, seed=M + bits)           # ragged tiles of w, a half chunk of K, two tasks a row


@pytest.mark.parametrize("N,K,g", [(8, 32, 32), (24, 96, 1), (40, 160, 4), (520, 768, 256), (16, 1024, 512), (2376, 2048, 2048),
                                   (136, 5504, 128), (2400, 4096, 4096), (72, 8192, 64), (48, 16384, 8192)])
@pytest.mark.parametrize("M", [1, 4, 24])
def test_shapes_and_blocks(M, N, K, g):
    check(M, N, K, 4, g, seed=M + N)


@pytest.mark.parametrize("M", [5, 16, 32])
@pytest.mark.parametrize("N,K,bits", [(4744, 544, 4), (7104, 160, 3), (7112, 160, 4), (2368, 2080, 5), (2376, 1056, 4), (4736, 288, 8), (4744, 288, 8),
                                      (5504, 5504, 4), (4744, 6176, 3)])
def test_rows_of_w_per_cta(M, N, K, bits):
    # either side of 16, 32 and 48 rows of w to a CTA that has an SM to itself; rows of w that go round its ring of 4 or 6
    # chunks more than once
    check(M, N, K, bits, 32, seed=M + N)


@pytest.mark.parametrize("M,N,K,bits", [(1, 9472, 256, 4), (1, 9480, 256, 4), (4, 9480, 1024, 2), (2, 4728, 2048, 4),
                                        (2, 4744, 2048, 1), (1, 2048, 3072, 4), (8, 9480, 3104, 1), (16, 9480, 1568, 2),
                                        (16, 14216, 64, 1), (17, 1192, 2080, 1), (24, 2376, 1056, 2), (24, 9480, 992, 4),
                                        (32, 9480, 1024, 8), (32, 14216, 1024, 4)])
def test_both_sides_of_the_routes(M, N, K, bits):
    # the last size of a route and the first of the next, on 148 SMs
    check(M, N, K, bits, 32, seed=M + K)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("out", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("trust", [0.0, 0.5, 1.3])
def test_types_and_trust_factors(dtype, out, trust):
    for M in (2, 20):
        check(M, 200, 1024, 4, 128, dtype, out, trust)
        check(M, 200, 1024, 8, 64, dtype, out, trust)


@pytest.mark.parametrize("bits", [1, 2])
@pytest.mark.parametrize("K,g", [(1024, 64), (2048, 128), (2048, 1024), (4096, 4096), (8320, 64), (16384, 128)])
@pytest.mark.parametrize("trust", [0.5, 1.3])
def test_byte_operands_of_one_and_two_bits(K, g, trust, bits):
    # every kernel that quantizes x in a launch of its own writes it as bytes here, and as E2M1 nibbles elsewhere
    check(12, 136, K, bits, g, trust=trust, seed=K + g)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("bits", [1, 4, 8])
@pytest.mark.parametrize("K,g", [(2048, 64), (2048, 128), (2048, 256), (2048, 2048), (4096, 4096), (16384, 128)])
def test_weights_that_change_between_calls(K, g, bits, dtype):
    """The kernel reads w ahead of its wait for the quantizer: what an earlier launch on the stream wrote, with nothing
    but the stream between them.  New codes in one buffer before every call; the operand that the call before has left;
    the operand that a call which quantizes w has left."""
    import paper_2502_05003_b200 as quest
    M, N, rounds = 24, 1040, 4
    gen = torch.Generator(device="cuda").manual_seed(K + bits)
    x = torch.randn((M, K), generator=gen, device="cuda").to(dtype)
    ws = [torch.randn((N, K), generator=gen, device="cuda").to(dtype) for _ in range(rounds)]
    want = []
    for w in ws:
        want.append(quest.quest_linear_fwd(x, w, bits, g)["y"])
        torch.cuda.synchronize()
    saved = quest.quest_linear_fwd(x, ws[0], bits, g, want_masks=False)
    saved = {k: torch.zeros_like(v) for k, v in saved.items() if k not in ("y", "mx", "mw")}
    work = quest.alloc_workspace(M, N, K, bits, bits)
    got = torch.zeros((3, 2, rounds, M, N), dtype=dtype, device="cuda")

    def layer_of(y, w=None, **cached):
        quest.quest_linear_fwd(x, w, bits, g, y=y, saved=saved, workspace=work, want_masks=False,
                               w_cached=None if w is not None else {"wq": saved["wq"], "sw": saved["sw"], **cached})
    torch.cuda.synchronize()
    for again in range(2):
        for i, w in enumerate(ws):
            quest.quest_quantize(w, bits, g, codes=saved["wq"], scales=saved["sw"], want_mask=False)
            layer_of(got[0, again, i])
            layer_of(got[1, again, i], operand_in_workspace=True)
            layer_of(got[2, again, i], w)
            layer_of(got[2, again, i], operand_in_workspace=True)
    torch.cuda.synchronize()
    for i in range(rounds):
        assert all(torch.equal(got[k, again, i], want[i]) for k in range(3) for again in range(2)), i


def same_values(a, b):
    if not a.is_floating_point():
        return torch.equal(a, b)
    return torch.equal(a.isnan(), b.isnan()) and torch.equal(a[~a.isnan()], b[~b.isnan()])


@pytest.mark.parametrize("bits", [1, 4, 8])
@pytest.mark.parametrize("M,K,g", [(1, 2048, 128), (2, 1024, 1024), (4, 512, 32), (20, 2048, 128)])
def test_rows_that_are_not_finite(M, K, g, bits):
    import paper_2502_05003_b200 as quest
    x, w = layer(40, 64, K, torch.bfloat16, M)
    x[0, 5] = float("nan")
    x[1, 7], x[1, K - 1] = float("inf"), float("-inf")
    x[3, 100] = float("-inf")
    full = quest.quest_linear_fwd(x, w, bits, g)
    got = quest.quest_linear_fwd(x[:M], None, bits, g, w_cached={"wq": full["wq"], "sw": full["sw"]})
    for key in ("xq", "sx", "mx", "y"):
        assert same_values(got[key], full[key][:M]), key


@pytest.mark.parametrize("bits", [1, 2, 3, 4, 8])
@pytest.mark.parametrize("M", [1, 20])
def test_scales_whose_product_is_close_to_the_smallest_normal_number(M, bits):
    import paper_2502_05003_b200 as quest
    x, w = layer(40, 64, 2048, torch.float32, bits)
    x, w = x * 1e-18, w * 5e-17
    full = quest.quest_linear_fwd(x, w, bits, 128)
    got = quest.quest_linear_fwd(x[:M], None, bits, 128, w_cached={"wq": full["wq"], "sw": full["sw"]})
    assert torch.equal(got["y"], full["y"][:M])


def test_against_the_oracle():
    import paper_2502_05003_b200 as quest
    for bits in (1, 4, 8):
        x, w = layer(5, 96, 1536, torch.float32, bits)
        ref = qo.linear_fwd(x.cpu().numpy(), w.cpu().numpy(), bits, 512, 1.0)
        cached = {"wq": torch.from_numpy(ref["wq"]).cuda(), "sw": torch.from_numpy(ref["sw"]).cuda()}
        got = quest.quest_linear_fwd(x, None, bits, 512, out_dtype=torch.float32, w_cached=cached)
        assert np.array_equal(got["xq"].cpu().numpy(), ref["xq"]) and np.array_equal(got["mx"].cpu().numpy(), ref["mx"])
        assert np.allclose(got["sx"].cpu().numpy(), ref["sx"], rtol=1e-6, atol=0)
        err = np.abs(got["y"].cpu().numpy().astype(np.float64) - ref["y"]).max()
        assert err <= 1e-5 * np.abs(ref["y"]).max()
