"""Arguments of the marshalled calls: what is converted, what is refused and with which exception."""
import numpy as np
import pytest
import torch

import oracle
import paper_2502_15779_b200 as rcp
from gen import synth
from helpers import f16_bits

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
N, K, M = 48, 256, 2


def _layer(group=0):
    codes, lut = (synth.make_layer_grouped(N, K, group, 1, "uniform", 1, device=DEV) if group
                  else synth.make_layer(N, K, 1, "uniform", 1, device=DEV))
    return rcp.rcp_pack_weights(codes), lut


def _buffers():
    return dict(xq=torch.empty(M, K // 2, dtype=torch.uint8, device=DEV), scale=torch.empty(M, dtype=torch.float16, device=DEV))


NUMBERS = [lambda v: v, float, np.int64, np.float32, torch.tensor, str]


@pytest.mark.parametrize("as_number", NUMBERS)
def test_numbers_are_taken_as_int_and_float_take_them(as_number):
    x = synth.make_activations(M, K, 2, device=DEV)
    ref = oracle.quantize_act(f16_bits(x), 64, 1.0)
    xq, scale = rcp.rcp_quantize_act(x, as_number(64), as_number(1))
    assert np.array_equal(xq.cpu().numpy(), ref["xq"]) and np.array_equal(f16_bits(scale), ref["scale"])
    for group in (0, 128):
        words, lut = _layer(group)
        b = _buffers()
        want = rcp.rcp_linear_w2a4(x, 64, 1.0, words, lut, group=group, **b)
        got = rcp.rcp_linear_w2a4(x, as_number(64), as_number(1), words, lut, group=as_number(group), **b)
        assert torch.equal(want, got)
    words, lut = _layer()
    y = torch.empty(M, N, dtype=torch.float16)
    b = _buffers()
    rcp.rcp_linear_w2a4_host(x.cpu(), as_number(64), as_number(1), words, lut, y, torch.empty_like(x), b["xq"], b["scale"],
                             torch.empty(M, N, dtype=torch.float16, device=DEV), rcp.make_workspace(M, N, K, DEV))
    torch.cuda.synchronize()
    assert torch.equal(y, rcp.rcp_linear_w2a4(x, 64, 1.0, words, lut, **_buffers()).cpu())


def test_what_is_no_number_is_refused():
    x = synth.make_activations(M, K, 2, device=DEV)
    with pytest.raises(TypeError):
        rcp.rcp_quantize_act(x, None, 1.0)
    with pytest.raises(ValueError):
        rcp.rcp_quantize_act(x, "a", 1.0)
    with pytest.raises(TypeError):
        rcp.rcp_quantize_act(x, 64, None)
    words, lut = _layer()
    with pytest.raises(TypeError):
        rcp.rcp_linear_w2a4(x, 64, 1.0, words, lut, group=None, **_buffers())


def _calls():
    """(call taking keyword buffers, its buffers by name as (dtype, elements)) of every marshalled entry point."""
    x = synth.make_activations(M, K, 2, device=DEV)
    words, lut = _layer()
    wordsg, lutg = _layer(128)
    codes3 = torch.randint(0, 8, (N, K), dtype=torch.uint8, device=DEV)
    words2, words1 = rcp.rcp_pack_weights3(codes3)
    lut3 = torch.randn(N, 8, device=DEV).half()
    xq, scale = rcp.rcp_quantize_act(x, 64, 1.0)
    h, u8, i8, f32, i32 = torch.float16, torch.uint8, torch.int8, torch.float32, torch.int32
    ws = (i32, 4)
    return {
        "quantize_act": (lambda **b: rcp.rcp_quantize_act(x, 64, 1.0, **b), dict(xq=(u8, M * K // 2), scale=(h, M))),
        "gemv": (lambda **b: rcp.rcp_gemv_w2a4(words, lut, xq, scale, variant="mma_only", **b),
                 dict(y=(h, M * N), workspace=ws, S_dbg=(i32, M * N * 4))),
        "grouped": (lambda **b: rcp.rcp_gemv_w2a4_grouped(wordsg, lutg, xq, scale, variant="dp4a", **b),
                    dict(y=(h, M * N), workspace=ws, S_dbg=(i32, M * N * (K // 128) * 4))),
        "w2a16": (lambda **b: rcp.rcp_gemv_w2a16(words, lut, x, **b),
                  dict(y=(h, M * N), digits=(i8, M * 4 * K), unit=(f32, M * 4), workspace=ws, S_dbg=(i32, 4 * M * N * 4))),
        "w3a4": (lambda **b: rcp.rcp_gemv_w3a4(words2, words1, lut3, xq, scale, **b), dict(y=(h, M * N), S_dbg=(i32, M * N * 8))),
        "linear": (lambda **b: rcp.rcp_linear_w2a4(x, 64, 1.0, words, lut, **b),
                   dict(y=(h, M * N), xq=(u8, M * K // 2), scale=(h, M), workspace=ws, S_dbg=(i32, M * N * 4))),
        "linear_grouped": (lambda **b: rcp.rcp_linear_w2a4(x, 64, 1.0, wordsg, lutg, group=128, **b),
                           dict(y=(h, M * N), xq=(u8, M * K // 2), scale=(h, M), workspace=ws, S_dbg=(i32, M * N * (K // 128) * 4))),
        "static": (lambda **b: rcp.rcp_gemv_w2a4_static(words, lut, xq, scale, **b), dict(y=(h, M * N))),
        "pack": (lambda **b: rcp.rcp_pack_weights(codes3 & 3, **b), dict(out=(i32, N * K // 16))),
    }


@pytest.mark.parametrize("name", ["quantize_act", "gemv", "grouped", "w2a16", "w3a4", "linear", "linear_grouped", "static", "pack"])
def test_buffers_too_small_or_of_another_kind_are_refused(name):
    call, spec = _calls()[name]
    good = {k: torch.zeros(n, dtype=t, device=DEV) for k, (t, n) in spec.items()}
    call(**good)
    torch.cuda.synchronize()
    for key, (dtype, n) in spec.items():
        with pytest.raises(ValueError):
            call(**dict(good, **{key: torch.zeros(n - 1, dtype=dtype, device=DEV)}))
        with pytest.raises(TypeError):
            call(**dict(good, **{key: torch.zeros(n, dtype=dtype)}))                                 # host memory
        with pytest.raises(TypeError):
            call(**dict(good, **{key: torch.zeros(2 * n, dtype=dtype, device=DEV)[::2]}))            # strided
        with pytest.raises(TypeError):
            call(**dict(good, **{key: 7}))
        if key != "workspace":
            with pytest.raises(TypeError):
                call(**dict(good, **{key: torch.zeros(n, dtype=torch.float64, device=DEV)}))
    torch.cuda.synchronize()


def test_buffers_that_are_larger_or_page_locked_are_taken():
    x = synth.make_activations(M, K, 2, device=DEV)
    words, lut = _layer()
    want = rcp.rcp_linear_w2a4(x, 64, 1.0, words, lut, **_buffers())
    y = torch.zeros(M + 3, N, dtype=torch.float16, device=DEV)
    xq = torch.zeros(M * K, dtype=torch.int8, device=DEV)
    rcp.rcp_linear_w2a4(x, 64, 1.0, words, lut, y=y, xq=xq, scale=torch.zeros(16, dtype=torch.float16, device=DEV),
                        workspace=torch.zeros(64, dtype=torch.uint8, device=DEV))
    assert torch.equal(y[:M], want) and not y[M:].any()
    pinned = torch.zeros(M, N, dtype=torch.float16).pin_memory()
    rcp.rcp_linear_w2a4(x, 64, 1.0, words, lut, y=pinned, **_buffers())
    torch.cuda.synchronize()
    assert torch.equal(pinned, want.cpu())


def test_host_form_checks_what_it_reads_and_writes():
    words, lut = _layer()
    good = dict(x_host=synth.make_activations(M, K, 2), had_block=64, clip_ratio=1.0, words=words, lut=lut,
                y_host=torch.zeros(M, N, dtype=torch.float16), x_dev=torch.empty(M, K, dtype=torch.float16, device=DEV),
                xq_dev=torch.empty(M, K // 2, dtype=torch.uint8, device=DEV), scale_dev=torch.empty(M, dtype=torch.float16, device=DEV),
                y_dev=torch.empty(M, N, dtype=torch.float16, device=DEV), workspace=rcp.make_workspace(M, N, K, DEV))
    rcp.rcp_linear_w2a4_host(**good)
    torch.cuda.synchronize()
    assert torch.equal(good["y_host"], rcp.rcp_linear_w2a4(good["x_host"].to(DEV), 64, 1.0, words, lut, **_buffers()).cpu())
    z = lambda *s, t=torch.float16: torch.zeros(*s, dtype=t, device=DEV)
    wrong = [
        (ValueError, dict(words=words[:, :8].contiguous())), (ValueError, dict(words=words.view(-1))), (TypeError, dict(words=words.cpu())),
        (TypeError, dict(words=words.float())), (TypeError, dict(words=words.t())), (ValueError, dict(lut=lut[1:])),
        (TypeError, dict(lut=lut.float())), (TypeError, dict(lut=None)), (TypeError, dict(x_host=z(M, K))),
        (TypeError, dict(x_host=synth.make_activations(K, M, 2).t())), (TypeError, dict(x_host=torch.zeros(M, K))),
        (ValueError, dict(x_host=synth.make_activations(1, M * K, 2)[0])), (ValueError, dict(y_host=torch.zeros(M, N - 1, dtype=torch.float16))),
        (TypeError, dict(y_host=torch.zeros(M, 2 * N, dtype=torch.float16)[:, ::2])), (TypeError, dict(y_host=z(M, N))),
        (ValueError, dict(x_dev=z(M, K - 1))), (ValueError, dict(xq_dev=z(M, K // 2 - 1, t=torch.uint8))), (ValueError, dict(scale_dev=z(M - 1))),
        (ValueError, dict(y_dev=z(M, N - 1))), (ValueError, dict(workspace=z(3, t=torch.int32))), (TypeError, dict(y_dev=z(M, N, t=torch.float32))),
    ]
    for error, change in wrong:
        with pytest.raises(error):
            rcp.rcp_linear_w2a4_host(**dict(good, **change))
    torch.cuda.synchronize()


@pytest.mark.parametrize("given", [False, True])
@pytest.mark.parametrize("bad,error", [(None, TypeError), (3, TypeError), ("1d", ValueError), ("0d", ValueError), ("host", TypeError)])
def test_operands_that_are_no_matrix(bad, error, given):
    """The same exceptions whether the result buffers are passed or allocated."""
    x = synth.make_activations(M, K, 2, device=DEV)
    words, lut = _layer()
    wordsg, lutg = _layer(128)
    words2, words1 = rcp.rcp_pack_weights3(torch.randint(0, 8, (N, K), dtype=torch.uint8, device=DEV))
    lut3 = torch.randn(N, 8, device=DEV).half()
    xq, scale = rcp.rcp_quantize_act(x, 64, 1.0)
    y = dict(y=torch.empty(M, N, dtype=torch.float16, device=DEV)) if given else {}
    ws = dict(workspace=rcp.make_workspace(M, N, K, DEV)) if given else {}
    dg = dict(digits=torch.empty(M, 4, K, dtype=torch.int8, device=DEV), unit=torch.empty(M, 4, device=DEV)) if given else {}

    def spoil(t):
        return {"1d": t.reshape(-1), "0d": t.reshape(-1)[0], "host": t.cpu()}.get(bad, bad) if isinstance(bad, str) else bad

    calls = [
        lambda: rcp.rcp_gemv_w2a4(spoil(words), lut, xq, scale, **y, **ws),
        lambda: rcp.rcp_gemv_w2a4(words, lut, spoil(xq), scale, **y, **ws),
        lambda: rcp.rcp_gemv_w2a4_grouped(spoil(wordsg), lutg, xq, scale, **y, **ws),
        lambda: rcp.rcp_gemv_w2a4_grouped(wordsg, lutg, spoil(xq), scale, **y, **ws),
        lambda: rcp.rcp_gemv_w2a16(spoil(words), lut, x, **y, **ws, **dg),
        lambda: rcp.rcp_gemv_w2a16(words, lut, spoil(x), **y, **ws, **dg),
        lambda: rcp.rcp_gemv_w3a4(spoil(words2), words1, lut3, xq, scale, **y),
        lambda: rcp.rcp_gemv_w3a4(words2, words1, lut3, spoil(xq), scale, **y),
        lambda: rcp.rcp_linear_w2a4(spoil(x), 64, 1.0, words, lut, **y, **ws, **(_buffers() if given else {})),
        lambda: rcp.rcp_linear_w2a4(x, 64, 1.0, spoil(words), lut, **y, **ws, **(_buffers() if given else {})),
        lambda: rcp.rcp_quantize_act(spoil(x), 64, 1.0, **(_buffers() if given else {})),
    ]
    for call in calls:
        with pytest.raises(error):
            call()
    torch.cuda.synchronize()
