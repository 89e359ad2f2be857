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
