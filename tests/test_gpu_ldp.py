"""GPU parity of rcp_ldp_export (partitioning quantizer -> packed codes and grids) against the CPU oracle:
codes and fp16 levels bit for bit; and the exported layer through the GEMV against the oracle's GEMV."""
import numpy as np
import pytest
import torch

import oracle
import paper_2502_15779_b200 as rcp
from gen import synth
from helpers import f16_bits

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _inputs(N, K, G, seed):
    g = torch.Generator(device="cpu")
    g.manual_seed(seed)
    u = torch.rand(N, K, generator=g, dtype=torch.float64) - 0.5
    w = (-0.02 * torch.sign(u) * torch.log1p(-2.0 * u.abs())).to(torch.float16)   # Laplace(0, 0.02)
    NG = K // G
    sb = torch.sigmoid(3.0 + torch.randn(N, NG, generator=g)).float()
    sg = torch.sigmoid(3.0 + torch.randn(N, NG, generator=g)).float()
    s1 = torch.sigmoid(-0.7 + 0.5 * torch.randn(N, NG, generator=g)).float()
    s2 = torch.sigmoid(0.5 * torch.randn(N, NG, generator=g)).float()
    return w, sb, sg, s1, s2


@pytest.mark.parametrize("N,K,G", [(1, 64, 16), (5, 128, 128), (33, 1024, 128), (17, 11008, 128), (64, 4096, 4096),
                                   (9, 2048, 64), (300, 512, 256), (3, 28672, 128), (2, 8192, 8192), (40, 384, 48)])
def test_ldp_export_bit_exact(N, K, G):
    w, sb, sg, s1, s2 = _inputs(N, K, G, N + K + G)
    if N > 2:
        w[1, :G] = 0.125            # a unit without range: code 0, four equal levels
        w[2, :G] = w[2, :G].abs()   # a unit whose minimum is positive
    ref = oracle.ldp_export(f16_bits(w), sb.numpy(), sg.numpy(), s1.numpy(), s2.numpy(), G)
    words, lut = rcp.rcp_ldp_export(w.to(DEV), sb.to(DEV), sg.to(DEV), s1.to(DEV), s2.to(DEV), G)
    assert np.array_equal(words.cpu().numpy().view(np.uint32), oracle.pack_weights(ref["codes"]))
    assert np.array_equal(f16_bits(lut), ref["lut"])
    assert len(np.unique(ref["codes"])) == 4


def test_ldp_export_at_the_uniform_initial_point_and_exact_thresholds():
    # weights on a grid of sixteenths over [0, 1], sigmoids 1/2: thresholds 1/4, 5/8, 7/8 are hit exactly
    G = 32
    w = (torch.arange(G, dtype=torch.float32) / 16.0).clamp(max=1.0).to(torch.float16)[None, :].repeat(2, 2).contiguous()
    half = torch.full((2, 2), 0.5, dtype=torch.float32)
    one = torch.ones(2, 2, dtype=torch.float32)
    ref = oracle.ldp_export(f16_bits(w), one.numpy(), one.numpy(), half.numpy(), half.numpy(), G)
    words, lut = rcp.rcp_ldp_export(w.to(DEV), one.to(DEV), one.to(DEV), half.to(DEV), half.to(DEV), G)
    assert np.array_equal(words.cpu().numpy().view(np.uint32), oracle.pack_weights(ref["codes"]))
    assert list(ref["codes"][0, :17]) == [0, 0, 0, 0, 1, 1, 1, 1, 1, 1, 2, 2, 2, 2, 3, 3, 3]
    assert lut[0, 0].tolist() == [0.0, 0.4375, 0.75, 1.0]


@pytest.mark.parametrize("N,K,G,M", [(200, 1024, 128, 1), (300, 4096, 128, 3), (150, 2048, 2048, 2)])
def test_exported_layer_through_the_gemv(N, K, G, M):
    w, sb, sg, s1, s2 = _inputs(N, K, G, 7 * N + M)
    words, lut = rcp.rcp_ldp_export(w.to(DEV), sb.to(DEV), sg.to(DEV), s1.to(DEV), s2.to(DEV), G)
    x = synth.make_activations(M, K, 11, device=DEV)
    B = 128
    xq, scale = rcp.rcp_quantize_act(x, B, 1.0)
    ref_q = oracle.ldp_export(f16_bits(w), sb.numpy(), sg.numpy(), s1.numpy(), s2.numpy(), G)
    qa = oracle.quantize_act(f16_bits(x), B, 1.0)
    w_ref = oracle.pack_weights(ref_q["codes"])
    if G == K:
        y = rcp.rcp_gemv_w2a4(words, lut.reshape(N, 4).contiguous(), xq, scale)
        ref = oracle.gemv_w2a4(w_ref, ref_q["lut"].reshape(N, 4), qa["xq"], qa["scale"])
    else:
        y = rcp.rcp_gemv_w2a4_grouped(words, lut, xq, scale, group=G)
        ref = oracle.gemv_w2a4_grouped(w_ref, ref_q["lut"], qa["xq"], qa["scale"], G)
    got = y.float().cpu().numpy().astype(np.float64)
    assert np.all(np.abs(got - ref["y"]) <= ref["tol"])
    # sanity: the 2-bit layer (untrained partition parameters) still follows the full-precision product
    full = (qa["q"].astype(np.float64) * qa["scale"].view(np.float16).astype(np.float64)[:, None]) @ w.numpy().astype(np.float64).T
    assert np.corrcoef(got.ravel(), full.ravel())[0, 1] > 0.6


@pytest.mark.parametrize("N,K,G,M", [(2500, 8192, 128, 1), (3000, 4096, 4096, 1), (700, 2048, 128, 4)])
def test_export_directly_followed_by_the_linear_call_on_one_stream(N, K, G, M):
    """The export kernel and the linear call back to back on one stream, nothing in between (the GEMV kernels
    start fetching the weights before the kernel in front of them has finished only if that kernel signals an
    early start, which the export kernel never does). Repeated, so that a stale read would show."""
    w, sb, sg, s1, s2 = _inputs(N, K, G, 3 * N + M)
    wd, sbd, sgd, s1d, s2d = (t.to(DEV) for t in (w, sb, sg, s1, s2))
    x = synth.make_activations(M, K, 13, device=DEV)
    B = K if G == K else 128
    ref_q = oracle.ldp_export(f16_bits(w), sb.numpy(), sg.numpy(), s1.numpy(), s2.numpy(), G)
    qa = oracle.quantize_act(f16_bits(x), B, 1.0)
    w_ref = oracle.pack_weights(ref_q["codes"])
    ref = (oracle.gemv_w2a4(w_ref, ref_q["lut"].reshape(N, 4), qa["xq"], qa["scale"]) if G == K
           else oracle.gemv_w2a4_grouped(w_ref, ref_q["lut"], qa["xq"], qa["scale"], G))
    words = torch.empty((N, K // 16), dtype=torch.int32, device=DEV)
    lut = torch.empty((N, K // G, 4), dtype=torch.float16, device=DEV)
    xq = torch.empty(M, K // 2, dtype=torch.uint8, device=DEV)
    scale = torch.empty(M, dtype=torch.float16, device=DEV)
    ws = rcp.make_workspace(M, N, K, DEV)
    L = rcp.lib()
    import ctypes as C
    st = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    for rep in range(5):
        words.fill_(-1)
        lut.fill_(float("nan"))
        torch.cuda.synchronize()
        assert L.rcp_ldp_export(wd.data_ptr(), sbd.data_ptr(), sgd.data_ptr(), s1d.data_ptr(), s2d.data_ptr(), N, K, G,
                                words.data_ptr(), lut.data_ptr(), st) == 0
        y = rcp.rcp_linear_w2a4(x, B, 1.0, words, lut.reshape(N, 4) if G == K else lut, group=0 if G == K else G,
                                xq=xq, scale=scale, workspace=ws)
        torch.cuda.synchronize()
        got = y.float().cpu().numpy().astype(np.float64)
        assert np.all(np.isfinite(got)) and np.all(np.abs(got - ref["y"]) <= ref["tol"]), f"repetition {rep}"


@pytest.mark.parametrize("N,K", [(1, 128), (1, 31 * 128), (1, 32 * 128), (3, 11 * 128), (257, 128), (40, 2048)])
def test_ldp_export_groups_of_128_at_tile_edges_and_hard_thresholds(N, K):
    """The form for units of 128 compares weights with the smallest fp16 number that reaches each threshold. Unit
    counts around its tiles of 32; thresholds that are hit exactly, that nothing or everything reaches, ranges so wide
    that the threshold lies among numbers far smaller than the range's rounding, subnormal ranges, signed zeros."""
    G = 128
    w, sb, sg, s1, s2 = _inputs(N, K, G, 5 * N + K)
    wv = w.view(N * K // G, G)
    for i in range(wv.shape[0]):
        a = (sb, sg, s1, s2)
        flat = [t.view(-1) for t in a]
        kind = i % 8
        if kind == 1:      # thresholds 1/4, 5/8, 7/8 of [0, 1] hit exactly
            wv[i] = (torch.arange(G) % 17 / 16.0).to(torch.float16)
            flat[0][i] = flat[1][i] = 1.0
            flat[2][i] = flat[3][i] = 0.5
        elif kind == 2:    # -60000 .. 60000 with a threshold near zero, met by subnormal weights of both signs
            wv[i] = (torch.arange(G) - 64).to(torch.float16) * 2.0 ** -24
            wv[i, 0], wv[i, 1] = -60000.0, 60000.0
            flat[0][i] = flat[1][i] = 1.0
            flat[2][i] = 0.999999 if i % 16 == 2 else 1.0
        elif kind == 3:    # t_1 = 0: everything reaches it; t_3 = 1
            flat[2][i], flat[3][i] = 0.0, 1.0
        elif kind == 4:    # subnormal weights only
            wv[i] = (torch.arange(G) * 7 % 53 - 20).to(torch.float16) * 2.0 ** -24
        elif kind == 5:    # no range, negative
            wv[i] = -0.25
        elif kind == 6:    # zeros of both signs and a positive maximum
            wv[i] = torch.where(torch.arange(G) % 2 == 0, 0.0, -0.0).to(torch.float16)
            wv[i, 5] = 0.5
    ref = oracle.ldp_export(f16_bits(w), sb.numpy(), sg.numpy(), s1.numpy(), s2.numpy(), G)
    words, lut = rcp.rcp_ldp_export(w.to(DEV), sb.to(DEV), sg.to(DEV), s1.to(DEV), s2.to(DEV), G)
    assert np.array_equal(words.cpu().numpy().view(np.uint32), oracle.pack_weights(ref["codes"]))
    # levels bit for bit, except that a zero level may carry either sign (which zero is the minimum is not defined)
    got = f16_bits(lut)
    assert np.all((got == ref["lut"]) | (((got | ref["lut"]) & 0x7FFF) == 0))


def _edge_units(wv, sig, kinds):
    """Every second unit of wv [units][128] becomes one of the edge cases."""
    sb, sg, s1, s2 = sig
    i = torch.arange(128)
    for u in range(0, wv.shape[0], 2):
        kind = kinds[(u // 2) % len(kinds)]
        if kind == "exact":        # thresholds 1/4, 5/8, 7/8 of [0, 1] hit exactly
            wv[u] = (i % 17 / 16.0).to(torch.float16)
            sb[u] = sg[u] = 1.0
            s1[u] = s2[u] = 0.5
        elif kind == "wide":       # a threshold among numbers far smaller than the rounding of the range
            wv[u] = (i - 64).to(torch.float16) * 2.0 ** -24
            wv[u, 0], wv[u, 1] = -60000.0, 60000.0
            sb[u] = sg[u] = 1.0
            s1[u] = 0.999999
        elif kind == "ends":       # t_1 = 0, t_3 = 1
            s1[u], s2[u] = 0.0, 1.0
        elif kind == "subnormal":
            wv[u] = (i * 7 % 53 - 20).to(torch.float16) * 2.0 ** -24
        elif kind == "flat":
            wv[u] = -0.25
        elif kind == "zeros":      # zeros of both signs, one of them the minimum
            wv[u] = torch.where(i % 2 == 0, 0.0, -0.0).to(torch.float16)
            wv[u, 5] = 0.5
        elif kind == "minus":      # zeros of both signs, one of them the maximum
            wv[u] = torch.where(i % 2 == 0, 0.0, -0.0).to(torch.float16)
            wv[u, 7] = -0.5


def _export_whole_and_in_pieces(w, sig, N, K):
    """The export of all rows in one call (tiles of units) and in calls of fewer than 4096 units (a warp per unit)."""
    args = [w.to(DEV)] + [t.view(N, K // 128).to(DEV) for t in sig]
    rows = 4095 // (K // 128)
    parts = [rcp.rcp_ldp_export(*[t[r:r + rows] for t in args], 128) for r in range(0, N, rows)]
    return rcp.rcp_ldp_export(*args, 128), (torch.cat([p[0] for p in parts]), torch.cat([p[1] for p in parts]))


@pytest.mark.parametrize("N,K", [(4096, 128), (4097, 128), (4127, 128), (1366, 384), (75776 + 33, 128), (300, 14336)])
def test_ldp_export_tiles_of_units_and_single_units_agree(N, K):
    """Both forms for groups of 128, bit for bit, signs of zero levels included; the first rows against the oracle too."""
    w, sb, sg, s1, s2 = _inputs(N, K, 128, N + K)
    sig = [t.reshape(-1) for t in (sb, sg, s1, s2)]
    _edge_units(w.view(-1, 128)[:400], sig, ["exact", "wide", "ends", "subnormal", "flat", "zeros", "minus"])
    whole, pieces = _export_whole_and_in_pieces(w, sig, N, K)
    assert torch.equal(whole[0], pieces[0])
    assert torch.equal(whole[1].view(torch.int16), pieces[1].view(torch.int16))
    n = 400 // (K // 128)
    ref = oracle.ldp_export(f16_bits(w[:n]), *[t.view(N, K // 128)[:n].numpy() for t in sig], 128)
    assert np.array_equal(whole[0][:n].cpu().numpy().view(np.uint32), oracle.pack_weights(ref["codes"]))
    # a zero level may carry either sign against the oracle (which zero is the minimum is not defined)
    got = f16_bits(whole[1][:n])
    assert np.all((got == ref["lut"]) | (((got | ref["lut"]) & 0x7FFF) == 0))


def test_ldp_export_units_of_nan_have_an_empty_range():
    """Nothing but NaN in a unit: no minimum and no maximum, so lo = +inf, no range, codes 0, four equal levels. A NaN among
    numbers is ignored by the range and gets code 0. Alike in both forms."""
    N, K = 4200, 128
    w, sb, sg, s1, s2 = _inputs(N, K, 128, 3)
    w[5] = w[4199] = float("nan")
    w[7, ::2] = float("nan")
    whole, pieces = _export_whole_and_in_pieces(w, [t.reshape(-1) for t in (sb, sg, s1, s2)], N, K)
    assert torch.equal(whole[0], pieces[0])
    assert torch.equal(whole[1].view(torch.int16), pieces[1].view(torch.int16))
    for row in (5, 4199):
        assert not whole[0][row].any() and torch.all(whole[1][row] == float("inf"))
    assert torch.isfinite(whole[1][7]).all()


def test_ldp_export_argument_errors():
    L = rcp.lib()
    z = torch.zeros(4096, dtype=torch.int32, device=DEV)
    p = z.data_ptr()
    f = L.rcp_ldp_export
    assert f(None, p, p, p, p, 4, 128, 128, p, p, None) == -1
    assert f(p, p, p, p, p, 0, 128, 128, p, p, None) == -2
    assert f(p, p, p, p, p, 4, 128, 48, p, p, None) == -2      # group does not divide K
    assert f(p, p, p, p, p, 4, 128, 8, p, p, None) == -2       # group below 16
    assert f(p + 2, p, p, p, p, 4, 128, 128, p, p, None) == -3
