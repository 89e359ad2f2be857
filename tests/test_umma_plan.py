"""Host logic of the GEMV on tcgen05: how a call's tokens are shared out over launches, and every launch's plan (rows, tensor
memory, shared memory, activations). No GPU needed: rcp_gemv_umma_plan only computes."""
import ctypes as C

import pytest

from paper_2502_15779_b200 import build
from gen.configs import CONFIGS

FIELDS = ("launched tokens stages smem nchunk part_chunks kpl bhalf bstep bgroup lg_m2 slots dcols acc_cols nbuf helpers off_bar off_misc "
          "off_red red_bytes off_bs bs_bytes off_qbuf nphase").split()
ITEM = 128 * 128        # an item of the ring: 128 lanes of 128 bytes


@pytest.fixture(scope="module")
def L():
    lib = C.CDLL(build.build())
    lib.rcp_gemv_umma_plan.argtypes = [C.c_int] * 5 + [C.POINTER(C.c_int), C.c_int]
    return lib


def plan(L, M, N, K, sms=148, block=0):
    buf = (C.c_int * 1600)()
    n = L.rcp_gemv_umma_plan(M, N, K, sms, block, buf, 1600)
    assert 2 <= n <= 1600, n
    at, launches = 2, []
    for _ in range(buf[1]):
        p = dict(zip(FIELDS, buf[at:at + len(FIELDS)]))
        at += len(FIELDS)
        p["phases"] = [tuple(buf[at + 9 * i: at + 9 * i + 9]) for i in range(p["nphase"])]
        at += 9 * p["nphase"]
        launches.append(p)
    assert at == n
    return buf[0], launches


def check(L, M, N, K, sms=148, block=0, qbytes=0):
    taken, launches = plan(L, M, N, K, sms, block)
    assert launches or not taken
    assert not launches or sum(p["launched"] for p in launches) == M
    for p in launches:
        m = p["tokens"]
        assert m == p["launched"], (M, N, K, "launched with a plan for another number of tokens", m, p["launched"])
        assert 1 << p["lg_m2"] >= m > (1 << p["lg_m2"]) // 2
        nxt, chunks = 0, -(-K // 512)
        assert p["nchunk"] == chunks and 1 <= p["nphase"] <= 5
        for gpc, first, total, ncta, reps, kp, items, ncol, ncol_f8 in p["phases"]:   # every group of 16 rows once, in order
            assert first == nxt and 1 <= ncta <= sms and -(-total // ncta) <= gpc <= 8
            assert gpc * kp <= 8 and kp & (kp - 1) == 0 and kp <= p["kpl"] and kp * items >= chunks > kp * (items - 1)
            # with 128 rows: kind::i8 takes 8 or a multiple of 16 columns, kind::f8f6f4 a multiple of 16
            assert ncol >= kp * (m + 1) and ncol <= p["dcols"] <= 256 and (ncol == 8 or ncol % 16 == 0)
            assert ncol_f8 >= ncol and ncol_f8 % 16 == 0 and ncol_f8 >= 16 and 2 * p["dcols"] + ncol_f8 <= p["acc_cols"]
            nxt += total * reps
        assert nxt == -(-N // 16)
        # tensor memory: slots of 128 columns at the top, sets of three accumulators below
        assert 2 <= p["slots"] <= 3 and 1 <= p["nbuf"] <= 4 and 128 * p["slots"] + p["acc_cols"] * p["nbuf"] <= 512
        # activations: rows of a half, halves of a step and steps of a group of chunks do not overlap; the last group is whole
        assert p["bhalf"] >= p["kpl"] * (m + 1) and p["bstep"] >= 8 * p["bhalf"] and p["bgroup"] >= 4 * p["bstep"]
        parts = -(-chunks // p["part_chunks"])
        assert p["part_chunks"] % p["kpl"] == 0 or parts == 1
        groups = -(-min(chunks, p["part_chunks"]) // p["kpl"])
        assert p["bs_bytes"] >= (groups * p["bgroup"] + max(ph[8] for ph in p["phases"])) * 16
        if parts > 1:
            assert p["nphase"] == 1 and p["phases"][0][4] == 1 and not block and p["part_chunks"] % p["phases"][0][5] == 0
        # shared memory
        assert 2 <= p["stages"] <= 12 and (not p["helpers"] or p["stages"] >= 5 and m <= 8)
        if any(ph[5] > 1 for ph in p["phases"]):
            assert p["red_bytes"] >= m * 3 * 128 * 4
        ends = [p["stages"] * ITEM, p["off_bar"], p["off_misc"], p["off_red"], p["off_red"] + p["red_bytes"], p["off_bs"],
                p["off_bs"] + p["bs_bytes"], p["off_qbuf"], p["off_qbuf"] + qbytes]
        assert ends == sorted(ends) and p["off_misc"] - p["off_bar"] >= 8 * (24 + 6 + 8 + 3) and p["off_red"] - p["off_misc"] >= 200
        assert p["off_bs"] % 16 == 0 and p["off_qbuf"] + qbytes + 1024 <= p["smem"] <= 232448
    if not block and sms == 148:
        n = L.rcp_linear_w2a4_launches(M, N, K, 1, 0)
        if taken & 2 and M > 1:
            assert n == 1 + len(launches)
    return taken, launches


def test_plans_of_all_benchmark_shapes(L):
    for cfg in CONFIGS:
        for layer in cfg.layers:
            for M in cfg.Ms:
                check(L, M, layer.N, layer.K)


@pytest.mark.parametrize("N", [1, 17, 256, 2368, 2369, 9473, 18944, 18945, 20000, 28417, 28672, 57344, 100003])
def test_plans_hold_for_all_tokens_and_channels(L, N):
    for K in [64, 512, 576, 4096, 5184, 8192, 11008, 14336, 20544, 20800, 20992, 24576, 28672, 32832, 40960, 51200, 65536]:
        for M in range(1, 17):
            check(L, M, N, K)


@pytest.mark.parametrize("sms", [1, 78, 132, 160])
def test_plans_for_other_sizes_of_gpu(L, sms):
    for N in (1, 300, 16 * 8 * sms, 16 * 8 * sms + 1, 28672):
        for K in (64, 4096, 20992, 65536):
            for M in (1, 2, 3, 7, 8, 13, 15, 16):
                check(L, M, N, K, sms)


def test_plans_with_the_quantizer_inside(L):
    for K, B, q in [(2048, 2048, 8832), (4096, 4096, 17536), (8192, 8192, 33024), (64, 64, 0), (5184, 64, 0), (11008, 128, 0), (16384, 512, 0)]:
        for N in (1, 300, 2369, 18944, 18945, 57344, 180000):
            check(L, 1, N, K, block=B, qbytes=q)


# Measured on B200: the first were slower on this kernel than on the streaming kernels (by 4 to 15 %; (rows, channels, tokens), as a
# linear call with a quantizer kernel and as a call on given activations), the others are faster by 10 % and more.
SLOWER_LINEAR = [(300, 28672, 3), (2368, 28672, 2), (2368, 28672, 3), (5000, 11008, 3), (5000, 20800, 6), (5000, 24576, 6), (5000, 40960, 8),
                 (5000, 65536, 8), (9001, 14336, 8), (9001, 24576, 8), (12288, 14336, 8), (12288, 20800, 8), (7000, 16384, 2), (10240, 12288, 5),
                 (10240, 16384, 5), (14000, 9216, 5)]
SLOWER_PLAIN = [(2368, 28672, 3), (5000, 11008, 2), (5000, 24576, 6), (5000, 40960, 8), (5000, 65536, 8), (12288, 20800, 8)]
FASTER_BOTH = [(57344, 8192, 2), (57344, 8192, 3), (57344, 8192, 8), (57344, 8192, 16), (8192, 28672, 3), (28672, 4096, 16), (9001, 28672, 3),
               (12288, 20800, 4), (8192, 28672, 8), (9001, 28672, 8), (5000, 28672, 2), (20000, 5184, 3), (9001, 11008, 9), (12288, 4096, 12)]


def test_the_choice_is_the_faster_kernel(L):
    for N, K, M in SLOWER_LINEAR:
        assert not plan(L, M, N, K)[0] & 2, (N, K, M)
    for N, K, M in SLOWER_PLAIN:
        assert not plan(L, M, N, K)[0] & 1, (N, K, M)
    for N, K, M in FASTER_BOTH:
        assert plan(L, M, N, K)[0] == 3, (N, K, M)


def test_uneven_launches(L):
    # fewer tokens take more chunks side by side, which pads K: by themselves seven tokens would not fit where eight do
    _, launches = check(L, 15, 28672, 20992)
    assert [p["launched"] for p in launches] == [8, 7]
    assert launches[1]["bhalf"] >= 8 * launches[1]["kpl"]


def test_refusals(L):
    buf = (C.c_int * 8)()
    assert L.rcp_gemv_umma_plan(0, 16, 64, 148, 0, buf, 8) == -2
    assert L.rcp_gemv_umma_plan(17, 16, 64, 148, 0, buf, 8) == -2
    assert L.rcp_gemv_umma_plan(1, 16, 100, 148, 0, buf, 8) == -2
    assert L.rcp_gemv_umma_plan(1, 16, 64, 148, 0, None, 8) == -1
    assert L.rcp_gemv_umma_plan(2, 16, 4096, 148, 4096, buf, 8) == -7
    assert L.rcp_gemv_umma_plan(1, 16, 4096, 148, 1024, buf, 8) == -7
