"""The GEMV on the fifth-generation tensor cores (variant "umma"): exact sums against the oracle at the edges of its tiles, of its
columns and of what fits in shared memory, in the production and in the guarded build; linear calls that run it,
with the quantizer inside and in front; and its neighbours on the stream. (The host's plans and its choice between the kernels: test_umma_plan.py.)"""
import ctypes as C
import os
import subprocess
import sys
import threading

import numpy as np
import pytest
import torch

import oracle
import paper_2502_15779_b200 as rcp
import test_gpu_streams_threads as streams
from gen import synth
from helpers import f16_bits

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# N, K, M: groups of 16 rows around the SMs and their rounds of eight, chunks of 512 around the lane blocks, tokens around the
# columns (8, 16, 32, 48) and the workers' fours; the last ones go through K in parts
CASES = [(1, 64, 1), (17, 192, 3), (16, 512, 1), (129, 576, 7), (300, 2048, 4), (2369, 1024, 2), (2368, 4096, 5), (4737, 1088, 9),
         (700, 8192, 8), (18945, 512, 1), (21300, 1024, 16), (333, 5184, 12), (64, 65536, 1), (300, 11008, 15), (300, 28672, 8),
         (2400, 14336, 16), (40, 65536, 7)]


def taken(M, N, K, B):   # whether a linear call runs this kernel; B: with the quantizer for such blocks inside, 0: behind it
    out = (C.c_int * 2)()
    assert rcp.lib().rcp_gemv_umma_plan(M, N, K, 0, B, out, 2) > 2
    return bool(out[0] & 2)


# several launches with an uneven last one (N, K, M): as many rows as make K in parts impossible
UNEVEN = [(28672, 20800, 15), (28672, 20992, 15), (20000, 14336, 13)]


def run_uneven(i):
    N, K, M = UNEVEN[i]
    g = torch.Generator(device=DEV)
    g.manual_seed(N + K)
    words = torch.randint(-2 ** 31, 2 ** 31 - 1, (N, K // 16), dtype=torch.int32, device=DEV, generator=g)
    lut = torch.sort(torch.randn(N, 4, device=DEV, generator=g) * 0.02, dim=1)[0].half()
    xq = torch.randint(0, 256, (M, K // 2), dtype=torch.uint8, device=DEV, generator=g)
    scale = (torch.rand(M, device=DEV, generator=g) * 0.1 + 0.01).half()
    ws = rcp.make_workspace(M, N, K, DEV)
    S = torch.full((M, N, 4), 77, dtype=torch.int32, device=DEV)
    checked = rcp.rcp_gemv_w2a4(words, lut, xq, scale, workspace=ws, variant="umma", S_dbg=S)
    y = rcp.rcp_gemv_w2a4(words, lut, xq, scale, workspace=ws, variant="umma")
    torch.cuda.synchronize()
    assert int(ws.abs().max()) == 0
    assert torch.equal(y.view(torch.int16), checked.view(torch.int16))
    want = rcp.rcp_gemv_w2a4(words, lut, xq, scale, workspace=ws, variant="simple")
    assert torch.equal(y.view(torch.int16), want.view(torch.int16))
    rows = torch.cat([torch.arange(0, N, 997, device=DEV), torch.tensor([N - 1], device=DEV)])
    ref = oracle.gemv_w2a4(words[rows].cpu().numpy().view(np.uint32), f16_bits(lut[rows]), xq.cpu().numpy(), f16_bits(scale))
    assert np.array_equal(S[:, rows].cpu().numpy(), ref["S"])


@pytest.mark.parametrize("i", range(len(UNEVEN)), ids=["x".join(map(str, c)) for c in UNEVEN])
def test_uneven_launches(i):
    run_uneven(i)


def run_case(i):
    N, K, M = CASES[i]
    codes, lut = synth.make_layer(N, K, 64, "uniform", 900 + i, device=DEV)
    words = rcp.rcp_pack_weights(codes)
    xq, scale = rcp.rcp_quantize_act(synth.make_activations(M, K, 900 + i, device=DEV), 64, 1.0)
    ws = rcp.make_workspace(M, N, K, DEV)
    S = torch.full((M, N, 4), 77, dtype=torch.int32, device=DEV)
    checked = rcp.rcp_gemv_w2a4(words, lut, xq, scale, workspace=ws, variant="umma", S_dbg=S)
    y = rcp.rcp_gemv_w2a4(words, lut, xq, scale, workspace=ws, variant="umma")
    torch.cuda.synchronize()
    assert int(ws.abs().max()) == 0
    assert np.array_equal(f16_bits(y), f16_bits(checked))
    ref = oracle.gemv_w2a4(words.cpu().numpy().view(np.uint32), f16_bits(lut), xq.cpu().numpy(), f16_bits(scale))
    assert np.array_equal(S.cpu().numpy(), ref["S"])
    assert np.all(np.abs(y.float().cpu().numpy().astype(np.float64) - ref["y"]) <= ref["tol"])


@pytest.mark.parametrize("i", range(len(CASES)), ids=["x".join(map(str, c)) for c in CASES])
def test_sums_are_the_oracles(i):
    run_case(i)


def in_guarded_build(what):
    from paper_2502_15779_b200 import build
    env = dict(os.environ, RCP_W2A4_LIB=build.build_checked(), PYTHONPATH=os.pathsep.join([ROOT, os.path.join(ROOT, "tests")]))
    subprocess.run([sys.executable, "-c", "import test_gpu_umma as t\n" + what], check=True, env=env, cwd=ROOT, timeout=900)


def test_guarded_build_reports_nothing():
    in_guarded_build("for i in range(len(t.CASES)): t.run_case(i)\nfor i in range(len(t.UNEVEN)): t.run_uneven(i)")


# A worker whose wait gives up (in the guarded build the status word can ask one for it) leaves with the code, and the other three
# warps of its tokens are not left at the barriers where the lane blocks of a row add up. One tile per CTA: nothing else waits.
def run_one_warp_gives_up():
    for N, K, M, warps in [(300, 4096, 1, (0, 3)), (2368, 8192, 3, (2,)), (500, 4096, 16, (5, 15))]:
        codes, lut = synth.make_layer(N, K, 64, "uniform", 5, device=DEV)
        words = rcp.rcp_pack_weights(codes)
        xq, scale = rcp.rcp_quantize_act(synth.make_activations(M, K, 5, device=DEV), 64, 1.0)
        ws = rcp.make_workspace(M, N, K, DEV)
        want = rcp.rcp_gemv_w2a4(words, lut, xq, scale, workspace=ws, variant="umma")
        for warp in warps:
            ws[0] = -1 - warp
            rcp.rcp_gemv_w2a4(words, lut, xq, scale, workspace=ws, variant="umma")
            torch.cuda.synchronize()
            assert int(ws[0]) == 3
            ws.zero_()
        y = rcp.rcp_gemv_w2a4(words, lut, xq, scale, workspace=ws, variant="umma")
        torch.cuda.synchronize()
        assert int(ws.abs().max()) == 0 and torch.equal(y.view(torch.int16), want.view(torch.int16))


def test_one_warp_gives_up():
    in_guarded_build("t.run_one_warp_gives_up()")


# Rings of two and three stages, whose stages are filled again as soon as they have been read: the sums of many calls in a row
# are those of the plain kernel.
@pytest.mark.parametrize("N,K,M", [(28672, 20992, 8), (28672, 20480, 7), (5217, 23040, 6), (20000, 11008, 12)])
def test_a_short_ring_keeps_what_is_being_read(N, K, M):
    g = torch.Generator(device=DEV)
    g.manual_seed(N + K)
    words = torch.randint(-2 ** 31, 2 ** 31 - 1, (N, K // 16), dtype=torch.int32, device=DEV, generator=g)
    lut = torch.sort(torch.randn(N, 4, device=DEV, generator=g) * 0.02, dim=1)[0].half()
    xq = torch.randint(0, 256, (M, K // 2), dtype=torch.uint8, device=DEV, generator=g)
    scale = (torch.rand(M, device=DEV, generator=g) * 0.1 + 0.01).half()
    ws = rcp.make_workspace(M, N, K, DEV)
    S, want = torch.empty(M, N, 4, dtype=torch.int32, device=DEV), torch.empty(M, N, 4, dtype=torch.int32, device=DEV)
    y = rcp.rcp_gemv_w2a4(words, lut, xq, scale, workspace=ws, variant="simple", S_dbg=want)
    ys = torch.empty(12, M, N, dtype=torch.float16, device=DEV)
    for rep in range(10):
        for out in ys:
            rcp.rcp_gemv_w2a4(words, lut, xq, scale, y=out, workspace=ws, variant="umma")
        rcp.rcp_gemv_w2a4(words, lut, xq, scale, workspace=ws, variant="umma", S_dbg=S)
        torch.cuda.synchronize()
        assert int(ws.abs().max()) == 0
        assert torch.equal(S, want), f"repetition {rep}"
        assert all(torch.equal(out.view(torch.int16), y.view(torch.int16)) for out in ys), f"repetition {rep}"


# Somebody else's small kernel behind a call, let in early, that takes all of the tensor memory of an SM before it waits for that
# call: it gets it when the call's CTA has given it back.
BEHIND = r"""
#include <cuda_runtime.h>
__global__ void behind(const short* y, short* copy, int n) {
  __shared__ unsigned at;
  const unsigned a = (unsigned)__cvta_generic_to_shared(&at);
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(a) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  for (int i = blockIdx.x * 32 + threadIdx.x; i < n; i += gridDim.x * 32) copy[i] = ((volatile const short*)y)[i];
  __syncwarp();
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(*(volatile unsigned*)&at) : "memory");
}
extern "C" int run_behind(const void* y, void* copy, int n, void* stream) {
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3(148);
  c.blockDim = dim3(32);
  c.stream = (cudaStream_t)stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  c.attrs = at;
  c.numAttrs = 1;
  return (int)cudaLaunchKernelEx(&c, behind, (const short*)y, (short*)copy, n);
}
"""


@pytest.fixture(scope="module")
def run_behind(tmp_path_factory):
    d = tmp_path_factory.mktemp("behind")
    (d / "b.cu").write_text(BEHIND)
    subprocess.run([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-O2", "--shared",
                    "-Xcompiler", "-fPIC", "-o", str(d / "b.so"), str(d / "b.cu")], check=True)
    lib = C.CDLL(str(d / "b.so"))
    lib.run_behind.argtypes = [C.c_void_p, C.c_void_p, C.c_int, C.c_void_p]
    return lib.run_behind


@pytest.mark.parametrize("N,K,M", [(40, 128, 1), (2368, 2048, 3), (57344, 8192, 1), (300, 28672, 8)])
def test_a_kernel_behind_that_takes_tensor_memory(run_behind, N, K, M):
    g = torch.Generator(device=DEV)
    g.manual_seed(N)
    words = torch.randint(-2 ** 31, 2 ** 31 - 1, (N, K // 16), dtype=torch.int32, device=DEV, generator=g)
    lut = torch.sort(torch.randn(N, 4, device=DEV, generator=g) * 0.02, dim=1)[0].half()
    xq = torch.randint(0, 256, (M, K // 2), dtype=torch.uint8, device=DEV, generator=g)
    scale = torch.full((M,), 0.1, dtype=torch.float16, device=DEV)
    ws = rcp.make_workspace(M, N, K, DEV)
    want = rcp.rcp_gemv_w2a4(words, lut, xq, scale, workspace=ws, variant="simple")
    y, copy = torch.zeros_like(want), torch.zeros_like(want)
    for rep in range(5):
        y.zero_()
        rcp.rcp_gemv_w2a4(words, lut, xq, scale, y=y, workspace=ws, variant="umma")
        assert run_behind(y.data_ptr(), copy.data_ptr(), y.numel(), torch.cuda.current_stream().cuda_stream) == 0
        torch.cuda.synchronize()
        assert int(ws.abs().max()) == 0
        assert torch.equal(copy.view(torch.int16), want.view(torch.int16)), rep


# shapes whose linear call runs as one kernel of this kind (large ones), every form of the quantizer inside
@pytest.mark.parametrize("N,K,B", [(60000, 8192, 8192), (90000, 4096, 4096), (180000, 2048, 2048), (90000, 5184, 64),
                                   (40000, 11008, 128)])
def test_linear_with_the_quantizer_inside(N, K, B):
    g = torch.Generator(device=DEV)
    g.manual_seed(N)
    words = torch.randint(-2 ** 31, 2 ** 31 - 1, (N, K // 16), dtype=torch.int32, device=DEV, generator=g)
    lut = torch.sort(torch.randn(N, 4, device=DEV, generator=g) * 0.02, dim=1)[0].half()
    x = synth.make_activations(1, K, 5, device=DEV)
    ws = rcp.make_workspace(1, N, K, DEV)
    assert taken(1, N, K, B)
    xq, scale = rcp.rcp_quantize_act(x, B, 1.0)
    want = rcp.rcp_gemv_w2a4(words, lut, xq, scale, workspace=ws, variant="dp4a")
    xq2, scale2 = torch.zeros_like(xq), torch.zeros_like(scale)
    y = rcp.rcp_linear_w2a4(x, B, 1.0, words, lut, xq=xq2, scale=scale2, workspace=ws)
    torch.cuda.synchronize()
    assert int(ws.abs().max()) == 0
    assert torch.equal(xq, xq2) and torch.equal(scale, scale2)
    assert np.array_equal(f16_bits(y), f16_bits(want))
    zero = rcp.rcp_linear_w2a4(torch.zeros_like(x), B, 1.0, words, lut, xq=xq2, scale=scale2, workspace=ws)
    assert not zero.any() and not xq2.any() and not scale2.any()


# Linear calls that run this kernel (N, K, B, M): its quantizer-inside forms, and the forms behind a quantizer, K at once and in parts,
# one and several launches. Results and sums, also those of the checked instantiations, are the plain kernel's.
LINEARS = [(60000, 8192, 8192, 1), (90000, 4096, 4096, 1), (180000, 2048, 2048, 1), (90000, 5184, 64, 1), (40000, 11008, 128, 1),
           (8192, 28672, 128, 1), (57344, 8192, 8192, 8), (8192, 28672, 128, 8), (28672, 4096, 4096, 16), (28672, 20992, 128, 15),
           (5000, 28672, 128, 12), (5000, 65536, 128, 2)]


def run_linear(i):
    N, K, B, M = LINEARS[i]
    inside = rcp.rcp_linear_w2a4_launches(M, N, K, B) == 1
    assert taken(M, N, K, B if inside else 0)
    g = torch.Generator(device=DEV)
    g.manual_seed(N + M)
    words = torch.randint(-2 ** 31, 2 ** 31 - 1, (N, K // 16), dtype=torch.int32, device=DEV, generator=g)
    lut = torch.sort(torch.randn(N, 4, device=DEV, generator=g) * 0.02, dim=1)[0].half()
    x = synth.make_activations(M, K, 6, device=DEV)
    ws = rcp.make_workspace(M, N, K, DEV)
    xq, scale = rcp.rcp_quantize_act(x, B, 1.0)
    want_S, S = (torch.full((M, N, 4), v, dtype=torch.int32, device=DEV) for v in (1, 2))
    want = rcp.rcp_gemv_w2a4(words, lut, xq, scale, workspace=ws, variant="simple", S_dbg=want_S)
    for S_dbg in (None, S):
        xq2, scale2 = torch.zeros_like(xq), torch.zeros_like(scale)
        y = rcp.rcp_linear_w2a4(x, B, 1.0, words, lut, xq=xq2, scale=scale2, workspace=ws, S_dbg=S_dbg)
        torch.cuda.synchronize()
        assert int(ws.abs().max()) == 0
        assert torch.equal(xq, xq2) and torch.equal(scale, scale2)
        assert torch.equal(y.view(torch.int16), want.view(torch.int16))
    assert torch.equal(S, want_S)


@pytest.mark.parametrize("i", range(len(LINEARS)), ids=["x".join(map(str, c)) for c in LINEARS])
def test_linear_calls(i):
    run_linear(i)


def test_linear_calls_in_the_guarded_build():
    in_guarded_build("for i in range(len(t.LINEARS)): t.run_linear(i)")


# Calls of this kernel beside one another and beside a streaming one: several streams, several host threads, a captured step
BESIDE = [(57344, 8192, 8192, 1), (57344, 8192, 8192, 8), (8192, 28672, 128, 3), (4096, 4096, 4096, 1), (28672, 4096, 4096, 16)]


def test_streams_threads_and_replays():
    probs = [streams._problem(N, K, B, M, 700 + i) for i, (N, K, B, M) in enumerate(BESIDE)]
    want = []
    for p in probs:
        streams._run(p)
        torch.cuda.synchronize()
        want.append(p["y"].clone())

    def check(what):
        torch.cuda.synchronize()
        for p, w in zip(probs, want):
            assert torch.equal(p["y"].view(torch.int16), w.view(torch.int16)), what
            assert int(p["ws"].abs().max()) == 0
            p["y"].zero_()
        torch.cuda.synchronize()

    lanes = [torch.cuda.Stream() for _ in probs]
    for rep in range(20):
        for p, st in zip(probs, lanes):
            with torch.cuda.stream(st):
                streams._run(p)
    check("streams")
    errors = []

    def worker(p, st):
        try:
            torch.cuda.set_device(0)
            with torch.cuda.stream(st):
                for rep in range(30):
                    streams._run(p)
                st.synchronize()
        except Exception as e:   # noqa: BLE001
            errors.append(repr(e))

    threads = [threading.Thread(target=worker, args=a) for a in zip(probs, lanes)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    check("threads")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for p in probs:
            streams._run(p)
    for rep in range(3):
        graph.replay()
        graph.replay()
        check(f"replay {rep}")


# Sums of fp32 products stay exact where they grow largest: every code 1 (the e4m3 reading is +2 throughout) against the largest
# activations over the longest K, then a few codes that change the last bits; +2 and -2 in long runs likewise.
@pytest.mark.parametrize("K", [65536, 28672])
def test_sums_at_the_ends_of_their_range(K):
    g = torch.Generator(device=DEV)
    g.manual_seed(K)
    N, M = 48, 2
    codes = torch.ones(N, K, dtype=torch.uint8, device=DEV)
    rnd = torch.randint(0, 4, (N, K), generator=g, device=DEV, dtype=torch.uint8)
    codes[1:8, -64:] = rnd[1:8, -64:]
    codes[8:16, ::129] = rnd[8:16, ::129]
    codes[16:24, K // 2:] = 3
    codes[24:32, 0::2] = 3
    codes[32:40] = 3 * (rnd[32:40] > 0).to(torch.uint8)
    codes[40:48] = 2 + rnd[40:48] // 3
    words = rcp.rcp_pack_weights(codes)
    lut = torch.sort(torch.randn(N, 4, device=DEV, generator=g) * 0.02, dim=1)[0].half()
    xq = torch.full((M, K // 2), 0x77, dtype=torch.uint8, device=DEV)
    xq[1, 1::3] = torch.randint(0, 256, xq[1, 1::3].shape, generator=g, device=DEV, dtype=torch.uint8)
    scale = torch.tensor([0.01, 0.02], dtype=torch.float16, device=DEV)
    S = torch.empty(M, N, 4, dtype=torch.int32, device=DEV)
    rcp.rcp_gemv_w2a4(words, lut, xq, scale, workspace=rcp.make_workspace(M, N, K, DEV), variant="umma", S_dbg=S)
    torch.cuda.synchronize()
    ref = oracle.gemv_w2a4(words.cpu().numpy().view(np.uint32), f16_bits(lut), xq.cpu().numpy(), f16_bits(scale))
    assert np.array_equal(S.cpu().numpy(), ref["S"])
