"""The C-ABI shared library loads and exports every function include/rcp.h declares (no GPU needed)."""
import ctypes
import os
import re
import shutil

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _declared_functions():
    text = open(os.path.join(ROOT, "include", "rcp.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(rcp_[a-z0-9_]+)\s*\(", text)))


@pytest.fixture(scope="module")
def libpath():
    from paper_2502_15779_b200 import build
    if not os.path.exists(build.LIB) and shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"):
        pytest.skip("no nvcc and no prebuilt library")
    return build.build()


def test_header_declares_the_three_hot_path_calls():
    names = _declared_functions()
    for required in ("rcp_pack_weights", "rcp_quantize_act", "rcp_gemv_w2a4"):
        assert required in names


def test_library_exports_every_declared_symbol(libpath):
    L = ctypes.CDLL(libpath)
    for name in _declared_functions():
        assert hasattr(L, name), name


def test_status_strings_and_workspace_query_run_without_gpu(libpath):
    L = ctypes.CDLL(libpath)
    L.rcp_status_str.restype = ctypes.c_char_p
    for code in range(0, -9, -1):
        assert L.rcp_status_str(code) not in (None, b"")
    L.rcp_gemv_workspace_bytes.restype = ctypes.c_size_t
    assert L.rcp_gemv_workspace_bytes(1, 0, 4096) == 0      # bad shape -> 0
    assert L.rcp_gemv_workspace_bytes(1, 4096, 100) == 0    # K % 64 != 0 -> 0
    assert L.rcp_gemv_workspace_bytes(1, 4096, 4096) % 16 == 0


def test_binding_fails_loudly_without_library(monkeypatch, tmp_path):
    from paper_2502_15779_b200 import binding
    monkeypatch.setattr(binding, "_lib", None)
    monkeypatch.setattr(binding, "LIB_PATH", str(tmp_path / "missing.so"))
    with pytest.raises(RuntimeError, match="no CPU or PyTorch fallback"):
        binding.lib()


def test_library_and_marshalling_module_are_of_one_header(libpath):
    from paper_2502_15779_b200 import build
    L = ctypes.CDLL(libpath)
    L.rcp_header_id.restype = ctypes.c_ulonglong
    assert L.rcp_header_id() == build.header_id() != 0
    assert os.path.exists(build.marshal_path())   # build() makes it as well


def test_binding_refuses_a_library_of_another_header(libpath, monkeypatch, tmp_path):
    """The marshalling module calls by address, with the prototypes it was compiled with."""
    from paper_2502_15779_b200 import binding
    monkeypatch.setattr(binding, "_m", None)
    monkeypatch.setattr(binding, "_lib", None)
    m = binding._native()
    other = ctypes.CFUNCTYPE(ctypes.c_ulonglong)(lambda: 12345)
    table = {name: ctypes.cast(getattr(binding.lib(), name), ctypes.c_void_p).value for name in binding._MARSHALLED}
    m.bind(table)
    with pytest.raises(RuntimeError, match="same include/rcp.h"):
        m.bind(dict(table, rcp_header_id=ctypes.cast(other, ctypes.c_void_p).value))
    m.bind(table)
    monkeypatch.setattr(binding, "_m", None)
    monkeypatch.setattr(binding, "_MARSHAL_PATH", str(tmp_path / "_marshal.of-another-torch.so"))
    with pytest.raises(RuntimeError, match="one Python and one torch"):
        binding._native()


def test_header_id_follows_declarations_alone(monkeypatch, tmp_path):
    from paper_2502_15779_b200 import build
    text = open(build.HEADER).read()
    was = build.header_id()
    for change, same in ((lambda t: t.replace("/*", "/* more", 1), True), (lambda t: t.replace("int M, int N", "int N, int M", 1), False)):
        p = tmp_path / "rcp.h"
        p.write_text(change(text))
        assert p.read_text() != text
        monkeypatch.setattr(build, "HEADER", str(p))
        assert (build.header_id() == was) == same
