"""Builds the CUDA library in-tree with nvcc for sm_100a (cross-compiles without a GPU), and the native argument
marshalling of the Python binding with the host compiler."""
import hashlib
import os
import re
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "librcp_w2a4.so")
LIB_CHECKED = os.path.join(HERE, "librcp_w2a4_checked.so")   # the guarded build (-DRCP_CHECKED), for tests
DRIVER = os.path.join(HERE, "e2e_driver")                     # host program: a decode step through the C ABI
HEADER = os.path.join(os.path.dirname(HERE), "include", "rcp.h")
SOURCES = ["rcp_api.cu"]


def header_id() -> int:
    """A number for the declarations of include/rcp.h (comments and spaces left out), compiled into the library and into the
    marshalling module, so that the module does not call a library of other signatures."""
    text = re.sub(r"/\*.*?\*/", " ", open(HEADER).read(), flags=re.S)
    return int(hashlib.sha1(" ".join(text.split()).encode()).hexdigest()[:15], 16)


def marshal_path() -> str:
    """csrc/binding.cpp as an extension module: good for one Python and one torch, which its name says."""
    import torch
    return os.path.join(HERE, f"_marshal.{sys.implementation.cache_tag}-torch{torch.__version__}.so")


def _newest_source_mtime() -> float:
    paths = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if not f.endswith(".cpp")]
    paths.append(HEADER)
    return max(os.path.getmtime(p) for p in paths)


def _compile(out: str, defines=(), verbose: bool = False) -> str:
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cmd = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
           "--shared", "-Xcompiler", "-fPIC", f"-DRCP_HEADER_ID={header_id()}ull", "-o", out] + [f"-D{d}" for d in defines] + \
          [os.path.join(CSRC, s) for s in SOURCES]
    if verbose:
        cmd.insert(1, "-Xptxas=-v")
    subprocess.check_call(cmd)
    return out


def build(force: bool = False, verbose: bool = False) -> str:
    """The library, and the module the binding calls it through; returns the library's path."""
    build_marshal(force)
    if not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= _newest_source_mtime():
        return LIB
    return _compile(LIB, verbose=verbose)


def build_checked(force: bool = False) -> str:
    """The guarded build: the same sources with -DRCP_CHECKED (shared-memory addresses and TMA requests of the
    streaming kernel checked against the host's layout; a violation is reported through the status word)."""
    if not force and os.path.exists(LIB_CHECKED) and os.path.getmtime(LIB_CHECKED) >= _newest_source_mtime():
        return LIB_CHECKED
    return _compile(LIB_CHECKED, defines=("RCP_CHECKED",))


def build_marshal(force: bool = False) -> str:
    src = os.path.join(CSRC, "binding.cpp")
    out = marshal_path()
    if not force and os.path.exists(out) and os.path.getmtime(out) >= max(os.path.getmtime(src), os.path.getmtime(HEADER)):
        return out
    import torch
    from torch.utils import cpp_extension
    flags = ["-I" + d for d in cpp_extension.include_paths()] + ["-I" + sysconfig.get_paths()["include"], "-I/usr/local/cuda/include"]
    libs = ["-L" + d for d in cpp_extension.library_paths()] + ["-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"]
    defines = [f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", f"-DRCP_HEADER_ID={header_id()}ull"]
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-fPIC", "-shared"] + defines + flags + ["-o", out, src] + libs)
    return out


def build_driver(force: bool = False) -> str:
    """The end-to-end driver (e2e_driver.cu): a C++ host program linked against the library, run by bench.py."""
    build()
    src = os.path.join(HERE, "e2e_driver.cu")
    if not force and os.path.exists(DRIVER) and os.path.getmtime(DRIVER) >= max(os.path.getmtime(src), os.path.getmtime(LIB)):
        return DRIVER
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    subprocess.check_call([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-O2", "-std=c++17", "-o", DRIVER, src,
                           "-L" + HERE, "-lrcp_w2a4", "-Xlinker", "-rpath", "-Xlinker", "$ORIGIN"])
    return DRIVER


if __name__ == "__main__":
    import sys
    print(build(force=True, verbose=True))
    print(marshal_path())
    print(build_driver(force=True))
    if "--checked" in sys.argv[1:]:
        print(build_checked(force=True))
