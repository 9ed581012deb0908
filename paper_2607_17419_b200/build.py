"""Build libkata.so in-tree with nvcc for sm_100a (cross-compiles without a GPU)."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
import warnings
from typing import Optional

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libkata.so")
HOST = os.path.join(HERE, "_kata_torch.so")      # the binding's tensor calls (csrc/kata_torch.cpp)
SOURCES = ["kata_api.cu", "kata_simt_quadratic.cu", "kata_simt_bwd.cu", "kata_simt_bwd_chunked.cu", "kata_simt_chunked.cu", "kata_simt_order1.cu", "kata_simt_attend.cu", "kata_tc.cu", "kata_tc_chunked.cu",
    "kata_tc_stream.cu", "kata_tc_stream_export.cu", "kata_tc_stream_restart.cu", "kata_tc_stream_state.cu", "kata_tc_attend.cu", "kata_tc_state.cu", "kata_tc_bwd.cu", "kata_tc_order1.cu", "kata_decode.cu", "kata_static.cu", "kata_selftest.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "--use_fast_math=false"]


def _nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def host_tag() -> Optional[str]:
    """What the native module is built for: it holds torch's C++ layouts and Python's.  None: there is no torch to build against."""
    try:
        import torch
    except ImportError:
        return None
    return f"kata_torch for torch {torch.__version__} {torch.version.git_version}, {sysconfig.get_config_var('SOABI')}"


def host_current() -> bool:
    """Whether the native module was built for the torch and the Python that run now (its tag is a string inside it)."""
    tag = host_tag()
    if tag is None or not os.path.exists(HOST):
        return False
    with open(HOST, "rb") as f:
        return tag.encode() + b"\0" in f.read()


def _newer_source(target: str) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(HERE, "..", "include", "kata.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def host_needs_build() -> bool:
    return host_tag() is not None and (_newer_source(HOST) or not host_current())


def needs_build() -> bool:
    return _newer_source(LIB) or host_needs_build()


def _host_command(obj: str) -> list:
    """Compiler call for the binding's native module."""
    import torch
    inc = os.path.join(os.path.dirname(torch.__file__), "include")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    return ["g++", "-O2", "-std=c++17", "-fPIC", "-fvisibility=hidden", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
            f'-DKATA_HOST_TAG="{host_tag()}"',
            "-isystem", inc, "-isystem", os.path.join(inc, "torch", "csrc", "api", "include"), "-isystem", os.path.join(cuda, "include"),
            "-isystem", sysconfig.get_path("include"), "-c", os.path.join(CSRC, "kata_torch.cpp"), "-o", obj]


def _host_link(obj: str) -> list:
    import torch
    lib = os.path.join(os.path.dirname(torch.__file__), "lib")
    return ["g++", "-shared", "-o", HOST, obj, "-L" + HERE, "-l:libkata.so", "-Wl,-rpath,$ORIGIN", "-L" + lib, "-lc10", "-lc10_cuda", "-ltorch_cpu",
            "-ltorch_python"]


def _build_host(objdir: str) -> None:
    """The binding's native module.  Without it (no compiler for it, no Python headers, a torch without CUDA) the binding's calls go
    through ctypes, so a failure is a warning."""
    if os.path.exists(HOST):
        os.remove(HOST)
    obj = os.path.join(objdir, "kata_torch.host.o")
    for command in (_host_command, _host_link):
        try:
            pr = subprocess.run(command(obj), stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
            failed, out = pr.returncode != 0, pr.stdout
        except OSError as e:
            failed, out = True, str(e)
        if failed:
            warnings.warn(f"{os.path.basename(HOST)} was not built, tensor calls will go through ctypes:\n{out}")
            return


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu into objects (in parallel) and link libkata.so next to this file, and the binding's native module."""
    objdir = os.path.join(HERE, "build")
    os.makedirs(objdir, exist_ok=True)
    if force or _newer_source(LIB):
        flags = [f for f in NVCC_FLAGS if not f.startswith("--use_fast_math")]
        procs = []
        objs = []
        for src in SOURCES:
            obj = os.path.join(objdir, src.replace(".cu", ".o"))
            objs.append(obj)
            cmd = [_nvcc(), *flags, "-c", os.path.join(CSRC, src), "-o", obj]
            if verbose:
                cmd.insert(1, "-Xptxas=-v")
            procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        failed = False
        for src, pr in procs:
            out, _ = pr.communicate()
            if pr.returncode != 0 or verbose:
                sys.stderr.write(f"--- {src} ---\n{out}\n")
            failed |= pr.returncode != 0
        if failed:
            raise RuntimeError("nvcc failed")
        subprocess.check_call([_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-o", LIB, *objs])
    if host_tag() is not None and (force or host_needs_build()):
        _build_host(objdir)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
