"""Builds libtik.so (the C-ABI library) with nvcc for sm_100a and its torch binding, in-tree."""
from __future__ import annotations

import concurrent.futures
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB_PATH = os.path.join(HERE, "libtik.so")
BIND_PATH = os.path.join(HERE, "_tikbind.so")      # CPython module that marshals torch tensors into libtik.so
BIND_SOURCE = "tik_bind.cpp"
SOURCES = ["tik_api.cu", "tik_attn.cu", "tik_attn_persist.cu", "tik_decode.cu", "tik_decode_cluster.cu", "tik_logprob.cu", "tik_static.cu", "tik_prep.cu", "tik_ffn.cu", "tik_linear.cu", "tik_attn_bwd.cu"]
HEADERS = ["tik_core.cuh", "tik_ptx.cuh", "tik_internal.h", os.path.join("..", "..", "include", "tik.h")]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-Xptxas", "-v"]


def _nvcc() -> str:
    exe = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(exe):
        raise RuntimeError("nvcc not found; libtik.so cannot be built")
    return exe


def _sources():
    return [s for s in SOURCES if os.path.exists(os.path.join(CSRC, s))]


def needs_build() -> bool:
    if not os.path.exists(LIB_PATH) or not os.path.exists(BIND_PATH):
        return True
    t = min(os.path.getmtime(LIB_PATH), os.path.getmtime(BIND_PATH))
    deps = [os.path.join(CSRC, f) for f in _sources() + HEADERS + [BIND_SOURCE]]
    return any(os.path.getmtime(d) > t for d in deps if os.path.exists(d))


def _build_bind() -> None:
    """The extension module: host C++ against torch's headers, linked to libtik.so beside it."""
    import sysconfig

    import torch
    inc = os.path.join(os.path.dirname(torch.__file__), "include")
    lib = os.path.join(os.path.dirname(torch.__file__), "lib")
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(_nvcc())))
    cmd = [shutil.which("g++") or "g++", "-O2", "-std=c++17", "-fPIC", "-shared",
           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch.compiled_with_cxx11_abi()),
           "-I" + inc, "-I" + os.path.join(inc, "torch", "csrc", "api", "include"),
           "-I" + sysconfig.get_paths()["include"], "-I" + os.path.join(cuda, "include"),
           os.path.join(CSRC, BIND_SOURCE), "-o", BIND_PATH, "-L" + HERE, "-l:libtik.so", "-Wl,-rpath,$ORIGIN",
           "-L" + lib, "-lc10", "-ltorch_cpu", "-lc10_cuda", "-ltorch_cuda", "-ltorch", "-ltorch_python"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("building %s failed:\n%s" % (os.path.basename(BIND_PATH), r.stderr))


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu under csrc/ and link them into libtik.so, then the extension module that
    binds it to torch; returns the library's path."""
    if not force and not needs_build():
        return LIB_PATH
    nvcc = _nvcc()
    os.makedirs(os.path.join(HERE, "build"), exist_ok=True)
    objs = [os.path.join(HERE, "build", src.replace(".cu", ".o")) for src in _sources()]

    def compile_one(src, obj):
        return subprocess.run([nvcc] + NVCC_FLAGS + ["-c", os.path.join(CSRC, src), "-o", obj], capture_output=True, text=True)

    logs = []
    with concurrent.futures.ThreadPoolExecutor(os.cpu_count() or 4) as pool:
        for src, r in zip(_sources(), pool.map(compile_one, _sources(), objs)):
            logs.append(r.stderr)
            if r.returncode != 0:
                raise RuntimeError("nvcc failed for %s:\n%s" % (src, r.stderr))
    cmd = [nvcc, "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", LIB_PATH] + objs
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("link failed:\n" + r.stderr)
    _build_bind()
    with open(os.path.join(HERE, "build", "ptxas.log"), "w") as f:
        f.write("\n".join(logs))
    if verbose:
        sys.stderr.write("\n".join(logs))
    return LIB_PATH


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
