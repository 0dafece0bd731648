"""Builds the CUDA library in-tree with nvcc for sm_100a (cross-compiles without a GPU), and the native half of its
Python binding with g++ against the installed PyTorch."""
import os
import re
import subprocess
import sys
import sysconfig

_HERE = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_HERE)
CSRC = os.path.join(_HERE, "csrc")
LIB_DIR = os.path.join(_HERE, "_lib")
LIB_PATH = os.path.join(LIB_DIR, "libtvm_attn.so")
SOURCES = ["tvm_attn_api.cu"]
BINDING_SOURCE = os.path.join(CSRC, "torch_binding.cpp")


def _newest_source_mtime():
    newest = 0.0
    for d in (CSRC, os.path.join(_ROOT, "include")):
        for name in os.listdir(d):
            newest = max(newest, os.path.getmtime(os.path.join(d, name)))
    return newest


def nvcc_command(out_path, extra=()):
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    return [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
            "-Xcompiler", "-fPIC", "-shared", "-I", os.path.join(_ROOT, "include"), "-I", CSRC,
            *extra, "-o", out_path, *[os.path.join(CSRC, s) for s in SOURCES]]


def binding_path():
    """Where the binding's native half lies.  It uses PyTorch's C++ interface, which changes from one build of PyTorch to the
    next, and CPython's: each pair has a file of its own, so that another PyTorch never loads an object made for this one."""
    import torch
    tag = "%s-%s-%s" % (torch.__version__, (torch.version.git_version or "")[:8], sys.implementation.cache_tag)
    return os.path.join(LIB_DIR, "_tvm_binding-%s.so" % re.sub(r"[^A-Za-z0-9.+-]", "_", tag))


def binding_command(out_path):
    import torch
    root = os.path.dirname(torch.__file__)
    libs = [os.path.join(root, "lib"), "/usr/local/cuda/lib64"]
    return [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
            "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI), "-I", os.path.join(_ROOT, "include"),
            "-isystem", os.path.join(root, "include"), "-isystem", os.path.join(root, "include", "torch", "csrc", "api", "include"),
            "-isystem", "/usr/local/cuda/include", "-isystem", sysconfig.get_paths()["include"], BINDING_SOURCE, "-o", out_path,
            *["-L" + d for d in libs], "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_cuda", "-ltorch", "-ltorch_python"]


def build_binding(force=False):
    """Compiles the binding's native half if there is none for this PyTorch or it is older than its source; returns its path."""
    path = binding_path()
    header = os.path.join(_ROOT, "include", "tvm_attn.h")
    if not force and os.path.exists(path) and os.path.getmtime(path) >= max(os.path.getmtime(f) for f in (BINDING_SOURCE, header)):
        return path
    _run(binding_command, path)
    return path


def _run(command, path, *args):
    """Runs command(temporary path, ...) and moves what it wrote to `path`; returns its messages."""
    os.makedirs(os.path.dirname(path), exist_ok=True)
    tmp = path + ".tmp.%d" % os.getpid()
    cmd = command(tmp, *args)
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("compilation failed:\n%s\n%s" % (" ".join(cmd), res.stderr[-8000:]))
    os.replace(tmp, path)
    return res.stderr


def build(force=False, verbose=False, out_path=None):
    """Compiles libtvm_attn.so if it is missing or older than its sources; returns its path.
    `out_path` writes the library somewhere else.  The binding's native half is built along with the in-tree library."""
    global_out = out_path or LIB_PATH
    if out_path is None:
        build_binding(force)
    if not force and os.path.exists(global_out) and os.path.getmtime(global_out) >= _newest_source_mtime():
        return global_out
    messages = _run(nvcc_command, global_out, ("-Xptxas", "-v") if verbose else ())
    if verbose:
        print(messages)
    return global_out


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
