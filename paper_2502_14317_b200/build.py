"""Builds libpc.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and _pc_host.so (host side of the binding) with the C++ compiler."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB_PATH = os.path.join(HERE, "libpc.so")
HOST_SOURCE = "pc_host.cpp"
SOURCES = ["pc_api.cu", "pc_prefill2.cu", "pc_parallel.cu", "pc_decode.cu", "pc_rope.cu", "pc_select_gather.cu", "pc_queue.cu", "pc_static_scratch.cu"]
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo",
    "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden", "--expt-relaxed-constexpr",
]


def host_path(torch_version) -> str:
    """_pc_host.so for this Python and that torch.  It is compiled against the C++ classes of one torch and the ABI of one Python, so their
    versions are part of its name: after an upgrade the file is not there, instead of one that is loaded and crashes."""
    return os.path.join(HERE, "_pc_host-torch%s%s" % (torch_version, sysconfig.get_config_var("EXT_SUFFIX")))


def _nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _older(path, sources) -> bool:
    sources = [os.path.join(CSRC, f) for f in sources] + [os.path.join(HERE, "..", "include", "pc.h"), os.path.join(HERE, "build.py")]
    return not os.path.exists(path) or any(os.path.getmtime(p) > os.path.getmtime(path) for p in sources)


def needs_build() -> bool:
    return _older(LIB_PATH, [f for f in os.listdir(CSRC) if f != HOST_SOURCE])


def _torch():
    """The installed torch; None where there is none, or one that cannot be loaded."""
    try:
        import torch
    except (ImportError, OSError):
        return None
    return torch


def _host_command(torch):
    """Command that compiles csrc/pc_host.cpp against that torch."""
    root = os.path.dirname(torch.__file__)
    inc = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"), sysconfig.get_paths()["include"]]
    lib = os.path.join(root, "lib")
    return [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
            "-D_GLIBCXX_USE_CXX11_ABI=%d" % torch._C._GLIBCXX_USE_CXX11_ABI, *("-isystem" + d for d in inc), os.path.join(CSRC, HOST_SOURCE),
            "-L" + lib, "-Wl,-rpath," + lib, "-ltorch_python", "-ltorch_cpu", "-lc10"]


def build_library(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu under csrc/ into one shared library, and beside it csrc/pc_host.cpp into _pc_host.so; returns the library's path.

    The library needs nvcc alone.  _pc_host.so, the host side of the binding's hot_path, needs torch, the Python headers and a C++ compiler: where
    one of them is missing or fails that is said on stderr, the library is built all the same, and hot_path raises PcError."""
    os.makedirs(os.path.join(HERE, "_build"), exist_ok=True)
    new_lib = os.path.join(HERE, "_build", os.path.basename(LIB_PATH))
    host, torch = None, _torch()
    if torch is None:
        sys.stderr.write("_pc_host.so is not built: torch cannot be imported\n")
    elif force or _older(host_path(torch.__version__), [HOST_SOURCE]):
        new_host = os.path.join(HERE, "_build", os.path.basename(host_path(torch.__version__)))
        try:
            host = subprocess.Popen(_host_command(torch) + ["-o", new_host], stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
        except OSError as e:
            sys.stderr.write("_pc_host.so is not built: %s\n" % e)
    procs, objs = [], []
    if force or needs_build():
        for src in SOURCES:
            obj = os.path.join(HERE, "_build", src.replace(".cu", ".o"))
            cmd = [_nvcc(), *NVCC_FLAGS, "-c", os.path.join(CSRC, src), "-o", obj]
            if verbose:
                cmd.insert(1, "-Xptxas=-v")
            procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
            objs.append(obj)
    failed = []
    for src, p in procs:
        out, _ = p.communicate()
        if verbose or p.returncode != 0:
            sys.stderr.write(out)
        if p.returncode != 0:
            failed.append(src)
    if host is not None:
        out, _ = host.communicate()
        if verbose or host.returncode != 0:
            sys.stderr.write(out)
        if host.returncode == 0:
            os.replace(new_host, host_path(torch.__version__))   # (a process that has the old one mapped keeps it)
        else:
            sys.stderr.write("_pc_host.so is not built: compiling %s failed\n" % HOST_SOURCE)
    if failed:
        raise RuntimeError("compiling %s failed" % ", ".join(failed))
    if objs:
        link = [_nvcc(), "-shared", "-o", new_lib, *objs, "-gencode", "arch=compute_100a,code=sm_100a"]
        r = subprocess.run(link, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
        if r.returncode != 0:
            sys.stderr.write(r.stdout)
            raise RuntimeError("link failed")
        os.replace(new_lib, LIB_PATH)
    return LIB_PATH


if __name__ == "__main__":
    print(build_library(force="--force" in sys.argv, verbose="-v" in sys.argv))
