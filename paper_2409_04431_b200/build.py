"""Builds libsigattn.so in-tree with nvcc for sm_100a (cross-compiles without a GPU), and the compiled host side of
the Python binding (_sigattn_host.so) against the installed torch."""
from __future__ import annotations

import importlib.util
import os
import shutil
import subprocess
import sys
import sysconfig

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG_DIR, "csrc")
LIB_PATH = os.path.join(PKG_DIR, "libsigattn.so")
HOST_PATH = os.path.join(PKG_DIR, "_sigattn_host.so")
SOURCES = ["sigattn_api.cu", "sigattn_fp32.cu", "sigattn_fwd_sm100.cu", "sigattn_fwd_single_sm100.cu", "sigattn_bwd_sm100.cu",
           "sigattn_decode_sm100.cu", "sigattn_short_fwd_sm100.cu", "sigattn_short_bwd_sm100.cu",
           "sigattn_static_scratch.cu", "sigattn_peer.cu"]
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-O3", "-std=c++17", "-lineinfo",
    "-Xcompiler", "-fPIC",
    "-Xcompiler", "-fvisibility=hidden",
]


def _nvcc() -> str:
    path = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(path):
        raise RuntimeError("nvcc not found: libsigattn.so cannot be built")
    return path


def _host_command() -> list[str]:
    """g++ command of the host module: torch's own headers and libraries, libsigattn.so from beside it."""
    torch_dir = list(importlib.util.find_spec("torch").submodule_search_locations)[0]
    inc = os.path.join(torch_dir, "include")
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(_nvcc())))
    return ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
            "-I", sysconfig.get_paths()["include"], "-isystem", inc,
            "-isystem", os.path.join(inc, "torch", "csrc", "api", "include"), "-isystem", os.path.join(cuda, "include"),
            os.path.join(CSRC, "host_calls.cpp"), "-o", HOST_PATH, "-L", os.path.join(torch_dir, "lib"),
            "-ltorch_python", "-ltorch_cpu", "-ltorch", "-lc10", "-lc10_cuda", "-L", PKG_DIR, "-lsigattn",
            "-Wl,-rpath,$ORIGIN"]


def _stale() -> bool:
    if not os.path.exists(LIB_PATH) or not os.path.exists(HOST_PATH):
        return True
    built = min(os.path.getmtime(LIB_PATH), os.path.getmtime(HOST_PATH))
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    deps.append(os.path.join(os.path.dirname(PKG_DIR), "include", "sigattn.h"))
    deps.append(os.path.abspath(__file__))
    return any(os.path.getmtime(d) > built for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every CUDA source into libsigattn.so (one object per source, in parallel), then the host module."""
    if not force and not _stale():
        return LIB_PATH
    nvcc = _nvcc()
    obj_dir = os.path.join(PKG_DIR, "build")
    os.makedirs(obj_dir, exist_ok=True)
    procs = []
    objs = []
    for src in SOURCES:
        obj = os.path.join(obj_dir, src.replace(".cu", ".o"))
        objs.append(obj)
        cmd = [nvcc, *NVCC_FLAGS, "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = False
    for src, proc in procs:
        out, _ = proc.communicate()
        if proc.returncode != 0:
            failed = True
            sys.stderr.write(f"nvcc failed on {src}:\n{out}\n")
        elif verbose or out.strip():
            sys.stderr.write(out)
    if failed:
        raise RuntimeError("libsigattn.so build failed")
    link = [nvcc, "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", LIB_PATH, *objs]
    subprocess.run(link, check=True)
    subprocess.run(_host_command(), check=True)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
