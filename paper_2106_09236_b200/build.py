"""Builds libpsattn.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a."""
from __future__ import annotations

import hashlib
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libpsattn.so")
NATIVE = os.path.join(HERE, "psattn_torch.so")       # the native side of the Python binding (a CPython module)
NATIVE_SOURCE = os.path.join(CSRC, "psattn_torch.cpp")
SOURCES = ["psattn_api.cu", "psattn_staged.cu", "psattn_noalloc.cu", "psattn_attend_tc.cu", "psattn_measure_mma.cu", "psattn_measure_shared.cu", "psattn_exact_measure.cu", "psattn_project.cu", "psattn_attend64.cu", "psattn_fused.cu", "psattn_fused_fp32.cu", "psattn_probe.cu", "psattn_project_out.cu"]
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC",
]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def built_from() -> bytes:
    """Digest of the flags and of the sources of libpsattn.so; the library holds it as a string."""
    h = hashlib.sha1(" ".join(NVCC_FLAGS).encode())
    files = sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh", ".h")))
    for path in files + [os.path.join(os.path.dirname(HERE), "include", "psattn.h")]:
        with open(path, "rb") as f:
            h.update(os.path.basename(path).encode() + f.read())
    return b"built from " + h.hexdigest().encode()


def needs_build() -> bool:
    """Missing, or built from other sources (by content: a file put back to an older state is older than the library)."""
    if not os.path.exists(LIB):
        return True
    with open(LIB, "rb") as f:
        return built_from() + b"\0" not in f.read()


def build(force: bool = False, verbose: bool = False, phase_stamps: bool = False, nvtx: bool = False) -> str:
    """Builds the library.  phase_stamps: a second library, libpsattn_stamps.so, whose kernels record per-phase
    times and their begin and end (-DPSATTN_PHASE_STAMPS); only the benchmark's --phases mode uses it.
    nvtx: a library, libpsattn_nvtx.so, with a named range around every compute entry point (-DPSATTN_NVTX) for
    timeline tools; load it with PSATTN_LIBRARY."""
    if phase_stamps:
        return _build_variant("libpsattn_stamps.so", ["-DPSATTN_PHASE_STAMPS"], ".stamps.o")
    if nvtx:
        return _build_variant("libpsattn_nvtx.so", ["-DPSATTN_NVTX"], ".nvtx.o", ["-ldl"])
    if not force and not needs_build():
        return LIB
    objs, key = [], built_from().decode()
    for src in SOURCES:
        obj = os.path.join(CSRC, src.replace(".cu", ".o"))
        cmd = [_nvcc(), *NVCC_FLAGS, '-DPSATTN_BUILT_FROM="%s"' % key, "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas")
            cmd.insert(2, "-v")
            print(" ".join(cmd), file=sys.stderr)
        subprocess.check_call(cmd)
        objs.append(obj)
    tmp = LIB + ".tmp.%d" % os.getpid()
    subprocess.check_call([_nvcc(), "-shared", "-o", tmp, *objs, "-lcudart"])
    os.replace(tmp, LIB)
    return LIB


def native_built_for() -> bytes:
    """What the native module is compiled against: the layout of torch's and Python's objects belongs to these versions."""
    import sysconfig

    import torch
    return ("built for torch %s, C++11 ABI %d, %s" % (torch.__version__, int(torch._C._GLIBCXX_USE_CXX11_ABI),
                                                      sysconfig.get_config_var("SOABI"))).encode()


def native_needs_build() -> bool:
    """Missing, older than its source, or compiled against another torch or Python (the module holds the text as a string)."""
    if not os.path.exists(NATIVE) or os.path.getmtime(NATIVE_SOURCE) > os.path.getmtime(NATIVE):
        return True
    with open(NATIVE, "rb") as f:
        return native_built_for() + b"\0" not in f.read()


def build_native(verbose: bool = False) -> str:
    """Builds the module that marshals torch tensors into the C calls (g++ against torch's headers; no CUDA code)."""
    import sysconfig

    import torch
    root = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(_nvcc())) if os.path.isabs(_nvcc()) else "/usr/local/cuda"
    inc = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
           sysconfig.get_paths()["include"], os.path.join(cuda, "include")]
    tmp = NATIVE + ".tmp.%d" % os.getpid()
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI),
           '-DPSATTN_BUILT_FOR="%s"' % native_built_for().decode(), *["-I" + i for i in inc],
           NATIVE_SOURCE, "-o", tmp, "-L" + os.path.join(root, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10",
           "-lc10_cuda", "-Wl,-rpath," + os.path.join(root, "lib")]
    if verbose:
        print(" ".join(cmd), file=sys.stderr)
    subprocess.check_call(cmd)
    os.replace(tmp, NATIVE)
    return NATIVE


def _build_variant(name: str, extra: list, suffix: str, link: list = ()) -> str:
    out = os.path.join(HERE, name)
    objs = []
    for src in SOURCES:
        obj = os.path.join(CSRC, src.replace(".cu", suffix))
        subprocess.check_call([_nvcc(), *NVCC_FLAGS, *extra, "-c", os.path.join(CSRC, src), "-o", obj])
        objs.append(obj)
    tmp = out + ".tmp.%d" % os.getpid()
    subprocess.check_call([_nvcc(), "-shared", "-o", tmp, *objs, "-lcudart", *link])
    os.replace(tmp, out)
    return out


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv, nvtx="--nvtx" in sys.argv))
    if "--force" in sys.argv or native_needs_build():
        print(build_native(verbose="-v" in sys.argv))
