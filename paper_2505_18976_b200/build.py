"""In-tree build of the sm_100a shared library ``libgrass_b200.so`` with nvcc, and of the ``_native`` extension (the
binding's per-call marshalling) with the host compiler."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
SO = os.path.join(HERE, "libgrass_b200.so")
NATIVE = os.path.join(HERE, "_native.so")
NATIVE_SRC = "binding_native.cpp"
SOURCES = ["grass_compress.cu", "grass_compress_rows.cu", "grass_sjlt_table.cu", "factgrass.cu", "factgrass_cluster.cu", "factgrass_persistent.cu", "grass_score.cu", "grass_score_tc.cu", "grass_score_bf16.cu", "grass_fim.cu", "grass_fim_gram.cu", "grass_fim_blocks.cu", "grass_util.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-cudart", "static"]


def _nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _stale(so: str = SO) -> bool:
    if not os.path.exists(so):
        return True
    t = os.path.getmtime(so)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)
            if (f == NATIVE_SRC if so == NATIVE else f.endswith((".cu", ".cuh", ".h")))]
    deps.append(os.path.join(os.path.dirname(HERE), "include", "grass.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def _native_cmd(out: str) -> list:
    """Host compiler command of the extension, against the headers and libraries of the installed torch."""
    from importlib.util import find_spec
    tdir = os.path.dirname(find_spec("torch").origin)
    inc = [os.path.join(tdir, "include"), os.path.join(tdir, "include", "torch", "csrc", "api", "include"),
           sysconfig.get_paths()["include"], os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")]
    return ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden", *["-I" + d for d in inc],
            os.path.join(CSRC, NATIVE_SRC), "-o", out, "-L" + os.path.join(tdir, "lib"), "-lc10", "-lc10_cuda",
            "-ltorch_cpu", "-ltorch_cuda", "-ltorch_python"]


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu for sm_100a and link them into one shared object next to this file, and the extension
    module beside it."""
    native = None
    if force or _stale(NATIVE):
        ntmp = NATIVE + f".tmp{os.getpid()}"
        native = subprocess.Popen(_native_cmd(ntmp))
    try:
        if force or _stale():
            _build_library(verbose)
    finally:
        if native is not None and native.wait() == 0:
            os.replace(ntmp, NATIVE)
    if native is not None and native.returncode != 0:
        raise RuntimeError("building the _native extension failed")
    return SO


def _build_library(verbose: bool) -> None:
    objs = []
    bdir = os.path.join(HERE, "_build")
    os.makedirs(bdir, exist_ok=True)
    procs = []
    for src in SOURCES:
        obj = os.path.join(bdir, src.replace(".cu", ".o"))
        cmd = [_nvcc(), *NVCC_FLAGS, "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas")
            cmd.insert(2, "-v")
        procs.append((cmd, subprocess.Popen(cmd)))
        objs.append(obj)
    for cmd, p in procs:
        if p.wait() != 0:
            raise RuntimeError("nvcc failed: " + " ".join(cmd))
    tmp = SO + f".tmp{os.getpid()}"
    subprocess.check_call([_nvcc(), "-shared", "-cudart", "static", "-o", tmp, *objs])
    os.replace(tmp, SO)


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
