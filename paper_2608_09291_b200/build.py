"""Builds the native code in-tree: the C-ABI CUDA library (nvcc, sm_100a) and, where torch is installed, the native module
of the Python front end on it (the calls that take tensors)."""
from __future__ import annotations

import importlib.util
import os
import subprocess
import sys
import sysconfig
import tempfile
from concurrent.futures import ThreadPoolExecutor
from pathlib import Path

PKG = Path(__file__).resolve().parent
CSRC = PKG / "csrc"
LIB = PKG / "libunionsparse.so"
EXT = PKG / "_us_torch.so"
# (source, extra flags, object): the kernels are one translation unit per N class and kind of K, so that they build in parallel
UNITS = [(CSRC / "us_api.cu", [], "us_api.o"), (CSRC / "us_encode.cpp", [], "us_encode.o"),
         (CSRC / "us_load.cu", [], "us_load.o"), (CSRC / "us_spmm_tc.cu", [], "us_spmm_tc.o")] + [
    (CSRC / "us_kernels.cu", [f"-DUS_NT={nt}", f"-DUS_ANY={a}"], f"us_kernels_nt{nt}_{a}.o") for nt in (1, 2, 4, 8) for a in (0, 1)]
HEADERS = [CSRC / "us_host.h", CSRC / "us_launch.h", CSRC / "us_load.h", CSRC / "us_device_encode.cuh",
           CSRC / "us_spmm_kernel.cuh", CSRC / "us_spmm_tc.cuh", CSRC / "us_spmm_ahead.cuh", CSRC / "us_quant_kernels.cuh",
           PKG.parent / "include" / "unionsparse.h"]
EXT_SOURCE = CSRC / "us_torch.cpp"


def nvcc_flags(verbose: bool = False) -> list[str]:
    cmd = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
           "-Xcompiler", "-fPIC,-O3,-Wall", "-cudart", "shared"]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    return cmd + os.environ.get("US_NVCC_FLAGS", "").split()


def ext_command(out: Path) -> list[str]:
    import torch
    from torch.utils import cpp_extension
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-Wall", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"]
    cmd += [f"-I{p}" for p in cpp_extension.include_paths("cuda")] + [f"-I{sysconfig.get_paths()['include']}"]
    cmd += [str(EXT_SOURCE), "-o", str(out)]
    for p in cpp_extension.library_paths("cuda"):
        cmd += [f"-L{p}", f"-Wl,-rpath,{p}"]
    return cmd + [f"-L{PKG}", "-l:libunionsparse.so", "-Wl,-rpath,$ORIGIN", "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_cuda",
                  "-ltorch", "-ltorch_python"]


def _newest(paths) -> float:
    return max(p.stat().st_mtime for p in paths)


def _lib_stale() -> bool:
    return not LIB.exists() or LIB.stat().st_mtime < _newest([u[0] for u in UNITS] + HEADERS)


def _ext_stale() -> bool:
    if importlib.util.find_spec("torch") is None:   # nothing to build it for
        return False
    return not EXT.exists() or EXT.stat().st_mtime < _newest([EXT_SOURCE, PKG.parent / "include" / "unionsparse.h"])


def is_stale() -> bool:
    return _lib_stale() or _ext_stale()


def _run(cmd: list[str], verbose: bool = False) -> None:
    r = subprocess.run(cmd, capture_output=True, text=True)
    if verbose:
        sys.stderr.write(r.stderr)
    if r.returncode != 0:
        raise RuntimeError(f"{cmd[0]} failed:\n" + r.stdout + r.stderr)


def build(force: bool = False, verbose: bool = False) -> Path:
    if force or verbose or _lib_stale():
        with tempfile.TemporaryDirectory() as tmp, ThreadPoolExecutor(len(UNITS)) as pool:
            objs = [str(Path(tmp) / o) for _, _, o in UNITS]
            jobs = [pool.submit(_run, ["nvcc", *nvcc_flags(verbose), *flags, "-c", str(src), "-o", obj], verbose)
                    for (src, flags, _), obj in zip(UNITS, objs)]
            for j in jobs:
                j.result()
            new = LIB.with_suffix(f".tmp{os.getpid()}.so")
            _run(["nvcc", *nvcc_flags(), "-shared", *objs, "-o", str(new)])
            os.replace(new, LIB)
    if importlib.util.find_spec("torch") is None:
        sys.stderr.write(f"torch is not installed: {EXT.name} (the calls that take tensors) is not built\n")
    elif force or verbose or _ext_stale():
        new = EXT.with_suffix(f".tmp{os.getpid()}.so")
        _run(ext_command(new))
        os.replace(new, EXT)
    return LIB


if __name__ == "__main__":
    build(force=True, verbose="-v" in sys.argv)
    print(LIB)
