"""Build the agx CUDA library (sm_100a only) into ``paper_2605_10380_b200/lib/libagx.so``, and the CPython module that marshals
its calls' arguments (``csrc/agx_torch.cpp``, host code only) into ``lib/agx_torch.so``.

Usage: ``python -m paper_2605_10380_b200.build [--force] [--verbose]``.  nvcc cross-compiles
without a GPU.  Objects are cached under ``_build/`` and rebuilt when a source or header is newer.
"""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor
from pathlib import Path

PKG = Path(__file__).resolve().parent
ROOT = PKG.parent
CSRC = PKG / "csrc"
OUT = PKG / "lib" / "libagx.so"
BINDING = PKG / "lib" / "agx_torch.so"
OBJ_DIR = PKG / "_build"

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden",
    f"-I{ROOT / 'include'}", f"-I{CSRC}",
]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    return "nvcc"


def sources():
    return sorted(CSRC.glob("*.cu"))


def _stale(target: Path, deps) -> bool:
    if not target.exists():
        return True
    t = target.stat().st_mtime
    return any(Path(d).stat().st_mtime > t for d in deps)


def _binding_command(out: Path):
    """g++ command of the argument-marshalling module (torch's headers give the tensors' addresses and the current stream)."""
    import torch
    base = Path(torch.__file__).resolve().parent
    cuda = Path(_nvcc()).resolve().parent.parent
    inc = [base / "include", base / "include" / "torch" / "csrc" / "api" / "include", cuda / "include",
           sysconfig.get_paths()["include"], ROOT / "include"]
    return [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
            f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", *(f"-I{i}" for i in inc),
            str(CSRC / "agx_torch.cpp"), "-o", str(out), f"-L{base / 'lib'}", "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]


def _binding_stamp() -> str:
    """What the argument-marshalling module is tied to besides its sources."""
    import torch
    return "\n".join([torch.__version__, sys.version, *_binding_command(BINDING)])


def _binding_stale() -> bool:
    stamp = OBJ_DIR / "agx_torch.stamp"
    return (_stale(BINDING, [CSRC / "agx_torch.cpp", ROOT / "include" / "agx.h"]) or not stamp.exists()
            or stamp.read_text() != _binding_stamp())


def build(force: bool = False, verbose: bool = False) -> Path:
    srcs = sources()
    headers = list(CSRC.glob("*.cuh")) + list((ROOT / "include").glob("*.h"))
    OBJ_DIR.mkdir(exist_ok=True)
    OUT.parent.mkdir(exist_ok=True)
    nvcc = _nvcc()
    jobs = []
    for src in srcs:
        obj = OBJ_DIR / (src.stem + ".o")
        if force or _stale(obj, [src] + headers):
            cmd = [nvcc, *NVCC_FLAGS, "-c", str(src), "-o", str(obj)]
            if verbose:
                cmd.insert(1, "-Xptxas")
                cmd.insert(2, "-v")
            jobs.append(cmd)

    binding_tmp = BINDING.with_suffix(f".tmp{os.getpid()}.so")
    if force or _binding_stale():
        jobs.append(_binding_command(binding_tmp))

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or r.returncode != 0:
            sys.stderr.write(" ".join(cmd) + "\n" + r.stdout + r.stderr)
        if r.returncode != 0:
            raise RuntimeError("compilation failed: " + " ".join(cmd))

    with ThreadPoolExecutor(max_workers=min(8, max(1, len(jobs)))) as ex:
        list(ex.map(run, jobs))
    if binding_tmp.exists():
        os.replace(binding_tmp, BINDING)
        (OBJ_DIR / "agx_torch.stamp").write_text(_binding_stamp())
    objs = [OBJ_DIR / (s.stem + ".o") for s in srcs]
    if force or jobs or _stale(OUT, objs):
        tmp = OUT.with_suffix(f".tmp{os.getpid()}.so")
        cmd = [nvcc, "-shared", "-o", str(tmp), *map(str, objs), "-gencode", "arch=compute_100a,code=sm_100a",
               "-Xcompiler", "-fPIC", "-cudart", "shared"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            sys.stderr.write(r.stdout + r.stderr)
            raise RuntimeError("link failed")
        os.replace(tmp, OUT)
    return OUT


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
