"""Build the CUDA library (csrc/*.cu -> libemu_gb300.so) in-tree for sm_103a."""
from __future__ import annotations

import os
import shutil
import subprocess
import tempfile
from pathlib import Path

PKG = Path(__file__).resolve().parent
ROOT = PKG.parent
SOURCES = sorted((PKG / "csrc").glob("*.cu"))
HEADERS = sorted((ROOT / "include").glob("*.h")) + sorted((PKG / "csrc").glob("*.cuh"))
LIB = PKG / "libemu_gb300.so"
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and Path(cand).exists():
            return cand
    raise RuntimeError("nvcc not found: the CUDA library cannot be built")


def stale() -> bool:
    if not LIB.exists():
        return True
    t = LIB.stat().st_mtime
    return any(p.stat().st_mtime > t for p in SOURCES + HEADERS + [Path(__file__)])


def build(force: bool = False, verbose: bool = False) -> Path:
    """Compile every CUDA source (in parallel) into one shared library (static cudart)."""
    if not force and not stale():
        return LIB
    tmp = LIB.with_name(f".{LIB.name}.{os.getpid()}.tmp")
    # (kernel templates are instantiated in one translation unit and launched from another)
    flags = [*ARCH, "-O3", "-lineinfo", "-std=c++17", "-static-global-template-stub=false", "-Xcompiler", "-fPIC",
             f"-I{ROOT / 'include'}"]
    if verbose:
        flags.insert(0, "-Xptxas=-v")
    with tempfile.TemporaryDirectory() as d:   # the translation units side by side
        objs = [Path(d) / (p.stem + ".o") for p in SOURCES]
        jobs = [subprocess.Popen([nvcc(), *flags, "-c", "-o", str(o), str(p)]) for o, p in zip(objs, SOURCES)]
        bad = [p.name for j, p in zip(jobs, SOURCES) if j.wait() != 0]
        if bad:
            raise RuntimeError(f"nvcc failed on {', '.join(bad)}")
        subprocess.check_call([nvcc(), *ARCH, "-shared", "-o", str(tmp), *map(str, objs)])
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
