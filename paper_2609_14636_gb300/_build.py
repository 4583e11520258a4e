"""In-tree build of libstride.so for sm_103a (nvcc, no cmake) and of the
Python module's native marshalling, _binding.<interpreter>.torch-<version>.so
(g++, torch's headers: it holds that interpreter's and that torch's layouts, so
another of either gets a file of its own).

Each .cu under csrc/ compiles to an object in parallel; the objects link into
paper_2609_14636_gb300/libstride.so against the shared CUDA runtime.  Either
build is skipped when its result is newer than its sources and headers.  The
library needs nvcc (and its host compiler) alone: without torch, or where
binding.cpp does not compile against it, only the marshalling is missing.
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sysconfig
import warnings
from concurrent.futures import ThreadPoolExecutor
from pathlib import Path

PKG = Path(__file__).resolve().parent
ROOT = PKG.parent
CSRC = PKG / "csrc"
INCLUDE = ROOT / "include"
BUILD = PKG / "_build"
LIB = PKG / "libstride.so"

ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden", "-Xptxas", "-v",
              "-I", str(INCLUDE), "-I", str(CSRC)]


def nvcc() -> str:
    cand = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    return cand


def sources() -> list[Path]:
    return sorted(CSRC.glob("*.cu"))


def _newer(out: Path, deps: list[Path]) -> bool:
    return out.exists() and all(p.stat().st_mtime <= out.stat().st_mtime for p in deps)


def up_to_date() -> bool:
    """Whether libstride.so is."""
    return _newer(LIB, sources() + sorted(CSRC.glob("*.cuh")) + sorted(CSRC.glob("*.h")) + sorted(INCLUDE.glob("*.h")))


def binding() -> Path:
    """The marshalling of this interpreter and the installed torch."""
    import torch

    return PKG / f"_binding.{sysconfig.get_config_var('SOABI')}.torch-{torch.__version__}.so"


def build_binding(force: bool = False) -> Path:
    """binding(), built if need be (against torch's headers and libraries)."""
    import torch

    out = binding()
    if not force and _newer(out, [CSRC / "binding.cpp"] + sorted(INCLUDE.glob("*.h"))):
        return out
    t = Path(torch.__file__).parent
    cuda = Path(nvcc()).resolve().parent.parent
    tmp = out.with_name(out.name + f".tmp{os.getpid()}")
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", "-I", str(INCLUDE), "-isystem",
           str(t / "include"), "-isystem", str(t / "include/torch/csrc/api/include"), "-isystem", str(cuda / "include"),
           "-isystem", sysconfig.get_paths()["include"], str(CSRC / "binding.cpp"), "-o", str(tmp), "-L", str(t / "lib"),
           "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"g++ failed for binding.cpp:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, out)
    return out


def build(force: bool = False, verbose: bool = False, defines: tuple = (), lib: Path | None = None,
          build_dir: Path | None = None) -> Path:
    """Compile and link.  `defines` adds -D flags (tuning knobs of the
    kernels); `lib`/`build_dir` redirect the output (default: in-tree, with
    the Python module's marshalling beside it; a warning says why where that
    cannot be built)."""
    if lib is not None:
        return _build_lib(Path(lib), BUILD if build_dir is None else Path(build_dir), defines, verbose)
    with ThreadPoolExecutor(max_workers=1) as ex:
        binding = ex.submit(build_binding, force)
        if force or defines or not up_to_date():
            _build_lib(LIB, BUILD if build_dir is None else Path(build_dir), defines, verbose)
        try:
            binding.result()
        except Exception as e:  # (no torch, no headers, no compiler: the calls take the general code)
            warnings.warn(f"native marshalling not built: {e}", RuntimeWarning, stacklevel=2)
    return LIB


def _build_lib(out_lib: Path, bdir: Path, defines: tuple, verbose: bool) -> Path:
    bdir.mkdir(parents=True, exist_ok=True)
    objs = []

    def compile_one(src: Path) -> tuple[Path, str]:
        obj = bdir / (src.stem + ".o")
        cmd = [nvcc(), *ARCH, *NVCC_FLAGS, *[f"-D{d}" for d in defines], "-c", str(src), "-o", str(obj)]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed for {src.name}:\n{r.stdout}\n{r.stderr}")
        return obj, r.stderr

    with ThreadPoolExecutor(max_workers=min(8, len(sources()))) as ex:
        results = list(ex.map(compile_one, sources()))
    log = []
    for obj, err in results:
        objs.append(obj)
        log.append(err)
    (bdir / "ptxas.log").write_text("\n".join(log))
    tmp = out_lib.with_name(out_lib.name + f".tmp{os.getpid()}")
    cmd = [nvcc(), *ARCH, "-shared", "-cudart", "shared", "-o", str(tmp), *map(str, objs)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, out_lib)
    if verbose:
        print("\n".join(log))
    return out_lib


if __name__ == "__main__":
    build(force=True, verbose=True)
    print(LIB)
