"""Builds the CUDA library in-tree with nvcc for sm_100a (cross-compiles without a GPU).

The kernels are templates with many instantiations; they are spread over translation units (one per encoder
mode and dither width, one per decoder variant and group size) that are compiled in parallel and linked into one shared library.
The Python calls (csrc/dq_calls.cpp) are a second, small library, linked against the first.
"""
from __future__ import annotations

import hashlib
import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor
from pathlib import Path

PKG = Path(__file__).resolve().parent
ROOT = PKG.parent
CSRC = PKG / "csrc"
LIB = PKG / "lib" / "libdq_b200.so"
CALLS = PKG / "lib" / "dq_calls.so"
OBJ = PKG / "lib" / "obj"
DEPS = sorted(CSRC.glob("*.cu*")) + sorted(CSRC.glob("*.h")) + sorted(CSRC.glob("*.cpp")) + [ROOT / "include" / "dq.h"]

NVCC_FLAGS = [
    "-std=c++17", "-O3",
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-lineinfo",
    "--fmad=false",          # every fused multiply-add in the kernels is written explicitly
    "-Xcompiler", "-fPIC",
]

# (object name, source, extra defines)
UNITS = [("dq_b200", "dq_b200.cu", [])]
UNITS += [(f"enc_m{m}_d{d}", "dq_encode_inst.cu", [f"-DDQ_INST_MODE={m}", f"-DDQ_INST_DITH={d}"])
          for m in (0, 1, 2, 3) for d in (32, 16)]
UNITS += [(f"dec_d{d}_r{r}_e{e}", "dq_decode_inst.cu", [f"-DDQ_INST_DITH={d}", f"-DDQ_INST_RUN={r}", f"-DDQ_INST_E={e}"])
          for d, r in ((32, 0), (32, 1), (32, 2), (16, 0), (16, 1), (16, 2), (0, 0)) for e in (32, 16, 8)]
UNITS += [(f"dec_one_d{d}", "dq_decode_one_inst.cu", [f"-DDQ_INST_DITH={d}"]) for d in (32, 16)]


def nvcc_path() -> str:
    cand = os.environ.get("NVCC") or "/usr/local/cuda/bin/nvcc"
    return cand if Path(cand).exists() else "nvcc"


def source_hash() -> str:
    """Content hash of everything the library is built from (sources, headers, flags)."""
    h = hashlib.sha256()
    for f in DEPS:
        h.update(f.name.encode())
        h.update(f.read_bytes())
    h.update(" ".join(NVCC_FLAGS).encode())
    return h.hexdigest()[:16]


def stale() -> bool:
    if not LIB.exists() or not CALLS.exists():
        return True
    t = min(LIB.stat().st_mtime, CALLS.stat().st_mtime)
    return any(d.stat().st_mtime > t for d in DEPS)


def _compile(unit, verbose: bool, obj_dir: Path = OBJ, extra_flags=()) -> Path:
    name, src, defs = unit
    obj = obj_dir / f"{name}.o"
    cmd = [nvcc_path(), *NVCC_FLAGS, *defs, *extra_flags, f"-I{ROOT / 'include'}", f"-I{CSRC}", "-c", "-o", str(obj),
           str(CSRC / src)]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    subprocess.run(cmd, check=True)
    return obj


def build(force: bool = False, verbose: bool = False, out: Path | None = None, extra_flags=()) -> Path:
    """Compiles every translation unit and links the shared library.  `out` / `extra_flags` build a variant
    (other tile or occupancy constants, see the DQ_* macros in csrc/) beside the default library."""
    if out is not None:
        return _build_to(Path(out), list(extra_flags), verbose)
    if not force and not stale():
        return LIB
    with ThreadPoolExecutor(max_workers=1) as pool:
        calls = pool.submit(_compile_calls)
        lib = _build_to(LIB, [], verbose)
        _link_calls(calls.result())
    return lib


def _compile_calls() -> Path:
    import torch
    from torch.utils.cpp_extension import include_paths
    OBJ.mkdir(parents=True, exist_ok=True)
    obj = OBJ / "dq_calls.o"
    inc = [*include_paths(), sysconfig.get_paths()["include"], str(Path(nvcc_path()).resolve().parents[1] / "include"),
           str(ROOT / "include")]
    abi = f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}"
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++20", "-O2", "-fPIC", "-fvisibility=hidden", abi,
                    *[f"-isystem{i}" for i in inc], "-c", "-o", str(obj), str(CSRC / "dq_calls.cpp")], check=True)
    return obj


def _link_calls(obj: Path) -> None:
    from torch.utils.cpp_extension import library_paths
    tmp = CALLS.with_suffix(f".{os.getpid()}.tmp")
    # torch's libraries are in the process before this one is loaded; libdq_b200.so lies beside it
    subprocess.run([os.environ.get("CXX", "g++"), "-shared", "-o", str(tmp), str(obj),
                    *[f"-L{d}" for d in library_paths()], "-ltorch_python", "-ltorch_cpu", "-ltorch", "-lc10_cuda",
                    "-lc10", f"-L{LIB.parent}", f"-l:{LIB.name}", "-Wl,-rpath,$ORIGIN"], check=True)
    os.replace(tmp, CALLS)


def _build_to(lib: Path, extra_flags, verbose: bool) -> Path:
    global OBJ
    obj_dir = OBJ if lib == LIB else lib.parent / (lib.stem + "_obj")
    obj_dir.mkdir(parents=True, exist_ok=True)
    jobs = int(os.environ.get("DQ_BUILD_JOBS", "0")) or min(len(UNITS), os.cpu_count() or 1)
    with ThreadPoolExecutor(max_workers=jobs) as pool:
        objs = list(pool.map(lambda u: _compile(u, verbose, obj_dir, extra_flags), UNITS))
    tmp = lib.with_suffix(f".{os.getpid()}.tmp")
    subprocess.run([nvcc_path(), "-shared", "-cudart", "static", "-gencode", "arch=compute_100a,code=sm_100a",
                    "-o", str(tmp), *[str(o) for o in objs]], check=True)
    os.replace(tmp, lib)
    return lib


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
