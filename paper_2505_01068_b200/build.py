"""Builds the sm_100a C-ABI library (libgsit.so) in-tree with nvcc; objects are compiled in parallel.  Beside it the CPython
extension `_native` (g++, torch headers) that hands torch tensors to the library."""
from __future__ import annotations

import os
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor
from pathlib import Path

PKG = Path(__file__).resolve().parent
CSRC = PKG / "csrc"
INCLUDE = PKG.parent / "include"
OBJ_DIR = PKG / "_build"
LIB = PKG / "libgsit.so"
SOURCES = ["gsit_api.cu", "attn_f32.cu", "attn_bf16.cu", "attn_tc.cu", "attn_tcs.cu", "linear.cu", "linear_f32.cu", "gemm_tc.cu", "fused_layer.cu", "fused_layer_tc.cu", "fused_layer_tc128.cu", "fused_rows.cu", "attn_mlp_rows.cu", "layer_static.cu", "stack_head.cu", "rows.cu"]
EXT_SOURCE = CSRC / "torch_ext.cpp"
EXT = PKG / "_native.so"
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-I", str(INCLUDE), "-I", str(CSRC)]


def _nvcc() -> str:
    cand = os.environ.get("NVCC") or "/usr/local/cuda/bin/nvcc"
    return cand if Path(cand).exists() else "nvcc"


def _stale(target: Path, deps) -> bool:
    if not target.exists():
        return True
    t = target.stat().st_mtime
    return any(Path(d).stat().st_mtime > t for d in deps)


def _ext_commands() -> list[list[str]]:
    """Compile and link lines of the extension; it finds libgsit.so beside itself and everything else in the torch that
    imports it."""
    import sysconfig

    import torch
    root = Path(torch.__file__).resolve().parent
    cuda = Path(_nvcc()).resolve().parent.parent
    inc = [INCLUDE, root / "include", root / "include" / "torch" / "csrc" / "api" / "include", cuda / "include",
           sysconfig.get_paths()["include"]]
    obj = str(OBJ_DIR / "torch_ext.o")
    cxx = os.environ.get("CXX", "g++")
    return [[cxx, "-O2", "-std=c++20", "-fPIC", "-fvisibility=hidden", "-w", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"]
            + [w for i in inc for w in ("-isystem", str(i))] + ["-c", str(EXT_SOURCE), "-o", obj],
            [cxx, "-shared", "-o", "{out}", obj, "-L" + str(PKG), "-l:" + LIB.name, "-L" + str(root / "lib"), "-ltorch_python", "-ltorch_cuda",
             "-ltorch_cpu", "-ltorch", "-lc10_cuda", "-lc10", "-L" + str(cuda / "lib64"), "-lcudart", "-Wl,-rpath,$ORIGIN"]]


def build(force: bool = False, verbose: bool = False) -> Path:
    OBJ_DIR.mkdir(exist_ok=True)
    headers = list(CSRC.glob("*.cuh")) + list(INCLUDE.glob("*.h")) + [Path(__file__)]
    jobs = []
    for src in SOURCES:
        obj = OBJ_DIR / (src[:-3] + ".o")
        if force or _stale(obj, [CSRC / src] + headers):
            cmd = [_nvcc()] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-c", str(CSRC / src), "-o", str(obj)]
            jobs.append(cmd)
    ext_obj, ext_jobs = OBJ_DIR / "torch_ext.o", []
    if force or _stale(ext_obj, [EXT_SOURCE, Path(__file__)] + list(INCLUDE.glob("*.h"))):
        ext_jobs.append(_ext_commands()[0])

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or r.returncode:
            sys.stderr.write(r.stdout + r.stderr)
        if r.returncode:
            raise RuntimeError("nvcc failed: " + " ".join(cmd))

    with ThreadPoolExecutor(max_workers=max(1, min(len(jobs) + len(ext_jobs), os.cpu_count() or 1))) as ex:
        list(ex.map(run, ext_jobs + jobs))
    objs = [str(OBJ_DIR / (s[:-3] + ".o")) for s in SOURCES]
    if force or jobs or _stale(LIB, objs):
        tmp = LIB.with_suffix(f".tmp{os.getpid()}.so")
        run([_nvcc(), "-shared", "-o", str(tmp)] + objs + ["-gencode", "arch=compute_100a,code=sm_100a"])
        os.replace(tmp, LIB)
    if force or ext_jobs or _stale(EXT, [ext_obj]):
        tmp = EXT.with_suffix(f".tmp{os.getpid()}.so")
        run([str(tmp) if w == "{out}" else w for w in _ext_commands()[1]])
        os.replace(tmp, EXT)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
