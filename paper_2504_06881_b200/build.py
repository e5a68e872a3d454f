"""Builds libtconv.so (CUDA kernels + C ABI) for sm_100a with nvcc, in-tree.

The tiled forward kernels are compiled as one translation unit per (mode, channel
combine) family, in parallel, and linked with the API unit into one shared library.
The autograd layer over it (csrc/torch_layers.cpp) becomes the extension module _tconv_torch.
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import subprocess
import sys
from pathlib import Path

PKG = Path(__file__).resolve().parent
ROOT = PKG.parent
CSRC = PKG / "csrc"
LIB = PKG / "libtconv.so"
EXT = PKG / "_tconv_torch.so"
# The compiler that nvcc takes for host code, whatever CXX says: one that links its C++ library statically puts a
# second copy of it beside torch's, and formatting a number for an error message then crashed.
HOST_CXX = "g++"
OBJ = PKG / "build"

# (exported launcher, tconv_mode_t, channel combine: 1 sum, 2 max, 3 min)
FWD_INSTANCES = [("fwd_inst_maxplus_sum", 0, 1), ("fwd_inst_maxplus_max", 0, 2),
                 ("fwd_inst_maxplus_min", 0, 3), ("fwd_inst_minplus_sum", 1, 1),
                 ("fwd_inst_minplus_max", 1, 2), ("fwd_inst_minplus_min", 1, 3),
                 ("fwd_inst_compound", 2, 1), ("fwd_inst_parallel", 3, 1)]


def _newest_source() -> float:
    files = list(CSRC.glob("*.cu")) + list(CSRC.glob("*.cpp")) + list(CSRC.glob("*.cuh")) + \
        list((ROOT / "include").glob("*.h")) + [Path(__file__)]
    return max(f.stat().st_mtime for f in files)


def _nvcc_base(verbose: bool):
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cmd = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo",
           "-Xcompiler", "-fPIC", "-I", str(ROOT / "include"), "-I", str(CSRC)]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    return cmd


def _torch_flags():
    """Include and link flags of the extension module: torch's headers and libraries, and the library beside it."""
    import sysconfig
    import torch
    root = Path(torch.__file__).resolve().parent
    cuda = Path(os.environ.get("CUDA_HOME", "/usr/local/cuda"))
    inc = [ROOT / "include", root / "include", root / "include/torch/csrc/api/include", cuda / "include",
           sysconfig.get_paths()["include"]]
    cc = ["-O2", "-std=c++17", "-fPIC", "-DTORCH_API_INCLUDE_EXTENSION_H",
          f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"]
    for d in inc:
        cc += ["-isystem" if d != inc[0] else "-I", str(d)]
    ld = ["-L", str(PKG), "-ltconv", "-L", str(root / "lib"), "-lc10", "-lc10_cuda", "-ltorch", "-ltorch_cpu",
          "-ltorch_cuda", "-ltorch_python", "-Wl,-rpath,$ORIGIN", f"-Wl,-rpath,{root / 'lib'}"]
    return cc, ld


def _compile(job):
    src, obj, defs, verbose = job
    if src.suffix == ".cpp":
        cmd = [HOST_CXX] + _torch_flags()[0] + ["-c", str(src), "-o", str(obj)]
    else:
        cmd = _nvcc_base(verbose) + defs + ["-c", str(src), "-o", str(obj)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    return obj, r.returncode, r.stdout + r.stderr


def build(force: bool = False, verbose: bool = False) -> Path:
    """Compile the library if it is missing or older than any source file."""
    if not force and all(f.exists() and f.stat().st_mtime >= _newest_source() for f in (LIB, EXT)):
        return LIB
    OBJ.mkdir(exist_ok=True)
    jobs = [(CSRC / "tconv_api.cu", OBJ / "tconv_api.o", [], verbose),
            (CSRC / "tconv_bwd_sum.cu", OBJ / "tconv_bwd_sum.o", [], verbose),
            (CSRC / "tconv3d_api.cu", OBJ / "tconv3d_api.o", [], verbose)]
    for name, mode, chan in FWD_INSTANCES:
        defs = [f"-DTCONV_INST_NAME={name}", f"-DTCONV_INST_MODE={mode}", f"-DTCONV_INST_CHAN={chan}"]
        jobs.append((CSRC / "tconv_fwd_inst.cu", OBJ / f"{name}.o", defs, verbose))
    ext_obj = OBJ / "torch_layers.o"
    jobs.append((CSRC / "torch_layers.cpp", ext_obj, [], verbose))
    log = []
    with cf.ThreadPoolExecutor(max_workers=min(len(jobs), os.cpu_count() or 4)) as ex:
        for obj, rc, out in ex.map(_compile, jobs):
            log.append(f"== {obj.name}\n{out}")
            if rc != 0:
                raise RuntimeError(f"nvcc failed for {obj.name}:\n{out}")
    if verbose:
        print("\n".join(log))
    tmp = LIB.with_suffix(f".{os.getpid()}.tmp.so")
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cmd = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "--cudart", "shared"] + \
          [str(j[1]) for j in jobs if j[1] != ext_obj] + ["-o", str(tmp)]
    subprocess.run(cmd, check=True)
    os.replace(tmp, LIB)
    tmp = EXT.with_suffix(f".{os.getpid()}.tmp.so")
    subprocess.run([HOST_CXX, "-shared", str(ext_obj)] + _torch_flags()[1] + ["-o", str(tmp)], check=True)
    os.replace(tmp, EXT)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
