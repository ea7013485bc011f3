"""Builds libcqt_b200.so (sm_100a) in-tree with nvcc.  Usage: python -m paper_2609_29119_b200.build [--force]"""
from __future__ import annotations

import concurrent.futures as cf
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(HERE, "build")
LIB = os.path.join(HERE, "libcqt_b200.so")
EXT = os.path.join(HERE, "_cqt_torch.so")        # Python side of the transform calls, linked to LIB and torch
SOURCES = ["band_two_pass.cu", "band_analysis.cu", "band_synthesis.cu", "layout.cpp", "api.cu", "band.cu", "band_chirp.cu", "band_split.cu", "band_pow2.cu", "band_smooth.cu", "long_fft_forward.cu", "long_fft_inverse.cu", "short_fft.cu", "slicq.cu", "static_ws.cu"]
# compiled once per class, direction and kind of launch (CQT_SMOOTH_KERNELS in band_smooth.cuh)
VARIANTS = [("band_smooth_kernel.cu", f"band_smooth_{c}{'sa'[a]}{'_chained' * h}.o", [f"-DCQT_CLASS={c}", f"-DCQT_ANALYSIS={a}", f"-DCQT_CHAINED={h}"])
            for c, a, h in ((0, 0, 0), (0, 0, 1), (0, 1, 0), (0, 1, 1), (1, 1, 0), (2, 1, 0), (4, 0, 0), (4, 1, 0))]
HEADERS = ["layout.hpp", "plan_types.h", "internal.hpp", "engine.cuh", "band_common.cuh", "long_common.cuh", "long_passes.cuh",
           "static_fft.cuh", "twiddle_rows.cuh", "codelets_gen.cuh", "table_upload.hpp",
           os.path.join("..", "..", "include", "cqt.h")]
SMOOTH_HEADERS = ["band_smooth.cuh", "band_shapes.cuh"]   # of the sources that start with band_smooth
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    raise RuntimeError("nvcc not found")


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False, debug_bounds: bool = False) -> str:
    """debug_bounds=True (or CQT_DEBUG_BOUNDS=1 in the environment) compiles the index self-checks in: an
    out-of-range index is recorded for cqt_plan_check and the access skipped (slower; for debugging only)."""
    debug_bounds = debug_bounds or os.environ.get("CQT_DEBUG_BOUNDS") == "1"
    flags_extra = ["-DCQT_DEBUG_BOUNDS"] if debug_bounds else []
    stamp = os.path.join(OBJ, "debug_bounds.stamp")
    os.makedirs(OBJ, exist_ok=True)
    if debug_bounds != os.path.exists(stamp):
        force = True
        if debug_bounds:
            open(stamp, "w").close()
        else:
            os.unlink(stamp)
    # the register codelets are written by a script; the header is not under version control
    gen = os.path.join(CSRC, "gen_codelets.py")
    gen_out = os.path.join(CSRC, "codelets_gen.cuh")
    if force or _stale(gen_out, [gen]):
        res = subprocess.run([sys.executable, gen, gen_out], capture_output=True, text=True)
        if res.returncode:
            sys.stderr.write(res.stdout + res.stderr)
            raise RuntimeError("gen_codelets.py failed")
    hdrs = [os.path.join(CSRC, h) for h in HEADERS]
    nvcc = _nvcc()
    jobs = []
    objs = []
    for s, o, flags in [(s, os.path.splitext(s)[0] + ".o", []) for s in SOURCES] + VARIANTS:
        src = os.path.join(CSRC, s)
        obj = os.path.join(OBJ, o)
        objs.append(obj)
        own = [os.path.join(CSRC, h) for h in SMOOTH_HEADERS] if s.startswith("band_smooth") else []
        if force or _stale(obj, [src] + hdrs + own):
            cmd = [nvcc] + NVCC_FLAGS + flags + flags_extra + (["-Xptxas", "-v"] if verbose else []) + ["-x", "cu", "-c", src, "-o", obj]
            jobs.append(cmd)
    if jobs:
        with cf.ThreadPoolExecutor(max_workers=min(8, len(jobs))) as ex:
            for cmd, res in zip(jobs, ex.map(lambda c: subprocess.run(c, capture_output=True, text=True), jobs)):
                if verbose or res.returncode:
                    sys.stderr.write(" ".join(cmd) + "\n" + res.stdout + res.stderr)
                if res.returncode:
                    raise RuntimeError("nvcc failed for " + cmd[-3])
    if jobs or force or _stale(LIB, objs):
        cmd = [nvcc, "-shared", "-o", LIB] + objs + ["-gencode", "arch=compute_100a,code=sm_100a"]
        res = subprocess.run(cmd, capture_output=True, text=True)
        if res.returncode:
            sys.stderr.write(res.stdout + res.stderr)
            raise RuntimeError("link failed")
    ext_src = os.path.join(CSRC, "torch_ext.cpp")
    if force or _stale(EXT, [ext_src, hdrs[-1]]):
        import sysconfig
        from torch.utils import cpp_extension as ce
        import torch
        libs = ce.library_paths()
        cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
               ext_src, "-o", EXT, "-I" + sysconfig.get_paths()["include"],
               "-I" + os.path.join(os.path.dirname(os.path.dirname(nvcc)), "include") if os.path.isabs(nvcc) else "-I/usr/local/cuda/include"]
        cmd += ["-I" + p for p in ce.include_paths()] + ["-L" + p for p in libs] + ["-Wl,-rpath," + p for p in libs]
        cmd += ["-L" + HERE, "-Wl,-rpath,$ORIGIN", "-lcqt_b200", "-ltorch_python", "-ltorch_cpu", "-ltorch", "-lc10", "-lc10_cuda"]
        res = subprocess.run(cmd, capture_output=True, text=True)
        if res.returncode:
            sys.stderr.write(res.stdout + res.stderr)
            raise RuntimeError("the torch extension failed to build")
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv, debug_bounds="--debug-bounds" in sys.argv))
