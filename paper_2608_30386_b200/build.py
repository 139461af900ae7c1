"""Build libdasc.so in-tree with nvcc for sm_100a (cross-compiles without a GPU)."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libdasc.so")
CALL = os.path.join(HERE, "_dasccall.so")   # CPython entry to the library's device calls
CALL_SOURCE = "pycall.c"
SOURCES = ["dasc_api.cu", "plan_host.cpp", "pack_restore.cu", "codec_int8.cu", "refresh_seq.cu", "refresh_chunked.cu"]
# sources compiled several times, side by side: object name and define of each translation unit
UNITS = {"refresh_seq.cu": [(f"refresh_seq_{d}", f"-DDASC_SEQ_DIM={d}") for d in (128, 64, 32)]}
HEADERS = [os.path.join(ROOT, "include", "dasc.h"), os.path.join(CSRC, "dasc_internal.h"),
           os.path.join(CSRC, "tcgen05_util.cuh"), os.path.join(CSRC, "launch.cuh")]

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-Xfatbin=-compress-all",
]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    return "nvcc"


def needs_build() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(CALL):
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(CALL))
    deps = [os.path.join(CSRC, s) for s in SOURCES + [CALL_SOURCE]] + HEADERS + [os.path.abspath(__file__)]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not needs_build():
        return LIB
    objdir = os.path.join(HERE, "build")
    os.makedirs(objdir, exist_ok=True)
    objs = []
    procs = []
    for s, name, *define in ((s, *u) for s in SOURCES for u in UNITS.get(s, [(os.path.splitext(s)[0],)])):
        obj = os.path.join(objdir, name + ".o")
        objs.append(obj)
        cmd = [_nvcc(), *NVCC_FLAGS, *define, "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-x", "cu", "-c",
               os.path.join(CSRC, s), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        procs.append((cmd, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = False
    for cmd, p in procs:
        out, _ = p.communicate()
        if p.returncode != 0 or verbose:
            sys.stderr.write(" ".join(cmd) + "\n" + out + "\n")
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    link = [_nvcc(), "-shared", "-o", LIB, *objs, "-gencode", "arch=compute_100a,code=sm_100a"]
    subprocess.run(link, check=True)
    subprocess.run([os.environ.get("CC", "gcc"), "-O2", "-shared", "-fPIC", "-I", sysconfig.get_paths()["include"],
                    "-I", os.path.join(ROOT, "include"), os.path.join(CSRC, CALL_SOURCE), "-o", CALL, "-L", HERE,
                    "-l:libdasc.so", "-Wl,-rpath,$ORIGIN"], check=True)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
