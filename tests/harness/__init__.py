"""Builds kernels.cu (one shared object per part) and loads the parts."""
import concurrent.futures as cf
import ctypes
import os
import subprocess

from paper_2406_10158_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))
PARTS = 5


def load(out_dir):
    """The parts' libraries, compiled into ``out_dir``; the engine must be built."""
    def one(part):
        so = os.path.join(str(out_dir), f"libkernels{part}.so")
        cmd = [build.nvcc(), *build.ARCH, "-O1", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", f"-DPART={part}",
               "-I", build.INCLUDE, "-I", build.CSRC, os.path.join(HERE, "kernels.cu"), "-o", so, build.LIB,
               "-Xlinker", "-rpath", "-Xlinker", build.OUT_DIR]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on part {part}:\n{r.stderr}")
        return so
    with cf.ThreadPoolExecutor(max_workers=PARTS) as ex:
        return [ctypes.CDLL(so) for so in ex.map(one, range(PARTS))]
