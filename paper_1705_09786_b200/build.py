"""Build step: compiles the sources under csrc/ into libampnet.so (in-tree) for sm_100a with nvcc."""
import glob
import os
import subprocess

_DIR = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(_DIR, "csrc", "ampnet.cu")
SRC_HOST = os.path.join(_DIR, "csrc", "ir_builders.cpp")
SRC_DIRECT = os.path.join(_DIR, "csrc", "engine_fast.cu")
SRC_WAVE = [os.path.join(_DIR, "csrc", f) for f in ("wave_engine.cu", "wave_forward.cu", "wave_moments.cu", "wave_split.cu", "wave_forward_split.cu", "wave_encode.cu")]
# whatever the sources include: every file beside them, and the public header
DEPS = sorted(glob.glob(os.path.join(_DIR, "csrc", "*"))) + [os.path.join(os.path.dirname(_DIR), "include", "ampnet.h")]
LIB = os.path.join(_DIR, "libampnet.so")


def up_to_date():
    return os.path.exists(LIB) and all(os.path.getmtime(LIB) >= os.path.getmtime(d) for d in DEPS)


def build(force=False, verbose=False):
    if not force and up_to_date():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
           "-Xcompiler", "-fPIC", "-shared", "-o", tmp, SRC, SRC_DIRECT, *SRC_WAVE, SRC_HOST]
    if verbose:
        cmd.insert(1, "-Xptxas=-v")
    subprocess.check_call(cmd)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
