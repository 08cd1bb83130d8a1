"""Compile the CUDA sources into paper_1908_06077_b200/libnuq.so for sm_100a."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libnuq.so")
SOURCES = ["nuq_api.cu", "nuq_encode.cu", "nuq_encode_fixed4.cu", "nuq_decode_chains.cu"]
OBJECTS = [os.path.join(HERE, f[:-3] + ".o") for f in SOURCES]          # compiled side by side, then linked
HEADERS = ["nuq_common.cuh", "nuq_async.cuh", "nuq_encode_common.cuh", "nuq_decode_common.cuh", "nuq_decode_fields.cuh", "nuq_launch.h", os.path.join("..", "..", "include", "nuq.h")]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "--fmad=false", "-Xcompiler", "-fPIC"]


def _stale():
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    files = [os.path.join(CSRC, f) for f in SOURCES + HEADERS] + [os.path.abspath(__file__)]
    return any(os.path.getmtime(f) > t for f in files)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not _stale():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    flags = NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else [])
    jobs = [subprocess.Popen([nvcc] + flags + ["-c", "-o", o, os.path.join(CSRC, f)]) for f, o in zip(SOURCES, OBJECTS)]
    failed = [f for f, job in zip(SOURCES, jobs) if job.wait()]
    if failed:
        raise RuntimeError("nvcc failed on " + ", ".join(failed))
    subprocess.run([nvcc] + NVCC_FLAGS + ["-shared", "-o", LIB] + OBJECTS, check=True)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
