"""Build libbifrost.so (sm_100a) in-tree with nvcc.  Cross-compiles without a GPU."""
import os
import subprocess
import sys
import tempfile

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libbifrost.so")
SOURCES = ["api.cu", "ntt.cu", "kernels.cu", "mac.cu", "mac_wide.cu", "encode.cu"]
HEADERS = ["bf_common.cuh", "bf_host.h", "mac_kernel.cuh", os.path.join("..", "..", "include", "bifrost.h")]


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, f) for f in SOURCES + HEADERS] + [os.path.abspath(__file__)]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not _stale():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    flags = ["-std=c++17", "-O3", "-lineinfo", "-gencode", "arch=compute_100a,code=sm_100a",
             "-Xcompiler", "-fPIC,-O2,-fno-fast-math"]
    if verbose:
        flags += ["-Xptxas", "-v"]
    with tempfile.TemporaryDirectory() as tmp:        # one compilation per source, side by side
        objs = [os.path.join(tmp, f + ".o") for f in SOURCES]
        jobs = [subprocess.Popen([nvcc, *flags, "-c", os.path.join(CSRC, f), "-o", o]) for f, o in zip(SOURCES, objs)]
        failed = [f for f, j in zip(SOURCES, jobs) if j.wait() != 0]
        if failed:
            raise RuntimeError("nvcc failed on " + ", ".join(failed))
        subprocess.run([nvcc, *flags, "-shared", "-o", LIB, *objs, "-lcudart"], check=True)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
