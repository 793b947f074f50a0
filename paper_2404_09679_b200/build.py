"""Builds libantdt.so (CUDA kernels for sm_100a + the host planner) in-tree with nvcc/gcc.

`python -m paper_2404_09679_b200.build` rebuilds; `build()` is a no-op when the library is
newer than every source.  nvcc cross-compiles without a GPU.
"""
import glob
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
INC = os.path.join(os.path.dirname(HERE), "include")
OBJ = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libantdt.so")
MARSHAL = os.path.join(HERE, "_marshal.so")  # Python objects -> the entry points' arguments

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-I", INC, "-I", CSRC]
GCC_FLAGS = ["-O2", "-std=c11", "-fPIC", "-ffp-contract=off", "-Wall", "-I", INC]


def _sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu"))), sorted(glob.glob(os.path.join(CSRC, "*.c")))


def _newest_dep():
    deps = glob.glob(os.path.join(CSRC, "*")) + glob.glob(os.path.join(INC, "*.h"))
    return max(os.path.getmtime(p) for p in deps)


def _marshal_command():
    import torch  # its headers and libraries
    root = os.path.dirname(torch.__file__)
    inc = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
           sysconfig.get_paths()["include"], "/usr/local/cuda/include", INC]
    return (["g++", "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"]
            + [x for i in inc for x in ("-isystem", i)] + [os.path.join(CSRC, "marshal.cpp"), "-o", MARSHAL, "-L", os.path.join(root, "lib"),
               "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"])


def build(force: bool = False, verbose: bool = False, ptxas_info: bool = False) -> str:
    if not force and all(os.path.exists(p) and os.path.getmtime(p) >= _newest_dep() for p in (LIB, MARSHAL)):
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    os.makedirs(OBJ, exist_ok=True)
    cu, c = _sources()
    hdr_time = max(os.path.getmtime(p) for p in
                   glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(INC, "*.h")))
    objs, procs = [], []
    for src in cu + c:
        obj = os.path.join(OBJ, os.path.basename(src) + ".o")
        objs.append(obj)
        if (not force and os.path.exists(obj)
                and os.path.getmtime(obj) >= max(os.path.getmtime(src), hdr_time)):
            continue
        if src.endswith(".cu"):
            cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if ptxas_info else []) + ["-c", src, "-o", obj]
        else:
            cmd = ["gcc"] + GCC_FLAGS + ["-c", src, "-o", obj]
        if verbose:
            print(" ".join(cmd), flush=True)
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT)))
    src = os.path.join(CSRC, "marshal.cpp")
    stale = not os.path.exists(MARSHAL) or os.path.getmtime(MARSHAL) < max(os.path.getmtime(src), os.path.getmtime(os.path.join(INC, "antdt.h")))
    if force or stale:
        procs.append((src, subprocess.Popen(_marshal_command(), stdout=subprocess.PIPE, stderr=subprocess.STDOUT)))
    else:
        os.utime(MARSHAL)
    failed = False
    for src, p in procs:
        out = p.communicate()[0].decode()
        if p.returncode != 0 or ptxas_info:
            sys.stderr.write(f"== {os.path.basename(src)}\n{out}\n")
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("libantdt.so: compilation failed")
    link = [nvcc, "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", LIB] + objs + ["-cudart", "static", "-lm"]
    subprocess.run(link, check=True)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True, ptxas_info="--ptxas" in sys.argv))
