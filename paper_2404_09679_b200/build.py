"""Builds libantdt.so (CUDA kernels for sm_100a + the host planner) in-tree with nvcc/gcc, and the
extension module _marshal, which hands the forward's arguments over natively (without it they go
through ctypes).

`python -m paper_2404_09679_b200.build` rebuilds; `build()` is a no-op when both are newer than every
source and the module is of this torch and Python.  nvcc cross-compiles without a GPU.
"""
import glob
import os
import shutil
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
INC = os.path.join(os.path.dirname(HERE), "include")
OBJ = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libantdt.so")
MARSHAL = os.path.join(HERE, "_marshal" + sysconfig.get_config_var("EXT_SUFFIX"))
MARSHAL_KEY = os.path.join(OBJ, "marshal.key")  # what MARSHAL was built against

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-I", INC, "-I", CSRC]
GCC_FLAGS = ["-O2", "-std=c11", "-fPIC", "-ffp-contract=off", "-Wall", "-I", INC]


def _sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu"))), sorted(glob.glob(os.path.join(CSRC, "*.c")))


def _newest_dep():
    deps = glob.glob(os.path.join(CSRC, "*")) + glob.glob(os.path.join(INC, "*.h"))
    return max(os.path.getmtime(p) for p in deps)


def _marshal_command(nvcc):
    import torch  # its headers and libraries
    root = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(shutil.which(nvcc) or nvcc)))
    inc = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
           sysconfig.get_paths()["include"], os.path.join(cuda, "include"), INC]
    return (["g++", "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
             f'-DANTDT_TORCH="{torch.__version__}"']
            + [x for i in inc for x in ("-isystem", i)] + [os.path.join(CSRC, "marshal.cpp"), "-o", MARSHAL, "-L", os.path.join(root, "lib"),
               "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"])


_NO_MARSHAL = "_marshal: not built; the forward's arguments go through ctypes"


def _marshal_key():
    try:
        import torch
    except ImportError:
        return "no torch"
    return f"torch {torch.__version__}, Python {sys.version}"


def _marshal_current(newer_than: float) -> bool:
    """The module is there, newer than its sources, and of this torch and Python."""
    if not os.path.exists(MARSHAL) or os.path.getmtime(MARSHAL) < newer_than or not os.path.exists(MARSHAL_KEY):
        return False
    with open(MARSHAL_KEY) as f:
        return f.read() == _marshal_key()


def build(force: bool = False, verbose: bool = False, ptxas_info: bool = False) -> str:
    marshal_src = os.path.join(CSRC, "marshal.cpp")
    marshal_current = not force and _marshal_current(max(os.path.getmtime(p) for p in (marshal_src, os.path.join(INC, "antdt.h"))))
    if not force and marshal_current and os.path.exists(LIB) and os.path.getmtime(LIB) >= _newest_dep():
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
    if not marshal_current:
        try:
            procs.append((marshal_src, subprocess.Popen(_marshal_command(nvcc), stdout=subprocess.PIPE, stderr=subprocess.STDOUT)))
        except (ImportError, OSError) as e:  # no torch, no g++
            sys.stderr.write(f"{_NO_MARSHAL} ({e})\n")
    failed = False
    for src, p in procs:
        out = p.communicate()[0].decode()
        if p.returncode != 0 or ptxas_info:
            sys.stderr.write(f"== {os.path.basename(src)}\n{out}\n")
        if src == marshal_src:
            if p.returncode == 0:
                with open(MARSHAL_KEY, "w") as f:
                    f.write(_marshal_key())
            else:  # the library does without it
                sys.stderr.write(f"{_NO_MARSHAL}\n")
            continue
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("libantdt.so: compilation failed")
    link = [nvcc, "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", LIB] + objs + ["-cudart", "static", "-lm"]
    subprocess.run(link, check=True)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True, ptxas_info="--ptxas" in sys.argv))
