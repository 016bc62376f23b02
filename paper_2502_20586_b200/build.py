"""Compile the CUDA library in-tree for sm_100a, ``paper_2502_20586_b200/libmxfp4_b200.so``, and the native host calls of the binding,
``_host_calls`` with the file name of this Python's extension modules."""
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libmxfp4_b200.so")
HOST = os.path.join(HERE, "_host_calls" + sysconfig.get_config_var("EXT_SUFFIX"))
HOST_UNTAGGED = os.path.join(HERE, "_host_calls.so")                     # any Python would load this: an earlier build's goes
HOST_SOURCE = os.path.join(CSRC, "host_calls.cpp")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")
HEADER = os.path.join(INCLUDE, "mxfp4.h")
SOURCES = ["api.cu", "gemm.cu", "gemm_pair.cu", "gemm_fused.cu", "quantize.cu", "quantize_tc.cu", "static_workspace.cu", "fp4_ceiling.cu", "bias_grad.cu", "gemm_f8.cu", "variants.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
              "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden", "--expt-relaxed-constexpr"]


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if not f.endswith(".cpp")] + [HEADER]
    return any(os.path.getmtime(d) > t for d in deps)


def host_stamp() -> str:
    """What the host calls are compiled against, besides their sources: inline code of torch's headers works on the running torch's objects."""
    import torch
    return f"host calls for torch {torch.__version__}, C++11 ABI {int(torch.compiled_with_cxx11_abi())}, {sys.implementation.cache_tag}"


def _host_stale() -> bool:
    if not os.path.exists(HOST) or any(os.path.getmtime(d) > os.path.getmtime(HOST) for d in (HOST_SOURCE, HEADER)):
        return True
    with open(HOST, "rb") as f:
        return host_stamp().encode() + b"\0" not in f.read()


def host_command(out: str, include: str = INCLUDE) -> list:
    """The compiler's command line for the host calls: C++ against the headers and libraries of the torch that imports them."""
    import torch
    root = os.path.dirname(torch.__file__)
    dirs = [include, os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"), sysconfig.get_paths()["include"]]
    return [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
            f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}", f'-DMXFP4_HOST_STAMP="{host_stamp()}"', *(f"-I{d}" for d in dirs), HOST_SOURCE, "-o", out,
            "-L" + os.path.join(root, "lib"), "-lc10", "-ltorch_cpu", "-ltorch_python"]


def build_host(force: bool = False) -> str:
    if not force and not _host_stale():
        return HOST
    subprocess.run(host_command(HOST + ".tmp"), check=True)
    os.replace(HOST + ".tmp", HOST)
    if HOST_UNTAGGED != HOST and os.path.exists(HOST_UNTAGGED):
        os.remove(HOST_UNTAGGED)
    return HOST


def build(force: bool = False, verbose: bool = False) -> str:
    build_host(force)
    return build_library(force, verbose)


def build_library(force: bool = False, verbose: bool = False) -> str:
    if not force and not _stale():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    flags = list(NVCC_FLAGS) + (["-Xptxas", "-v"] if verbose else [])
    objs = []
    procs = []
    for src in SOURCES:
        obj = os.path.join(CSRC, src.replace(".cu", ".o"))
        objs.append(obj)
        procs.append(subprocess.Popen([nvcc, *flags, "-c", os.path.join(CSRC, src), "-o", obj]))
    for p in procs:
        if p.wait() != 0:
            raise RuntimeError("nvcc failed")
    subprocess.run([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-o", LIB + ".tmp", *objs], check=True)
    os.replace(LIB + ".tmp", LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
