"""Build libzipvl.so in-tree with nvcc for sm_100a (cross-compiles without a GPU), and _native.so,
the extension module that hands torch tensors to it, with g++."""
import glob
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libzipvl.so")
NATIVE = os.path.join(HERE, "_native.so")
NATIVE_SRC = os.path.join(CSRC, "binding.cpp")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
         "--use_fast_math", "-Xcompiler", "-fPIC", "-Xcompiler", "-Wall", "-shared",
         "-cudart", "shared"]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def stale():
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    if not os.path.exists(NATIVE) or os.path.getmtime(NATIVE) < os.path.getmtime(NATIVE_SRC):
        return True
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + \
        glob.glob(os.path.join(HERE, "..", "include", "*.h"))
    return any(os.path.getmtime(p) > t for p in deps)


def native_command():
    import torch
    t = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(NVCC))
    inc = [sysconfig.get_paths()["include"], f"{t}/include", f"{t}/include/torch/csrc/api/include", f"{cuda}/include"]
    return ["g++", "-O2", "-std=c++17", "-fPIC", "-Wall", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}",
            *[a for p in inc for a in ("-isystem", p)], "-c", NATIVE_SRC, "-o", NATIVE_SRC[:-4] + ".o"]


def native_link():
    import torch
    lib = os.path.join(os.path.dirname(torch.__file__), "lib")
    return ["g++", "-shared", "-o", NATIVE + ".tmp", NATIVE_SRC[:-4] + ".o", f"-L{lib}", "-ltorch_python", "-ltorch_cpu",
            "-lc10_cuda", "-lc10", LIB, "-Wl,-rpath,$ORIGIN"]


def build(force=False, verbose=False):
    if not force and not stale():
        return LIB
    objs = []
    procs = []
    for src in sources():
        obj = src[:-3] + ".o"
        cmd = [NVCC, *[f for f in FLAGS if f != "-shared"], "-c", src, "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        procs.append((src, subprocess.Popen(cmd)))
        objs.append(obj)
    procs.append((NATIVE_SRC, subprocess.Popen(native_command())))
    for src, p in procs:
        if p.wait() != 0:
            raise RuntimeError(f"compiler failed on {src}")
    subprocess.run([NVCC, "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-cudart", "shared",
                    "-Xlinker", "-soname=libzipvl.so", "-o", LIB + ".tmp", *objs], check=True)
    os.replace(LIB + ".tmp", LIB)
    subprocess.run(native_link(), check=True)
    os.replace(NATIVE + ".tmp", NATIVE)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
