"""Builds libfastpool.so (the C-ABI library) from csrc/ with nvcc for sm_100a, in-tree."""
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libfastpool.so")
NATIVE = os.path.join(HERE, "_native.so")          # Python module: argument marshalling of the calls of a layer step
SOURCES = ["pool.cu", "swap.cu", "sgmv.cu", "sgmv_tc.cu", "attention.cu", "attention_tc2.cu", "tmap.cu", "lora_linear.cu", "lora_skinny.cu", "swapper.cu", "tree.cu", "cache_sim.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "--use_fast_math", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", CSRC]


def _stale(obj, deps):
    if not os.path.exists(obj):
        return True
    t = os.path.getmtime(obj)
    return any(os.path.getmtime(d) > t for d in deps)


def build(verbose=False, force=False):
    """Compile every .cu under csrc/ and link libfastpool.so; returns the library path."""
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    headers = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    headers.append(os.path.join(ROOT, "include", "fastpool.h"))
    bdir = os.path.join(HERE, "_build")
    os.makedirs(bdir, exist_ok=True)
    objs, procs = [], []
    for src in SOURCES:
        s = os.path.join(CSRC, src)
        o = os.path.join(bdir, src.replace(".cu", ".o"))
        objs.append(o)
        if force or _stale(o, [s] + headers):
            cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-c", s, "-o", o]
            procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = False
    for src, p in procs:
        out, _ = p.communicate()
        if verbose or p.returncode != 0:
            sys.stderr.write(f"--- {src}\n{out}\n")
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    if procs or not os.path.exists(LIB):
        subprocess.check_call([nvcc, "-shared", "-o", LIB] + objs + ["-lcudart"])
    src = os.path.join(CSRC, "native.cpp")
    if force or _native_stale(src):
        _build_native(src)
    return LIB


def _native_tag():
    """What the module is built against: it links torch's C++ libraries and Python's."""
    from importlib.metadata import version
    return f"fastpool-native python {sys.version_info[0]}.{sys.version_info[1]} torch {version('torch')}"


def _native_stale(src):
    if _stale(NATIVE, [src, os.path.join(ROOT, "include", "fastpool.h")]):
        return True
    with open(NATIVE, "rb") as f:
        return _native_tag().encode() + b"\0" not in f.read()


def _build_native(src):
    import sysconfig
    import torch
    tdir = os.path.dirname(torch.__file__)
    inc = [os.path.join(ROOT, "include"), sysconfig.get_paths()["include"], os.path.join(tdir, "include"),
           os.path.join(tdir, "include", "torch", "csrc", "api", "include"), "/usr/local/cuda/include"]
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", f'-DFL_NATIVE_TAG="{_native_tag()}"', f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", src, "-o", NATIVE]
    cmd += [f for i in inc for f in ("-isystem" if "torch" in i else "-I", i)]
    cmd += ["-L", HERE, "-l:libfastpool.so", "-L", os.path.join(tdir, "lib"), "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda",
            "-Wl,-rpath,$ORIGIN", "-Wl,-rpath," + os.path.join(tdir, "lib")]
    subprocess.check_call(cmd)


if __name__ == "__main__":
    print(build(verbose="-v" in sys.argv, force="-f" in sys.argv))
