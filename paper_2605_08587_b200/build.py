"""Build libkla_b200.so in-tree with nvcc for sm_100a (cross-compiles without a GPU)."""
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libkla_b200.so")
HOST = os.path.join(HERE, "_host.so")   # native half of the Python binding (csrc/host.cpp)
SOURCES = ["api.cu", "decode.cu", "chunk_mma.cu", "chunk_wy.cu", "segscan.cu", "static_scratch.cu", "token_scan.cu", "bwd_scan.cu", "bwd_chunk.cu"]
HEADERS = [os.path.join(CSRC, "common.cuh"), os.path.join(CSRC, "umma.cuh"), os.path.join(CSRC, "chunk_pieces.cuh"), os.path.join(CSRC, "scan_pieces.cuh"), os.path.join(CSRC, "solve_pieces.cuh"), os.path.join(CSRC, "mma_pieces.cuh"), os.path.join(ROOT, "include", "kla.h")]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-I" + os.path.join(ROOT, "include"), "-I" + CSRC]


def _newest_source_mtime():
    paths = [os.path.join(CSRC, s) for s in SOURCES + ["host.cpp"]] + [h for h in HEADERS if os.path.exists(h)] + [__file__]
    return max(os.path.getmtime(p) for p in paths)


def _host_compile_cmd(obj):
    import sysconfig

    import torch
    inc = os.path.join(os.path.dirname(torch.__file__), "include")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(shutil.which("nvcc")))), "include")
    return ["g++", "-O2", "-std=c++17", "-fPIC", "-fvisibility=hidden", "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI),
            "-I" + os.path.join(ROOT, "include"), "-isystem", inc, "-isystem", os.path.join(inc, "torch", "csrc", "api", "include"),
            "-isystem", cuda, "-isystem", sysconfig.get_paths()["include"], "-c", os.path.join(CSRC, "host.cpp"), "-o", obj]


def build(force: bool = False, verbose: bool = False) -> str:
    if (not force) and all(os.path.exists(x) and os.path.getmtime(x) >= _newest_source_mtime() for x in (LIB, HOST)):
        return LIB
    objdir = os.path.join(HERE, "_build")
    os.makedirs(objdir, exist_ok=True)
    procs = []
    for s in SOURCES:
        obj = os.path.join(objdir, s.replace(".cu", ".o"))
        cmd = ["nvcc"] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-c", os.path.join(CSRC, s), "-o", obj]
        procs.append((s, obj, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    host_obj = os.path.join(objdir, "host.o")
    procs.append(("host.cpp", host_obj, subprocess.Popen(_host_compile_cmd(host_obj), stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    objs = []
    for s, obj, pr in procs:
        out, _ = pr.communicate()
        if verbose or pr.returncode != 0:
            sys.stderr.write(out)
        if pr.returncode != 0:
            raise RuntimeError("nvcc failed on " + s)
        if s != "host.cpp":
            objs.append(obj)
    tmp = LIB + ".tmp.%d" % os.getpid()
    subprocess.run(["nvcc", "-shared", "-o", tmp] + objs + ["-lcudart"], check=True)
    os.replace(tmp, LIB)
    import torch
    tlib = os.path.join(os.path.dirname(torch.__file__), "lib")
    tmp = HOST + ".tmp.%d" % os.getpid()
    subprocess.run(["g++", "-shared", "-o", tmp, host_obj, "-L" + HERE, "-l:" + os.path.basename(LIB), "-L" + tlib, "-lc10", "-lc10_cuda",
                    "-ltorch_cpu", "-ltorch_python", "-Wl,-rpath,$ORIGIN"], check=True)   # torch's own libraries: loaded by import torch
    os.replace(tmp, HOST)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
