"""Builds libstructkv.so (sm_100a, nvcc) and _native.so (the binding's calls, g++ against torch's headers) in-tree.
Run: python -m paper_2604_06746_b200.build"""
import importlib.metadata
import os
import platform
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libstructkv.so")
NATIVE = os.path.join(HERE, "_native.so")
SOURCES = ["api.cu", "score_simt.cu", "score_tc.cu", "score_tc_d64_one.cu",
           "score_tc_d64_many.cu", "score_tc_d128_one.cu", "score_tc_d128_many.cu", "score_res.cu",
           "score_res_d64.cu", "score_res_d128.cu", "score_short_d64.cu", "score_short_d128.cu", "score_reduce.cu",
           "select.cu", "compact.cu", "aggregate.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-Xcompiler", "-fno-gnu-unique", "-Wno-deprecated-gpu-targets"]


def native_for():
    """What _native.so is compiled against; it carries the text."""
    return f"structkv binding for torch {importlib.metadata.version('torch')}, python {platform.python_version()}"


def needs_build():
    if not (os.path.exists(LIB) and os.path.exists(NATIVE)):
        return True
    with open(NATIVE, "rb") as f:
        if native_for().encode() + b"\0" not in f.read():
            return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(NATIVE))
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(ROOT, "include", "structkv.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def native_commands():
    """Compilation and linking of _native.so; it finds the library beside itself."""
    import torch
    from torch.utils import cpp_extension
    cxx, obj = os.environ.get("CXX", "g++"), os.path.join(HERE, "_build", "native.o")
    inc = cpp_extension.include_paths() + ["/usr/local/cuda/include", sysconfig.get_paths()["include"], os.path.join(ROOT, "include")]
    abi = int(torch._C._GLIBCXX_USE_CXX11_ABI)
    libs = [f"-L{p}" for p in cpp_extension.library_paths()] + ["-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"]
    return ([cxx, "-O2", "-std=c++17", "-fPIC", f"-D_GLIBCXX_USE_CXX11_ABI={abi}",
             f'-DSTRUCTKV_NATIVE_FOR="{native_for()}"', *[f"-isystem{i}" for i in inc], "-c",
             os.path.join(CSRC, "native.cpp"), "-o", obj],
            [cxx, "-shared", "-o", NATIVE, obj, f"-L{HERE}", "-lstructkv", "-Wl,-rpath,$ORIGIN", *libs])


def build(force=False, verbose=False):
    if not force and not needs_build():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    objs = []
    build_dir = os.path.join(HERE, "_build")
    os.makedirs(build_dir, exist_ok=True)
    native_compile, native_link = native_commands()
    procs = [("native.cpp", subprocess.Popen(native_compile, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True))]
    for src in SOURCES:
        obj = os.path.join(build_dir, src.replace(".cu", ".o"))
        objs.append(obj)
        cmd = [nvcc, *NVCC_FLAGS, "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-c",
               os.path.join(CSRC, src), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = False
    for src, p in procs:
        out, _ = p.communicate()
        if p.returncode != 0 or verbose:
            sys.stderr.write(f"--- {src}\n{out}\n")
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    subprocess.check_call([nvcc, "-shared", "-o", LIB, *objs, "-cudart", "static"])
    subprocess.check_call(native_link)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
