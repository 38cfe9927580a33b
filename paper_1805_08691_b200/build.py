"""Compile libq8.so (CUDA kernels + C ABI) for sm_100a with nvcc, and the module that marshals torch tensors into its most
frequent calls (_q8native.*.so), both in-tree."""
import os
import shutil
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libq8.so")
SOURCES = ["q8_api.cu", "q8_elementwise.cu", "q8_conv_direct.cu", "q8_conv_splitk.cu", "q8_conv_static.cu", "q8_conv_umma.cu", "q8_conv_fused.cu", "q8_conv_gather.cu", "q8_conv_packed.cu", "q8_mma_rate.cu", "q8_selftest.cu", "q8_detect.cu", "q8_record.cu"]
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "-fmad=false",
         "-Xcompiler", "-fPIC,-ffp-contract=off,-fno-fast-math", "-I", os.path.join(ROOT, "include"), "-I", CSRC]


def native_path() -> str:
    """The marshalling module of this interpreter and this torch: it holds tensors by their C++ layout, so another build of
    either looks for, and makes, another file."""
    import torch
    version = "".join(c if c.isalnum() or c in ".+" else "_" for c in torch.__version__)
    return os.path.join(HERE, f"_q8native.{sysconfig.get_config_var('SOABI')}.torch{version}.{(torch.version.git_version or '')[:8]}"
                              f".abi{int(torch._C._GLIBCXX_USE_CXX11_ABI)}.so")


def _cuda_include():
    """Where cuda_runtime.h is: CUDA_HOME, beside nvcc, or the usual place."""
    nvcc = shutil.which("nvcc")
    homes = [os.environ.get("CUDA_HOME"), nvcc and os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "/usr/local/cuda"]
    return next((d for d in (os.path.join(h, "include") for h in homes if h) if os.path.exists(os.path.join(d, "cuda_runtime.h"))), None)


def _cxx():
    return shutil.which(os.environ.get("CXX") or "g++") or shutil.which("c++")


def _native_command(out):
    import torch  # only its headers and libraries: the module is linked against the torch that will load it
    t = os.path.dirname(torch.__file__)
    system = [sysconfig.get_paths()["include"], os.path.join(t, "include"), os.path.join(t, "include", "torch", "csrc", "api", "include"),
              _cuda_include()]
    return [_cxx(), "-O2", "-std=c++17", "-fPIC", "-shared", "-Wall", "-Wextra",
            f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", "-I" + os.path.join(ROOT, "include"),
            *(w for d in system if d for w in ("-isystem", d)),
            os.path.join(CSRC, "q8_python.cpp"), "-o", out, "-L" + os.path.join(t, "lib"),
            "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"]


def _older(path, deps) -> bool:
    return not os.path.exists(path) or any(os.path.getmtime(d) > os.path.getmtime(path) for d in deps)


def _native_stale() -> bool:
    return _older(native_path(), [os.path.join(CSRC, "q8_python.cpp"), os.path.join(ROOT, "include", "q8.h"), __file__])


def _stale() -> bool:
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f != "q8_python.cpp"] + [os.path.join(ROOT, "include", "q8.h"), __file__]
    return _older(LIB, deps)


def build_native(force: bool = False) -> str:
    """The marshalling module alone, which needs a C++ compiler and no nvcc."""
    path = native_path()
    if not force and not _native_stale():
        return path
    if _cxx() is None:
        raise RuntimeError("no C++ compiler (CXX, g++ or c++)")
    part = f"{path}.{os.getpid()}"   # (renamed when whole: another process may be loading the module)
    pr = subprocess.run(_native_command(part), stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    sys.stderr.write(pr.stdout)
    if pr.returncode != 0:
        raise RuntimeError("the compiler failed")
    os.replace(part, path)
    return path


def build(force: bool = False, verbose: bool = False) -> str:
    with ThreadPoolExecutor(1) as pool:   # beside nvcc
        native = pool.submit(build_native, force)
        if force or _stale():
            _build_library(verbose)
    native.result()
    return LIB


def _build_library(verbose):
    objs = []
    procs = []
    for src in SOURCES:
        obj = os.path.join(HERE, "_build", src.replace(".cu", ".o"))
        os.makedirs(os.path.dirname(obj), exist_ok=True)
        cmd = ["nvcc", *FLAGS, "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
        objs.append(obj)
    failed = False
    for src, pr in procs:
        out, _ = pr.communicate()
        if verbose or pr.returncode != 0:
            sys.stderr.write(out)
        failed |= pr.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    subprocess.run(["nvcc", "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-o", LIB, *objs], check=True)


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
