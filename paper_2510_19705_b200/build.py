"""In-tree build of the C-ABI library (libhsd.so) for sm_100a with nvcc alone, and of the binding's native calls with the C++
compiler, where torch is installed (the library needs none of it)."""
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libhsd.so")
HEADER = os.path.join(HERE, "..", "include", "hsd.h")
HOST_SRC = os.path.join(HERE, "native", "host_calls.cpp")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
FLAGS = ["-std=c++17", "-O3", "-lineinfo", "-gencode", "arch=compute_100a,code=sm_100a", "-Xcompiler", "-fPIC",
         "--cudart", "static", "--expt-extended-lambda", "--expt-relaxed-constexpr"]


def sources():
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cu", ".cpp")))


def _torch():
    try:
        import torch
    except ImportError:
        return None
    return torch


def host_path():
    """The binding's native calls, built against this Python and this torch (None without torch)."""
    torch = _torch()
    return torch and os.path.join(HERE, "_host_calls.%s.torch-%s.so" % (sysconfig.get_config_var("SOABI"), torch.__version__))


def _older(target, deps):
    return not os.path.exists(target) or any(os.path.getmtime(d) > os.path.getmtime(target) for d in deps)


def _library_is_old():
    return _older(LIB, [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [HEADER])


def _host_is_old():
    return host_path() is not None and _older(host_path(), [HOST_SRC, HEADER])


def needs_build():
    return _library_is_old() or _host_is_old()


def host_command():
    """g++ command of the binding's native calls: torch's headers and libraries, no device code."""
    torch = _torch()
    root = os.path.dirname(torch.__file__)
    lib = os.path.join(root, "lib")
    cuda = os.path.dirname(os.path.dirname(NVCC))
    inc = [sysconfig.get_paths()["include"], os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
           os.path.join(cuda, "include")]
    return [os.environ.get("CXX", "g++"), "-std=c++17", "-O2", "-fPIC", "-shared", "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI)] + \
        ["-isystem" + d for d in inc] + [HOST_SRC, "-o", host_path(), "-L" + lib, "-Wl,-rpath," + lib, "-ltorch_python", "-ltorch_cpu", "-lc10_cuda", "-lc10"]


def _finish(src, proc, verbose):
    out, _ = proc.communicate()
    if verbose or proc.returncode != 0:
        sys.stderr.write(out)
    if proc.returncode != 0:
        raise RuntimeError("the compiler failed on " + src)


def _start(cmd):
    return subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)


def build_library(verbose=False):
    """Compile every CUDA source into libhsd.so."""
    os.makedirs(os.path.join(HERE, "build"), exist_ok=True)
    objs, procs = [], []
    for src in sources():
        objs.append(os.path.join(HERE, "build", os.path.basename(src) + ".o"))
        extra = os.environ.get("HSD_NVCC_EXTRA", "").split()
        procs.append((src, _start([NVCC] + FLAGS + extra + (["-Xptxas", "-v"] if verbose else []) + ["-c", src, "-o", objs[-1]])))
    for src, p in procs:
        _finish(src, p, verbose)
    subprocess.run([NVCC, "-shared", "--cudart", "static", "-gencode", "arch=compute_100a,code=sm_100a", "-o", LIB] + objs, check=True)


def build(force=False, verbose=False):
    """Bring the library and, where torch is installed, the binding's native calls up to date; returns the library's path."""
    if force or _library_is_old():
        build_library(verbose)
    if _host_is_old() or (force and host_path()):
        _finish(HOST_SRC, _start(host_command()), verbose)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
