"""Build libptqtp.so in-tree with nvcc for sm_100a and the marshalling extension of the binding with the host compiler (no JIT cache, no
torch extension machinery)."""
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libptqtp.so")
SOURCES = ["api.cu", "pack.cu", "pack2.cu", "gemv.cu", "gemv2.cu", "gemv3.cu", "pack3.cu", "gemv4.cu", "gemv5.cu", "gemm7.cu", "gemm8.cu", "skinny3.cu", "decompose.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden", "--shared", "-cudart", "shared"]


def _nvcc():
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def marshal_path():
    """The extension's file, which belongs to one Python and one torch: it is made of the headers of both."""
    import torch
    return os.path.join(HERE, "_marshal-%s%s" % (torch.__version__, sysconfig.get_config_var("EXT_SUFFIX")))


def _stale(target, sources):
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in sources + [os.path.join(ROOT, "include", "ptqtp.h")])


def library_stale():
    return _stale(LIB, [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cu", ".h"))])


def marshal_stale():
    try:
        return _stale(marshal_path(), [os.path.join(CSRC, "marshal.cpp")])
    except ImportError:
        return False                                     # without torch nobody calls it


def needs_build():
    return library_stale() or marshal_stale()


def build_marshal():
    """Compile csrc/marshal.cpp against the torch that is installed."""
    import torch
    root = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(_nvcc())) if os.path.isabs(_nvcc()) else "/usr/local/cuda"
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI), '-DPTQTP_TORCH_VERSION="%s"' % torch.__version__, "-I", os.path.join(ROOT, "include"),
           "-I", sysconfig.get_paths()["include"], "-isystem", os.path.join(cuda, "include"), "-isystem", os.path.join(root, "include"),
           "-isystem", os.path.join(root, "include", "torch", "csrc", "api", "include"), os.path.join(CSRC, "marshal.cpp"),
           "-L", os.path.join(root, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python", "-o", marshal_path()]
    res = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    if res.returncode != 0:
        raise RuntimeError("%s failed\n%s" % (cmd[0], res.stdout))


def build(force=False, verbose=False, extra=()):
    """Compile every CUDA source into paper_2509_16989_b200/libptqtp.so and the marshalling extension, what is not up to date of the two;
    returns the library's path.  The library needs no torch; the binding runs without the extension, only slower, so where that cannot be
    built (no host compiler, no torch or Python headers) a message is printed."""
    if force or library_stale():
        cmd = [_nvcc()] + NVCC_FLAGS + list(extra) + ["-I", os.path.join(ROOT, "include"), "-I", CSRC]
        if verbose:
            cmd += ["-Xptxas", "-v"]
        cmd += [os.path.join(CSRC, s) for s in SOURCES] + ["-o", LIB]
        res = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
        if verbose or res.returncode != 0:
            sys.stderr.write(res.stdout)
        if res.returncode != 0:
            raise RuntimeError("nvcc failed building libptqtp.so")
    if force or marshal_stale():
        try:
            build_marshal()
        except (ImportError, OSError, RuntimeError) as e:
            if not isinstance(e, ImportError) and os.path.exists(marshal_path()):           # of older sources
                os.remove(marshal_path())
            sys.stderr.write("the marshalling extension was not built, plain calls of the binding take the slower way: %s\n" % e)
    return LIB


if __name__ == "__main__":
    build(force=True, verbose="-v" in sys.argv)
    print(LIB)
