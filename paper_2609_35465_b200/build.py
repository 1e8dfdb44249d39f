"""Builds the CUDA library in-tree, paper_2609_35465_b200/libtetra_b200.so (sm_100a), and the native half of the
Python binding, _binding.so.

nvcc cross-compiles without a GPU.  Run:  python -m paper_2609_35465_b200.build
"""
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libtetra_b200.so")
BINDING = os.path.join(HERE, "_binding.so")
SOURCES = ["tetra_tables.cpp", "tetra_decode.cu", "tetra_gemv.cu", "tetra_list.cu", "tetra_batched.cu", "tetra_api.cu", "tetra_noalloc.cu", "q4_gemv.cu", "q4_list.cu", "tetra_encode.cu"]
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo",
         "-Xcompiler", "-fPIC", "-Xcompiler", "-Wall", "--use_fast_math"]


def built_for() -> str:
    """What the binding is tied to; the file holds this text, and tetra.py asks for it before the first call."""
    import torch
    return "torch %s, Python %d.%d" % (torch.__version__, sys.version_info[0], sys.version_info[1])


def _stale() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(BINDING):
        return True
    with open(BINDING, "rb") as f:
        if built_for().encode() not in f.read():
            return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(BINDING))
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if not f.endswith(".o")]  # the objects are the build's own
    deps += [os.path.join(os.path.dirname(HERE), "include", h) for h in ("tetra.h", "tetra_q4.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def _binding_command(out: str):
    """g++ command for csrc/binding.cpp against the installed torch and this interpreter."""
    import torch
    root = os.path.dirname(torch.__file__)
    inc, lib = os.path.join(root, "include"), os.path.join(root, "lib")
    cuda = os.path.dirname(os.path.dirname(NVCC))
    return [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
            "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI), '-DTETRA_BUILT_FOR="%s"' % built_for(),
            "-isystem", inc, "-isystem", os.path.join(inc, "torch", "csrc", "api", "include"),
            "-isystem", os.path.join(cuda, "include"), "-isystem", sysconfig.get_paths()["include"],
            os.path.join(CSRC, "binding.cpp"), "-o", out, "-L" + lib, "-ltorch_python", "-ltorch_cuda", "-ltorch_cpu", "-lc10_cuda", "-lc10",
            "-ldl"]


def build(force: bool = False, verbose: bool = False) -> str:
    if not (force or _stale()):
        return LIB
    flags = list(FLAGS) + os.environ.get("TETRA_EXTRA_FLAGS", "").split()
    if verbose:
        flags += ["-Xptxas", "-v"]
    # built beside their place and moved there whole: a program that is running keeps the library it has loaded
    tmp_lib, tmp_binding = ["%s.tmp.%d" % (path, os.getpid()) for path in (LIB, BINDING)]
    objs = []
    procs = []
    try:
        for src in SOURCES:
            obj = os.path.join(CSRC, os.path.splitext(src)[0] + ".o")
            objs.append(obj)
            procs.append(subprocess.Popen([NVCC] + flags + ["-c", os.path.join(CSRC, src), "-o", obj], cwd=CSRC))
        procs.append(subprocess.Popen(_binding_command(tmp_binding)))
        if any([p.wait() != 0 for p in procs]):
            raise RuntimeError("the compiler failed")
        subprocess.run([NVCC, "-shared", "-o", tmp_lib] + objs + ["-lcudart"], check=True, cwd=CSRC)
        os.replace(tmp_lib, LIB)
        os.replace(tmp_binding, BINDING)
    finally:  # a failed or interrupted build leaves nothing beside the sources
        for p in procs:
            if p.poll() is None:
                p.terminate()
                p.wait()
        for tmp in (tmp_lib, tmp_binding):
            if os.path.exists(tmp):
                os.remove(tmp)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
