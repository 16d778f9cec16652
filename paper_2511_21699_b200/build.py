"""Builds libcacheback.so (the C-ABI library) in-tree with nvcc for sm_100a, and libcacheback_debug.so, the same sources
compiled with -DCB_DEBUG (range checks on indices taken from memory, guard areas behind the workspace regions), and
_binding.so, the Python module with the host side of the step calls (csrc/cb_binding.cpp, g++ against torch's headers)."""
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
SO = os.path.join(HERE, "libcacheback.so")
SO_DEBUG = os.path.join(HERE, "libcacheback_debug.so")
SO_BINDING = os.path.join(HERE, "_binding.so")
SOURCES = ["cb_api.cu", "cb_table.cu", "cb_accept.cu", "cb_kv.cu", "cb_branches.cu", "cb_frozen.cu", "cb_frozen_build.cu", "cb_attn.cu", "cb_attn_tc.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", CSRC]


def _stale(target, deps):
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build_binding(force=False):
    import torch
    src = os.path.join(CSRC, "cb_binding.cpp")
    # The module is tied to torch's C++ classes and to the interpreter, so what it was built against lies beside it.
    against = "torch %s, %s, C++11 ABI %d\n" % (torch.__version__, sys.implementation.cache_tag, int(torch._C._GLIBCXX_USE_CXX11_ABI))
    stamp = SO_BINDING + ".stamp"
    built = open(stamp).read() if os.path.exists(stamp) else None
    if not force and built == against and not _stale(SO_BINDING, [src, os.path.join(ROOT, "include", "cacheback.h"), os.path.abspath(__file__)]):
        return SO_BINDING
    t = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
    inc = [os.path.join(ROOT, "include"), os.path.join(t, "include"), os.path.join(t, "include", "torch", "csrc", "api", "include"),
           os.path.join(cuda, "include"), sysconfig.get_paths()["include"]]
    tmp = SO_BINDING + ".tmp%d" % os.getpid()
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI)] +
                          [x for i in inc for x in ("-isystem" if i.startswith(t) else "-I", i)] +
                          [src, "-o", tmp, "-L", os.path.join(t, "lib"), "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"])
    os.replace(tmp, SO_BINDING)
    with open(stamp + ".tmp%d" % os.getpid(), "w") as f:
        f.write(against)
    os.replace(stamp + ".tmp%d" % os.getpid(), stamp)
    return SO_BINDING


def build(force=False, verbose=False, debug=False):
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    so, suffix, extra = (SO_DEBUG, ".dbg.o", ["-DCB_DEBUG"]) if debug else (SO, ".o", [])
    hdrs = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    hdrs.append(os.path.join(ROOT, "include", "cacheback.h"))
    objs = []
    procs = []
    for s in SOURCES:
        src = os.path.join(CSRC, s)
        obj = os.path.join(CSRC, s.replace(".cu", suffix))
        objs.append(obj)
        if force or _stale(obj, [src] + hdrs):
            cmd = [nvcc] + NVCC_FLAGS + extra + (["-Xptxas", "-v"] if verbose else []) + ["-c", src, "-o", obj]
            procs.append((s, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    for s, p in procs:
        out, _ = p.communicate()
        if verbose or p.returncode != 0:
            sys.stderr.write(out)
        if p.returncode != 0:
            raise RuntimeError("nvcc failed on %s" % s)
    if force or procs or _stale(so, objs):
        tmp = so + ".tmp%d" % os.getpid()
        subprocess.check_call([nvcc, "-shared", "-o", tmp] + objs + ["-gencode", "arch=compute_100a,code=sm_100a"])
        os.replace(tmp, so)
    build_binding(force)
    return so


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv, debug=True))
