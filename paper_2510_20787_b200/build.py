"""Build ``liblte.so`` (the C-ABI CUDA library, nvcc for sm_100a) and ``_binding.so`` (its Python binding, g++) in-tree.

Usage: ``python -m paper_2510_20787_b200.build [--force] [--verbose]``.
Object files are cached per source under ``csrc/build`` and rebuilt when the source or a header is newer.
"""
import concurrent.futures
import glob
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")
LIB = os.path.join(HERE, "liblte.so")
BINDING = os.path.join(HERE, "_binding.so")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
         "-Xcompiler", "-fPIC", "-I", INCLUDE, "-I", CSRC]


def _newer(target, deps):
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def _built_for(target, tag):
    with open(target, "rb") as f:
        return tag.encode() in f.read()


def build_binding(force=False, verbose=False):
    """The CPython module over ``liblte.so``: needs torch's headers and libraries, no CUDA compiler.  It uses torch's C++ interface, so it
    carries the versions it was built for (torch's, Python's) as a string and is built again for others."""
    import torch
    src = os.path.join(CSRC, "binding.cpp")
    tag = "lte binding for torch %s, %s" % (torch.__version__, sys.implementation.cache_tag)
    if not force and not _newer(BINDING, [src, LIB, os.path.join(INCLUDE, "lte.h")]) and _built_for(BINDING, tag):
        return BINDING
    troot = os.path.dirname(torch.__file__)
    tmp = BINDING + ".tmp.%d" % os.getpid()
    cmd = (["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI),
            '-DLTE_BUILT_FOR="%s"' % tag, src, "-o", tmp]
           + ["-I" + d for d in (INCLUDE, sysconfig.get_paths()["include"])]
           + ["-isystem" + d for d in (os.path.join(troot, "include"), os.path.join(troot, "include", "torch", "csrc", "api", "include"),
                                       os.path.join(os.path.dirname(os.path.dirname(NVCC)), "include"))]
           + ["-L" + os.path.join(troot, "lib"), "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10_cuda", "-lc10",
              "-L" + HERE, "-l:liblte.so", "-Wl,-rpath,$ORIGIN"])
    r = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or r.returncode:
        sys.stderr.write(" ".join(cmd) + "\n" + r.stdout + r.stderr)
    if r.returncode:
        raise RuntimeError("g++ failed for binding.cpp")
    os.replace(tmp, BINDING)
    return BINDING


def build(force=False, verbose=False):
    srcs = sorted(glob.glob(os.path.join(CSRC, "*.cu")))
    hdrs = glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(INCLUDE, "*.h"))
    objdir = os.path.join(CSRC, "build")
    os.makedirs(objdir, exist_ok=True)
    jobs = []
    objs = []
    for s in srcs:
        o = os.path.join(objdir, os.path.basename(s)[:-3] + ".o")
        objs.append(o)
        if force or _newer(o, [s] + hdrs):
            cmd = [NVCC] + FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-c", s, "-o", o]
            jobs.append(cmd)

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        return cmd, r

    with concurrent.futures.ThreadPoolExecutor(max_workers=min(8, max(1, len(jobs)))) as ex:
        for cmd, r in ex.map(run, jobs):
            if verbose or r.returncode:
                sys.stderr.write(" ".join(cmd) + "\n" + r.stdout + r.stderr)
            if r.returncode:
                raise RuntimeError("nvcc failed for " + cmd[-3])
    if jobs or force or _newer(LIB, objs):
        tmp = LIB + ".tmp.%d" % os.getpid()
        subprocess.check_call([NVCC, "-shared", "-o", tmp] + objs + ["-lcudart"])
        os.replace(tmp, LIB)
    build_binding(force, verbose)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
