"""Build libbfhe.so in-tree with nvcc for sm_103a (one -gencode, parallel TUs).

Usage: python -m paper_2204_12201_gb300.build   (or build() from Python)
The library lands in paper_2204_12201_gb300/_lib/libbfhe.so; objects in _build/.
"""

import concurrent.futures as cf
import os
import shutil
import subprocess
import sys

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIBDIR = os.path.join(PKG, "_lib")
OBJDIR = os.path.join(ROOT, "_build")
# (object, source, defines): the kernels of ntt.cu and ext_pm.cu compile as several objects in parallel
UNITS = [("host", "host.cu", []), ("kernels", "kernels.cu", []), ("ext", "ext.cu", []), ("api", "api.cu", [])]
UNITS += [("ext_pm%d" % p, "ext_pm.cu", ["-DBFHE_EXT_PM_PART=%d" % p]) for p in range(5)]
UNITS += [("ntt%d" % p, "ntt.cu", ["-DBFHE_NTT_PART=%d" % p]) for p in range(5)]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-Xcompiler", "-O2"]


def _nvcc():
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def lib_path():
    return os.path.join(LIBDIR, "libbfhe.so")


def _stale(obj, srcs):
    if not os.path.exists(obj):
        return True
    t = os.path.getmtime(obj)
    return any(os.path.getmtime(s) > t for s in srcs)


def build(verbose=False, force=False):
    nvcc = _nvcc()
    os.makedirs(LIBDIR, exist_ok=True)
    os.makedirs(OBJDIR, exist_ok=True)
    headers = [os.path.join(CSRC, h) for h in os.listdir(CSRC) if h.endswith((".cuh", ".h"))]
    headers.append(os.path.join(ROOT, "include", "bfhe.h"))
    jobs = []
    for name, src, defs in UNITS:
        s = os.path.join(CSRC, src)
        o = os.path.join(OBJDIR, name + ".o")
        if force or _stale(o, [s] + headers):
            jobs.append([nvcc, *ARCH, *FLAGS, *defs, "-c", s, "-o", o])

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed:\n" + " ".join(cmd) + "\n" + r.stdout + r.stderr)
        if verbose:
            sys.stdout.write(r.stdout + r.stderr)

    with cf.ThreadPoolExecutor(max_workers=len(UNITS)) as ex:
        list(ex.map(run, jobs))
    objs = [os.path.join(OBJDIR, name + ".o") for name, _, _ in UNITS]
    lib = lib_path()
    if force or jobs or _stale(lib, objs):
        tmp = lib + ".tmp"
        run([nvcc, *ARCH, "-shared", "-o", tmp, *objs, "-lcudart"])
        os.replace(tmp, lib)
    return lib


def build_demo():
    """Compile examples/abi_demo.c against the library (plain C through the ABI); returns its path."""
    lib = build()
    cc = shutil.which("gcc") or shutil.which("cc")
    if cc is None:
        raise RuntimeError("no C compiler")
    cuda = os.path.dirname(os.path.dirname(_nvcc()))
    out = os.path.join(LIBDIR, "abi_demo")
    cmd = [cc, "-O2", "-I", os.path.join(ROOT, "include"), "-I", os.path.join(cuda, "include"),
           os.path.join(PKG, "examples", "abi_demo.c"), "-o", out, "-L", LIBDIR, "-lbfhe",
           "-L", os.path.join(cuda, "lib64"), "-lcudart", "-Wl,-rpath," + LIBDIR]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("demo build failed:\n" + " ".join(cmd) + "\n" + r.stdout + r.stderr)
    return out, lib


if __name__ == "__main__":
    print(build(verbose="-v" in sys.argv, force="-f" in sys.argv))
