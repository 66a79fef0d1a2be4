"""Build the CUDA library in-tree for sm_100a with nvcc (cross-compiles without a GPU)."""
import glob
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
LIB = os.path.join(HERE, "libcadnn.so")
FAST = os.path.join(HERE, "_fastcall" + sysconfig.get_config_var("EXT_SUFFIX"))   # native argument marshalling of the binding
FAST_SOURCE = os.path.join(HERE, "csrc", "fastcall.c")
SOURCES = sorted(glob.glob(os.path.join(HERE, "csrc", "*.cu")))
HEADERS = sorted(glob.glob(os.path.join(HERE, "csrc", "*.h"))) + [os.path.join(ROOT, "include", "cadnn.h")]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
              "-shared", "-Xcompiler", "-fPIC", "-I" + os.path.join(ROOT, "include")]


def stale():
    if not os.path.exists(LIB) or not os.path.exists(FAST):
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(FAST))
    return any(os.path.getmtime(f) > t for f in SOURCES + HEADERS + [FAST_SOURCE])


def build_fast():
    """Compile the CPython extension against the library next to it."""
    tmp = FAST + ".tmp%d" % os.getpid()
    subprocess.check_call([os.environ.get("CC", "gcc"), "-O2", "-fPIC", "-shared", "-I" + sysconfig.get_paths()["include"],
                           "-I" + os.path.join(ROOT, "include"), FAST_SOURCE, "-o", tmp, "-L" + HERE, "-l:" + os.path.basename(LIB),
                           "-Wl,-rpath,$ORIGIN"])
    os.replace(tmp, FAST)


def build(force=False, verbose=False):
    """Compile every .cu under csrc/ into libcadnn.so, and the binding's extension; returns the library's path."""
    if not force and not stale():
        return LIB
    nvcc = os.environ.get("NVCC", "nvcc")
    objs = []
    procs = []
    bdir = os.path.join(HERE, "_build")
    os.makedirs(bdir, exist_ok=True)
    for src in SOURCES:
        obj = os.path.join(bdir, os.path.basename(src) + ".o")
        objs.append(obj)
        cmd = [nvcc] + [f for f in NVCC_FLAGS if f != "-shared"] + (["-Xptxas", "-v"] if verbose else []) + ["-c", src, "-o", obj]
        procs.append((cmd, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT)))
    for cmd, p in procs:
        out, _ = p.communicate()
        if verbose or p.returncode:
            sys.stderr.write(out.decode(errors="replace"))
        if p.returncode:
            raise RuntimeError("nvcc failed: " + " ".join(cmd))
    tmp = LIB + ".tmp%d" % os.getpid()
    subprocess.check_call([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-o", tmp] + objs)
    os.replace(tmp, LIB)
    build_fast()
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
