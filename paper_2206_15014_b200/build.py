"""Builds libnmsparse.so (the C-ABI library) in-tree with nvcc for sm_100a."""
from __future__ import annotations

import importlib.machinery
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libnmsparse.so")
SOURCES = ("api.cu", "pack.cu", "quant_act.cu", "gemm.cu", "probe.cu")
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
         "-Xcompiler", "-fPIC", "--ftz=false", "--prec-div=true",
         "--prec-sqrt=true"]


# Other builds of the same sources: "trace" compiles time stamps into the GEMM kernels (nm_debug_set_trace),
# "shortwait" gives every device-side wait a limit of about a millisecond (the timeout test runs against it).
VARIANTS = {"": [], "trace": ["-DNM_TRACE"], "shortwait": ["-DNM_WAIT_LIMIT=(1ll<<21)", "-DNM_TEST_HOOKS"]}


# Extension module of the Python binding (csrc/marshal.c): plain C against the interpreter's headers, under this interpreter's tag, so that
# no other one loads it.  The binding is complete without it, and the library is built where it cannot be.
MARSHAL = os.path.join(HERE, "_marshal" + importlib.machinery.EXTENSION_SUFFIXES[0])


def build_marshal(force: bool = False) -> str | None:
    deps = (os.path.join(CSRC, "marshal.c"), os.path.join(os.path.dirname(HERE), "include", "nmsparse.h"), os.path.abspath(__file__))
    if not force and os.path.exists(MARSHAL) and os.path.getmtime(MARSHAL) >= max(map(os.path.getmtime, deps)):
        return MARSHAL
    tmp = MARSHAL + f".tmp{os.getpid()}"
    try:
        subprocess.check_call([os.environ.get("CC", "gcc"), "-O2", "-Wall", "-shared", "-fPIC", "-I" + sysconfig.get_paths()["include"],
                               deps[0], "-o", tmp])
    except (OSError, subprocess.CalledProcessError) as e:
        sys.stderr.write(f"{os.path.basename(MARSHAL)} not built ({e}): calls go through ctypes\n")
        return None
    os.replace(tmp, MARSHAL)
    return MARSHAL


def lib_path(variant: str = "") -> str:
    return LIB if not variant else os.path.join(HERE, f"libnmsparse_{variant}.so")


def _stale(lib: str = LIB) -> bool:
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh"))]
    deps.append(os.path.join(os.path.dirname(HERE), "include", "nmsparse.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False, variant: str = "") -> str:
    LIB = lib_path(variant)
    build_marshal(force)
    if not force and not _stale(LIB):
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    objs = []
    procs = []
    suffix = f".{variant}.o" if variant else ".o"
    for src in SOURCES:
        obj = os.path.join(CSRC, src.replace(".cu", suffix))
        cmd = [nvcc, *FLAGS, *VARIANTS[variant], "-c", os.path.join(CSRC, src), "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT)))
        objs.append(obj)
    for src, p in procs:
        out, _ = p.communicate()
        if verbose or p.returncode:
            sys.stderr.write(out.decode())
        if p.returncode:
            raise RuntimeError(f"nvcc failed on {src}")
    tmp = LIB + f".tmp{os.getpid()}"
    subprocess.check_call([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-o", tmp, *objs, "-cudart", "static"])
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    variant = sys.argv[sys.argv.index("--variant") + 1] if "--variant" in sys.argv else ""
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv, variant=variant))
