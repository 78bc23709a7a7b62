"""Builds libtreeverify.so (sm_100a only) in-tree with nvcc.

    python -m paper_2603_08088_b200.build [--force] [--verbose]

Every .cu under csrc/ is compiled to an object file under csrc/build/ and
linked into paper_2603_08088_b200/libtreeverify.so; csrc/calls.cpp (argument
marshalling for Python) becomes paper_2603_08088_b200/_calls.so, which links to
it.  Objects are rebuilt when their source or a header is newer, _calls.so also
when it was made for another torch or Python.  The library itself needs neither:
where torch cannot be imported, _calls.so is left out.
"""
import os
import shutil
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
OBJ = os.path.join(CSRC, "build")
LIB = os.path.join(PKG, "libtreeverify.so")
CALLS = os.path.join(PKG, "_calls.so")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden",
    "-I", os.path.join(ROOT, "include"), "-I", CSRC,
]


def _nvcc():
    exe = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(exe):
        raise RuntimeError("nvcc not found; the treeverify library cannot be built")
    return exe


def _calls_commands():
    """Compile and link commands of _calls.so (torch's headers and libraries are those of the running Python)."""
    import torch
    root = os.path.dirname(torch.__file__)
    lib, inc = os.path.join(root, "lib"), os.path.join(root, "include")
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(_nvcc())))
    made_for = f"torch {torch.__version__} {torch.__file__}, Python {sys.version}"
    obj = os.path.join(OBJ, "calls.o")
    abi = int(torch._C._GLIBCXX_USE_CXX11_ABI)
    compile_cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-fvisibility=hidden", f"-D_GLIBCXX_USE_CXX11_ABI={abi}",
                   "-I", os.path.join(ROOT, "include"), "-isystem", os.path.join(cuda, "include"),
                   "-isystem", sysconfig.get_paths()["include"]]
    compile_cmd += ["-isystem", inc, "-isystem", os.path.join(inc, "torch", "csrc", "api", "include")]
    compile_cmd += ["-c", os.path.join(CSRC, "calls.cpp"), "-o", obj]
    link_cmd = ["g++", "-shared", "-o", CALLS, obj, "-L", PKG, "-l:libtreeverify.so", "-L", lib, "-ltorch_python", "-ltorch_cpu",
                "-lc10", "-lc10_cuda", "-Wl,-rpath,$ORIGIN", "-Wl,-rpath," + lib]
    return obj, compile_cmd, link_cmd, made_for


def _calls_stale(obj, made_for):
    """Whether _calls.so has to be made again: its sources are newer, or it is for another torch or Python."""
    stamp = obj + ".for"
    if not (os.path.exists(CALLS) and os.path.exists(obj) and os.path.exists(stamp)) or open(stamp).read() != made_for:
        return True
    sources = (os.path.join(CSRC, "calls.cpp"), os.path.join(ROOT, "include", "treeverify.h"))
    return os.path.getmtime(obj) < max(os.path.getmtime(s) for s in sources)


def _newest_header():
    inc = os.path.join(ROOT, "include")
    hdrs = [os.path.join(inc, f) for f in os.listdir(inc) if f.endswith(".h")]
    hdrs += [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    return max(os.path.getmtime(h) for h in hdrs)


def build(force=False, verbose=False):
    extra = os.environ.get("TV_NVCC_EXTRA", "").split()      # e.g. -DNAME=value for tuning builds
    if extra:
        force = True
    os.makedirs(OBJ, exist_ok=True)
    nvcc = _nvcc()
    srcs = sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))
    hdr_time = _newest_header()
    jobs = []
    objs = []
    for s in srcs:
        src = os.path.join(CSRC, s)
        obj = os.path.join(OBJ, s[:-3] + ".o")
        objs.append(obj)
        if force or not os.path.exists(obj) or os.path.getmtime(obj) < max(os.path.getmtime(src), hdr_time):
            cmd = [nvcc] + NVCC_FLAGS + extra + (["-Xptxas", "-v"] if verbose else []) + ["-c", src, "-o", obj]
            jobs.append(cmd)

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0 or verbose:
            sys.stderr.write(" ".join(cmd) + "\n" + r.stdout + r.stderr)
        if r.returncode != 0:
            raise RuntimeError(cmd[0] + " failed for " + cmd[-3])

    try:
        calls_obj, calls_compile, calls_link, made_for = _calls_commands()
        calls_stale = force or _calls_stale(calls_obj, made_for)
    except ImportError as e:
        sys.stderr.write(f"_calls.so is not built: {e}\n")
        calls_stale = False
    cu_jobs = len(jobs)
    if calls_stale:
        jobs.append(calls_compile)

    with ThreadPoolExecutor(max_workers=min(8, max(1, len(jobs)))) as ex:
        list(ex.map(run, jobs))
    if cu_jobs or not os.path.exists(LIB):
        cmd = [nvcc, "-shared", "-o", LIB] + objs + ["-gencode", "arch=compute_100a,code=sm_100a", "-lcudart_static", "-ldl", "-lrt", "-lpthread"]
        run(cmd)
    if calls_stale:
        run(calls_link)
        with open(calls_obj + ".for", "w") as f:
            f.write(made_for)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
