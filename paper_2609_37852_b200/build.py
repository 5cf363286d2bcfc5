"""Builds the C-ABI library ``libattnfp8.so`` in-tree with nvcc for sm_100a, and beside it ``_marshal.so``,
the C++ side of ``binding`` (argument marshalling, compiled against the installed torch).

Usage: ``python -m paper_2609_37852_b200.build`` (or ``build()`` from Python).
Sources are compiled to objects in parallel and linked into
``paper_2609_37852_b200/libattnfp8.so``; nothing is installed elsewhere.
"""
import concurrent.futures
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OUT = os.path.join(HERE, "libattnfp8.so")
MARSHAL = os.path.join(HERE, "_marshal.so")
OBJ_DIR = os.path.join(HERE, "build")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo",
    "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr",
]


def _nvcc():
    path = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(path):
        raise RuntimeError("nvcc not found: the CUDA extension cannot be built")
    return path


def sources():
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cu"))


def _stale(target, deps):
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build(force=False, verbose=False):
    """Compile every .cu under csrc/ and link the shared library.  Returns its path."""
    nvcc = _nvcc()
    os.makedirs(OBJ_DIR, exist_ok=True)
    headers = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    headers.append(os.path.join(os.path.dirname(HERE), "include", "attn_fp8.h"))
    jobs = []
    objs = []
    for src in sources():
        obj = os.path.join(OBJ_DIR, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        if force or _stale(obj, [src] + headers):
            cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-c", src, "-o", obj]
            jobs.append(cmd)

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        return cmd, r

    with concurrent.futures.ThreadPoolExecutor(max_workers=8) as ex:
        for cmd, r in ex.map(run, jobs):
            if verbose or r.returncode:
                sys.stderr.write(" ".join(cmd) + "\n" + r.stdout + r.stderr)
            if r.returncode:
                raise RuntimeError("nvcc failed for " + cmd[-3])
    if jobs or force or _stale(OUT, objs):
        cmd = [nvcc, "-shared", "-o", OUT] + objs + ["-gencode", "arch=compute_100a,code=sm_100a"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode:
            sys.stderr.write(r.stdout + r.stderr)
            raise RuntimeError("link failed")
    build_marshal(force, verbose)
    return OUT


def marshal_key():
    """The interpreter and torch build that a compiled marshalling module works with."""
    import sysconfig
    import torch
    return "torch %s, C++11 ABI %d, %s" % (torch.__version__, int(torch.compiled_with_cxx11_abi()), sysconfig.get_config_var("EXT_SUFFIX"))


def marshal_built_for(path=None):
    """The key that the module at `path` was compiled for; None when there is no such file or it names none."""
    mark = b"marshal built for: "
    try:
        with open(path or MARSHAL, "rb") as f:
            data = f.read()
    except OSError:
        return None
    at = data.find(mark)
    return data[at + len(mark):data.index(b"\0", at)].decode() if at >= 0 else None


def build_marshal(force=False, verbose=False):
    """Compile csrc/marshal.cpp into an extension module linked against the library and torch's own."""
    src = os.path.join(CSRC, "marshal.cpp")
    key = marshal_key()
    if not force and marshal_built_for() == key and not _stale(MARSHAL, [src, os.path.join(os.path.dirname(HERE), "include", "attn_fp8.h")]):
        return
    import sysconfig
    import torch
    from torch.utils import cpp_extension
    inc = cpp_extension.include_paths() + [sysconfig.get_paths()["include"],
                                           os.path.join(os.path.dirname(os.path.dirname(_nvcc())), "include")]
    lib = os.path.join(os.path.dirname(torch.__file__), "lib")
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch.compiled_with_cxx11_abi()), '-DMARSHAL_BUILT_FOR="%s"' % key]
    for d in inc:
        cmd += ["-isystem", d]
    cmd += [src, "-o", MARSHAL, "-L" + HERE, "-lattnfp8", "-L" + lib, "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python",
            "-Wl,-rpath,$ORIGIN", "-Wl,-rpath," + lib]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or r.returncode:
        sys.stderr.write(" ".join(cmd) + "\n" + r.stdout + r.stderr)
    if r.returncode:
        raise RuntimeError("the marshalling module did not compile")


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
