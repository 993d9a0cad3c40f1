"""Compile the CUDA library (sm_100a) and the binding's native marshaller in-tree: paper_2606_12370_b200/libbebop.so
and paper_2606_12370_b200/_bebop_host.so."""
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libbebop.so")
HOST = os.path.join(HERE, "_bebop_host.so")
HOST_FOR = HOST + ".for"       # the versions it was made for
SOURCES = ["bebop_api.cu", "bebop_general.cu", "bebop_redraw.cu", "bebop_pipe.cu", "bebop_fuse.cu",
           "bebop_seq.cu"]
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
         "-Xcompiler", "-fPIC", "-shared"]


def _deps():
    out = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    out.append(os.path.join(os.path.dirname(HERE), "include", "bebop.h"))
    return out


def _run(cmd, out, verbose):
    """Run a compiler that writes `out` (under another name until it is complete)."""
    tmp = out + ".tmp.%d" % os.getpid()
    r = subprocess.run(cmd + ["-o", tmp], capture_output=True, text=True)
    if verbose or r.returncode != 0:
        sys.stderr.write(r.stdout + r.stderr)
    if r.returncode != 0:
        raise RuntimeError("%s failed" % cmd[0])
    os.replace(tmp, out)


def _fresh(out, deps):
    return os.path.exists(out) and all(os.path.getmtime(out) >= os.path.getmtime(d) for d in deps)


def _host_made_for() -> str:
    """What the native marshaller is compiled against: it uses internals of torch and of CPython, whose layout another
    version may change."""
    import torch
    return "torch %s at %s, python %s\n" % (torch.__version__, os.path.dirname(torch.__file__), sysconfig.get_config_var("SOABI"))


def _host_fresh() -> bool:
    src = os.path.join(CSRC, "bebop_host.cpp")
    if not _fresh(HOST, [src, os.path.join(os.path.dirname(HERE), "include", "bebop.h")]) or not os.path.exists(HOST_FOR):
        return False
    with open(HOST_FOR) as f:
        return f.read() == _host_made_for()


def build_host(force: bool = False, verbose: bool = False) -> str:
    """The native marshaller: a CPython module against torch's headers and libraries."""
    src = os.path.join(CSRC, "bebop_host.cpp")
    if force or not _host_fresh():
        import torch
        root = os.path.dirname(torch.__file__)
        inc = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
               sysconfig.get_paths()["include"], os.path.join(os.path.dirname(os.path.dirname(NVCC)), "include")]
        _run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI)] +
             ["-I" + d for d in inc] + [src, "-L" + os.path.join(root, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"],
             HOST, verbose)
        with open(HOST_FOR, "w") as f:
            f.write(_host_made_for())
    return HOST


def build(force: bool = False, verbose: bool = False) -> str:
    build_host(force, verbose)
    if not force and _fresh(LIB, _deps()):
        return LIB
    extra = os.environ.get("BEBOP_NVCC_EXTRA", "").split()
    _run([NVCC] + FLAGS + extra + (["-Xptxas", "-v"] if verbose else []) + [os.path.join(CSRC, s) for s in SOURCES], LIB, verbose)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
