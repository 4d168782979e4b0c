"""In-tree build of libfocus_b200.so (nvcc, sm_100a only) and of the module in front of it (g++).  ``python -m paper_2604_03260_b200.build``."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libfocus_b200.so")
MARSHAL = os.path.join(HERE, "_marshal" + sysconfig.get_config_var("EXT_SUFFIX"))     # (other interpreters do not look for that name)
SOURCES = ["api.cu", "assign.cu", "assign_hidden.cu", "sinkhorn.cu", "decode.cu", "tiles.cu", "tiles_sorted.cu", "attn_sm100.cu", "selftest.cu",
           "tma_host.cu", "noalloc.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    raise RuntimeError("nvcc not found")


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def marshal_abi() -> str:
    """What the module depends on beside its source: it reads torch's tensor objects by their layout."""
    import torch
    return f"{torch.__version__} {torch.version.git_version} {sysconfig.get_config_var('SOABI')}"


def _marshal_cmd(out: str) -> list:
    """csrc/marshal.cpp: a Python module that reads torch tensors and calls the library (whose addresses it is given)"""
    import torch
    t = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(_nvcc())) if os.path.sep in _nvcc() else "/usr/local/cuda"
    return (["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
             f'-DFOCUS_BUILT_FOR="{marshal_abi()}"',
             "-I", os.path.join(ROOT, "include"), "-I", os.path.join(t, "include"), "-I", os.path.join(t, "include", "torch", "csrc", "api", "include"),
             "-I", os.path.join(cuda, "include"), "-I", sysconfig.get_paths()["include"], os.path.join(CSRC, "marshal.cpp"), "-o", out,
             "-L", os.path.join(t, "lib"), "-ltorch_python", "-ltorch", "-lc10", "-lc10_cuda"])


def _marshal_stamp() -> str:
    return os.path.join(HERE, "_build", "marshal.cmd")


def marshal_stale() -> bool:
    """the module is missing, older than its sources, or made by another command (another torch or Python among them)"""
    if _stale(MARSHAL, [os.path.join(CSRC, "marshal.cpp"), os.path.join(ROOT, "include", "focus.h")]) or not os.path.exists(_marshal_stamp()):
        return True
    with open(_marshal_stamp()) as f:
        return f.read() != "\n".join(_marshal_cmd(MARSHAL))


def build_marshal(force: bool = False) -> bool:
    """The module, where torch's headers and g++ are to hand; without it the binding makes the same calls through ctypes."""
    try:
        if force or marshal_stale():
            tmp = MARSHAL + ".tmp%d" % os.getpid()
            subprocess.check_call(_marshal_cmd(tmp))
            os.replace(tmp, MARSHAL)
            with open(_marshal_stamp(), "w") as f:
                f.write("\n".join(_marshal_cmd(MARSHAL)))
        return True
    except (ImportError, OSError, subprocess.CalledProcessError) as e:
        print(f"csrc/marshal.cpp not built, calls go through ctypes: {e}", file=sys.stderr)
        if os.path.exists(MARSHAL):             # of an older source or another torch
            os.remove(MARSHAL)
        return False


def build(force: bool = False, verbose: bool = False) -> str:
    headers = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    headers.append(os.path.join(ROOT, "include", "focus.h"))
    objdir = os.path.join(HERE, "_build")
    os.makedirs(objdir, exist_ok=True)
    objs = []
    procs = []
    for src in SOURCES:
        s = os.path.join(CSRC, src)
        o = os.path.join(objdir, src.replace(".cu", ".o"))
        objs.append(o)
        if force or _stale(o, [s] + headers):
            cmd = [_nvcc()] + NVCC_FLAGS + ["-I", os.path.join(ROOT, "include"), "-I", CSRC, "-c", s, "-o", o]
            if verbose:
                cmd.insert(1, "-Xptxas=-v")
            procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = False
    for src, p in procs:
        out, _ = p.communicate()
        if out.strip():
            print(f"--- {src}\n{out}", file=sys.stderr)
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    if force or procs or _stale(LIB, objs):
        tmp = LIB + ".tmp%d" % os.getpid()
        subprocess.check_call([_nvcc(), "-shared", "-o", tmp] + objs)
        os.replace(tmp, LIB)
    build_marshal(force)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
