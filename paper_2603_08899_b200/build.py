"""Build libconfu.so (the C-ABI CUDA library) in-tree for sm_100a with nvcc, and the native module its Python calls go
through (_calls*.so, g++)."""
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libconfu.so")
SOURCES = ["api.cu", "plan.cu", "attn_generic.cu", "attn_tc.cu", "attn_tc2.cu", "attn_narrow.cu", "attn_fp8.cu", "combine.cu", "accept.cu", "accept_walk.cu", "accept_static.cu", "compact.cu", "moe.cu", "selftest.cu"]
HEADERS = [os.path.join(CSRC, "common.cuh"), os.path.join(CSRC, "attn_tc.cuh"), os.path.join(CSRC, "tc_ptx.cuh"), os.path.join(CSRC, "tc_walk.cuh"), os.path.join(CSRC, "accept.cuh"), os.path.join(CSRC, "walk.cuh"),
           os.path.join(ROOT, "include", "confu.h")]

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
              "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", CSRC]


CALLS_SRC = os.path.join(CSRC, "python_calls.cpp")
CALLS = os.path.join(HERE, "_calls" + sysconfig.get_config_var("EXT_SUFFIX"))


def build_calls(force: bool = False) -> str:
    """The native module behind binding.py; links to libconfu.so next to it and to torch's Python library."""
    header = os.path.join(ROOT, "include", "confu.h")
    if not force and os.path.exists(CALLS) and os.path.getmtime(CALLS) >= max(os.path.getmtime(p) for p in (CALLS_SRC, header)):
        return CALLS
    import torch
    from torch.utils import cpp_extension
    nvcc = _nvcc()
    cuda = os.path.dirname(os.path.dirname(nvcc)) if os.path.isabs(nvcc) else "/usr/local/cuda"
    inc = cpp_extension.include_paths() + [sysconfig.get_paths()["include"], os.path.join(cuda, "include"), os.path.join(ROOT, "include")]
    lib = os.path.join(os.path.dirname(torch.__file__), "lib")
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-w", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"]
    cmd += [f"-I{d}" for d in inc] + [CALLS_SRC, "-o", CALLS, f"-L{HERE}", "-lconfu", "-Wl,-rpath,$ORIGIN", f"-L{lib}",
                                      "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
    subprocess.run(cmd, check=True)
    return CALLS


def _nvcc():
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def build(force: bool = False, verbose: bool = False) -> str:
    srcs = [os.path.join(CSRC, s) for s in SOURCES]
    if not force and os.path.exists(LIB):
        newest = max(os.path.getmtime(p) for p in srcs + HEADERS)
        if os.path.getmtime(LIB) >= newest:
            build_calls()
            return LIB
    objdir = os.path.join(HERE, "_build")
    os.makedirs(objdir, exist_ok=True)
    objs = []
    procs = []
    for s in srcs:
        o = os.path.join(objdir, os.path.basename(s) + ".o")
        objs.append(o)
        cmd = [_nvcc()] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-c", s, "-o", o]
        procs.append((cmd, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    for cmd, p in procs:
        out, _ = p.communicate()
        if verbose or p.returncode:
            sys.stderr.write(out)
        if p.returncode:
            raise RuntimeError("nvcc failed: " + " ".join(cmd))
    link = [_nvcc(), "-shared", "-o", LIB] + objs + ["-gencode", "arch=compute_100a,code=sm_100a", "-cudart", "static"]
    subprocess.run(link, check=True)
    build_calls(force)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
