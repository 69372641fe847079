"""Builds libwpp.so in-tree with nvcc for sm_100a (cross-compiles without a GPU)."""
import os
import shlex
import shutil
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libwpp.so")
SOURCES = ["wpp_plan.cpp", "wpp_waves.cpp", "wpp_hints.cu", "wpp_api.cu", "wpp_append_combine.cu", "wpp_attention.cu", "wpp_attention_small.cu",
           "wpp_kda.cu", "wpp_kda_tc.cu", "wpp_kda_group.cu"]
CALL_SOURCE = os.path.join(CSRC, "wpp_call.c")          # Python module that marshals the calls of every layer
CALL = os.path.join(HERE, "_wpp_call" + sysconfig.get_config_var("EXT_SUFFIX"))
HEADERS = ["wpp_host.h", "wpp_plan_format.h", "wpp_device.h", "wpp_ptx.cuh", "wpp_kda_blocks.cuh", os.path.join("..", "..", "include", "wpp.h")]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", shutil.which("nvcc")):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def _cc() -> list:
    """The C compiler's command: CC (with its options), else gcc or cc."""
    for cand in (shlex.split(os.environ.get("CC", "")), ["gcc"], ["cc"]):
        if cand and shutil.which(cand[0]):
            return cand
    raise RuntimeError("no C compiler found (CC, gcc, cc)")


def is_stale() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(CALL):
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(CALL))
    deps = [os.path.join(CSRC, s) for s in SOURCES + HEADERS] + [CALL_SOURCE]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False, defines=(), out: str = None) -> str:
    """Compile the library; `defines` (a list of NAME=VALUE strings) and `out` build a variant beside it."""
    if out is None and not force and not is_stale():
        return LIB
    if out is None:
        tmp = CALL + f".tmp{os.getpid()}"
        subprocess.check_call(_cc() + ["-O2", "-Wall", "-Wextra", "-shared", "-fPIC", "-fvisibility=hidden",
                               "-I", sysconfig.get_paths()["include"], CALL_SOURCE, "-o", tmp])
        os.replace(tmp, CALL)
    target = out or LIB
    tmp = target + f".tmp{os.getpid()}"
    cmd = [_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo",
           "-shared", "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=default", "-cudart", "static",
           "-x", "cu"]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += [f"-D{d}" for d in defines]
    cmd += [os.path.join(CSRC, s) for s in SOURCES] + ["-o", tmp]
    subprocess.check_call(cmd)
    os.replace(tmp, target)
    return target


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
