"""Builds libssd.so (the C-ABI CUDA library) for sm_100a with nvcc, and _ssd_call.so (the
marshalling of torch tensors for its hot calls) with the host compiler, both in-tree."""
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libssd.so")
CALL = os.path.join(HERE, "_ssd_call.so")
HEADER = os.path.join(os.path.dirname(HERE), "include", "ssd.h")
SOURCES = ["ssd_api.cu", "ssd_ctc.cu", "ssd_verify.cu", "ssd_verify_static.cu", "ssd_decide.cu", "ssd_verify_ee.cu",
           "ssd_readspan.cu"]
CALL_SOURCE = os.path.join(CSRC, "ssd_call.cpp")
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "--use_fast_math=false", "-Xcompiler", "-fPIC", "-shared", "-cudart", "shared"]


def built_for() -> str:
    """What _ssd_call.so has to have been built with to be usable here: it sees torch's C++ types."""
    import torch
    return "torch %s, %s" % (torch.__version__, sysconfig.get_config_var("SOABI"))


def _other_torch() -> bool:
    with open(CALL, "rb") as f:
        return b"_ssd_call for " + built_for().encode() + b"\0" not in f.read()


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def _run(cmd, target: str, tmp: str, verbose: bool) -> None:
    r = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or r.returncode != 0:
        sys.stderr.write(r.stdout + r.stderr)
    if r.returncode != 0:
        raise RuntimeError("building %s failed" % os.path.basename(target))
    os.replace(tmp, target)


def build(force: bool = False, verbose: bool = False) -> str:
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if not f.endswith(".cpp")] + [HEADER]
    if force or _stale(LIB, deps):
        nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
        tmp = LIB + ".tmp.%d" % os.getpid()
        flags = [f for f in NVCC_FLAGS if not f.startswith("--use_fast_math")]
        _run([nvcc] + flags + (["-Xptxas", "-v"] if verbose else []) +
             [os.path.join(CSRC, s) for s in SOURCES] + ["-Xlinker", "-soname=libssd.so", "-o", tmp],
             LIB, tmp, verbose)
    if force or _stale(CALL, [CALL_SOURCE, HEADER]) or _other_torch():
        import torch
        root = os.path.dirname(torch.__file__)
        cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
        inc = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
               os.path.join(cuda, "include"), sysconfig.get_paths()["include"]]
        tmp = CALL + ".tmp.%d" % os.getpid()
        _run([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
              "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI),
              '-DSSD_BUILT_FOR="%s"' % built_for()] +
             [f for d in inc for f in ("-isystem", d)] + [CALL_SOURCE, "-o", tmp, "-L" + HERE, "-l:libssd.so",
              "-L" + os.path.join(root, "lib"), "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda",
              "-Wl,-rpath,$ORIGIN"], CALL, tmp, verbose)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
