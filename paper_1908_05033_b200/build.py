"""Compile the CUDA sources into paper_1908_05033_b200/libdsq_b200.so for
sm_100a with nvcc (cross-compiles without a GPU), and the native side of the
Python binding into paper_1908_05033_b200/_dsq_host.so."""
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libdsq_b200.so")
HOST_LIB = os.path.join(HERE, "_dsq_host.so")
HOST_SOURCE = "dsq_host.cpp"
OBJ_DIR = os.path.join(HERE, "_build")
SOURCES = ["dsq_elementwise.cu", "dsq_dwconv.cu", "dsq_tc.cu", "dsq_conv3.cu", "dsq_pw.cu", "dsq_gemm8.cu",
           "dsq_wgemm_small.cu", "dsq_gemm_small.cu", "dsq_conv_small.cu",
           "dsq_soft.cu", "dsq_plan.cu", "dsq_workspace.cu"]
HEADERS = ["dsq_common.cuh", "dsq_conv_rule.h", "dsq_epilogue.cuh", "dsq_fragments.cuh", "dsq_gemm8_rule.h", "dsq_ptx.cuh", "dsq_tc_common.cuh",
           "dsq_tc_host.h", "dsq_hooks.h", "dsq_launch.h", "dsq_plan.h",
           os.path.join("..", "..", "include", "dsq.h")]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo",
              "-std=c++17", "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC",
              "-Xcompiler", "-fvisibility=default", "--fmad=false"]


def _stale(lib, files) -> bool:
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    return any(os.path.getmtime(os.path.join(CSRC, f)) > t for f in files)


def _build_cuda(verbose: bool) -> None:
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    os.makedirs(OBJ_DIR, exist_ok=True)
    objects = [os.path.join(OBJ_DIR, f + ".o") for f in SOURCES]
    flags = NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else [])
    jobs = [subprocess.Popen([nvcc] + flags + ["-c", os.path.join(CSRC, f), "-o", o])
            for f, o in zip(SOURCES, objects) if verbose or _stale(o, [f] + HEADERS)]
    if any([j.wait() for j in jobs]):
        raise subprocess.CalledProcessError(1, "nvcc")
    subprocess.run([nvcc] + NVCC_FLAGS + ["-shared", "-o", LIB] + objects, check=True)


def _build_host() -> None:
    import torch
    root = os.path.dirname(os.path.abspath(torch.__file__))
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared",
           "-fvisibility=hidden", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           "-I", os.path.join(root, "include"),
           "-I", os.path.join(root, "include", "torch", "csrc", "api", "include"),
           "-I", sysconfig.get_paths()["include"], "-I", os.path.join(cuda, "include"),
           os.path.join(CSRC, HOST_SOURCE), "-o", HOST_LIB,
           "-L", os.path.join(root, "lib"), "-ltorch_python", "-ltorch_cpu", "-ltorch", "-lc10",
           "-lc10_cuda", "-L", HERE, "-l:" + os.path.basename(LIB), "-Wl,-rpath,$ORIGIN"]
    subprocess.run(cmd, check=True, cwd=HERE)


def build(force: bool = False, verbose: bool = False) -> str:
    if force and os.path.isdir(OBJ_DIR):
        for f in os.listdir(OBJ_DIR):
            os.unlink(os.path.join(OBJ_DIR, f))
    if force or _stale(LIB, SOURCES + HEADERS):
        _build_cuda(verbose)
    if force or _stale(HOST_LIB, [HOST_SOURCE] + HEADERS):
        _build_host()
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
