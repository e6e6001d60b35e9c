"""In-tree build of libhmar.so (nvcc, sm_100a only) and of the compiled half of the Python binding (g++, against torch)."""
import os
import shutil
import subprocess
import sys
import sysconfig

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG_DIR, "csrc")
LIB_PATH = os.environ.get("HMAR_LIBRARY") or os.path.join(PKG_DIR, "libhmar.so")
CHECKED_LIB_PATH = os.path.join(PKG_DIR, "libhmar_check.so")     # the same sources with -DHMAR_BOUNDS_CHECK (tests)
SOURCES = ["api.cu", "schedule.cpp", "simt_kernels.cu", "tc_dispatch.cu", "fwd_sm100.cu", "bwd_sm100.cu", "noalloc_bwd.cu", "step_small.cu", "recon.cu"]

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC", "-Xcompiler", "-Wall", "-shared",
]


def _nvcc():
    path = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(path):
        raise RuntimeError("nvcc not found; the HMAR CUDA library cannot be built")
    return path


def needs_build(path=None):
    path = path or LIB_PATH
    if not os.path.exists(path):
        return True
    lib_time = os.path.getmtime(path)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    deps.append(os.path.join(PKG_DIR, "..", "include", "hmar.h"))
    return any(os.path.getmtime(d) > lib_time for d in deps)


def build(force=False, verbose=False, checked=False):
    """Compile every CUDA source of the library into paper_2506_04421_b200/libhmar.so, or, with `checked`, into
    libhmar_check.so: the build whose kernels compare every address they form with its tensor's extent."""
    target = CHECKED_LIB_PATH if checked else os.path.join(PKG_DIR, "libhmar.so")
    if not force and not needs_build(target):
        return target
    cmd = [_nvcc()] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + (["-DHMAR_BOUNDS_CHECK"] if checked else [])
    cmd += [os.path.join(CSRC, s) for s in SOURCES] + ["-o", target]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
        raise RuntimeError("nvcc failed building libhmar.so")
    if verbose:
        sys.stderr.write(res.stdout + res.stderr)
    if not checked:
        build_host(force)
    return target


def host_path():
    """The binding's compiled module; its name holds what it was compiled against."""
    import torch
    return os.path.join(PKG_DIR, "_hmar_host-%s-%s.so" % (sysconfig.get_config_var("SOABI"), torch.__version__))


def build_host(force=False):
    """Compile csrc/host_binding.cpp unless it is up to date; returns the module's path."""
    target = host_path()
    deps = [os.path.join(CSRC, "host_binding.cpp"), os.path.join(PKG_DIR, "..", "include", "hmar.h")]
    if not force and os.path.exists(target) and all(os.path.getmtime(d) <= os.path.getmtime(target) for d in deps):
        return target
    import torch
    root = os.path.dirname(os.path.abspath(torch.__file__))
    cuda = os.path.dirname(os.path.dirname(_nvcc()))
    partial = "%s.%d" % (target, os.getpid())              # another process may be loading or building the same file
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-Wall", "-D_GLIBCXX_USE_CXX11_ABI=%d" % torch._C._GLIBCXX_USE_CXX11_ABI]
    cmd += ["-I" + d for d in (os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
                               sysconfig.get_paths()["include"], os.path.join(cuda, "include"))]
    cmd += [deps[0], "-L" + os.path.join(root, "lib"), "-ltorch_python", "-lc10_cuda", "-ltorch", "-ltorch_cpu", "-lc10", "-o", partial]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
        raise RuntimeError("g++ failed building the binding's compiled module")
    os.replace(partial, target)
    return target


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
