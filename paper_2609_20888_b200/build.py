"""Build the C-ABI library `libeta_b200.so` in-tree with nvcc for sm_100a."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import tempfile
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libeta_b200.so")
HEADER = os.path.join(os.path.dirname(HERE), "include", "eta.h")


# Copies of the library for tests.  Two in which a consumer warp, of the streaming kernel or of the one-kernel step, skips a
# barrier arrival and the bounded waits are short (2^16 polls, a few milliseconds), so that a give-up path runs and can be checked.
GIVEUP_LIB = os.path.join(HERE, "libeta_b200_test_giveup.so")
GIVEUP_FLAGS = ["-DETA_TEST_SKIP_FLUSH_ARRIVE", "-DETA_TEST_GENERAL_PATH", "-DETA_WAIT_LIMIT=65536"]
GIVEUP_STEP_LIB = os.path.join(HERE, "libeta_b200_test_giveup_step.so")
GIVEUP_STEP_FLAGS = ["-DETA_TEST_SKIP_STAGE_ARRIVE", "-DETA_WAIT_LIMIT=65536"]
# And one that takes the general path whatever the size: small problems reach its edges too.
GENERAL_LIB = os.path.join(HERE, "libeta_b200_test_general.so")
GENERAL_FLAGS = ["-DETA_TEST_GENERAL_PATH"]


def sources() -> list[str]:
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def needs_build(lib: str = LIB) -> bool:
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + [HEADER]
    return any(os.path.getmtime(p) > t for p in deps)


def build(force: bool = False, verbose: bool = False, lib: str = LIB, extra_flags: tuple = ()) -> str:
    if lib == LIB:
        build_torch_module(force)
    if not force and not needs_build(lib):
        return lib
    cmd = [os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), *os.environ.get("ETA_NVCC_FLAGS", "").split(),
           "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "-Xcompiler", "-fPIC"]
    cmd += (["-Xptxas", "-v"] if verbose else []) + list(extra_flags)
    # a compiler per source file, side by side: two files with instances by the dozen take most of the time
    with tempfile.TemporaryDirectory() as tmp, ThreadPoolExecutor(os.cpu_count() or 1) as pool:
        objects = [os.path.join(tmp, os.path.basename(src) + ".o") for src in sources()]
        list(pool.map(lambda so: subprocess.run([*cmd, "-c", so[0], "-o", so[1]], check=True), zip(sources(), objects)))
        subprocess.run([*cmd, "-shared", "-o", lib, *objects], check=True)
    return lib


# The marshalling of a decode step's calls for torch: a Python module of its own, compiled by the host compiler.
TORCH_MODULE = os.path.join(HERE, "_eta_torch.so")
TORCH_SOURCE = os.path.join(CSRC, "eta_torch.cpp")


# It is linked against torch's C++ interface and the interpreter's: beside it stands what it was built for.
TORCH_STAMP = os.path.join(HERE, "_eta_torch.built_for")


def torch_stamp() -> str:
    import sysconfig

    import torch
    return f"torch {torch.__version__} {sysconfig.get_config_var('SOABI')}"


def torch_module_is_current() -> bool:
    deps = [TORCH_SOURCE, HEADER]
    if not (os.path.exists(TORCH_MODULE) and os.path.exists(TORCH_STAMP)):
        return False
    if any(os.path.getmtime(p) > os.path.getmtime(TORCH_MODULE) for p in deps):
        return False
    with open(TORCH_STAMP) as f:
        return f.read() == torch_stamp()


def build_torch_module(force: bool = False) -> str:
    if not force and torch_module_is_current():
        return TORCH_MODULE
    import sysconfig

    import torch
    root = os.path.dirname(torch.__file__)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-o", TORCH_MODULE, TORCH_SOURCE,
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"]
    for inc in (os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
                os.path.join(cuda, "include"), sysconfig.get_paths()["include"]):
        cmd += ["-isystem", inc]
    cmd += ["-L" + os.path.join(root, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"]
    subprocess.run(cmd, check=True)
    with open(TORCH_STAMP, "w") as f:
        f.write(torch_stamp())
    return TORCH_MODULE


def build_giveup_variant(force: bool = False) -> str:
    return build(force=force, lib=GIVEUP_LIB, extra_flags=tuple(GIVEUP_FLAGS))


def build_giveup_step_variant(force: bool = False) -> str:
    return build(force=force, lib=GIVEUP_STEP_LIB, extra_flags=tuple(GIVEUP_STEP_FLAGS))


def build_general_variant(force: bool = False) -> str:
    return build(force=force, lib=GENERAL_LIB, extra_flags=tuple(GENERAL_FLAGS))


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
