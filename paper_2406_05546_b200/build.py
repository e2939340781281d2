"""Compile the CUDA library in-tree: paper_2406_05546_b200/libps_b200.so (sm_100a only), and the binding's argument
marshalling, _marshal, an extension of the running Python (with its headers and the C compiler that nvcc calls as well)."""
import glob
import os
import subprocess
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libps_b200.so")
MARSHAL = os.path.join(HERE, "_marshal" + sysconfig.get_config_var("EXT_SUFFIX"))      # the suffix names the Python it was built for
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale():
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not _stale():
        return LIB
    cmd = [NVCC, "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
           "-Xcompiler", "-fPIC", "-shared",
           "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-o", LIB] + sources()
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
    subprocess.run(cmd, check=True)
    return LIB


def build_marshal(force: bool = False) -> str:
    src, header = os.path.join(CSRC, "marshal.c"), os.path.join(ROOT, "include", "ps.h")
    if force or not os.path.exists(MARSHAL) or any(os.path.getmtime(d) > os.path.getmtime(MARSHAL) for d in (src, header)):
        subprocess.run([os.environ.get("CC", "gcc"), "-O2", "-shared", "-fPIC", "-I", sysconfig.get_paths()["include"], "-I", os.path.join(ROOT, "include"),
                        "-o", MARSHAL, src], check=True)
    return MARSHAL


if __name__ == "__main__":
    import sys
    print(build(force=True, verbose="-v" in sys.argv), build_marshal(force=True))
