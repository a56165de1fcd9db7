"""Builds C++ source over the device headers for the host (device_on_host.h) and loads it."""
import ctypes
import os
import pathlib
import subprocess

HERE = pathlib.Path(__file__).resolve().parent
CSRC = HERE.parent / "paper_2107_12027_gb300" / "csrc"
CUDA = pathlib.Path(os.environ.get("CUDA_HOME", "/usr/local/cuda"))


def load(src, tmp, name="h"):
    cpp, so = pathlib.Path(tmp) / (name + ".cpp"), pathlib.Path(tmp) / (name + ".so")
    cpp.write_text('#include "device_on_host.h"\n' + src)
    # (frames of 8 x 8 arrays: -O1 keeps the build to seconds)
    subprocess.run(["g++", "-O1", "-std=c++17", "-fpermissive", "-w", "-ffp-contract=off", "-shared", "-fPIC", "-I", str(HERE),
                    "-I", str(CSRC), "-I", str(HERE.parent / "include"), "-I", str(CUDA / "include"), "-o", str(so),
                    str(cpp)], check=True)
    return ctypes.CDLL(str(so))
