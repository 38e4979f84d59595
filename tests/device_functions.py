"""Builds tests/device_functions.cu (single device functions of the library as
C entry points) into a folder and loads it."""
import ctypes
import os
import subprocess

from paper_2101_06769_gb300 import build as B

SOURCE = os.path.join(os.path.dirname(os.path.abspath(__file__)), "device_functions.cu")


def load(folder):
    so = os.path.join(str(folder), "device_functions.so")
    subprocess.run([B._nvcc()] + B.ARCH + B.FLAGS + ["-Xcompiler", "-fvisibility=default", "-I", B.CSRC, "-shared",
                                                    SOURCE, "-o", so], check=True)
    return ctypes.CDLL(so)
