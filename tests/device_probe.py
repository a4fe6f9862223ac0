"""Builds device_probe.cu (device functions of the library as kernels of their own) and loads it."""
import ctypes
import functools
import os
import subprocess

from paper_1605_01715_gb300 import build as kb, capi

HERE = os.path.dirname(os.path.abspath(__file__))


@functools.lru_cache(maxsize=1)
def lib():
    capi.lib()
    os.makedirs(kb.BUILD, exist_ok=True)
    src = os.path.join(HERE, "device_probe.cu")
    out = os.path.join(kb.BUILD, "device_probe.%d.so" % os.getpid())
    subprocess.run([kb.NVCC, "-shared", *kb.FLAGS, "-o", out, src, kb.LIB, "-Xlinker", "-rpath," + os.path.dirname(kb.LIB)],
                   check=True)
    loaded = ctypes.CDLL(out)
    os.remove(out)
    return loaded
