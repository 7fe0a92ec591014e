"""Compiles a piece of test CUDA around the library's device headers (nvcc, the library's flags for
its FP64 arithmetic) and loads it; and numpy arrays as arguments of its functions."""
import ctypes
import os
import subprocess

import numpy as np

from paper_2509_03313_gb300 import build

PRELUDE = """#include <cuda_runtime.h>
#include <vector>
// device copies of host arrays, freed with the object
struct Arrays {
  std::vector<void*> dev;
  cudaError_t err = cudaSuccess;
  template <class T> T* in(const T* h, long n) { T* p = out(h, n); if (!err) err = cudaMemcpy(p, h, n * sizeof(T), cudaMemcpyHostToDevice); return p; }
  template <class T> T* out(const T*, long n) { void* p = nullptr; if (!err) err = cudaMalloc(&p, n * sizeof(T)); dev.push_back(p); return static_cast<T*>(p); }
  template <class T> void back(T* h, const T* p, long n) { if (!err) err = cudaGetLastError(); if (!err) err = cudaMemcpy(h, p, n * sizeof(T), cudaMemcpyDeviceToHost); }
  ~Arrays() { for (void* p : dev) cudaFree(p); }
};
"""


def load(directory, source):
    cu, so = os.path.join(str(directory), "test.cu"), os.path.join(str(directory), "test.so")
    with open(cu, "w", encoding="utf-8") as f:
        f.write(PRELUDE + source)
    include = os.path.join(os.path.dirname(build.HERE), "include")
    r = subprocess.run([build.nvcc(), *build.ARCH, *build.COMMON, "--fmad=false", "-shared", "-I", build.CSRC, "-I", include,
                        cu, "-o", so], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(so)


def call(fn, *args):
    """Arrays by address, integers as long; the function returns a cudaError_t."""
    e = fn(*[a.ctypes.data_as(ctypes.c_void_p) if isinstance(a, np.ndarray) else ctypes.c_long(int(a)) for a in args])
    assert e == 0, f"CUDA error {e}"
