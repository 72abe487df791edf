"""Runs a script with a cudaMalloc that fails for chosen sizes: `deny(lo, hi)` in
the script makes every request of lo..hi bytes return out of memory, on the host,
with the GPU's memory as it is (a preloaded stand-in that forwards all others)."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <dlfcn.h>
#include <stddef.h>
static size_t lo = 1, hi = 0;
void deny(size_t a, size_t b) { lo = a; hi = b; }
int cudaMalloc(void** p, size_t n) {
  static int (*real)(void**, size_t);
  if (!real) real = (int (*)(void**, size_t))dlsym(dlopen("libcudart.so.13", RTLD_LAZY), "cudaMalloc");
  if (n >= lo && n <= hi) return 2; /* cudaErrorMemoryAllocation */
  return real(p, n);
}
"""

PRELUDE = """
import ctypes, os
import numpy as np
import torch
from paper_1606_03416_gb300 import dgchefsi as D
from paper_1606_03416_gb300 import inputs as G
_fake = ctypes.CDLL(os.environ["LD_PRELOAD"])
_fake.deny.argtypes = [ctypes.c_size_t, ctypes.c_size_t]
deny = _fake.deny
"""


def run(tmp_path, script):
    src, lib = tmp_path / "fake.c", tmp_path / "libfake.so"
    src.write_text(SOURCE)
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", str(lib), str(src), "-ldl"], check=True)
    r = subprocess.run([sys.executable, "-c", PRELUDE + script], cwd=ROOT, capture_output=True, text=True, timeout=300,
                       env={**os.environ, "LD_PRELOAD": str(lib)})
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    return r.stdout
