"""The launch rules that live in the kernels' headers, called on the CPU: a
small library is compiled from the headers themselves."""
import ctypes
import os
import subprocess

import pytest

from paper_2609_11923_gb300 import build

SOURCE = r"""
#include "batch.cuh"
extern "C" unsigned resident_size(long long nodes, unsigned T) {
  // the near-root part of a chance root over `nodes` terminals and one set
  cfr::InstDesc in = {};
  in.n_nodes = (int)nodes;
  in.n_int = 1;
  in.n_sets = 1;
  in.n_slots = 2;
  in.n_dec = 1;
  in.n_chance = 1;
  return cfr::resident_size(in, T);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    src, so = str(d / "rules.cu"), str(d / "rules.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.check_call([build.NVCC] + build.ARCH + ["-O0", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-I", build.CSRC,
                                                       src, "-o", so])
    return ctypes.CDLL(so)


@pytest.mark.parametrize("T", [4, 8])
@pytest.mark.parametrize("nodes", [1 << 28, (1 << 29) + 3, (1 << 30) + 64, (1 << 31) - 3])
def test_no_width_of_a_chance_root_wraps_the_resident_bytes(lib, nodes, T):
    lib.resident_size.argtypes = [ctypes.c_longlong, ctypes.c_uint]
    lib.resident_size.restype = ctypes.c_uint
    assert lib.resident_size(nodes, T) == 0
    # just below what shared memory holds, and just above
    fits = (190 * 1024 - 512) // T
    assert nodes * T > lib.resident_size(fits, T) >= fits * T
    assert lib.resident_size(190 * 1024 // T, T) == 0
