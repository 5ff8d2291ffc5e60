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
// per instance: nodes, sets, depths, chain, resident, 0 FP32, 1 FP64, 2 a best response
extern "C" void plan(int n, const long long *load, int least, int sms, int four, int eight, int sixteen, int *out) {
  std::vector<cfr::BatchLoad> l(n);
  for (int i = 0; i < n; ++i) {
    const long long *x = load + 6 * i;
    l[i] = cfr::BatchLoad{x[0], x[1], x[2], x[3], x[4] != 0, x[5] != 0, x[5] == 2, 1.0};
  }
  cfr::ClusterRoom r;
  r.sms = sms;
  r.four = four;
  r.eight = eight;
  r.sixteen = sixteen;
  const std::vector<int> c = cfr::plan_clusters(l, least, r);
  for (int i = 0; i < n; ++i) out[i] = c[i];
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


ROOM = (152, 34, 16, 7)  # SMs, and clusters of 4, 8 and 16 CTAs that run at once


def ctas(lib, loads, least=1, room=ROOM):
    flat = [x for load in loads for x in load]
    out = (ctypes.c_int * len(loads))()
    lib.plan(len(loads), (ctypes.c_longlong * len(flat))(*flat), least, *room, out)
    return list(out)


def test_depths_are_paid_for_in_every_ctas_barriers(lib):
    # 300 chains of 100 depths side by side: one CTA 696 us an iteration, 16 of them 881
    assert ctas(lib, [(60301, 100, 101, 30000, 0, 0)]) == [1]
    assert ctas(lib, [(81, 40, 40, 40, 1, 0)]) == ctas(lib, [(201, 100, 100, 100, 1, 1)]) == [1]
    # a large endgame and a random tree: 16 CTAs (64 us, by two 375; 90, by one 742)
    assert ctas(lib, [(920440, 4380, 5, 532, 0, 0)]) == ctas(lib, [(275507, 33629, 11, 140, 0, 0)]) == [16]
    # FP64 is worth a cluster far earlier (10,000 nodes: 142 us, by 16 CTAs 50)
    assert ctas(lib, [(10241, 1334, 8, 90, 1, 1)])[0] >= 8 and ctas(lib, [(10414, 400, 5, 41, 1, 0)]) == [1]
    # a cluster of two loses more to its barriers than it shares, one of 16 gains (23 us, 26, 18)
    assert ctas(lib, [(21178, 620, 5, 60, 0, 0)]) == [16]
    # long sets are walked by a group each wherever its CTA is
    assert ctas(lib, [(13801, 6, 3, 600, 0, 1)]) == [1]


@pytest.mark.parametrize("room,most", [((152, 34, 16, 0), 8), ((152, 34, 0, 0), 4), ((152, 0, 0, 0), 2)])
@pytest.mark.parametrize("n", [1, 40, 500])
def test_no_cluster_that_the_device_cannot_hold(lib, n, room, most):
    loads = [(920440, 4380, 5, 532, 0, 0)] + [(200000, 3520, 5, 532, 0, 0)] * (n - 1)
    got = max(ctas(lib, loads, room=room))
    assert got == most if n < 500 else got <= most  # 500 alike fill the GPU as they are


def test_the_least_ctas_are_everyones(lib):
    assert min(ctas(lib, [(300, 30, 5, 12, 1, 0), (920440, 4380, 5, 532, 0, 0)], least=4)) >= 4


def test_growth_that_does_not_bring_the_end_forward_is_taken_back(lib):
    alike = (10241, 1334, 8, 60, 0, 0)  # 40 random trees: 16 CTAs would be faster, and there is room for a few
    assert ctas(lib, [alike])[0] > 1 and ctas(lib, [alike] * 40) == [1] * 40
    # the largest still grows beside them
    assert ctas(lib, [(920440, 4380, 5, 532, 0, 0)] + [alike] * 40)[0] == 16


def test_best_responses_of_small_trees_stay_in_one_cta(lib):
    # by one CTA or 16 alike for 3,385 nodes alone (70 us), 1,810 and 222 us for 920,440
    assert ctas(lib, [(3385, 458, 7, 50, 0, 2)] * 16) == [1] * 16
    assert ctas(lib, [(920440, 4380, 5, 412, 0, 2)]) == [16]
