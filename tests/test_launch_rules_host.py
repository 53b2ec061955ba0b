"""The rules that choose between launch forms, compiled for the host: clusters for the FP64 projected problems only
while every CTA of every running call has an SM, projected problems in launches of bounded size, FP32
sums of the adjoint over at most 128 pairs."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1603_06855_gb300", "csrc")
HARNESS = r"""
#include "launch_rules.h"
extern "C" int chunks(int pairs, int wave, int most) { return adj_chunks(pairs, wave, most); }
extern "C" int per_launch(long long nk, int sms) { return rr_problems_per_launch(nk, sms); }
extern "C" int clusters(int n, int m, long long nk, long long others, int sms) { return rr64_uses_clusters(n, m, nk, others, sms); }
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("rules")
    src, lib = d / "h.cpp", d / "libh.so"
    src.write_text(HARNESS)
    subprocess.run([cxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(lib)], check=True,
                   capture_output=True)
    so = ctypes.CDLL(str(lib))
    so.clusters.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_longlong, ctypes.c_longlong, ctypes.c_int]
    so.per_launch.argtypes = [ctypes.c_longlong, ctypes.c_int]
    return so


def test_clusters_alone_and_beside_others(rules):
    for sms in (148, 152):
        most = sms // 8
        assert rules.clusters(48, 16, most, 0, sms) and not rules.clusters(48, 16, most + 1, 0, sms)
        assert not rules.clusters(16, 16, 1, 0, sms)  # no products to share
        for others in (0, 4, most - 1, most, 60, 10**6):  # a batch's other designs
            assert rules.clusters(48, 16, 1, others, sms) == (others <= most - 1)


def test_projected_problems_per_launch(rules):
    for nk in (1, 152, 2431, 2432):
        assert rules.per_launch(nk, 152) == nk
    for nk in (2433, 65535):
        assert rules.per_launch(nk, 152) == 2432


def test_adjoint_sums(rules):
    most = 64
    for pairs in (1, 20, 128, 129, 720, 2000, 4096, 6000, 8192, 65535 * 24):
        for wave in range(1, min(32, pairs) + 1):
            chunks = rules.chunks(pairs, wave, most)
            assert wave <= chunks <= most and chunks % wave == 0
            if pairs <= 128 * most // 2:
                assert -(-pairs // chunks) <= 128
            assert -(-pairs // chunks) <= max(128, -(-pairs // (most // 2)))
