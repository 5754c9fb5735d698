"""Host-side rules of the library (no GPU needed): inline functions of its
internal header, called through a small C++ shared object."""

import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = os.path.join(ROOT, "paper_2608_29748_gb300", "csrc", "internal.h")

SOURCE = """
#include "%s"
extern "C" int path(long long B, long long K, long long d, int direct, int gate_dense_e, int pairs) {
  return retrace::cond_path(B, K, d, direct != 0, gate_dense_e != 0, pairs);
}
extern "C" long long split_bytes(long long B, long long K, long long d) {
  return (long long)retrace::pair_split_bytes(B, K, d, 2);
}
"""
SWAP, ONE_SM, PAIR = 0, 1, 2


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(nvcc)))
    where = tmp_path_factory.mktemp("rules")
    src, so = str(where / "rules.cpp"), str(where / "rules.so")
    with open(src, "w") as f:
        f.write(SOURCE % HEADER)
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(cuda, "include"), "-o", so, src], check=True)
    lib = ctypes.CDLL(so)
    lib.path.argtypes = [ctypes.c_longlong] * 3 + [ctypes.c_int] * 3
    lib.split_bytes.argtypes, lib.split_bytes.restype = [ctypes.c_longlong] * 3, ctypes.c_longlong
    return lib


def test_conditioning_path(rules):
    """Kernels by rows and features, and what a device without room for a pair
    of CTAs takes."""
    assert rules.path(64, 16, 4096, 0, 0, 76) == SWAP            # 960 rows x 4096 <= 2^22
    assert rules.path(69, 16, 4096, 0, 0, 76) == PAIR            # 1035 x 4096 > 2^22
    assert rules.path(274, 16, 256, 0, 0, 76) == PAIR            # 4110 rows > 4096
    assert rules.path(69, 16, 4096, 0, 1, 76) == ONE_SM
    assert rules.path(274, 16, 264, 0, 1, 76) == PAIR            # per-position e, d no multiple of 256
    assert rules.path(4, 16, 1 << 20, 1, 0, 76) == SWAP          # direct rows
    for d, dense, want in ((4096, 0, SWAP), (4104, 0, SWAP), (4104, 1, SWAP), (4096, 1, ONE_SM)):
        assert rules.path(256, 16, d, 0, dense, 0) == want       # no pair fits


def test_pair_kernel_has_its_split_partials(rules):
    """Every bf16 shape that runs on CTA pairs without column checks has the
    workspace of its split tiles: the line to the small-R kernels (rows times
    features) and the workspace's (rows and tiles) are stated apart."""
    pairs = 0
    for d in range(256, 20481, 256):
        # Rows around both lines: 2^22 / d, 4096, and whole tiles of 256.
        for line in {2**22 // d, 4096, *range(256, 4097, 256)}:
            for rows in range(max(line - 17, 1), line + 18):
                if rules.path(rows, 2, d, 0, 0, 76) == PAIR:
                    pairs += 1
                    assert rules.split_bytes(rows, 2, d) > 0, (rows, d)
    assert pairs > 10000
