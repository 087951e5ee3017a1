"""The bit-sliced scattering expressions of the CUDA path, compiled for the
host, against the oracle's 256-entry tables: every node byte x both
chiralities (no GPU needed)."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def host_scatter(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = tmp_path_factory.mktemp("hs") / "libhost_scatter.so"
    subprocess.run([nvcc, "-shared", "-Xcompiler", "-fPIC", "-std=c++17", "-o", str(out),
                    os.path.join(HERE, "csrc", "host_scatter.cu")], check=True)
    lib = ctypes.CDLL(str(out))
    lib.host_scatter_words.argtypes = [ctypes.c_void_p, ctypes.c_uint32, ctypes.c_uint32, ctypes.c_uint32,
                                       ctypes.c_void_p]
    lib.host_scatter_words.restype = None
    lib.host_scatter_saturated_words.argtypes = [ctypes.c_void_p, ctypes.c_uint32, ctypes.c_uint32, ctypes.c_void_p]
    lib.host_scatter_saturated_words.restype = None
    return lib


@pytest.mark.parametrize("rules,mask", [(2, 0xFFFFFFFF), (1, 0), (3, None)])
def test_bitsliced_scatter_equals_table(host_scatter, oracle_mod, rules, mask):
    tables = [oracle_mod.table(0, rules=rules), oracle_mod.table(1, rules=rules)]
    states = np.arange(256, dtype=np.uint32)
    # 8 words x 32 nodes cover all 256 bytes; a chirality pattern per run
    for chi_pattern in (0x00000000, 0xFFFFFFFF, 0xA5A5A5A5, 0x0F0F33CC):
        for wi in range(8):
            nodes = states[32 * wi:32 * wi + 32]
            planes = np.array([int(((nodes >> k) & 1) @ (1 << np.arange(32, dtype=np.uint64)))
                               for k in range(7)], dtype=np.uint32)
            solid = np.uint32(int(((nodes >> 7) & 1) @ (1 << np.arange(32, dtype=np.uint64))))
            out = np.zeros(7, dtype=np.uint32)
            if rules == 3:
                host_scatter.host_scatter_saturated_words(planes.ctypes.data, int(solid), chi_pattern, out.ctypes.data)
            else:
                host_scatter.host_scatter_words(planes.ctypes.data, int(solid), chi_pattern, mask, out.ctypes.data)
            for j in range(32):
                b = int(nodes[j])
                chi = (chi_pattern >> j) & 1
                got = sum(((int(out[k]) >> j) & 1) << k for k in range(7)) | (b & 0x80)
                assert got == int(tables[chi][b]), (b, chi)


@pytest.mark.parametrize("rules", [1, 2, 3])
def test_fluid_networks_equal_table(tmp_path, oracle_mod, rules):
    """The networks of words without solid nodes: all 128 fluid states x both
    chiralities."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = tmp_path / "libhost_fluid_scatter.so"
    subprocess.run([nvcc, "-shared", "-Xcompiler", "-fPIC", "-std=c++17", "-o", str(out),
                    os.path.join(HERE, "csrc", "host_fluid_scatter.cu")], check=True)
    lib = ctypes.CDLL(str(out))
    lib.host_fluid_scatter_words.argtypes = [ctypes.c_int, ctypes.c_void_p, ctypes.c_uint32, ctypes.c_void_p]
    lib.host_fluid_scatter_words.restype = None
    tables = [oracle_mod.table(0, rules=rules), oracle_mod.table(1, rules=rules)]
    for first in range(0, 128, 32):
        nodes = np.arange(first, first + 32, dtype=np.uint32)
        planes = np.array([int(((nodes >> k) & 1) @ (1 << np.arange(32, dtype=np.uint64))) for k in range(7)],
                          dtype=np.uint32)
        for chi_pattern in (0x00000000, 0xFFFFFFFF, 0xA5A5A5A5):
            got = np.zeros(7, dtype=np.uint32)
            lib.host_fluid_scatter_words(rules, planes.ctypes.data, chi_pattern, got.ctypes.data)
            for j, node in enumerate(nodes):
                byte = sum(((int(got[k]) >> j) & 1) << k for k in range(7))
                assert byte == int(tables[(chi_pattern >> j) & 1][node]), (int(node), (chi_pattern >> j) & 1)
