"""The shared memory of the 2 x 2 form of a run of layers (csrc/chain_quad_layout.h), checked on the CPU: for every height that form takes and every
number of images a group may have, no operand lies outside what the launch asks for."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("chain_quad") / "check.so")
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    include = os.path.join(os.path.dirname(os.path.dirname(nvcc)), "include")
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", include, "-o", so, os.path.join(ROOT, "tests", "chain_quad_layout_check.cpp")])
    lib = ctypes.CDLL(so)

    def run(G, H, W):
        tiles, smem, msg = ctypes.c_int(), ctypes.c_uint(), ctypes.create_string_buffer(256)
        return lib.check_chain_quad(G, H, W, ctypes.byref(tiles), ctypes.byref(smem), msg), tiles.value, smem.value, msg.value.decode()
    return run


@pytest.mark.parametrize("H", range(2, 66, 2))                  # 64: the most a run of layers takes
def test_operands_lie_in_shared_memory(check, H):
    for G in range(1, 100):
        rc, tiles, smem, msg = check(G, H, 32)
        assert rc >= 0, (G, msg)
        if rc == 1:
            break
    assert G > 1, "one image fits"                              # (then a run of such images is planned)
