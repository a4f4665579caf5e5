"""The placement of a whole network in shared memory (csrc/net_plan.cpp), checked on the CPU: over depths, pruning ratios and every way
of giving images to CTAs, nothing that is still read is written over - also where one of a CTA's two images is ahead of the other."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CHOICES = [(1, 4, 8), (1, 2, 8), (1, 1, 16), (2, 1, 8)]          # images per CTA, CTAs per image, warps per image


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("net_plan") / "check.so")
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    include = os.path.join(os.path.dirname(os.path.dirname(nvcc)), "include")
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", include, "-o", so, os.path.join(ROOT, "tests", "net_plan_check.cpp"),
                           os.path.join(ROOT, "paper_2010_16165_b200", "csrc", "net_plan.cpp")])
    lib = ctypes.CDLL(so)

    def run(hw, widths, per_stage, ratios, choice, meet_off=0):
        keep, conv = [widths[0]], 1
        for K in widths:
            for _ in range(per_stage):
                keep += [K - int(np.floor(ratios[conv] * K + 1e-9)), K]
                conv += 2
        msg = ctypes.create_string_buffer(256)
        rc = lib.check_net_plan(hw, len(widths), (ctypes.c_int * len(widths))(*widths), per_stage, (ctypes.c_int * len(keep))(*keep), *choice, meet_off, msg)
        return rc, msg.value.decode()
    return run


@pytest.mark.parametrize("choice", CHOICES)
@pytest.mark.parametrize("per_stage", [1, 2, 3, 5, 9, 18])
def test_nothing_is_overwritten(check, per_stage, choice):
    rng = np.random.default_rng(per_stage)
    n = 6 * per_stage + 2
    ratios = [np.full(n, p / 100) for p in range(0, 62, 3 if per_stage < 9 else 6)]
    ratios += [rng.uniform(lo, 0.6, n) for lo in (0.0, 0.2, 0.4) for _ in range(4)]
    for r in ratios:
        rc, msg = check(32, (16, 32, 64), per_stage, r, choice)
        assert rc == 0, (r[:3], msg)                            # every one of these networks fits


@pytest.mark.parametrize("choice", CHOICES)
@pytest.mark.parametrize("hw, widths", [(32, (8, 8, 8)), (32, (9, 17, 33)), (32, (7, 24, 40)), (32, (16, 48, 56)), (32, (24, 40, 64)), (16, (24, 64)),
                                        (16, (33, 50)), (8, (64,)), (8, (12,))])
def test_other_widths(check, hw, widths, choice):
    for per_stage in (1, 2, 4):
        for p in (0.0, 0.25, 0.5):
            rc, msg = check(hw, widths, per_stage, np.full(6 * per_stage + 2, p), choice)
            assert rc >= 0, (per_stage, p, msg)


def test_the_check_sees_an_image_that_clears_what_the_other_still_reads(check):
    """ResNet-32 at 0.2: without waiting for the second image, the first one clears filters that the second has still to read."""
    rc, msg = check(32, (16, 32, 64), 5, np.full(32, 0.2), (2, 1, 8), meet_off=1)
    assert rc == -1 and "filters overwritten" in msg
