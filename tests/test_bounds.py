"""The lower bounds that end a round's merges (merged_bound), against the cells that
the update formula makes: the kernel's own source, compiled for the host.

A bound above a cell would let a merge go ahead of a smaller cell; the margins
are there for the formula's roundings.  The planted mistake, a bound without its
margin, has to show on the same operands.
"""
import ctypes
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
COUNT = 1_000_000


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    gxx = shutil.which("g++")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if gxx is None or not os.path.exists(os.path.join(include, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    so = str(tmp_path_factory.mktemp("bounds") / "bounds.so")
    subprocess.run([gxx, "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-isystem", include,
                    os.path.join(HERE, "bounds_probe.cpp"), "-o", so], check=True)
    lib = ctypes.CDLL(so)
    lib.bounds_check.argtypes = [ctypes.c_int, ctypes.c_ulonglong, ctypes.c_longlong,
                                 ctypes.POINTER(ctypes.c_longlong)]
    lib.bounds_check.restype = None
    lib.bound_of.argtypes = [ctypes.c_int] + [ctypes.c_float] * 6
    lib.bound_of.restype = ctypes.c_uint
    return lib


@pytest.mark.parametrize("link", range(6))
def test_no_cell_lies_below_its_bound(probe, link):
    out = (ctypes.c_longlong * 4)()
    probe.bounds_check(link, 11 + link, COUNT, out)
    below, margin_needed, useless, no_cells = out
    assert below == 0
    assert margin_needed > 0  # a bound without its margin is caught on these operands
    assert useless == 0  # (and a bound of zero everywhere would be)
    assert no_cells == 0


@pytest.mark.parametrize("link", range(6))
@pytest.mark.parametrize("value", [0.0, 1e-40, 1e-33, 3.4e38, float("inf"), float("nan")])
def test_values_without_a_margin_give_no_bound(probe, link, value):
    """Too small for a relative margin, or not finite: bound 0 (single linkage's
    margin is one of the largest value: above a small one the bound is 0 too)."""
    assert probe.bound_of(link, value, value, 3.0, 8.0, 0.0, value) == 0
    # a part of NaN cells makes NaN cells, above every number: the other's bound may stand
    assert probe.bound_of(link, value, 1.0, 3.0, 8.0, 0.5, 1.0) <= 0x3f800000 or value > 1.0
