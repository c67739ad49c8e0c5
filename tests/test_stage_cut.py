"""The stage kernel's work items (csrc/stage_cut.h) on the host: whatever cut the launch rule
chooses, for any number of blocks and every kind of kernel, its items cover each plane of each block
exactly once, in sizes that do not grow along the list."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
# kernels as the rule sees them: FP64, planes come as primitives, source terms, CTAs per SM
KERNELS = {"hd64": (1, 0, 0, 2), "mhd64": (1, 0, 0, 1), "srhd64": (1, 1, 0, 1), "ffhd64": (1, 0, 1, 2),
           "hd32": (0, 0, 0, 3), "mhd32": (0, 0, 0, 2), "srhd32": (0, 1, 0, 3), "ffhd32": (0, 0, 1, 3)}


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    out = str(tmp_path_factory.mktemp("shim") / "libcutshim.so")
    subprocess.run([gxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-o", out, os.path.join(HERE, "cut_shim.cpp")],
                   check=True)
    return C.CDLL(out)


def _cut(shim, nblk, *kernel, sms=152):
    out = np.zeros(5, dtype=np.int32)
    shim.shim_cut(nblk, sms, *kernel, C.c_void_p(out.ctypes.data))
    return [int(v) for v in out]


def _covers(shim, nblk, n1, a, m, items):
    it = np.full((items, 3), -1, dtype=np.int32)
    shim.shim_items(nblk, n1, a, m, C.c_void_p(it.ctypes.data))
    assert np.all(np.diff(it[:, 2]) <= 0) and it[:, 2].min() >= 1
    seen = np.zeros((nblk, 17), dtype=np.int64)          # +1 at an item's start, -1 behind its end
    np.add.at(seen, (it[:, 0], it[:, 1]), 1)
    np.add.at(seen, (it[:, 0], it[:, 1] + it[:, 2]), -1)
    cover = np.cumsum(seen, axis=1)
    assert np.all(cover[:, :16] == 1) and np.all(cover[:, 16] == 0)


@pytest.mark.parametrize("kernel", sorted(KERNELS))
def test_items_cover_every_plane_once(shim, kernel):
    for nblk in list(range(1, 700)) + [1000, 1250, 1728, 4096, 47178]:
        n1, a, m, items, whole = _cut(shim, nblk, *KERNELS[kernel])
        _covers(shim, nblk, n1, a, m, items)
        assert whole == (n1 == nblk or a == 16)


@pytest.mark.parametrize("kernel", sorted(KERNELS))
def test_cut_fits_the_launch_it_is_for(shim, kernel):
    """An autotuned batch may launch fewer CTAs per SM than fit; the cut is formed for those. With one
    per SM a lone item is no slower than others, so one or two blocks per SM stay whole."""
    *kind, fit = KERNELS[kernel]
    for ctas in range(1, fit + 1):
        for nblk in list(range(1, 700, 7)) + [1000, 1250, 4096]:
            n1, a, m, items, whole = _cut(shim, nblk, *kind, ctas)
            _covers(shim, nblk, n1, a, m, items)
    assert _cut(shim, 152, *kind, 1)[4] and _cut(shim, 304, *kind, 1)[4]


def test_every_size_of_items(shim):
    for nblk, n1 in ((1, 0), (7, 3), (305, 152), (4000, 3952)):
        for a in range(1, 17):
            m = 16 // a
            _covers(shim, nblk, n1, a, m, n1 + (nblk - n1) * (m + (16 % a > 0)))


def test_division_of_large_item_numbers(shim):
    """The block of an item comes from a product instead of a quotient: exact up to 2^28 items."""
    for m in range(1, 17):
        inv = ((1 << 32) + m - 1) // m
        v = np.concatenate([np.arange(4096), (1 << 28) - 1 - np.arange(4096)]).astype(np.uint64)
        assert np.array_equal(v * np.uint64(inv) >> np.uint64(32), v // np.uint64(m))
