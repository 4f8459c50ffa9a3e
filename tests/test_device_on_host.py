"""Device functions of common.cuh on the CPU (`device_on_host.cpp`)."""
import ctypes
import os
import re
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_2408_15562_b200", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("device_on_host") / "libdevice_on_host.so")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-I" + os.path.join(ROOT, "include"), "-I" + CSRC, "-I/usr/local/cuda/include",
                           os.path.join(HERE, "device_on_host.cpp"), "-o", out])
    return ctypes.CDLL(out)


@pytest.mark.parametrize("hi", [1, 2, 3, 4, 5, 8, 11])
@pytest.mark.parametrize("late", [0, 1])
def test_four_positions_of_a_row(lib, hi, late):
    """Inside the row its values, outside of it the padding and no load; nothing of a row that may have been written late goes by the
    read-only path, which is for data that nobody writes while the kernel runs."""
    raw = np.arange(16 + 4, dtype=np.float32)
    row = raw[(-raw.ctypes.data // 4) % 4:]
    for j in range(-4, 13, 4):
        out = np.empty(4, np.float32)
        by_read_only = lib.load4(ctypes.c_void_p(row.ctypes.data), j, hi, late, ctypes.c_void_p(out.ctypes.data))
        want = [row[i] if 0 <= i < hi else -1.0 for i in range(j, j + 4)]
        assert by_read_only >= 0 and out.tolist() == want
        assert not (late and by_read_only)


def test_the_walk_takes_rows_that_the_scan_brings_as_late_ones(lib):
    """The walk behind a scan by the trees is resident while that scan writes rows of host logits to the device: the type of its rows
    keeps them from the read-only loads, and so from every function that takes a plain pointer."""
    assert lib.late_row_is_a_pointer() == 0
    walk = open(os.path.join(CSRC, "accept_walk.cu")).read()
    assert re.search(r"struct LogitsRow<true> \{ typedef FspadLateRow T; \}", walk)
    assert re.findall(r"args\.logits\b[^;]*", walk) == ["args.logits + row0 * V}"] and "const Row lg{args.logits" in walk


@pytest.mark.parametrize("vocab", [1, 2, 3, 4, 5, 6, 7, 9])
def test_units_loaded_whole_lie_in_the_array(lib, vocab):
    """The scan by the trees loads a row's units of four whole where they end in a row behind it, however short those rows are: all
    that it loads whole lies in the array, and every unit of the row that does is loaded whole."""
    for rows in range(1, 8):
        for row in range(rows):
            start = row * vocab
            j0 = -(start & 3)
            units = (vocab - j0 + 3) // 4
            whole = [i for i in range(units) if start + j0 + 4 * i + 4 <= rows * vocab]
            for n in range(units + 1):
                assert max(0, lib.whole_units(rows, row, vocab, j0, n)) == len([i for i in whole if i < n]), (rows, row, n)
