"""Row placement of the sliced storage (host code, compiled here): every row
once at the positions in front of the padding, which the kernels that run over
one position per row rely on."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from oracle_cases import hierarchy

NEVER, ALWAYS, AUTO = 0, 1, 2


@pytest.fixture(scope="module")
def place(root, tmp_path_factory):
    d = tmp_path_factory.mktemp("placement")
    src, lib = d / "place.cpp", d / "place.so"
    src.write_text('#include "placement.h"\n'
                   'extern "C" int place(const int* rp, long n, int how, int* order) {\n'
                   "  bamg::Placement p = bamg::place_rows(std::vector<int>(rp, rp + n + 1), n, how);\n"
                   "  std::copy(p.order.begin(), p.order.end(), order);\n"
                   "  return p.sorted;\n}\n")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I",
                    os.path.join(root, "paper_2606_24748_gb300", "csrc"), str(src), "-o", str(lib)], check=True)
    fn = ctypes.CDLL(str(lib)).place

    def run(lengths, how):
        n = len(lengths)
        rp = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
        order = np.full((n + 31) // 32 * 32, -7, dtype=np.int32)
        ip = ctypes.POINTER(ctypes.c_int)
        how = fn(rp.ctypes.data_as(ip), ctypes.c_long(n), how, order.ctypes.data_as(ip))
        return order, bool(how)

    return run


def check(place, lengths, how):
    order, is_sorted = place(lengths, how)
    n = len(lengths)
    assert (order[n:] == -1).all()
    assert np.array_equal(np.sort(order[:n]), np.arange(n))
    if not is_sorted:
        assert np.array_equal(order[:n], np.arange(n))
    return is_sorted


@pytest.mark.parametrize("last", [1, 2, 31, 32, 33, 63, 500, 1023, 1024])
@pytest.mark.parametrize("windows", [0, 1, 3])
@pytest.mark.parametrize("width", [0, 1, 30, 60])
def test_padding_stays_last(place, last, windows, width):
    """Windows of 1,024 uneven rows (40 and 3 blocks in turn), then a part of
    a window whose rows are narrower or wider than all others."""
    lengths = np.concatenate([np.tile([40, 3], 512 * windows), np.full(last, width)]).astype(int)
    assert check(place, lengths, ALWAYS)
    check(place, lengths, AUTO)
    assert not check(place, lengths, NEVER)


def test_padding_stays_last_on_random_rows(place):
    rng = np.random.default_rng(3)
    for n in (1, 31, 32, 100, 1025, 1057, 5000):
        for _ in range(5):
            lengths = rng.integers(0, rng.integers(1, 80), n)
            check(place, lengths, ALWAYS)
            check(place, lengths, AUTO)


@pytest.mark.parametrize("ne,order,aggregation", [(6, 2, "geometric"), (12, 1, "mis"), (13, 1, "geometric")])
def test_padding_stays_last_on_hierarchies(place, ne, order, aggregation):
    for level in hierarchy(ne, order=order, aggregation=aggregation).levels[:-1]:
        check(place, np.diff(level.P.rowptr), ALWAYS)
        check(place, np.diff(level.A.rowptr), AUTO)


def test_slices_go_from_wide_to_narrow(place):
    lengths = np.tile([40, 3, 17, 0, 27], 512)
    order, _ = place(lengths, ALWAYS)
    widths = lengths[order].reshape(-1, 32).max(1)
    assert (np.diff(widths[:lengths.size // 32]) <= 0).all()
