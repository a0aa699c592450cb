"""The commands that the blocks of the interaction-matrix rows write (csrc/row_parts.h, compiled for the
host): over all parts of the commands each one is written exactly once, by a zero run or by its DM's band,
whatever lies at the parts' bounds."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include "row_parts.h"
using namespace mcao;
// counts[c]: times command c is written; returns the writes outside the writer's own part
extern "C" int cover(int n_cmd, int n_parts, int n_dms, const int* c0, const int* c1, int* counts) {
    int stray = 0;
    for (int z = 0; z < n_parts; ++z) {
        const CmdRange p = command_part(n_cmd, n_parts, z);
        CmdRange b[8];
        auto write = [&](CmdRange r) {
            for (int c = r.lo; c < r.hi; ++c) {
                ++counts[c];
                stray += c < p.lo || c >= p.hi;
            }
        };
        for (int m = 0; m < n_dms; ++m) write(b[m] = band_in_part(p, c0[m], c1[m]));
        for (int m = 0; m <= n_dms; ++m) write(zeros_between(p, m ? b + m - 1 : nullptr, m < n_dms ? b + m : nullptr));
    }
    return stray;
}
"""


@pytest.fixture(scope="module")
def cover(tmp_path_factory):
    d = tmp_path_factory.mktemp("row_parts")
    (d / "cover.cpp").write_text(SRC)
    so = str(d / "cover.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_1608_00386_gb300", "csrc"),
                    str(d / "cover.cpp"), "-o", so], check=True)
    return ctypes.CDLL(so).cover


def _check(cover, sizes, bands, parts):
    """DMs of `sizes` commands, band rows of DM m at commands bands[m] counted from its first."""
    cmd0 = np.concatenate([[0], np.cumsum(sizes)])[:-1].astype(np.int32)
    n_cmd = sum(sizes)
    c = (cmd0[:, None] + np.asarray(bands, np.int32).reshape(-1, 2)).astype(np.int32)
    lo, hi = np.ascontiguousarray(c[:, 0]), np.ascontiguousarray(c[:, 1])
    counts = np.zeros(n_cmd + 1, np.int32)
    p = lambda a: a.ctypes.data_as(ctypes.POINTER(ctypes.c_int))
    stray = cover(n_cmd, parts, len(sizes), p(lo), p(hi), p(counts))
    assert stray == 0 and np.all(counts[:-1] == 1) and counts[-1] == 0, (sizes, bands, parts)


@pytest.mark.parametrize("parts", range(1, 17))
def test_every_command_is_written_once(cover, parts):
    # the 39 m system's DMs with whole bands (a 2 x 2 sensor sees the whole pupil) and with narrow ones
    eelt = [5402, 1441, 1208]
    _check(cover, eelt, [(0, s) for s in eelt], parts)
    _check(cover, eelt, [(700, 900), (0, 40), (1200, 1208)], parts)
    rng = np.random.default_rng(parts)
    for _ in range(200):
        sizes = [int(rng.integers(0, 60)) for _ in range(rng.integers(1, 5))]
        bands = [sorted(int(rng.integers(0, s + 1)) for _ in range(2)) for s in sizes]   # empty ones too
        _check(cover, sizes, bands, parts)
