"""The index arithmetic of csrc/row_walk.h, compiled for the host: which entries the lanes of the kernels load."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# Walks a row as the kernels do, every lane of every warp after the other.
HOST = r"""
#include "row_walk.h"
using namespace b2sp;

// The window-table pass over a row of the last pattern (`last`) or an earlier one of a batch.  loads[p] += 1 for every position
// that is loaded; 0: one outside [0, count).
extern "C" int table_row(const int *row_ptr, int row, long long nnz, int batch, int last, unsigned misalign, int count, unsigned char *loads)
{
    const int beg = row_ptr[row], end = row_ptr[row + 1];
    const TableRow tr(beg, end, load_limit(end, last ? batch - 1 : 0, batch, nnz), misalign);
    for (int p0 = tr.first; p0 < tr.end; p0 += kMasksChunk)
        for (int lane = 0; lane < 32; ++lane) {
            const int p = p0 + kMasksRun * lane;
            if (p >= tr.end) break;
            for (int i = 0; i < kMasksRun; ++i)
                if (tr.wide(p) || tr.has(p + i)) {
                    if (p + i < 0 || p + i >= count) return 0;
                    loads[p + i] += 1;
                }
        }
    return 1;
}
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    d = tmp_path_factory.mktemp("row_walk")
    src, lib = d / "host.cpp", d / "host.so"
    src.write_text(HOST)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-fwrapv", "-shared", "-fPIC", "-o", str(lib), str(src),
                           "-I" + os.path.join(ROOT, "paper_2311_00368_b200", "csrc")])
    return ctypes.CDLL(str(lib))


@pytest.mark.parametrize("misalign", [0, 1, 2, 3])
@pytest.mark.parametrize("batch,last,slack", [(1, 1, 0), (3, 0, 5), (3, 1, 1), (3, 1, 4), (3, 1, 7), (2, 1, 300)])
def test_the_table_pass_stays_inside_the_pattern(host, batch, last, slack, misalign):
    """A pattern of a batch has a slot of nnz_stride elements, but the last one's array may end with its last entry."""
    rng = np.random.default_rng(slack)
    for lens in ([1], [3], [8], [5, 0, 12], [300, 2, 1], list(rng.integers(0, 40, 30)), [256, 255, 257, 9]):
        rp = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
        count = int(rp[-1])
        for row in range(len(lens)):
            loads = np.zeros(count + slack, np.uint8)
            assert host.table_row(rp.ctypes.data_as(ctypes.c_void_p), row, ctypes.c_longlong(count + slack), batch, last, misalign,
                                  count if last else count + slack, loads.ctypes.data_as(ctypes.c_void_p)), (lens, row)
            assert (loads[rp[row]:rp[row + 1]] == 1).all()
