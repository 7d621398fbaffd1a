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
    const unsigned end = row_ptr[row + 1] + misalign;
    const TableRow tr{row_ptr[row] + misalign, end, load_limit(end, last ? batch - 1 : 0, batch, nnz)};
    for (unsigned p0 = tr.first(); p0 < tr.end; p0 += kMasksChunk)
        for (int lane = 0; lane < 32; ++lane) {
            const unsigned p = p0 + kMasksRun * lane;
            if (p >= tr.end) break;
            for (unsigned i = 0; i < kMasksRun; ++i)
                if (tr.wide(p) || tr.has(p + i)) {
                    const long long at = (long long)(p + i) - misalign;
                    if (at < 0 || at >= count) return 0;
                    loads[at] += 1;
                }
        }
    return 1;
}

// One row [beg, end) of a pattern that ends with it, `warps` warps sharing it.  0: a load behind the pattern, or more iterations
// than the row has chunks.
extern "C" int table_row_at(int beg, int end, unsigned misalign, int warps, unsigned char *loads)
{
    const TableRow tr{beg + misalign, end + misalign, load_limit(end + misalign, 0, 1, end)};
    for (int warp = 0; warp < warps; ++warp) {
        int iterations = 0;
        for (unsigned p0 = tr.first() + kMasksChunk * warp; p0 < tr.end; p0 += kMasksChunk * warps) {
            if (++iterations > (end - beg) / (int)kMasksChunk + 2) return 0;
            for (int lane = 0; lane < 32; ++lane) {
                const unsigned p = p0 + kMasksRun * lane;
                if (p >= tr.end) break;
                for (unsigned i = 0; i < kMasksRun; ++i) {
                    if (tr.has(p + i)) loads[p + i - tr.beg] += 1;
                    else if (tr.wide(p) && p + i >= tr.end) return 0;
                }
            }
        }
    }
    return 1;
}

// A row kernel's walk over a row [beg, end): every entry is taken once, and a prefetch that says it is inside the row is.
extern "C" int row_chunks(int beg, int end, int warps, int size, unsigned char *taken)
{
    for (int warp = 0; warp < warps; ++warp) {
        int iterations = 0;
        for (RowChunks r(beg, end, warp, warps, size); r.more(); r.advance()) {
            if (++iterations > (end - beg) / size + 1) return 0;
            for (int i = 0; i < (int)r.count(); ++i) taken[(long long)r.at + i - beg] += 1;
            for (int lane = 0; lane < 32; ++lane) {
                const bool inside = (long long)r.at + warps * size + lane < end;
                if ((r.next(lane) < r.end) != inside || (lane < r.behind()) != inside) return 0;
            }
        }
    }
    return 1;
}

extern "C" int block_rows(int block, int rows, int blocks)   // rows that a block walks; -1: one that does not exist
{
    int n = 0;
    for (BlockRows b(block, rows, blocks); b.more(); b.advance()) {
        if ((long long)b.row < 0 || (long long)b.row >= rows || ++n > 4) return -1;
    }
    return n;
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


@pytest.mark.parametrize("warps", [1, 4])
@pytest.mark.parametrize("length", [1, 31, 700, 2500])
def test_the_table_pass_ends_at_the_largest_positions(host, length, warps):
    """The last entry of a row may be number 2^31 - 2: steps past it must not wrap round."""
    for end in (2 ** 31 - 1, 2 ** 31 - 2, 2 ** 31 - 260, 2 ** 31 - 1030):
        for misalign in range(4):
            loads = np.zeros(length, np.uint8)
            assert host.table_row_at(end - length, end, misalign, warps, loads.ctypes.data_as(ctypes.c_void_p)), end
            assert (loads == 1).all()


@pytest.mark.parametrize("size", [4, 12, 16, 32])
@pytest.mark.parametrize("length", [1, 16, 33, 64, 65, 129, 700])
def test_the_row_kernels_take_every_entry_once(host, length, size):
    for end in (length, 1000 + length, 2 ** 31 - 1, 2 ** 31 - 2, 2 ** 31 - 100, 2 ** 31 - 160):
        taken = np.zeros(length, np.uint8)
        assert host.row_chunks(end - length, end, 4, size, taken.ctypes.data_as(ctypes.c_void_p)), end
        assert (taken == 1).all()


@pytest.mark.parametrize("rows,blocks,block,want", [(10, 10, 9, 1), (10, 4, 1, 3), (2 ** 31 - 1, 2 ** 31 - 1, 2 ** 31 - 2, 1),
                                                    (2 ** 30 + 5, 2 ** 30 + 5, 2 ** 30 + 4, 1), (2 ** 30, 2 ** 30, 7, 1)])
def test_a_block_walks_its_rows(host, rows, blocks, block, want):
    assert host.block_rows(block, rows, blocks) == want
