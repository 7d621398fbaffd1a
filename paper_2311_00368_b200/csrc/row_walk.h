// Which entries of a CSR row a warp or a lane takes, and which of them it may load: the index arithmetic of kernels, free of
// CUDA so that the host can run it too (tests/test_row_walk.py walks whole patterns and checks every position).
#pragma once

#ifdef __CUDACC__
#define B2SP_HD __host__ __device__ __forceinline__
#else
#define B2SP_HD inline
#endif

namespace b2sp {

// ---- window table: the runs of a row -----------------------------------------------------------
// Positions are counted from the 16-byte boundary at or before the pattern's first entry, so that runs that begin at a multiple
// of four are aligned wherever the array begins, and unsigned: a pattern may have 2^31 - 1 entries, and a step past the last of
// them still fits.
constexpr unsigned kMasksRun = 8;                // consecutive entries of a lane
constexpr unsigned kMasksChunk = 32 * kMasksRun; // entries of a warp's iteration

// Entries of a pattern below this position may be loaded along with a row that ends at `end`.  A single pattern has `nnz` entries;
// in a batch `nnz` is the distance between the patterns' arrays, and the last array may end with its last entry (the rule that
// costs nothing: a load of the last pattern's own entry count ran 4% to 10% longer, a row's own end for all rows up to 6%).
B2SP_HD unsigned load_limit(unsigned end, int pattern, int batch, unsigned nnz)
{
    return batch > 1 && pattern == batch - 1 ? end : nnz;
}

struct TableRow {
    unsigned beg, end;   // the row's entries
    unsigned limit;      // of the entries that may be loaded

    // where lane 0's first run begins: at the row or up to three entries before it
    B2SP_HD unsigned first() const { return beg & ~3u; }
    // the run at p .. p + 7 may be loaded sixteen bytes at a time (the first four positions may lie before the array)
    B2SP_HD bool wide(unsigned p) const { return p >= 4 && p + kMasksRun <= limit; }
    B2SP_HD bool has(unsigned p) const { return p >= beg && p < end; }
};

// ---- row kernels ---------------------------------------------------------------------------------
// Rows and positions are unsigned here too: both may number 2^31 - 1, and a step past the last one still fits.
// The rows of a block of a grid of `blocks`: block, block + blocks, ...
struct BlockRows {
    unsigned row, rows, step;
    B2SP_HD BlockRows(unsigned block, unsigned rows_, unsigned blocks) : row(block), rows(rows_), step(blocks) {}
    B2SP_HD bool more() const { return row < rows; }
    B2SP_HD void advance() { row += step; }
};

// The chunks of a row [beg, end) that warp `warp` of `warps` takes: every warps-th one.
struct RowChunks {
    unsigned at, end, step, size;   // the chunk begins at `at`
    B2SP_HD RowChunks(unsigned beg, unsigned end_, unsigned warp, unsigned warps, unsigned size_)
        : at(beg + warp * size_), end(end_), step(warps * size_), size(size_)
    {
    }
    B2SP_HD bool more() const { return at < end; }
    B2SP_HD void advance() { at += step; }
    B2SP_HD int count() const { return (int)(end - at < size ? end - at : size); }
    B2SP_HD unsigned next(int i) const { return at + step + i; }   // entry i of the warp's next chunk (behind the row: not < end)
    B2SP_HD int behind() const { return (int)(end - at) - (int)step; }   // entries of the row from the next chunk on (0 or less: none)
};

}  // namespace b2sp
