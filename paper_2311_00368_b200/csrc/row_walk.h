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
constexpr int kMasksRun = 8;                // consecutive entries of a lane
constexpr int kMasksChunk = 32 * kMasksRun; // entries of a warp's iteration

// Entries of a pattern below this position may be loaded along with a row that ends at `end`.  A single pattern has `nnz` entries;
// in a batch `nnz` is the distance between the patterns' arrays, and the last array may end with its last entry (the rule that
// costs nothing: a load of the last pattern's own entry count ran 4% to 10% longer, a row's own end for all rows up to 6%).
B2SP_HD int load_limit(int end, long long pattern, long long batch, long long nnz)
{
    return batch > 1 && pattern == batch - 1 ? end : (int)nnz;
}

struct TableRow {
    int beg, end;   // the row's entries
    int limit;      // of the entries that may be loaded
    int first;      // where lane 0's first run begins: at the row or up to three entries before it, on a 16-byte boundary

    // `misalign`: elements between a 16-byte boundary and the pattern's first entry
    B2SP_HD TableRow(int beg_, int end_, int limit_, unsigned misalign)
        : beg(beg_), end(end_), limit(limit_), first(beg_ - (int)(((unsigned)beg_ + misalign) & 3u))
    {
    }
    // the run at p .. p + 7 may be loaded sixteen bytes at a time
    B2SP_HD bool wide(int p) const { return p >= 0 && p <= limit - kMasksRun; }
    B2SP_HD bool has(int p) const { return p >= beg && p < end; }
};

}  // namespace b2sp
