// Support kernels of the dense-tile (tensor-core) family.
//
// Idea of the family: at 10-30% density a 128 x 32 window of S is a dense tile with 70-90% zeros, and
// the 5th-generation tensor cores multiply it by a dense tile an order of magnitude faster than the
// FP32 pipes can walk its nonzeros.  fp32 accuracy is kept by splitting every operand into two tf32
// numbers (x = hi + lo) and issuing three MMAs per product: hi*hi + lo*hi + hi*lo.
//
// Pieces here (the tile kernel itself is in tile_fused.cuh):
//   tile_masks_kernel      per row and 32-column window: first CSR position + occupancy bit mask
//                          (needs strictly increasing columns in a row; sets a flag otherwise)
//   split_dense_kernel     dense fp32 operands -> zero-padded (hi, lo) tf32 copies
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "ptx_sm100.cuh"
#include "row_walk.h"
#include "tile_dispatch.h"

namespace b2sp {

constexpr int kTileKC = 32;       // columns of S per pipeline stage (one 128-byte swizzle row of tf32)
// Flag words of the tile pre-passes (the gate of the row-kernel fallback reads the first two, see row_kernels.cuh):
constexpr int kFlagUnsorted = 0;   // != 0: the window table is unusable (a row's columns are not strictly increasing,
                                   // or the table belongs to other arrays); stays set until the table is rebuilt
constexpr int kFlagNotFinite = 1;  // != 0: a dense operand of this call holds a non-finite value; cleared by the fallback
constexpr int kFlagGateReaders = 2;  // CTAs of the gated fallback that have read the flags so far

// ---- table signature ------------------------------------------------------------------------------------
struct PatternSignature {
    int magic, M, K, Wk;
    long long nnz;
    const int *row_ptr, *col_idx;
    long long batch, rp_stride, nz_stride;   // a batch of patterns (see tile_masks_kernel); 1, 0, 0 for a single one
};
constexpr int kPatternMagic = 0x62327370;

// ---- window table -------------------------------------------------------------------------------
// T[r*Wk + w] = (first CSR position of row r whose column is >= 32w, occupancy bit mask of the column
// window [32w, 32w+32): bit b set <=> column 32w+b is stored).
// A row has one mask word per window in shared memory.  First sweep: lane l of a warp reads eight consecutive
// entries (two 16-byte loads, the next eight in flight meanwhile) and ORs each entry's bit into its window's word.
// Second sweep: a lane takes two windows; the position of a window is the row start plus the entries of all earlier
// windows (a prefix sum over the pop counts).  Every window of every row is written, so the table needs no clearing.
// The table is only meaningful when the columns of each row are strictly increasing and in range;
// the first sweep checks exactly that and sets flags[kFlagUnsorted] if not.
constexpr int kMasksMaxWk = 24 * 1024;                // the mask row must fit in the shared memory a block may ask for (96 KB)
constexpr int kMasksMaxSmem = kMasksMaxWk * 4;
constexpr int kMasksRows = 8;                         // rows (= warps) of a tile_masks_kernel<false> block
constexpr unsigned kMasksOwn = 2048;                       // entries of its row that a warp of such a block reads by itself
constexpr int kMasksSharedWarps = 4;                  // warps of a tile_masks_kernel<true> block
__host__ __device__ constexpr int masks_row_words(int Wk) { return (Wk + 127) & ~127; }   // (cleared sixteen bytes per lane)

// Entries p .. p + 7: sixteen-byte loads where all of them may be read (p is chosen so that their addresses are aligned), single
// ones of the row otherwise.
__device__ __forceinline__ void masks_load_run(const int *__restrict__ col_idx, const TableRow &row, unsigned p, int (&v)[kMasksRun])
{
    if (p >= row.end) return;
    if (row.wide(p)) {
#pragma unroll
        for (unsigned i = 0; i < kMasksRun; i += 4) {
            const int4 x = __ldg(reinterpret_cast<const int4 *>(col_idx + p + i));
            v[i] = x.x; v[i + 1] = x.y; v[i + 2] = x.z; v[i + 3] = x.w;
        }
    } else {
#pragma unroll
        for (unsigned i = 0; i < kMasksRun; ++i)
            if (row.has(p + i)) v[i] = __ldg(col_idx + p + i);
    }
}

// ORs the bits of a lane's run c (entries p .. p + 7) into the row's words (shared-memory address `words`).  `prev` = the
// entry before the run, `interior` (the same for the whole warp): every lane's run is inside the row.  false: the row is not
// strictly increasing or out of range (a table with such a row is not used).  Neighbouring lanes are eight entries apart,
// so that they hardly ever OR into the same word at the same time (consecutive entries mostly share one).
template <bool BRANCH_FREE>
__device__ __forceinline__ bool masks_or_run(const int (&c)[kMasksRun], int prev, unsigned p, const TableRow &row, int K, uint32_t words, bool interior)
{
    auto or_bit = [&](int col) { ptx::red_or_shared(words + 4 * (col >> 5), __funnelshift_l(0u, 1u, col)); };   // 1 << (column within the window)
    if (interior) {
        bool ok = (p <= row.beg || c[0] > prev) && c[0] >= 0 && c[kMasksRun - 1] < K;   // (in order, so the others are in range too)
#pragma unroll
        for (int i = 1; i < kMasksRun; ++i) ok = ok && c[i] > c[i - 1];
        if (!ok) return false;
#pragma unroll
        for (int i = 0; i < kMasksRun; ++i) or_bit(c[i]);
        return true;
    }
    // An end of the row: some of the entries are not in it.  (What the two ways cost: at tile_masks_kernel.)
    bool bad = false;
    if constexpr (BRANCH_FREE) {
#pragma unroll
        for (int i = 0; i < kMasksRun; ++i) {
            const bool in_row = row.has(p + i), in_range = (unsigned)c[i] < (unsigned)K;
            const bool in_order = p + i == row.beg || c[i] > (i == 0 ? prev : c[i == 0 ? 0 : i - 1]);
            bad |= in_row & !(in_range & in_order);
            ptx::red_or_shared_if(words + 4 * (c[i] >> 5), __funnelshift_l(0u, 1u, c[i]), in_row & in_range);
        }
    } else {
#pragma unroll
        for (int i = 0; i < kMasksRun; ++i) {
            if (!row.has(p + i)) continue;
            const bool in_range = (unsigned)c[i] < (unsigned)K;
            bad |= !in_range || (p + i != row.beg && c[i] <= (i == 0 ? prev : c[i == 0 ? 0 : i - 1]));
            if (in_range) or_bit(c[i]);
        }
    }
    return !bad;
}

// Blocks of the form with a warp per row that share an SM.
constexpr int masks_blocks_per_sm(bool six) { return (six ? 48 : 40) / kMasksRows; }

// A batch of `sig.batch` patterns of the same M and K (row_ptr arrays `sig.rp_stride` elements apart, each
// starting at 0; col_idx arrays `sig.nz_stride` elements apart) gives one table per pattern, stacked:
// T[(b*M + r)*Wk + w], positions relative to the pattern's own col_idx array.
//
// SHARED = false: a block of eight warps has eight rows, a warp to each, which meet once, between the sweeps, to hear whether
// one of the rows is long: a warp reads the first kMasksOwn entries of its row by itself, and what is left of longer rows is
// dealt to all eight warps, so that a long row is not one warp's chain of iterations.  SHARED = true: the four warps of a block
// share one row throughout, for few rows (which would leave the GPU idle otherwise), for long ones and for rows whose words
// fill the shared memory.
// What bounds it: instruction issue (82% of the slots at 32768 rows of 820 entries, 2.7 TB/s; about 30 instructions per
// 32 entries, the row's fixed part included).  Measured, against a block of four warps per row with two barriers and
// branches per entry (one 16-byte load per lane and step): 32768 x 8192 at 20% 88 -> 62 us, eight patterns of 4096 x 4096
// at 20% 61 -> 41 us (those do not begin on 16-byte boundaries), 16384 x 512 at 20% 18 -> 13.5 us, power-law 8192 x 8192 at
// 30% (SHARED) 38.6 -> 31 us.
//
// SIX: of the form with a warp per row, six blocks per SM (40 registers) instead of five (48).  The ends of rows are handled without
// branches where the registers allow it, and a row of 410 entries has two chunks, both of them ends.  Five blocks and no branches
// against six with branches, inputs in L2: 4096 x 4096 at 10% 8.5 against 9.6 us, 8192 x 8192 at 20% 18.6 against 20.4, 16384 x 4096 at 20% 20.7
// against 22.6, 32768 x 512 at 20% 20.7 against 21.8; power-law 8192 x 8192 at 30% (SHARED) 31.0 against 33.0.  Six blocks without branches
// spill: 32768 x 512 at 5% 22.7, 4096 x 30000 at 3% 16.5 against 14.7.
template <bool SHARED, bool SIX = false>
__global__ void __launch_bounds__(SHARED ? kMasksSharedWarps * 32 : kMasksRows * 32, SHARED ? 8 : masks_blocks_per_sm(SIX))
tile_masks_kernel(int M, int K, int Wk, long long nnz, const int *__restrict__ row_ptr0,
                  const int *__restrict__ col_idx0, int2 *__restrict__ T, int *__restrict__ flags,
                  PatternSignature sig, PatternSignature *__restrict__ sig_out)
{
    extern __shared__ __align__(16) unsigned mask_rows[];
    // (inside a stateless tile op the operand-split kernel is launched as a programmatic dependent of this
    // one: the two touch different data and may overlap; that kernel waits for this grid before it ends)
    ptx::launch_dependents();
    if (blockIdx.x == 0 && threadIdx.x == 0) *sig_out = sig;   // what the table is built from
    constexpr unsigned kFull = 0xffffffffu;
    constexpr bool BRANCH_FREE = !SIX;
    constexpr int WARPS = SHARED ? kMasksSharedWarps : 1;       // warps of a row
    constexpr int ROWS = SHARED ? 1 : kMasksRows;               // rows of the block at a time
    __shared__ int warp_total[WARPS];
    __shared__ uint4 rest[ROWS];                                // of each row: problem, first entry, first entry not read yet, end
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int words = masks_row_words(Wk);
    unsigned *mask = mask_rows + (SHARED ? 0 : warp * words);
    const uint32_t mask_smem = ptx::smem_u32(mask);
    bool bad = false;
    const long long rows_all = (long long)M * sig.batch;
    for (long long row0 = (long long)blockIdx.x * ROWS; row0 < rows_all; row0 += (long long)gridDim.x * ROWS) {
        const long long rowg = row0 + (SHARED ? 0 : warp);
        const bool live = SHARED || rowg < rows_all;
        // (no 64-bit division, which is a library call, where it can be avoided)
        const int pb = sig.batch == 1 || !live ? 0 : rows_all < 0x7fffffffll ? (int)((unsigned)rowg / (unsigned)M) : (int)(rowg / M);
        const int row = live ? (int)(rowg - (long long)pb * M) : 0;
        const int *__restrict__ row_ptr = row_ptr0 + pb * sig.rp_stride;
        // (from the 16-byte boundary at or before the problem's first entry, see row_walk.h)
        auto aligned_down = [](const int *p) { return reinterpret_cast<const int *>(reinterpret_cast<uintptr_t>(p) & ~uintptr_t(15)); };
        auto misalignment = [](const int *p) { return (unsigned)(reinterpret_cast<uintptr_t>(p) >> 2) & 3u; };
        const int *__restrict__ col_idx = aligned_down(col_idx0 + pb * sig.nz_stride);
        const unsigned misalign = misalignment(col_idx0 + pb * sig.nz_stride);
        const int beg = live ? __ldg(row_ptr + row) : 0, end = live ? __ldg(row_ptr + row + 1) : 0;
        const TableRow tr{(unsigned)beg + misalign, (unsigned)end + misalign, load_limit((unsigned)end + misalign, pb, (int)sig.batch, (unsigned)nnz)};
        int c[kMasksRun], c_next[kMasksRun];
        unsigned p0 = tr.first();
        const unsigned own_end = SHARED || tr.end - p0 <= kMasksOwn ? tr.end : p0 + kMasksOwn;
#pragma unroll
        for (int i = 0; i < kMasksRun; ++i) c_next[i] = 0;
        if (SHARED) p0 += kMasksChunk * warp;
        if (beg < end) masks_load_run(col_idx, tr, p0 + kMasksRun * lane, c_next);
        else p0 = own_end;
        for (int w = (SHARED ? (int)threadIdx.x : lane) * 4; w < words; w += WARPS * 128)
            *reinterpret_cast<uint4 *>(mask + w) = make_uint4(0u, 0u, 0u, 0u);
        if (!SHARED && lane == 0) rest[warp] = make_uint4((unsigned)pb, tr.beg, beg < end ? own_end : tr.end, tr.end);
        if (SHARED) __syncthreads();
        else __syncwarp();
        int carry = 0;   // the last entry of the warp's previous iteration
        for (; p0 < own_end; p0 += kMasksChunk * WARPS) {
            const unsigned p = p0 + kMasksRun * lane;
#pragma unroll
            for (int i = 0; i < kMasksRun; ++i) c[i] = c_next[i];
            if (p0 + kMasksChunk * WARPS < own_end) masks_load_run(col_idx, tr, p + kMasksChunk * WARPS, c_next);
            int prev = __shfl_up_sync(kFull, c[kMasksRun - 1], 1);
            if (lane == 0) prev = !SHARED ? carry : p > tr.beg ? __ldg(col_idx + p - 1) : 0;
            if (!SHARED) carry = __shfl_sync(kFull, c[kMasksRun - 1], 31);
            bad |= !masks_or_run<BRANCH_FREE>(c, prev, p, tr, K, mask_smem, p0 >= tr.beg && p0 + kMasksChunk <= tr.end);
        }
        if (SHARED) {
            __syncthreads();
        } else if (__syncthreads_or(beg < end && own_end < tr.end)) {
            // some of the block's rows are longer: their other entries, in chunks dealt to the warps in turn
            unsigned turn = 0;   // chunks of the rows before
            for (int r = 0; r < ROWS; ++r) {
                const uint4 q = rest[r];
                if (q.z >= q.w) continue;
                const int *__restrict__ ci = aligned_down(col_idx0 + q.x * sig.nz_stride);
                const TableRow other{q.y, q.w, q.w};
                const unsigned chunks = (q.w - q.z + kMasksChunk - 1) / kMasksChunk;
                for (unsigned j = (warp - turn) & (ROWS - 1); j < chunks; j += ROWS) {
                    const unsigned pc = q.z + j * kMasksChunk, p = pc + kMasksRun * lane;
                    masks_load_run(ci, other, p, c);
                    int prev = __shfl_up_sync(kFull, c[kMasksRun - 1], 1);
                    if (lane == 0) prev = __ldg(ci + p - 1);
                    bad |= !masks_or_run<BRANCH_FREE>(c, prev, p, other, K, ptx::smem_u32(mask_rows + r * words), pc + kMasksChunk <= q.w);
                }
                turn += chunks;
            }
            __syncthreads();
        }
        int run = beg;
        int2 *Trow = T + rowg * Wk;
        const bool pairs = ((rowg * Wk) & 1) == 0;   // the row's records are 16-byte aligned in twos
        // (Two windows per lane: a warp's stores are contiguous.  With four per lane each store writes half of every 32-byte sector
        // it touches: 32768 x 2048 at 10% 21.0 -> 22.7 us, 4096 x 60000 at 1% 24.7 -> 27.7, 2500 x 98304 at 1% 18.9 -> 20.6; only
        // few long runs of windows gained, 32768 x 8192 at 5% 35.0 -> 33.2.)
        if (live)
            for (int w0 = 0; w0 < Wk; w0 += WARPS * 64) {
                const int w = w0 + 2 * (SHARED ? (int)threadIdx.x : lane);
                const uint2 m = w < words ? *reinterpret_cast<const uint2 *>(mask + w) : make_uint2(0u, 0u);
                const int n0 = __popc(m.x), cnt = n0 + __popc(m.y);
                int incl = cnt;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const int t = __shfl_up_sync(kFull, incl, d);
                    if (lane >= d) incl += t;
                }
                int before = 0, all;
                if (!SHARED) {
                    all = __shfl_sync(kFull, incl, 31);
                } else {
                    if (lane == 31) warp_total[warp] = incl;
                    __syncthreads();
                    all = 0;
#pragma unroll
                    for (int i = 0; i < WARPS; ++i) {
                        const int t = warp_total[i];
                        if (i < warp) before += t;
                        all += t;
                    }
                }
                const int pos = run + before + incl - cnt;
                if (pairs && w + 1 < Wk) {
                    *reinterpret_cast<int4 *>(Trow + w) = make_int4(pos, (int)m.x, pos + n0, (int)m.y);
                } else {
                    if (w < Wk) Trow[w] = make_int2(pos, (int)m.x);
                    if (w + 1 < Wk) Trow[w + 1] = make_int2(pos + n0, (int)m.y);
                }
                run += all;
                if (SHARED) __syncthreads();   // warp_total is reused
            }
        if (row0 + (long long)gridDim.x * ROWS < rows_all) __syncthreads();   // the words and `rest` are reused
    }
    if (bad) atomicExch(&flags[kFlagUnsorted], 1);
}

// True when the workspace holds a table built from exactly these arrays.
__device__ __forceinline__ bool signature_matches(const PatternSignature &want, const PatternSignature *have)
{
    const PatternSignature h = *have;
    return h.magic == want.magic && h.M == want.M && h.K == want.K && h.Wk == want.Wk && h.nnz == want.nnz &&
           h.row_ptr == want.row_ptr && h.col_idx == want.col_idx && h.batch == want.batch &&
           h.rp_stride == want.rp_stride && h.nz_stride == want.nz_stride;
}

// ---- dense operand split ----------------------------------------------------------------------------
// X [rows x cols] (ld) -> hi, lo in a column-blocked layout: element (r, c) lives at
// ((c/32)*rows_p + r)*32 + c%32, i.e. [cols_p/32][rows_p][32] floats, zero in the padding
// (rows_p >= rows, cols_p >= cols, cols_p % 32 == 0).  One 32-float group of a row is one
// 128-byte swizzle row for TMA, and the whole thing is a plain packed 3-D tensor.
// A batch of `batch` equally sized operands, `batch_stride` elements apart, is stacked along the rows:
// [cols_p/32][batch * rows_p][32].
// bf16 operands (dtype 1) are exact in tf32: hi is the value itself and no lo copy is written.
// One launch handles up to three jobs (blockIdx.y picks the job) and, being the first kernel of
// every tile op, also clears the workspace's device status word (unless `status` is NULL: the second
// kernel of a two-phase op keeps what the first one reported).
//
// The dense-tile kernels multiply whole windows of S, positions without a stored entry included (by
// zero), so an Inf or NaN anywhere in a dense operand -- also in a row no stored entry refers to -- or a
// value so close to FLT_MAX that its tf32 hi part rounds to Inf would turn into NaN in outputs that
// Eq. 1-3 leave finite.  Every job therefore also looks at what it reads, and a job with `check_only`
// (the A operand, which the tile kernel splits itself) does nothing else: a non-finite hi part raises
// the fallback flag, and the row kernels, which touch exactly the entries the equations name, produce
// the result.
struct SplitJob {
    const void *X;
    long long ld;
    int rows, cols;
    float *hi, *lo;
    int rows_p, cols_p;
    int batch;                // operands stacked along the rows (1: a single operand)
    long long batch_stride;   // elements between consecutive operands of the batch
    int dtype;                // kDenseF32 / kDenseBf16
    int check_only;           // look for non-finite values, write nothing
};


// It also compares the signature stored beside a prepared window table with the arrays of this call
// (`chk.have` != NULL) and raises the fallback flag on a mismatch: the flags are then final before the tile
// kernel starts, which lets the gated fallback run beside it.
struct TableCheck {
    PatternSignature want;
    const PatternSignature *have;   // NULL: nothing to check (the table was built by this call)
    int *flags;
    int after_prepass;              // launched as a programmatic dependent of the pattern pre-pass of the same call:
                                    // this grid must not complete before that one (the tile kernel waits for this grid only)
};

struct SplitJobs {
    SplitJob j[2];    // operands to split (blockIdx.y picks one)
    int n;
    SplitJob check;   // a check_only job done on the side by the blocks of job 0 (no blocks of its own: the launch
    int has_check;    // stays one wave of blocks, and the tile kernel behind it waits for this grid to end)
};

__device__ __forceinline__ bool tf32_hi_not_finite(uint32_t hi) { return (hi & 0x7f800000u) == 0x7f800000u; }

// One job of split_dense_kernel, walked by the blocks (gridDim.x of them) of one blockIdx.y.  True: a non-finite hi part was seen.
__device__ __forceinline__ bool split_job(const SplitJob &j)
{
    const bool bf16 = j.dtype == kDenseBf16;
    // 16-byte loads of four fp32 (or 8-byte loads of four bf16) need the alignment for every operand of the batch
    const bool vec = (j.ld & 3) == 0 && (j.batch_stride & 3) == 0 &&
                     (reinterpret_cast<uintptr_t>(j.X) & (bf16 ? 7 : 15)) == 0;
    const long long rows_all = (long long)j.batch * j.rows_p;
    const long long groups = rows_all * (j.cols_p >> 2);  // float4 groups
    const bool small = groups < 0x7fffffffll;
    bool bad = false;
    for (long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x; g < groups;
         g += (long long)gridDim.x * blockDim.x) {
        const int q = (int)(g & 7);                 // float4 inside the 32-float group
        const long long rg = g >> 3;                // (column group, stacked row) pair
        int b, r, c;
        if (small) {   // 32-bit index arithmetic (64-bit divisions are library calls: they were most of this kernel's time)
            const unsigned rg32 = (unsigned)rg, cg = rg32 / (unsigned)rows_all, rs = rg32 - cg * (unsigned)rows_all;
            b = j.batch == 1 ? 0 : (int)(rs / (unsigned)j.rows_p);
            r = (int)(rs - (unsigned)b * (unsigned)j.rows_p);
            c = (int)cg * 32 + q * 4;
        } else {
            const long long rs = rg % rows_all;
            b = (int)(rs / j.rows_p);
            r = (int)(rs % j.rows_p);
            c = (int)(rg / rows_all) * 32 + q * 4;
        }
        uint32_t h[4] = {0, 0, 0, 0}, l[4] = {0, 0, 0, 0};
        if (r < j.rows && c < j.cols) {
            const long long at = (long long)b * j.batch_stride + (long long)r * j.ld + c;
            float x[4] = {0.f, 0.f, 0.f, 0.f};
            if (bf16) {
                const unsigned short *src = static_cast<const unsigned short *>(j.X) + at;
                if (vec && c + 3 < j.cols) {
                    const uint2 u = __ldg(reinterpret_cast<const uint2 *>(src));
                    x[0] = __uint_as_float(u.x << 16); x[1] = __uint_as_float(u.x & 0xffff0000u);
                    x[2] = __uint_as_float(u.y << 16); x[3] = __uint_as_float(u.y & 0xffff0000u);
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (c + i < j.cols) x[i] = __uint_as_float((uint32_t)__ldg(src + i) << 16);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) h[i] = __float_as_uint(x[i]);   // bf16 is exact in tf32
            } else {
                const float *src = static_cast<const float *>(j.X) + at;
                if (vec && c + 3 < j.cols) {
                    const float4 f = __ldg(reinterpret_cast<const float4 *>(src));
                    x[0] = f.x; x[1] = f.y; x[2] = f.z; x[3] = f.w;
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (c + i < j.cols) x[i] = __ldg(src + i);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) ptx::split_tf32(x[i], h[i], l[i]);
            }
            bad |= tf32_hi_not_finite(h[0]) || tf32_hi_not_finite(h[1]) || tf32_hi_not_finite(h[2]) || tf32_hi_not_finite(h[3]);
        }
        if (!j.check_only) {
            reinterpret_cast<uint4 *>(j.hi)[g] = make_uint4(h[0], h[1], h[2], h[3]);
            if (j.lo) reinterpret_cast<uint4 *>(j.lo)[g] = make_uint4(l[0], l[1], l[2], l[3]);
        }
    }
    return bad;
}

__global__ void split_dense_kernel(SplitJobs jobs, int *__restrict__ status, TableCheck chk)
{
    ptx::launch_dependents();   // the tile kernel may take its SMs; it waits for this grid before it reads anything
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) {
        if (status) *status = 0;
        if (chk.have && !signature_matches(chk.want, chk.have)) atomicExch(&chk.flags[kFlagUnsorted], 1);
    }
    bool bad = split_job(jobs.j[blockIdx.y]);
    if (jobs.has_check && blockIdx.y == 0) bad |= split_job(jobs.check);
    if (bad) atomicExch(&chk.flags[kFlagNotFinite], 1);
    if (chk.after_prepass) ptx::wait_for_primary_grid();
}

}  // namespace b2sp
