// CUDA-core "row" kernels for SPMM / SDDMM / FusedMM over CSR (sm_100a).
//
// One CTA of kRowWarps warps owns one sparse row (and one slab of output columns).  The row's
// (col_idx, values) segment is consumed in chunks of 32 entries -- the paper's VLC = 32 -- one
// entry per lane, loaded coalesced and handed round by warp shuffles.  The warps of the CTA
// take alternate chunks (the paper's "NT threads share a row's nonzeros") and, for SPMM and
// FusedMM, their partial output rows are combined through shared memory in a fixed order, so
// results are deterministic.  Rows are visited in the order given by `row_order` (longest
// first, produced by the binning kernels below) or in natural order when it is NULL.
// `clear`, when not NULL, points at the workspace's status word, which the kernel resets (a call whose only
// launch is this kernel cannot fail on the device).
// `gate`, when not NULL, points at three device words (used when the row family is only the fallback of
// the dense-tile family): the kernel does nothing if words 0 and 1 are both 0.  Word 0 says that the
// window table cannot be used and stays as it is; word 1 says that a dense operand of this call holds a
// non-finite value and is per call: the last CTA of this grid to have read it clears it (word 2 counts
// the readers), so that the next call on the workspace starts clean without a launch of its own.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "row_walk.h"

namespace b2sp {

constexpr int kRowWarps = 4;
constexpr int kRowThreads = kRowWarps * 32;
constexpr int kBuckets = 32;
constexpr unsigned kFull = 0xffffffffu;
// Longest A_i that is staged in shared memory, by the elements that a load takes.  Fewer than four mean two to four times as many
// loads, and then the few CTAs that fit on an SM beside a long A_i lose to a lane per entry (us, staged and a lane per entry, 2000 x
// 2000 at 2%: Kd = 16001 sddmm 2850 and 3520, 20001 5000 and 4500, 20002 2580 and 4320, 30002 7940 and 6510; N = 33 fusedmm 16001
// 2720 and 3630, 30001 14700 and 6680; N = 34 20002 2760 and 4160, 30002 8340 and 6260).
__host__ __device__ constexpr int max_staged_kd(int V) { return V == 4 ? 40960 : V == 2 ? 24576 : 16384; }

// ------------------------------------------------------------------------------------------
// Row binning (work assignment): counting sort of the rows by length bucket
// bucket(len) = number of significant bits of len, longest bucket first.
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ int bucket_of(int len) { return len <= 0 ? 0 : 32 - __clz(len); }

// Programmatic dependent launches: the binning kernels and the row kernel that follows them are chained so
// that each is placed, and does what does not need its predecessor's output, while the predecessor runs.
__device__ __forceinline__ void grid_release_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void grid_wait_for_primary() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// A batch of independent problems of the same sizes in one launch (FusedMM only): blockIdx.z is the problem,
// whose arrays start `*` elements after those of problem 0.  All zero for a single problem.
struct RowBatch {
    long long rp, nz, A, B, D, O;
};
struct NoBatch {};   // what a single-problem kernel takes in RowBatch's place (no parameter bytes, no arithmetic)
template <bool BATCHED> struct BatchArg { using type = NoBatch; };
template <> struct BatchArg<true> { using type = RowBatch; };

// True when a gated launch has nothing to do (see the top of this file).  Called by every thread of the CTA.
__device__ __forceinline__ bool gate_closed(int *gate)
{
    if (!gate) return false;
    __shared__ int gate_word;
    if (threadIdx.x == 0) {
        volatile int *g = gate;
        gate_word = g[0] | g[1];
        __threadfence();   // the read above is performed before this CTA is counted as a reader
        const unsigned readers = gridDim.x * gridDim.y * gridDim.z;
        if ((unsigned)atomicAdd(gate + 2, 1) == readers - 1) {
            g[2] = 0;
            g[1] = 0;
        }
    }
    __syncthreads();
    return gate_word == 0;
}

__global__ void bin_count_kernel(int M, const int *__restrict__ row_ptr, int *__restrict__ count)
{
    __shared__ int h[kBuckets];
    grid_release_dependents();
    if (threadIdx.x < kBuckets) h[threadIdx.x] = 0;
    __syncthreads();
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < (unsigned)M) atomicAdd(&h[bucket_of(row_ptr[i + 1] - row_ptr[i])], 1);
    __syncthreads();
    if (threadIdx.x < kBuckets && h[threadIdx.x]) atomicAdd(&count[threadIdx.x], h[threadIdx.x]);
}

__global__ void bin_scatter_kernel(int M, const int *__restrict__ row_ptr,
                                   const int *__restrict__ count, int *__restrict__ cursor,
                                   int *__restrict__ row_order)
{
    __shared__ int h[kBuckets];
    __shared__ int base[kBuckets];
    if (threadIdx.x < kBuckets) h[threadIdx.x] = 0;
    __syncthreads();
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
    int b = 0, r = 0;
    if (i < (unsigned)M) {
        b = bucket_of(row_ptr[i + 1] - row_ptr[i]);
        r = atomicAdd(&h[b], 1);
    }
    __syncthreads();
    grid_wait_for_primary();     // the counts of the whole matrix (bin_count_kernel)
    grid_release_dependents();   // the row kernel behind this one waits for this grid before it reads the order
    if (threadIdx.x < kBuckets) {
        int mine = threadIdx.x, start = 0;
        for (int j = kBuckets - 1; j > mine; --j) start += count[j];
        base[mine] = h[mine] ? start + atomicAdd(&cursor[mine], h[mine]) : 0;
    }
    __syncthreads();
    if (i < (unsigned)M) row_order[base[b] + r] = (int)i;
}

// ------------------------------------------------------------------------------------------
// helpers
// ------------------------------------------------------------------------------------------
// Dense operands are fp32 or bfloat16 (DT below); sums and outputs are always fp32.  A bf16 value is the top
// half of the fp32 value it stands for, so widening it is exact.
struct bf16_t { unsigned short bits; };
__device__ __forceinline__ float4 ldg4(const float *p) { return __ldg(reinterpret_cast<const float4 *>(p)); }
__device__ __forceinline__ float4 ldg4(const bf16_t *p)   // four consecutive elements, 8-byte aligned
{
    const uint2 u = __ldg(reinterpret_cast<const uint2 *>(p));
    return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u),
                       __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xffff0000u));
}
__device__ __forceinline__ float2 ldg2(const float *p) { return __ldg(reinterpret_cast<const float2 *>(p)); }
__device__ __forceinline__ float2 ldg2(const bf16_t *p)   // two consecutive elements, 4-byte aligned
{
    const unsigned u = __ldg(reinterpret_cast<const unsigned *>(p));
    return make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u));
}
__device__ __forceinline__ float ldg1(const float *p) { return __ldg(p); }
__device__ __forceinline__ float ldg1(const bf16_t *p)
{
    return __uint_as_float((uint32_t)__ldg(reinterpret_cast<const unsigned short *>(p)) << 16);
}


// V consecutive elements of a dense row, widened to fp32: what a lane loads, multiplies and stores at a time.  V = 4 where
// every row of every operand begins on a four-element boundary and has whole groups of four, V = 2 where that holds for
// pairs, V = 1 for any width, leading dimension and address.
template <int V> struct alignas(4 * V) VecF { float e[V]; };
template <int V, typename DT>
__device__ __forceinline__ VecF<V> ldgv(const DT *p)
{
    VecF<V> r;
    if constexpr (V == 4) {
        const float4 f = ldg4(p);
        r.e[0] = f.x; r.e[1] = f.y; r.e[2] = f.z; r.e[3] = f.w;
    } else if constexpr (V == 2) {
        const float2 f = ldg2(p);
        r.e[0] = f.x; r.e[1] = f.y;
    } else {
        r.e[0] = ldg1(p);
    }
    return r;
}

template <int V>
__device__ __forceinline__ void fma_v(VecF<V> &acc, float s, const VecF<V> &v)
{
#pragma unroll
    for (int i = 0; i < V; ++i) acc.e[i] = fmaf(s, v.e[i], acc.e[i]);
}

template <int V>
__device__ __forceinline__ float dot_v(const VecF<V> &a, const VecF<V> &b, float acc)
{
#pragma unroll
    for (int i = 0; i < V; ++i) acc = fmaf(a.e[i], b.e[i], acc);
    return acc;
}

// Geometry of the SPMM sweep.  SPLIT sub-warps of LPN = 32/SPLIT lanes each take alternate
// entries of a chunk; a lane owns U groups of V columns: col0 + (sl + LPN*u)*V.
template <int V, int U, int SPLIT>
struct SweepGeom {
    static constexpr int LPN = 32 / SPLIT;
    static constexpr int SLAB = LPN * V * U;
};

// Two forms of the row kernels.  Short rows are cut into a chunk for each warp, and their partial chunks, which is all they
// have, keep several entries' loads in flight.  That takes registers and a chunk length known at run time only, which long rows
// pay for and have no use for: their form has chunks of 32 and the plainest loops for what is left of a row.  Where both are
// instantiated the host chooses by the average row length (short_rows in b2sp_api.cu).

// One chunk (up to 32 entries, lane l holds entry l: column k, scalar s) of the Alg. 2 SAXPY
// sweep.  SRC(j) gives the lane that holds entry j's scalar.
template <int V, int U, int SPLIT, bool PERMUTED, bool SHORT, typename DT>
__device__ __forceinline__ void saxpy_chunk(VecF<V> (&acc)[U], int k, float s, int cnt,
                                            const DT *__restrict__ Dcol, int64_t ldd,
                                            bool (&live)[U], int sub)
{
    constexpr int LPN = 32 / SPLIT;
    constexpr int STEPS = 32 / SPLIT;
    if (cnt == 32) {
#pragma unroll 8
        for (int jj = 0; jj < STEPS; ++jj) {
            int j = jj * SPLIT + sub;
            int src = PERMUTED ? ((j & 3) * 8 + (j >> 2)) : j;
            int kk = __shfl_sync(kFull, k, j);
            float ss = __shfl_sync(kFull, s, src);
            const DT *d = Dcol + (int64_t)kk * ldd;
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (live[u]) fma_v<V>(acc[u], ss, ldgv<V>(d + u * LPN * V));
        }
    } else if constexpr (SHORT) {
        // Entries whose loads are in flight together.  It is a matter of registers, which the full chunks then miss, and was
        // measured: single or pair elements four (two: 1501 x 2903 x 71 spmm 24.8 -> 27.5 us); SPMM with whole warps two (one:
        // power law 8192 x 8192 at 10% x 256 382 -> 442 us), but one with four groups per lane (two: 77 registers instead of 62,
        // 1024 x 1024 at 25% x 512 29.5 -> 38.5 us, 8192 x 8192 at 30% 1.68 -> 1.74 ms); FusedMM and sub-warps one (two: power law
        // 8192 x 8192 at 10% x 64 spmm 156 -> 205 us, 8192 x 8192 at 5%, Kd = N = 32, fusedmm 90 -> 97 us).
        constexpr int BATCH = V < 4 ? 4 : !PERMUTED && SPLIT == 1 && U < 4 ? 2 : 1;
        for (int jj = 0; jj * SPLIT < cnt; jj += BATCH) {
            VecF<V> d[BATCH][U];
            float ss[BATCH];
#pragma unroll
            for (int i = 0; i < BATCH; ++i) {
                const int j = (jj + i) * SPLIT + sub;
                const int src = PERMUTED ? ((j & 3) * 8 + (j >> 2)) : j;
                const int kk = __shfl_sync(kFull, k, j & 31);
                ss[i] = __shfl_sync(kFull, s, src & 31);
                const DT *p = Dcol + (int64_t)kk * ldd;
#pragma unroll
                for (int u = 0; u < U; ++u) d[i][u] = j < cnt && live[u] ? ldgv<V>(p + u * LPN * V) : VecF<V>{};
            }
#pragma unroll
            for (int i = 0; i < BATCH; ++i)
                if ((jj + i) * SPLIT + sub < cnt) {
#pragma unroll
                    for (int u = 0; u < U; ++u) fma_v<V>(acc[u], ss[i], d[i][u]);
                }
        }
    } else {
        for (int jj = 0; jj < STEPS; ++jj) {
            const int j = jj * SPLIT + sub;
            const int src = PERMUTED ? ((j & 3) * 8 + (j >> 2)) : j;
            const int kk = __shfl_sync(kFull, k, j);
            const float ss = __shfl_sync(kFull, s, src);
            if (j < cnt) {
                const DT *d = Dcol + (int64_t)kk * ldd;
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (live[u]) fma_v<V>(acc[u], ss, ldgv<V>(d + u * LPN * V));
            }
        }
    }
}

// Entries of a row that a warp takes at a time: 32; in the form for short rows a quarter of a row of 64 or fewer, rounded up to
// groups of four (those of sddmm_chunk), so that the four warps share it: a row of 25 entries was one warp's serial chain while
// three idled (256 x 256 at 10%, Kd = N = 64, fusedmm: 7.1 -> 4.0 us; 4096 x 512 at 5%, Kd = 100, N = 250: 66 -> 32 us).  Between
// 65 and about 110 entries the warps' parts are uneven (65: 32, 32, 1 and 0); with the line at 128 instead, rows of 102 lost their
// full chunks' eight loads in flight (3072 x 1024 x 32 spmm 7.1 -> 7.5 us).
template <bool SHORT>
__device__ __forceinline__ int chunk_of(int len) { return !SHORT || len > 64 ? 32 : ((len + 4 * kRowWarps - 1) / (4 * kRowWarps)) * 4; }

// Combine the sub-warps of a warp, then the warps of the CTA (fixed order), and store the row.
template <int V, int U, int SPLIT>
__device__ __forceinline__ void reduce_and_store_row(VecF<V> (&acc)[U], VecF<V> *red, int warp,
                                                     int lane, float *__restrict__ Orow,
                                                     bool (&live)[U])
{
    constexpr int LPN = 32 / SPLIT;
#pragma unroll
    for (int off = 16; off >= LPN; off >>= 1) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
#pragma unroll
            for (int i = 0; i < V; ++i) acc[u].e[i] += __shfl_xor_sync(kFull, acc[u].e[i], off);
        }
    }
    if (lane < LPN) {
#pragma unroll
        for (int u = 0; u < U; ++u) red[(warp * U + u) * LPN + lane] = acc[u];
    }
    __syncthreads();
    if (warp == 0 && lane < LPN) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (!live[u]) continue;
            VecF<V> r = red[u * LPN + lane];
#pragma unroll
            for (int w = 1; w < kRowWarps; ++w) {
                const VecF<V> t = red[(w * U + u) * LPN + lane];
#pragma unroll
                for (int i = 0; i < V; ++i) r.e[i] += t.e[i];
            }
            *reinterpret_cast<VecF<V> *>(Orow + u * LPN * V) = r;
        }
    }
}

// ------------------------------------------------------------------------------------------
// SPMM  (Alg. 2; N, ldd, ldo multiples of V, D and O aligned to V elements)
// ------------------------------------------------------------------------------------------
template <int V, int U, int SPLIT, bool SHORT, typename DT>
__global__ void __launch_bounds__(kRowThreads)
spmm_row_kernel(int N, const int *__restrict__ row_ptr, const int *__restrict__ col_idx,
                const float *__restrict__ values, const DT *__restrict__ D, int64_t ldd,
                float *__restrict__ O, int64_t ldo, const int *__restrict__ row_order,
                int *__restrict__ gate, int nrows, int *__restrict__ clear)
{
    using G = SweepGeom<V, U, SPLIT>;
    __shared__ VecF<V> red[kRowWarps * U * G::LPN];
    if (gate_closed(gate)) return;
    if (clear && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *clear = 0;
    if (row_order) grid_wait_for_primary();   // launched behind the binning pass: its row order
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int sub = lane / G::LPN, sl = lane % G::LPN;
    for (BlockRows br(blockIdx.x, nrows, gridDim.x); br.more(); br.advance()) {
        const int row = row_order ? row_order[br.row] : (int)br.row;
        const int col0 = blockIdx.y * G::SLAB + sl * V;
        bool live[U];
        VecF<V> acc[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            live[u] = col0 + u * G::LPN * V < N;
            acc[u] = VecF<V>{};
        }
        const int beg = row_ptr[row], end = row_ptr[row + 1];
        const DT *Dcol = D + col0;
        // the next chunk's indices and values are fetched before the current chunk is consumed
        // (the role of the paper's prefetch of the next ja/avalues block)
        int k = 0;
        float s = 0.f;
        const int chunk = chunk_of<SHORT>(end - beg);
        RowChunks rc(beg, end, warp, kRowWarps, chunk);
        {
            const unsigned p = rc.at + lane;
            if (p < rc.end) {
                k = __ldg(col_idx + p);
                s = __ldg(values + p);
            }
        }
        for (; rc.more(); rc.advance()) {
            const unsigned pn = rc.next(lane);
            int kn = 0;
            float sn = 0.f;
            if (pn < rc.end) {
                kn = __ldg(col_idx + pn);
                sn = __ldg(values + pn);
            }
            saxpy_chunk<V, U, SPLIT, false, SHORT, DT>(acc, k, s, rc.count(), Dcol, ldd, live, sub);
            k = kn;
            s = sn;
        }
        reduce_and_store_row<V, U, SPLIT>(acc, red, warp, lane, O + (int64_t)row * ldo + col0, live);
        __syncthreads();   // shared memory is reused by the next row
    }
}

// ------------------------------------------------------------------------------------------
// SDDMM  (Alg. 1; Kd, lda, ldb multiples of V, A and B aligned to V elements)
//
// A group of 8 lanes computes one sampled dot product: lane t of the group owns elements
// (t + 8u)*V .. +V-1 of the Kd-vector.  KU > 0: A_i is held in KU groups of registers per lane
// (Kd <= 8*V*KU).  KU == 0: any Kd, A_i staged in shared memory.  In a chunk of 32 entries,
// group g takes entries 4r + g (r = 0..7); after the 3-step butterfly every lane of the
// group has the sum and lane t keeps round t's, so lane 8g + t ends up holding entry 4t + g.
// ------------------------------------------------------------------------------------------
template <int V, int KU, bool SHORT, bool FUSED, typename DT>
__device__ __forceinline__ float sddmm_chunk(const VecF<V> (&areg)[KU > 0 ? KU : 1],
                                             const float *__restrict__ a_smem, int Kd, int k,
                                             const DT *__restrict__ B, int64_t ldb, int lane, int cnt)
{
    const int g = lane >> 3, t = lane & 7;
    float mine = 0.f;
    auto keep = [&](int r, float part) {
        part += __shfl_xor_sync(kFull, part, 1);
        part += __shfl_xor_sync(kFull, part, 2);
        part += __shfl_xor_sync(kFull, part, 4);
        if (r == t) mine = part;
    };
    if constexpr (KU == 0) {
        // Long dot products: R rounds go through the elements together, so that their loads are in flight at the same time and
        // A_i is read from shared memory once for all of them.  Round after round, with whatever loads the compiler then kept in
        // flight: 300 x 300 at 20%, Kd = 8000 sddmm 272 us, now 125; 4000 x 500 at 30%, Kd = 1024 230 and 149; with the elements
        // unrolled by two instead of four 144 and 157.
        auto rounds = [&](auto count, int r) {
            constexpr int R = decltype(count)::value;
            const DT *b[R];
            float part[R];
#pragma unroll
            for (int i = 0; i < R; ++i) {
                b[i] = B + (int64_t)__shfl_sync(kFull, k, 4 * (r + i) + g) * ldb;
                part[i] = 0.f;
            }
#pragma unroll 4
            for (int e = t * V; e < Kd; e += 8 * V) {
                const VecF<V> a = *reinterpret_cast<const VecF<V> *>(a_smem + e);
#pragma unroll
                for (int i = 0; i < R; ++i) part[i] = dot_v<V>(a, ldgv<V>(b[i] + e), part[i]);
            }
#pragma unroll
            for (int i = 0; i < R; ++i) keep(r + i, part[i]);
        };
        const int all = (cnt + 3) >> 2;
        int r = 0;
        for (; r + 4 <= all; r += 4) rounds(std::integral_constant<int, 4>(), r);
        for (; r + 2 <= all; r += 2) rounds(std::integral_constant<int, 2>(), r);
        if (r < all) rounds(std::integral_constant<int, 1>(), r);
    } else {
        auto round = [&](int r) {
            const int kq = __shfl_sync(kFull, k, 4 * r + g);
            const DT *b = B + (int64_t)kq * ldb + t * V;
            float part = 0.f;
#pragma unroll
            for (int u = 0; u < KU; ++u)
                if ((t + 8 * u) * V < Kd) part = dot_v<V>(areg[u], ldgv<V>(b + u * 8 * V), part);
            keep(r, part);
        };
        if constexpr (!SHORT) {   // (rounds behind the end of the row read row 0 of B)
#pragma unroll 4
            for (int r = 0; r < 8; ++r) round(r);
        } else if constexpr (!FUSED && KU == 8 && sizeof(DT) == 4) {
            // four rounds at a time and no second loop: with it 128 < Kd <= 256 took longer than with eight rounds for every chunk,
            // this way less (4096 x 1024 at 20%, Kd = 256: 73.0, 68.2 and 59.9 us; rows of 40 entries: 19.1, 34.9 and 20.9)
#pragma unroll 1
            for (int r0 = 0; 4 * r0 < cnt; r0 += 4) {
#pragma unroll
                for (int r = 0; r < 4; ++r) round(r0 + r);
            }
        } else if (cnt == 32) {
#pragma unroll 4
            for (int r = 0; r < 8; ++r) round(r);
        } else {   // (one loop for both, its length known only at run time, cost full chunks a quarter of their speed)
#pragma unroll 2
            for (int r = 0; r < (cnt + 3) >> 2; ++r) round(r);
        }
    }
    return mine;  // lane 8g+t: dot product of entry 4t+g
}

template <int V, int KU, typename DT>
__device__ __forceinline__ void load_a_row(VecF<V> (&areg)[KU > 0 ? KU : 1], float *a_smem,
                                           const DT *__restrict__ Arow, int Kd, int lane)
{
    if (KU > 0) {
        const int t = lane & 7;
#pragma unroll
        for (int u = 0; u < (KU > 0 ? KU : 1); ++u)
            areg[u] = (t + 8 * u) * V < Kd ? ldgv<V>(Arow + (t + 8 * u) * V) : VecF<V>{};
    } else {
        for (int e = threadIdx.x * V; e < Kd; e += kRowThreads * V)
            *reinterpret_cast<VecF<V> *>(a_smem + e) = ldgv<V>(Arow + e);
        __syncthreads();
    }
}

template <int V, int KU, bool SHORT, typename DT>
__global__ void __launch_bounds__(kRowThreads)
sddmm_row_kernel(int Kd, const int *__restrict__ row_ptr, const int *__restrict__ col_idx,
                 const float *s_values, const DT *__restrict__ A, int64_t lda,
                 const DT *__restrict__ B, int64_t ldb, float *out_values,
                 const int *__restrict__ row_order, int *__restrict__ gate, int nrows, int *__restrict__ clear)
{
    extern __shared__ float4 dyn_smem[];
    float *a_smem = reinterpret_cast<float *>(dyn_smem);
    if (gate_closed(gate)) return;
    if (clear && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *clear = 0;
    if (row_order) grid_wait_for_primary();   // launched behind the binning pass: its row order
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (BlockRows br(blockIdx.x, nrows, gridDim.x); br.more(); br.advance()) {
        const int row = row_order ? row_order[br.row] : (int)br.row;
        const int beg = row_ptr[row], end = row_ptr[row + 1];
        VecF<V> areg[KU > 0 ? KU : 1];
        load_a_row<V, KU, DT>(areg, a_smem, A + (int64_t)row * lda, Kd, lane);
        const int slot = (lane & 7) * 4 + (lane >> 3);  // entry of the chunk this lane ends up holding
        const int chunk = chunk_of<SHORT>(end - beg);
        for (RowChunks rc(beg, end, warp, kRowWarps, chunk); rc.more(); rc.advance()) {
            const unsigned p = rc.at + lane;
            int k = p < rc.end ? __ldg(col_idx + p) : 0;
            const int cnt = rc.count();
            float dp = sddmm_chunk<V, KU, SHORT, false, DT>(areg, a_smem, Kd, k, B, ldb, lane, cnt);
            const unsigned q = rc.at + slot;
            if (slot < cnt) out_values[q] = s_values ? s_values[q] * dp : dp;
        }
        __syncthreads();   // shared memory is reused by the next row
    }
}

// Kd too long for A_i in shared memory (max_staged_kd): one lane per entry, serial dot product.
template <typename DT>
__global__ void __launch_bounds__(kRowThreads)
sddmm_row_scalar_kernel(int Kd, const int *__restrict__ row_ptr, const int *__restrict__ col_idx,
                        const float *s_values, const DT *__restrict__ A, int64_t lda,
                        const DT *__restrict__ B, int64_t ldb, float *out_values,
                        const int *__restrict__ row_order, int *__restrict__ gate, int nrows, int *__restrict__ clear)
{
    if (gate_closed(gate)) return;
    if (clear && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *clear = 0;
    if (row_order) grid_wait_for_primary();   // launched behind the binning pass: its row order
    for (BlockRows br(blockIdx.x, nrows, gridDim.x); br.more(); br.advance()) {
        const int row = row_order ? row_order[br.row] : (int)br.row;
        const int beg = row_ptr[row], end = row_ptr[row + 1];
        const DT *a = A + (int64_t)row * lda;
        for (unsigned p = beg + threadIdx.x; p < (unsigned)end; p += kRowThreads) {
            const DT *b = B + (int64_t)__ldg(col_idx + p) * ldb;
            float dp = 0.f;
            for (int l = 0; l < Kd; ++l) dp = fmaf(ldg1(a + l), ldg1(b + l), dp);
            out_values[p] = s_values ? s_values[p] * dp : dp;
        }
        __syncthreads();   // shared memory is reused by the next row
    }
}

// ------------------------------------------------------------------------------------------
// FusedMM  (Alg. 3): per chunk, the SDDMM values stay in registers (one per lane) and are the
// scalars of the SAXPY sweep over the same staged column indices; C never reaches memory.
// ------------------------------------------------------------------------------------------
template <int V, int KU, int U, int SPLIT, bool SHORT, bool BATCHED, typename DT>
__global__ void __launch_bounds__(kRowThreads)
fusedmm_row_kernel(int Kd, int N, const int *__restrict__ row_ptr, const int *__restrict__ col_idx,
                   const float *__restrict__ s_values, const DT *__restrict__ A, int64_t lda,
                   const DT *__restrict__ B, int64_t ldb, const DT *__restrict__ D,
                   int64_t ldd, float *__restrict__ O, int64_t ldo,
                   const int *__restrict__ row_order, int *__restrict__ gate, int nrows, int *__restrict__ clear,
                   typename BatchArg<BATCHED>::type batch)
{
    using G = SweepGeom<V, U, SPLIT>;
    extern __shared__ float4 dyn_smem[];
    if (gate_closed(gate)) return;
    if constexpr (BATCHED) {   // this problem's arrays
        const long long pb = blockIdx.z;
        row_ptr += pb * batch.rp; col_idx += pb * batch.nz; if (s_values) s_values += pb * batch.nz;
        A += pb * batch.A; B += pb * batch.B; D += pb * batch.D; O += pb * batch.O;
    }
    if (clear && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *clear = 0;
    if (row_order) grid_wait_for_primary();   // launched behind the binning pass: its row order
    VecF<V> *red = reinterpret_cast<VecF<V> *>(dyn_smem);                // kRowWarps*U*LPN
    float *a_smem = reinterpret_cast<float *>(red + kRowWarps * U * G::LPN);  // Kd (KU == 0)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int sub = lane / G::LPN, sl = lane % G::LPN;
    for (BlockRows br(blockIdx.x, nrows, gridDim.x); br.more(); br.advance()) {
        const int row = row_order ? row_order[br.row] : (int)br.row;
        const int col0 = blockIdx.y * G::SLAB + sl * V;
        bool live[U];
        VecF<V> acc[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            live[u] = col0 + u * G::LPN * V < N;
            acc[u] = VecF<V>{};
        }
        const int beg = row_ptr[row], end = row_ptr[row + 1];
        VecF<V> areg[KU > 0 ? KU : 1];
        load_a_row<V, KU, DT>(areg, a_smem, A + (int64_t)row * lda, Kd, lane);
        const int slot = (lane & 7) * 4 + (lane >> 3);
        const DT *Dcol = D + col0;
        int k = 0;
        float sv = 1.f;
        const int chunk = chunk_of<SHORT>(end - beg);
        RowChunks rc(beg, end, warp, kRowWarps, chunk);
        {
            const unsigned p = rc.at + lane, q = rc.at + slot;
            if (p < rc.end) k = __ldg(col_idx + p);
            if (s_values && q < rc.end) sv = __ldg(s_values + q);
        }
        for (; rc.more(); rc.advance()) {
            const unsigned pn = rc.next(lane), qn = rc.next(slot);
            // (the same test in two ways: with the first the long form for 64 < Kd <= 128 spilled a register on bfloat16, 102 -> 116 us
            // at 450 entries a row; with the second it did for Kd = N = 32, 48.6 -> 51.3 us)
            constexpr bool BY_COUNT = !SHORT && KU >= 4;
            const bool has_p = BY_COUNT ? lane < rc.behind() : pn < rc.end, has_q = BY_COUNT ? slot < rc.behind() : qn < rc.end;
            int kn = has_p ? __ldg(col_idx + pn) : 0;
            float svn = (s_values && has_q) ? __ldg(s_values + qn) : 1.f;
            const int cnt = rc.count();
            float cv = sv * sddmm_chunk<V, KU, SHORT, true, DT>(areg, a_smem, Kd, k, B, ldb, lane, cnt);
            saxpy_chunk<V, U, SPLIT, true, SHORT, DT>(acc, k, cv, cnt, Dcol, ldd, live, sub);
            k = kn;
            sv = svn;
        }
        reduce_and_store_row<V, U, SPLIT>(acc, red, warp, lane, O + (int64_t)row * ldo + col0, live);
        __syncthreads();   // shared memory is reused by the next row
    }
}

// Kd too long for A_i in shared memory: lane-per-entry dot products, then a scalar sweep.
template <typename DT>
__global__ void __launch_bounds__(kRowThreads)
fusedmm_row_scalar_kernel(int Kd, int N, const int *__restrict__ row_ptr,
                          const int *__restrict__ col_idx, const float *__restrict__ s_values,
                          const DT *__restrict__ A, int64_t lda, const DT *__restrict__ B,
                          int64_t ldb, const DT *__restrict__ D, int64_t ldd,
                          float *__restrict__ O, int64_t ldo, const int *__restrict__ row_order,
                          int *__restrict__ gate, int nrows, int *__restrict__ clear, RowBatch batch)
{
    __shared__ float red[kRowWarps][128];
    if (gate_closed(gate)) return;
    {   // this problem's arrays
        const long long pb = blockIdx.z;
        row_ptr += pb * batch.rp; col_idx += pb * batch.nz; if (s_values) s_values += pb * batch.nz;
        A += pb * batch.A; B += pb * batch.B; D += pb * batch.D; O += pb * batch.O;
    }
    if (clear && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *clear = 0;
    if (row_order) grid_wait_for_primary();   // launched behind the binning pass: its row order
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (BlockRows br(blockIdx.x, nrows, gridDim.x); br.more(); br.advance()) {
        const int row = row_order ? row_order[br.row] : (int)br.row;
        const int col0 = blockIdx.y * 128 + lane;
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        const int beg = row_ptr[row], end = row_ptr[row + 1];
        const DT *a = A + (int64_t)row * lda;
        for (RowChunks rc(beg, end, warp, kRowWarps, 32); rc.more(); rc.advance()) {
            const unsigned p = rc.at + lane;
            int k = 0;
            float cv = 0.f;
            if (p < rc.end) {
                k = __ldg(col_idx + p);
                const DT *b = B + (int64_t)k * ldb;
                for (int l = 0; l < Kd; ++l) cv = fmaf(ldg1(a + l), ldg1(b + l), cv);
                if (s_values) cv *= __ldg(s_values + p);
            }
            const int cnt = rc.count();
            for (int j = 0; j < cnt; ++j) {
                int kk = __shfl_sync(kFull, k, j);
                float ss = __shfl_sync(kFull, cv, j);
                const DT *d = D + (int64_t)kk * ldd + col0;
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (col0 + 32 * u < N) acc[u] = fmaf(ss, ldg1(d + 32 * u), acc[u]);
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) red[warp][lane + 32 * u] = acc[u];
        __syncthreads();
        if (warp == 0) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (col0 + 32 * u >= N) continue;
                float r = red[0][lane + 32 * u];
                for (int w = 1; w < kRowWarps; ++w) r += red[w][lane + 32 * u];
                O[(int64_t)row * ldo + col0 + 32 * u] = r;
            }
        }
        __syncthreads();   // shared memory is reused by the next row
    }
}

// ------------------------------------------------------------------------------------------
// CSR validation (debug helper)
// ------------------------------------------------------------------------------------------
__global__ void validate_csr_kernel(int M, int K, long long nnz, const int *__restrict__ row_ptr,
                                    const int *__restrict__ col_idx, int *__restrict__ flag)
{
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    long long stride = (long long)gridDim.x * blockDim.x;
    bool bad = false;
    if (i == 0) bad |= row_ptr[0] != 0 || (long long)row_ptr[M] != nnz;
    for (long long r = i; r < M; r += stride) bad |= row_ptr[r + 1] < row_ptr[r];
    for (long long p = i; p < nnz; p += stride) {
        int c = col_idx[p];
        bad |= c < 0 || c >= K;
    }
    if (bad) atomicExch(flag, 1);
}

}  // namespace b2sp
