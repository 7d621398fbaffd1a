// C-ABI entry points of libb2sp: argument checks, workspace carving, kernel dispatch.
// See include/b2sp.h (and include/b2sp_debug.h) for the contract of every function.
#include "../../include/b2sp_debug.h"

#include <algorithm>
#include <climits>
#include <cstdlib>
#include <cstdint>
#include <mutex>
#include <type_traits>

#include "row_kernels.cuh"
#include "tile_dispatch.h"

namespace b2sp {

// ---- workspace layout ---------------------------------------------------------------------
// [0, 128)    int count[32]      row-length histogram            (zeroed per call)
// [128, 256)  int cursor[32]     scatter cursors                 (zeroed per call)
// [256, 512)  int status[64]     status[0] = device status word, status[1] = validate flag
// [512, ...)  int row_order[M]   rows, longest bucket first
constexpr size_t kHeaderBytes = 512;

inline size_t align256(size_t x) { return (x + 255) & ~size_t(255); }
inline size_t row_workspace_bytes(int M) { return align256(kHeaderBytes + sizeof(int) * (size_t)M); }

struct Workspace {
    int *count, *cursor, *status, *row_order;
};

inline Workspace carve(void *ws)
{
    char *b = static_cast<char *>(ws);
    Workspace w;
    w.count = reinterpret_cast<int *>(b);
    w.cursor = reinterpret_cast<int *>(b + 128);
    w.status = reinterpret_cast<int *>(b + 256);
    w.row_order = reinterpret_cast<int *>(b + kHeaderBytes);
    return w;
}

thread_local int g_last_algo[3] = {-1, -1, -1};
thread_local int g_last_launches[3] = {0, 0, 0};

// The most elements (4, 2 or 1) that may be loaded at a time from a row-major operand of this width: every row begins on such
// a boundary and has whole groups of them.
template <typename DT> inline int vec_width(const DT *p, int width, int64_t ld, int64_t batch_stride = 0)
{
    const int64_t odd = (int64_t)(reinterpret_cast<uintptr_t>(p) / sizeof(DT)) | width | ld | batch_stride;
    return (odd & 3) == 0 ? 4 : (odd & 1) == 0 ? 2 : 1;
}
template <typename DT> constexpr int dense_dtype() { return sizeof(DT) == 2 ? kDenseBf16 : kDenseF32; }

inline b2sp_status check_launch()
{
    return cudaGetLastError() == cudaSuccess ? B2SP_OK : B2SP_ERR_CUDA;
}

b2sp_status check_workspace(void *ws, size_t have, size_t need)
{
    if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255) != 0 || have < need) return B2SP_ERR_WORKSPACE;
    return B2SP_OK;
}

// Enqueue the binning pass; returns the row order pointer (NULL for natural order).
b2sp_status bin_rows(int M, const int *row_ptr, const Workspace &w, cudaStream_t st, int *launches)
{
    if (cudaMemsetAsync(w.count, 0, 512, st) != cudaSuccess) return B2SP_ERR_CUDA;
    const unsigned blocks = ((unsigned)M + 255u) / 256u;
    bin_count_kernel<<<blocks, 256, 0, st>>>(M, row_ptr, w.count);
    {   // a programmatic dependent of the counting kernel (it waits for the counts where it needs them)
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(blocks);
        cfg.blockDim = dim3(256);
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        cudaLaunchKernelEx(&cfg, bin_scatter_kernel, M, row_ptr, (const int *)w.count, w.cursor, w.row_order);
    }
    *launches += 2;
    return check_launch();
}

// Launches `kern`; a gated launch (the row family as the dense-tile family's device-side fallback) is marked as a
// programmatic dependent of the tile kernel before it: the tile kernel lets its dependents go as soon
// as it has read the gate's flags, which are final before it starts, so the fallback (which almost always
// finds its gate closed and exits) runs beside the tile kernel instead of after it.  A launch behind the binning
// pass (`order` given) is a programmatic dependent of it too: the kernel waits for the row order at its top.
template <class... KArgs, class... Args>
inline void launch_row(void (*kern)(KArgs...), dim3 grid, size_t smem, cudaStream_t st, bool dependent, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(kRowThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = dependent ? attr : nullptr;
    cfg.numAttrs = dependent ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kern, KArgs(args)...);
}

// A gated launch (the row family as the dense-tile family's fallback) almost always finds its gate
// closed: it gets a small grid whose blocks walk the rows, so that the usual case costs little.
inline unsigned gated_blocks(unsigned rows, int *gate, unsigned nbatch = 1)
{
    unsigned cap = 148u * 4u / (nbatch ? nbatch : 1);   // (every CTA of a gated grid counts itself at the gate: keep them few)
    if (cap < 16u) cap = 16u;
    return gate && rows > cap ? cap : rows;
}

template <int V, int U, int SPLIT, bool SHORT, typename DT>
void launch_spmm(dim3 grid, cudaStream_t st, int N, const int *row_ptr, const int *col_idx,
                 const float *values, const DT *D, int64_t ldd, float *O, int64_t ldo,
                 const int *order, int *gate, int *clear)
{
    const int nrows = (int)grid.x;
    grid.x = gated_blocks(grid.x, gate);
    launch_row(spmm_row_kernel<V, U, SPLIT, SHORT, DT>, grid, 0, st, gate != nullptr || order != nullptr, N, row_ptr, col_idx, values, D, ldd, O, ldo, order,
               gate, nrows, clear);
}

// Column geometry for a width N: U groups of V columns per lane, SPLIT sub-warps.
// (V < 4, rows that are not aligned groups of four: loads of two or one elements are two to four times as many, but even the
// single ones beat a lane per dot product: 1501 x 2903 at 12%, fusedmm Kd = 51, N = 71 68 -> 42 us, Kd = 50, N = 70 71 -> 37 us,
// on the device alone.  SPMM with 65 to 128 columns and 100 to 350 entries a row is 4% to 6% slower: x 70 23.6 -> 24.8 us.)
struct Geom { int U, SPLIT, slab; };
inline Geom pick_geom(int N, int V)
{
    if (V == 4) {
        if (N <= 32) return {1, 4, 32};
        if (N <= 64) return {1, 2, 64};
        if (N <= 128) return {1, 1, 128};
        if (N <= 256) return {2, 1, 256};
        return {4, 1, 512};
    }
    if (V == 2) {
        if (N <= 32) return {1, 2, 32};
        if (N <= 64) return {1, 1, 64};
        return {2, 1, 128};
    }
    if (N <= 16) return {1, 2, 16};
    if (N <= 32) return {1, 1, 32};
    if (N <= 64) return {2, 1, 64};
    return {4, 1, 128};
}

// Register groups of A_i per lane (0: A_i in shared memory).
inline int pick_ku(int Kd, int V)
{
    if (Kd <= 64) return 8 / V;
    if (Kd <= 128) return 16 / V;
    return V == 4 && Kd <= 256 ? 8 : 0;
}

// Where the form of a row kernel for long rows exists (see row_kernels.cuh), and up to which average row length the form for short
// rows is chosen beside it.  Measured over 40 to 1600 entries a row (4096 rows), us of the short and the long form; every width
// that is missing here is served better, or as well, by the form for short rows over the whole range.
template <int V, int U, int SPLIT> constexpr bool spmm_has_long() { return V == 4 && (SPLIT == 2 || U >= 2); }
template <int V, int KU, typename DT> constexpr bool sddmm_has_long() { return V == 4 && (KU == 2 || (KU == 8 && sizeof(DT) == 2)); }
// (The kernels for batches are others, and so are their registers: four problems of 3877 x 3877 at 267 entries a row, fp32, short and
// long, Kd = N = 64 151 / 168 us, Kd = 128, N = 512 650 / 736, Kd = N = 256 500 / 706.)
template <int V, int KU, int U, int SPLIT, bool BATCHED, typename DT> constexpr bool fused_has_long()
{
    constexpr bool F32 = sizeof(DT) == 4;
    return V == 4 && (KU == 2 ? U <= 2 && !(BATCHED && F32 && SPLIT == 2)
                      : KU == 4 ? SPLIT == 1 && !(BATCHED && F32 && U == 4) : KU == 8 && U == 2 && F32 && !BATCHED);
}
inline bool short_rows(long long nnz, int M, int entries) { return nnz <= (long long)entries * M; }
// x 64: 130 entries 15.0 / 15.3, 300 27.3 / 26.0; power law 8192 x 8192 at 10% 156 / 134.  x 256: 130 entries 31.9 / 33.3, 205
// 46.3 / 44.8, 1600 314 / 300, but with less than a wave of rows the loads in flight are worth more (300 x 4096, 614 entries: 26.6 /
// 30.2).  x 512: 40 entries 24.0 / 32.7, 80 39.7 / 39.8; bf16 60 entries 30.0 / 29.0, 205 71.8 / 67.9.
template <int U, int SPLIT> inline bool spmm_short(long long nnz, int M)
{
    return short_rows(nnz, M, U == 4 ? 72 : 144) || (U == 2 && M < 148 * 10);
}
// Kd = 64: 100 entries 12.4 / 12.7, 130 15.5 / 15.1; bf16 Kd = 256: 100 35.8 / 36.8, 205 64.0 / 62.5.
inline bool sddmm_short(long long nnz, int M) { return short_rows(nnz, M, 128); }
// Kd = N = 64: 130 entries 27.2 / 30.3, 205 38.2 / 37.2, 1600 224 / 207; Kd = N = 128: 60 28.4 / 35.5, 100 36.8 / 36.5, 205 63.8 / 58.8,
// 1600 382 / 333 (1024 x 1024 at 20%: 25.8 / 18.6); Kd = 128, N = 256: 130 54.5 / 58.5, 205 77.5 / 75.0.  Rows of 128 bytes or less:
// Kd = N = 32: 60 13.5 / 14.8, 80 15.6 / 15.2, 450 52.8 / 48.6; bf16 Kd = N = 64: 60 17.4 / 17.8, 100 20.5 / 19.6, 900 128 / 113.
template <typename DT> inline bool fused_short(long long nnz, int M, int N) { return short_rows(nnz, M, N * (int)sizeof(DT) <= 128 ? 72 : 144); }

template <int V, int KU, bool SHORT, typename DT>
void launch_sddmm(dim3 grid, cudaStream_t st, int Kd, const int *row_ptr, const int *col_idx,
                  const float *sv, const DT *A, int64_t lda, const DT *B, int64_t ldb,
                  float *out, const int *order, int *gate, int *clear)
{
    size_t smem = KU == 0 ? sizeof(float) * (size_t)((Kd + 3) & ~3) : 0;
    const int nrows = (int)grid.x;
    grid.x = gated_blocks(grid.x, gate);
    launch_row(sddmm_row_kernel<V, KU, SHORT, DT>, grid, smem, st, gate != nullptr || order != nullptr, Kd, row_ptr, col_idx, sv, A, lda, B, ldb, out, order,
               gate, nrows, clear);
}

template <int V, int KU, int U, int SPLIT, bool SHORT, typename DT>
b2sp_status launch_fused(dim3 grid, cudaStream_t st, int Kd, int N, const int *row_ptr,
                         const int *col_idx, const float *sv, const DT *A, int64_t lda,
                         const DT *B, int64_t ldb, const DT *D, int64_t ldd, float *O,
                         int64_t ldo, const int *order, int *gate, int *clear, const RowBatch &rb)
{
    size_t smem = sizeof(VecF<V>) * kRowWarps * U * (32 / SPLIT) +
                  (KU == 0 ? sizeof(float) * (size_t)((Kd + 3) & ~3) : 0);
    const bool batched = grid.z > 1;
    auto kern_b = fusedmm_row_kernel<V, KU, U, SPLIT, SHORT, true, DT>;
    auto kern_1 = fusedmm_row_kernel<V, KU, U, SPLIT, SHORT, false, DT>;
    if (smem > 48 * 1024) {
        if (smem > 200 * 1024) return B2SP_ERR_UNSUPPORTED;
        if (cudaFuncSetAttribute(batched ? reinterpret_cast<const void *>(kern_b) : reinterpret_cast<const void *>(kern_1),
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
            return B2SP_ERR_CUDA;
    }
    const int nrows = (int)grid.x;
    grid.x = gated_blocks(grid.x, gate, grid.z);
    if (batched)
        launch_row(kern_b, grid, smem, st, gate != nullptr || order != nullptr, Kd, N, row_ptr, col_idx, sv, A, lda, B, ldb, D, ldd, O, ldo,
                   order, gate, nrows, clear, rb);
    else
        launch_row(kern_1, grid, smem, st, gate != nullptr || order != nullptr, Kd, N, row_ptr, col_idx, sv, A, lda, B, ldb, D, ldd, O, ldo,
                   order, gate, nrows, clear, NoBatch{});
    return B2SP_OK;
}

template <int V, int KU, int U, int SPLIT, typename DT, class... Args>
b2sp_status launch_fused_form(bool is_short, dim3 grid, Args... args)
{
    constexpr bool one = fused_has_long<V, KU, U, SPLIT, false, DT>(), many = fused_has_long<V, KU, U, SPLIT, true, DT>();
    if constexpr (one || many) {
        if (!is_short && (grid.z > 1 ? many : one)) return launch_fused<V, KU, U, SPLIT, false, DT>(grid, args...);
    }
    return launch_fused<V, KU, U, SPLIT, true, DT>(grid, args...);
}

template <int V, int KU, typename DT, class... Args>
b2sp_status dispatch_fused_geom(const Geom &g, Args... args)
{
    if constexpr (V == 4) {
        if (g.SPLIT == 4) return launch_fused_form<V, KU, 1, 4, DT>(args...);
    }
    if (g.SPLIT == 2) return launch_fused_form<V, KU, 1, 2, DT>(args...);
    if (g.U == 1) return launch_fused_form<V, KU, 1, 1, DT>(args...);
    if constexpr (V == 2) return launch_fused_form<V, KU, 2, 1, DT>(args...);
    else if (g.U == 2) return launch_fused_form<V, KU, 2, 1, DT>(args...);
    else return launch_fused_form<V, KU, 4, 1, DT>(args...);
}

// `args`: is_short and launch_fused's.
template <int V, typename DT, class... Args>
b2sp_status dispatch_fused_ku(const Geom &g, int Kd, Args... args)
{
    const int ku = pick_ku(Kd, V);
    if (ku == 8 / V) return dispatch_fused_geom<V, 8 / V, DT>(g, args...);
    if (ku == 16 / V) return dispatch_fused_geom<V, 16 / V, DT>(g, args...);
    if constexpr (V == 4) {
        if (ku == 8) return dispatch_fused_geom<V, 8, DT>(g, args...);
    }
    return dispatch_fused_geom<V, 0, DT>(g, args...);
}

b2sp_status zero_rows(float *O, int64_t ldo, int M, int N, cudaStream_t st)
{
    if (M == 0 || N == 0) return B2SP_OK;
    return cudaMemset2DAsync(O, sizeof(float) * (size_t)ldo, 0, sizeof(float) * (size_t)N, (size_t)M,
                             st) == cudaSuccess
               ? B2SP_OK
               : B2SP_ERR_CUDA;
}

bool bad_csr_args(int M, int K, long long nnz, const int *row_ptr, const int *col_idx)
{
    if (M < 0 || K < 0 || nnz < 0 || nnz > (long long)INT_MAX) return true;
    if (M > 0 && !row_ptr) return true;
    if (nnz > 0 && (!col_idx || K == 0 || M == 0)) return true;
    return false;
}

}  // namespace b2sp

using namespace b2sp;

extern "C" int b2sp_version(void) { return 100; }

extern "C" const char *b2sp_status_string(b2sp_status s)
{
    switch (s) {
    case B2SP_OK: return "ok";
    case B2SP_ERR_INVALID_ARG: return "invalid argument";
    case B2SP_ERR_UNSUPPORTED: return "unsupported for these arguments";
    case B2SP_ERR_BAD_CSR: return "malformed CSR";
    case B2SP_ERR_CUDA: return "CUDA error";
    case B2SP_ERR_WORKSPACE: return "workspace missing, misaligned or too small";
    case B2SP_ERR_TIMEOUT: return "device-side wait timed out";
    case B2SP_ERR_TOO_LARGE: return "problem exceeds the library's built-in scratch array";
    }
    return "unknown status";
}

// The FusedMM tile kernel owns one 128-column tile of O and recomputes S (.) A B^T for each of them
// (tensor memory holds O, P, P' and A for one tile only).  Past two tiles that costs more than
// writing the sampled values once: measured at N = 512 on the 8192^2 / 30% workload, 717 us fused
// against 134 + 430 us for SDDMM into a scratch C and SPMM on C.  So wide outputs take the two
// phases inside one call (same window table, same fallback), and C lives in the workspace.
// With two tiles (128 < N <= 256) the line was drawn on an earlier fused kernel (N = 256, Kd = 128, two phases against fused: 8192^2
// 315 against 342 us).  With the kernels of today the two phases are the slower form at most sizes they are taken at, bfloat16 operands
// above all: 8192^2 at 30% 344 against 322 us (bfloat16 297 against 239), 16384 x 2048 at 30% 189 against 169 (177 / 137), 4096 x 8192 181
// against 165 (167 / 132), 32768 x 1024 234 against 200 (215 / 164), 32768 x 4096 at 20% 684 against 651 (566 / 470); only without stored
// values at 16384 x 8192 are they equal (577 / 581).  Below the line: 4096^2 92 against 85, 8192 x 4096 at Kd = 64 156 against 122, 2048^2 46
// against 33.
static bool fusedmm_two_phase(int M, int K, int Kd, int N)
{
    return N > 256 || (N > 128 && Kd > 64 && (double)M * (double)K >= 3.0e7);
}

// Workspace of the dense-tile family for an op (0: these sizes are outside the family).
static size_t tile_workspace_bytes(int op, int M, int K, int Kd, int N, long long nnz, size_t row_bytes)
{
    FusedPlan p = op == B2SP_OP_SPMM    ? plan_fused_tile(M, K, 0, N, nnz, row_bytes, true)
                  : op == B2SP_OP_SDDMM ? plan_fused_tile(M, K, Kd, 0, nnz, row_bytes, false)
                                        : plan_fused_tile(M, K, Kd, N, nnz, row_bytes, true);
    if (!p.feasible) return 0;
    if (op == B2SP_OP_FUSEDMM && fusedmm_two_phase(M, K, Kd, N)) {
        TwoPhasePlan t = plan_two_phase(M, K, Kd, N, nnz, row_bytes);
        if (t.feasible && t.bytes > p.bytes) return t.bytes;
    }
    return p.bytes;
}

static int tile_width(int op, int Kd, int N) { return op == B2SP_OP_SPMM ? N : op == B2SP_OP_SDDMM ? Kd : (Kd < N ? Kd : N); }

extern "C" size_t b2sp_workspace_bytes_algo(int op, int algo, int M, int K, int Kd, int N, long long nnz)
{
    if (op < 0 || op > 2 || M < 0 || K < 0 || Kd < 0 || N < 0 || nnz < 0) return 0;
    if (algo < B2SP_ALGO_AUTO || algo > B2SP_ALGO_TILE_PREPARED) return 0;
    const size_t rows = row_workspace_bytes(M);
    if (algo == B2SP_ALGO_ROW || algo == B2SP_ALGO_ROW_NAT) return rows;
    const size_t tile = tile_workspace_bytes(op, M, K, Kd, N, nnz, rows);
    if (algo == B2SP_ALGO_TILE || algo == B2SP_ALGO_TILE_PREPARED) return tile;
    return tile > rows && tile_profitable(op, M, K, tile_width(op, Kd, N), nnz) ? tile : rows;
}

extern "C" size_t b2sp_workspace_bytes(int op, int M, int K, int Kd, int N, long long nnz)
{
    if (op < 0 || op > 2 || M < 0 || K < 0 || Kd < 0 || N < 0 || nnz < 0) return 0;
    const size_t rows = row_workspace_bytes(M);
    const size_t tile = tile_workspace_bytes(op, M, K, Kd, N, nnz, rows);
    return tile > rows ? tile : rows;
}

extern "C" int b2sp_last_algo(int op) { return op >= 0 && op < 3 ? g_last_algo[op] : -1; }
extern "C" int b2sp_last_launches(int op) { return op >= 0 && op < 3 ? g_last_launches[op] : 0; }

// The row family under AUTO: the binning pass (two small launches, ~10 us) orders the rows longest
// first, which only pays when the CTAs of the row kernel need several waves on the GPU.
static int auto_row_algo(int M) { return M <= 4096 ? B2SP_ALGO_ROW_NAT : B2SP_ALGO_ROW; }

// Enqueues the row-family SPMM.  `gate` != NULL makes it a device-side fallback.
template <typename DT>
static b2sp_status spmm_rows(int M, int N, long long nnz, const int *row_ptr, const int *col_idx, const float *values,
                             const DT *D, long long ldd, float *O, long long ldo, const int *order,
                             int *gate, int *clear, cudaStream_t st)
{
    const int V = std::min(vec_width(D, N, ldd), vec_width(O, N, ldo));
    const Geom g = pick_geom(N, V);
    dim3 grid((unsigned)M, (unsigned)((N + g.slab - 1) / g.slab));
    auto launch = [&](auto v, auto u, auto split) {
        constexpr int V_ = decltype(v)::value, U_ = decltype(u)::value, S_ = decltype(split)::value;
        if constexpr (spmm_has_long<V_, U_, S_>()) {
            if (!spmm_short<U_, S_>(nnz, M)) {
                launch_spmm<V_, U_, S_, false, DT>(grid, st, N, row_ptr, col_idx, values, D, ldd, O, ldo, order, gate, clear);
                return;
            }
        }
        launch_spmm<V_, U_, S_, true, DT>(grid, st, N, row_ptr, col_idx, values, D, ldd, O, ldo, order, gate, clear);
    };
#define B2SP_S(V_, U_, S_) launch(std::integral_constant<int, V_>(), std::integral_constant<int, U_>(), std::integral_constant<int, S_>())
    if (V == 4) {
        if (g.SPLIT == 4) B2SP_S(4, 1, 4);
        else if (g.SPLIT == 2) B2SP_S(4, 1, 2);
        else if (g.U == 1) B2SP_S(4, 1, 1);
        else if (g.U == 2) B2SP_S(4, 2, 1);
        else B2SP_S(4, 4, 1);
    } else if (V == 2) {
        if (g.SPLIT == 2) B2SP_S(2, 1, 2);
        else if (g.U == 1) B2SP_S(2, 1, 1);
        else B2SP_S(2, 2, 1);
    } else {
        if (g.SPLIT == 2) B2SP_S(1, 1, 2);
        else if (g.U == 1) B2SP_S(1, 1, 1);
        else if (g.U == 2) B2SP_S(1, 2, 1);
        else B2SP_S(1, 4, 1);
    }
#undef B2SP_S
    return check_launch();
}

template <typename DT>
static b2sp_status spmm_impl(int M, int K, int N, long long nnz, const int *row_ptr, const int *col_idx,
                             const float *values, const DT *D, long long ldd, float *O, long long ldo,
                             void *workspace, size_t workspace_bytes, int algo, void *stream)
{
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (bad_csr_args(M, K, nnz, row_ptr, col_idx) || N < 0) return B2SP_ERR_INVALID_ARG;
    if (algo < B2SP_ALGO_AUTO || algo > B2SP_ALGO_TILE_PREPARED) return B2SP_ERR_INVALID_ARG;
    const bool prepared = algo == B2SP_ALGO_TILE_PREPARED;
    if (prepared) algo = B2SP_ALGO_TILE;
    if (M > 0 && N > 0 && (!O || ldo < N)) return B2SP_ERR_INVALID_ARG;
    if (nnz > 0 && N > 0 && (!values || !D || ldd < N)) return B2SP_ERR_INVALID_ARG;
    const size_t row_bytes = row_workspace_bytes(M);
    b2sp_status rc = check_workspace(workspace, workspace_bytes, row_bytes);
    if (rc != B2SP_OK) return rc;
    FusedPlan plan;   // SPMM runs through the FusedMM tile pipeline with P' = the stored values (Kd = 0)
    if (algo == B2SP_ALGO_TILE || (algo == B2SP_ALGO_AUTO && tile_profitable(B2SP_OP_SPMM, M, K, N, nnz)))
        plan = plan_fused_tile(M, K, 0, N, nnz, row_bytes, true);
    int use = algo == B2SP_ALGO_AUTO ? auto_row_algo(M) : algo;
    if (plan.feasible && workspace_bytes >= plan.bytes) use = B2SP_ALGO_TILE;
    else if (algo == B2SP_ALGO_TILE) return plan.feasible ? B2SP_ERR_WORKSPACE : B2SP_ERR_UNSUPPORTED;
    g_last_algo[B2SP_OP_SPMM] = use;
    int launches = 0;
    g_last_launches[B2SP_OP_SPMM] = 0;
    if (M == 0 || N == 0) return B2SP_OK;
    if (nnz == 0) return zero_rows(O, ldo, M, N, st);

    Workspace w = carve(workspace);
    if (use == B2SP_ALGO_TILE) {
        rc = fused_tile(plan, prepared, 2, M, K, 0, N, nnz, row_ptr, col_idx, values, nullptr, 0, nullptr, 0, D, ldd,
                        O, ldo, workspace, st, &launches, false, BatchDesc(), dense_dtype<DT>());
        if (rc != B2SP_OK) return rc;
        // device-side fallback: runs only if the pre-pass found rows that are not strictly sorted
        int *gate = reinterpret_cast<int *>(static_cast<char *>(workspace) + kWsTileFlagsOffset);
        rc = spmm_rows(M, N, nnz, row_ptr, col_idx, values, D, ldd, O, ldo, nullptr, gate, nullptr, st);
        g_last_launches[B2SP_OP_SPMM] = launches + 1;
        return rc;
    }
    const int *order = nullptr;
    int *clear = nullptr;
    if (use == B2SP_ALGO_ROW) {
        rc = bin_rows(M, row_ptr, w, st, &launches);
        if (rc != B2SP_OK) return rc;
        order = w.row_order;
    } else {   // no binning pass: the row kernel itself resets the status word
        clear = reinterpret_cast<int *>(static_cast<char *>(workspace) + kWsStatusOffset);
    }
    rc = spmm_rows(M, N, nnz, row_ptr, col_idx, values, D, ldd, O, ldo, order, nullptr, clear, st);
    g_last_launches[B2SP_OP_SPMM] = launches + 1;
    return rc;
}

// Picks the SDDMM kernel that holds A_i for this Kd.
template <int V, typename DT>
static b2sp_status dispatch_sddmm_ku(bool is_short, dim3 grid, cudaStream_t st, int Kd, const int *row_ptr, const int *col_idx, const float *s_values,
                                     const DT *A, long long lda, const DT *B, long long ldb, float *out_values, const int *order,
                                     int *gate, int *clear)
{
    const int ku = pick_ku(Kd, V);
#define B2SP_C(KU_, SHORT_) launch_sddmm<V, KU_, SHORT_, DT>(grid, st, Kd, row_ptr, col_idx, s_values, A, lda, B, ldb, out_values, order, gate, clear)
    auto launch = [&](auto groups) {
        constexpr int KU = decltype(groups)::value;
        if constexpr (sddmm_has_long<V, KU, DT>()) {
            if (!is_short) { B2SP_C(KU, false); return; }
        }
        B2SP_C(KU, true);
    };
    if (ku == 8 / V) { launch(std::integral_constant<int, 8 / V>()); return B2SP_OK; }
    if (ku == 16 / V) { launch(std::integral_constant<int, 16 / V>()); return B2SP_OK; }
    if constexpr (V == 4) {
        if (ku == 8) { launch(std::integral_constant<int, 8>()); return B2SP_OK; }
    }
    const size_t smem = sizeof(float) * (size_t)((Kd + 3) & ~3);
    if (smem > 48 * 1024 &&
        cudaFuncSetAttribute(sddmm_row_kernel<V, 0, true, DT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return B2SP_ERR_CUDA;
    B2SP_C(0, true);
#undef B2SP_C
    return B2SP_OK;
}

// Enqueues the row-family SDDMM.  `gate` != NULL makes it a device-side fallback.
template <typename DT>
static b2sp_status sddmm_rows(int M, int Kd, long long nnz, const int *row_ptr, const int *col_idx, const float *s_values,
                              const DT *A, long long lda, const DT *B, long long ldb,
                              float *out_values, const int *order, int *gate, int *clear, cudaStream_t st)
{
    dim3 grid((unsigned)M);
    const int V = std::min(vec_width(A, Kd, lda), vec_width(B, Kd, ldb));
    if (Kd > max_staged_kd(V)) {
        grid.x = gated_blocks(grid.x, gate);
        launch_row(sddmm_row_scalar_kernel<DT>, grid, 0, st, gate != nullptr || order != nullptr, Kd, row_ptr, col_idx, s_values, A, lda, B, ldb,
                   out_values, order, gate, M, clear);
        return check_launch();
    }
    const b2sp_status rc =
        V == 4 ? dispatch_sddmm_ku<4, DT>(sddmm_short(nnz, M), grid, st, Kd, row_ptr, col_idx, s_values, A, lda, B, ldb, out_values, order, gate, clear)
        : V == 2 ? dispatch_sddmm_ku<2, DT>(sddmm_short(nnz, M), grid, st, Kd, row_ptr, col_idx, s_values, A, lda, B, ldb, out_values, order, gate, clear)
                 : dispatch_sddmm_ku<1, DT>(sddmm_short(nnz, M), grid, st, Kd, row_ptr, col_idx, s_values, A, lda, B, ldb, out_values, order, gate, clear);
    if (rc != B2SP_OK) return rc;
    return check_launch();
}

template <typename DT>
static b2sp_status sddmm_impl(int M, int K, int Kd, long long nnz, const int *row_ptr, const int *col_idx,
                              const float *s_values, const DT *A, long long lda, const DT *B,
                              long long ldb, float *out_values, void *workspace, size_t workspace_bytes,
                              int algo, void *stream)
{
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (bad_csr_args(M, K, nnz, row_ptr, col_idx) || Kd < 0) return B2SP_ERR_INVALID_ARG;
    if (algo < B2SP_ALGO_AUTO || algo > B2SP_ALGO_TILE_PREPARED) return B2SP_ERR_INVALID_ARG;
    const bool prepared = algo == B2SP_ALGO_TILE_PREPARED;
    if (prepared) algo = B2SP_ALGO_TILE;
    if (nnz > 0 && !out_values) return B2SP_ERR_INVALID_ARG;
    if (nnz > 0 && Kd > 0 && (!A || !B || lda < Kd || ldb < Kd)) return B2SP_ERR_INVALID_ARG;
    const size_t row_bytes = row_workspace_bytes(M);
    b2sp_status rc = check_workspace(workspace, workspace_bytes, row_bytes);
    if (rc != B2SP_OK) return rc;
    FusedPlan plan;
    if (algo == B2SP_ALGO_TILE || (algo == B2SP_ALGO_AUTO && tile_profitable(B2SP_OP_SDDMM, M, K, Kd, nnz)))
        plan = plan_fused_tile(M, K, Kd, 0, nnz, row_bytes, false);
    int use = algo == B2SP_ALGO_AUTO ? auto_row_algo(M) : algo;
    if (plan.feasible && workspace_bytes >= plan.bytes) use = B2SP_ALGO_TILE;
    else if (algo == B2SP_ALGO_TILE) return plan.feasible ? B2SP_ERR_WORKSPACE : B2SP_ERR_UNSUPPORTED;
    g_last_algo[B2SP_OP_SDDMM] = use;
    int launches = 0;
    g_last_launches[B2SP_OP_SDDMM] = 0;
    if (M == 0 || nnz == 0) return B2SP_OK;
    if (Kd == 0)
        return cudaMemsetAsync(out_values, 0, sizeof(float) * (size_t)nnz, st) == cudaSuccess
                   ? B2SP_OK
                   : B2SP_ERR_CUDA;

    Workspace w = carve(workspace);
    if (use == B2SP_ALGO_TILE) {
        rc = fused_tile(plan, prepared, 0, M, K, Kd, 0, nnz, row_ptr, col_idx, s_values, A, lda, B, ldb, nullptr, 0,
                        out_values, 0, workspace, st, &launches, false, BatchDesc(), dense_dtype<DT>());
        if (rc != B2SP_OK) return rc;
        int *gate = reinterpret_cast<int *>(static_cast<char *>(workspace) + kWsTileFlagsOffset);
        rc = sddmm_rows(M, Kd, nnz, row_ptr, col_idx, s_values, A, lda, B, ldb, out_values, nullptr, gate, nullptr, st);
        g_last_launches[B2SP_OP_SDDMM] = launches + 1;
        return rc;
    }
    const int *order = nullptr;
    int *clear = nullptr;
    if (use == B2SP_ALGO_ROW) {
        rc = bin_rows(M, row_ptr, w, st, &launches);
        if (rc != B2SP_OK) return rc;
        order = w.row_order;
    } else {   // no binning pass: the row kernel itself resets the status word
        clear = reinterpret_cast<int *>(static_cast<char *>(workspace) + kWsStatusOffset);
    }
    rc = sddmm_rows(M, Kd, nnz, row_ptr, col_idx, s_values, A, lda, B, ldb, out_values, order, nullptr, clear, st);
    g_last_launches[B2SP_OP_SDDMM] = launches + 1;
    return rc;
}

// Enqueues the row-family FusedMM.  `gate` != NULL makes it a device-side fallback.
template <typename DT>
static b2sp_status fused_rows(int M, int Kd, int N, long long nnz, const int *row_ptr, const int *col_idx,
                              const float *s_values, const DT *A, long long lda, const DT *B,
                              long long ldb, const DT *D, long long ldd, float *O, long long ldo,
                              const int *order, int *gate, int *clear, cudaStream_t st,
                              int nbatch = 1, const RowBatch &rb = RowBatch{0, 0, 0, 0, 0, 0})
{
    b2sp_status rc = B2SP_OK;
    const int V = std::min({vec_width(A, Kd, lda, rb.A), vec_width(B, Kd, ldb, rb.B), vec_width(D, N, ldd, rb.D), vec_width(O, N, ldo, rb.O)});
    if (Kd > max_staged_kd(V)) {
        dim3 grid(gated_blocks((unsigned)M, gate, (unsigned)nbatch), (unsigned)((N + 127) / 128), (unsigned)nbatch);
        launch_row(fusedmm_row_scalar_kernel<DT>, grid, 0, st, gate != nullptr || order != nullptr, Kd, N, row_ptr, col_idx, s_values, A, lda, B, ldb,
                   D, ldd, O, ldo, order, gate, M, clear, rb);
        return check_launch();
    }
    const Geom g = pick_geom(N, V);
    dim3 grid((unsigned)M, (unsigned)((N + g.slab - 1) / g.slab), (unsigned)nbatch);
    const bool is_short = fused_short<DT>(nnz, M, N);
    rc = V == 4 ? dispatch_fused_ku<4, DT>(g, Kd, is_short, grid, st, Kd, N, row_ptr, col_idx, s_values, A, lda, B, ldb, D, ldd, O, ldo, order, gate, clear, rb)
         : V == 2 ? dispatch_fused_ku<2, DT>(g, Kd, is_short, grid, st, Kd, N, row_ptr, col_idx, s_values, A, lda, B, ldb, D, ldd, O, ldo, order, gate, clear, rb)
                  : dispatch_fused_ku<1, DT>(g, Kd, is_short, grid, st, Kd, N, row_ptr, col_idx, s_values, A, lda, B, ldb, D, ldd, O, ldo, order, gate, clear, rb);
    if (rc != B2SP_OK) return rc;
    return check_launch();
}

template <typename DT>
static b2sp_status fusedmm_impl(int M, int K, int Kd, int N, long long nnz, const int *row_ptr,
                                const int *col_idx, const float *s_values, const DT *A, long long lda,
                                const DT *B, long long ldb, const DT *D, long long ldd, float *O,
                                long long ldo, void *workspace, size_t workspace_bytes, int algo,
                                void *stream)
{
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (bad_csr_args(M, K, nnz, row_ptr, col_idx) || Kd < 0 || N < 0) return B2SP_ERR_INVALID_ARG;
    if (algo < B2SP_ALGO_AUTO || algo > B2SP_ALGO_TILE_PREPARED) return B2SP_ERR_INVALID_ARG;
    const bool prepared = algo == B2SP_ALGO_TILE_PREPARED;
    if (prepared) algo = B2SP_ALGO_TILE;
    if (M > 0 && N > 0 && (!O || ldo < N)) return B2SP_ERR_INVALID_ARG;
    if (nnz > 0 && N > 0 && (!D || ldd < N)) return B2SP_ERR_INVALID_ARG;
    if (nnz > 0 && N > 0 && Kd > 0 && (!A || !B || lda < Kd || ldb < Kd)) return B2SP_ERR_INVALID_ARG;
    const size_t row_bytes = row_workspace_bytes(M);
    b2sp_status rc = check_workspace(workspace, workspace_bytes, row_bytes);
    if (rc != B2SP_OK) return rc;
    FusedPlan plan;
    if (algo == B2SP_ALGO_TILE || (algo == B2SP_ALGO_AUTO && tile_profitable(B2SP_OP_FUSEDMM, M, K, Kd < N ? Kd : N, nnz)))
        plan = plan_fused_tile(M, K, Kd, N, nnz, row_bytes, true);
    int use = algo == B2SP_ALGO_AUTO ? auto_row_algo(M) : algo;
    if (plan.feasible && workspace_bytes >= plan.bytes) use = B2SP_ALGO_TILE;
    else if (algo == B2SP_ALGO_TILE) return plan.feasible ? B2SP_ERR_WORKSPACE : B2SP_ERR_UNSUPPORTED;
    g_last_algo[B2SP_OP_FUSEDMM] = use;
    int launches = 0;
    g_last_launches[B2SP_OP_FUSEDMM] = 0;
    if (M == 0 || N == 0) return B2SP_OK;
    if (nnz == 0 || Kd == 0) return zero_rows(O, ldo, M, N, st);  // empty dot products are 0

    Workspace w = carve(workspace);
    if (use == B2SP_ALGO_TILE) {
        TwoPhasePlan two;
        if (fusedmm_two_phase(M, K, Kd, N)) two = plan_two_phase(M, K, Kd, N, nnz, row_bytes);
        if (two.feasible && workspace_bytes >= two.bytes) {
            float *C = reinterpret_cast<float *>(static_cast<char *>(workspace) + two.off_c);
            rc = fused_tile(two.sddmm, prepared, 0, M, K, Kd, 0, nnz, row_ptr, col_idx, s_values, A, lda, B, ldb, nullptr, 0,
                            C, 0, workspace, st, &launches, false, BatchDesc(), dense_dtype<DT>());
            if (rc != B2SP_OK) return rc;
            rc = fused_tile(two.spmm, true, 2, M, K, 0, N, nnz, row_ptr, col_idx, C, nullptr, 0, nullptr, 0, D, ldd, O, ldo,
                            workspace, st, &launches, /*keep_status=*/true, BatchDesc(), dense_dtype<DT>());
        } else {
            rc = fused_tile(plan, prepared, 1, M, K, Kd, N, nnz, row_ptr, col_idx, s_values, A, lda, B, ldb, D, ldd, O, ldo,
                            workspace, st, &launches, false, BatchDesc(), dense_dtype<DT>());
        }
        if (rc != B2SP_OK) return rc;
        int *gate = reinterpret_cast<int *>(static_cast<char *>(workspace) + kWsTileFlagsOffset);
        rc = fused_rows(M, Kd, N, nnz, row_ptr, col_idx, s_values, A, lda, B, ldb, D, ldd, O, ldo, nullptr, gate, nullptr, st);
        g_last_launches[B2SP_OP_FUSEDMM] = launches + 1;
        return rc;
    }
    const int *order = nullptr;
    int *clear = nullptr;
    if (use == B2SP_ALGO_ROW) {
        rc = bin_rows(M, row_ptr, w, st, &launches);
        if (rc != B2SP_OK) return rc;
        order = w.row_order;
    } else {   // no binning pass: the row kernel itself resets the status word
        clear = reinterpret_cast<int *>(static_cast<char *>(workspace) + kWsStatusOffset);
    }
    rc = fused_rows(M, Kd, N, nnz, row_ptr, col_idx, s_values, A, lda, B, ldb, D, ldd, O, ldo, order, nullptr, clear, st);
    g_last_launches[B2SP_OP_FUSEDMM] = launches + 1;
    return rc;
}

// ---- the entry points: fp32 and bfloat16 dense operands -------------------------------------------------
extern "C" b2sp_status b2sp_spmm(int M, int K, int N, long long nnz, const int *row_ptr, const int *col_idx,
                                 const float *values, const float *D, long long ldd, float *O, long long ldo,
                                 void *workspace, size_t workspace_bytes, int algo, void *stream)
{
    return spmm_impl<float>(M, K, N, nnz, row_ptr, col_idx, values, D, ldd, O, ldo, workspace, workspace_bytes, algo, stream);
}
extern "C" b2sp_status b2sp_sddmm(int M, int K, int Kd, long long nnz, const int *row_ptr, const int *col_idx,
                                  const float *s_values, const float *A, long long lda, const float *B,
                                  long long ldb, float *out_values, void *workspace, size_t workspace_bytes,
                                  int algo, void *stream)
{
    return sddmm_impl<float>(M, K, Kd, nnz, row_ptr, col_idx, s_values, A, lda, B, ldb, out_values, workspace,
                             workspace_bytes, algo, stream);
}
extern "C" b2sp_status b2sp_fusedmm(int M, int K, int Kd, int N, long long nnz, const int *row_ptr,
                                    const int *col_idx, const float *s_values, const float *A, long long lda,
                                    const float *B, long long ldb, const float *D, long long ldd, float *O,
                                    long long ldo, void *workspace, size_t workspace_bytes, int algo,
                                    void *stream)
{
    return fusedmm_impl<float>(M, K, Kd, N, nnz, row_ptr, col_idx, s_values, A, lda, B, ldb, D, ldd, O, ldo, workspace,
                               workspace_bytes, algo, stream);
}
extern "C" b2sp_status b2sp_spmm_bf16(int M, int K, int N, long long nnz, const int *row_ptr, const int *col_idx,
                                      const float *values, const void *D, long long ldd, float *O, long long ldo,
                                      void *workspace, size_t workspace_bytes, int algo, void *stream)
{
    return spmm_impl<bf16_t>(M, K, N, nnz, row_ptr, col_idx, values, static_cast<const bf16_t *>(D), ldd, O, ldo,
                             workspace, workspace_bytes, algo, stream);
}
extern "C" b2sp_status b2sp_sddmm_bf16(int M, int K, int Kd, long long nnz, const int *row_ptr, const int *col_idx,
                                       const float *s_values, const void *A, long long lda, const void *B,
                                       long long ldb, float *out_values, void *workspace, size_t workspace_bytes,
                                       int algo, void *stream)
{
    return sddmm_impl<bf16_t>(M, K, Kd, nnz, row_ptr, col_idx, s_values, static_cast<const bf16_t *>(A), lda,
                              static_cast<const bf16_t *>(B), ldb, out_values, workspace, workspace_bytes, algo, stream);
}
extern "C" b2sp_status b2sp_fusedmm_bf16(int M, int K, int Kd, int N, long long nnz, const int *row_ptr,
                                         const int *col_idx, const float *s_values, const void *A, long long lda,
                                         const void *B, long long ldb, const void *D, long long ldd, float *O,
                                         long long ldo, void *workspace, size_t workspace_bytes, int algo,
                                         void *stream)
{
    return fusedmm_impl<bf16_t>(M, K, Kd, N, nnz, row_ptr, col_idx, s_values, static_cast<const bf16_t *>(A), lda,
                                static_cast<const bf16_t *>(B), ldb, static_cast<const bf16_t *>(D), ldd, O, ldo,
                                workspace, workspace_bytes, algo, stream);
}

// ---- batched FusedMM --------------------------------------------------------------------------------
namespace {

bool bad_batch_args(int batch, int M, int K, long long nnz_stride, const int *row_ptr, long long row_ptr_stride,
                    const int *col_idx)
{
    if (batch < 1 || M < 0 || K < 0 || nnz_stride < 0 || nnz_stride > (long long)INT_MAX) return true;
    if (M > 0 && !row_ptr) return true;
    if (row_ptr_stride != 0 && row_ptr_stride < (long long)M + 1) return true;
    if (nnz_stride > 0 && (!col_idx || K == 0 || M == 0)) return true;
    return false;
}

FusedPlan plan_batched(int batch, int M, int K, int Kd, int N, long long nnz_stride)
{
    if (N > 256) return FusedPlan();   // wide outputs: not on the dense-tile family in a batch
    return plan_fused_tile(M, K, Kd, N, nnz_stride, row_workspace_bytes(M), true, batch);
}

}  // namespace

extern "C" size_t b2sp_workspace_bytes_batched(int batch, int M, int K, int Kd, int N, long long nnz_stride)
{
    if (batch < 1 || M < 0 || K < 0 || Kd < 0 || N < 0 || nnz_stride < 0) return 0;
    const size_t rows = row_workspace_bytes(M);
    const FusedPlan p = plan_batched(batch, M, K, Kd, N, nnz_stride);
    return p.feasible && p.bytes > rows ? p.bytes : rows;
}

extern "C" b2sp_status b2sp_prepare_pattern_batched(int batch, int M, int K, long long nnz_stride, const int *row_ptr,
                                         long long row_ptr_stride, const int *col_idx, void *workspace,
                                         size_t workspace_bytes, void *stream)
{
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (bad_batch_args(batch, M, K, nnz_stride, row_ptr, row_ptr_stride, col_idx) || M == 0 || K == 0 || nnz_stride == 0)
        return B2SP_ERR_INVALID_ARG;
    const size_t need = pattern_table_offset(M) + pattern_table_bytes(M, K, batch);
    b2sp_status rc = check_workspace(workspace, workspace_bytes, need);
    if (rc != B2SP_OK) return rc;
    int launches = 0;
    BatchDesc bd;
    bd.count = batch; bd.rp = row_ptr_stride; bd.nz = row_ptr_stride == 0 ? 0 : nnz_stride;   // a shared pattern
    return pattern_pass(false, M, K, nnz_stride, row_ptr, col_idx, workspace, st, &launches, bd);
}

template <typename DT>
static b2sp_status fusedmm_batched_impl(int batch, int M, int K, int Kd, int N, long long nnz_stride,
                                        const int *row_ptr, long long row_ptr_stride, const int *col_idx,
                                        const float *s_values, const DT *A, long long lda, long long stride_a,
                                        const DT *B, long long ldb, long long stride_b, const DT *D, long long ldd,
                                        long long stride_d, float *O, long long ldo, long long stride_o, void *workspace,
                                        size_t workspace_bytes, int algo, void *stream)
{
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (bad_batch_args(batch, M, K, nnz_stride, row_ptr, row_ptr_stride, col_idx) || Kd < 0 || N < 0)
        return B2SP_ERR_INVALID_ARG;
    if (algo < B2SP_ALGO_AUTO || algo > B2SP_ALGO_TILE_PREPARED) return B2SP_ERR_INVALID_ARG;
    const bool prepared = algo == B2SP_ALGO_TILE_PREPARED;
    if (prepared) algo = B2SP_ALGO_TILE;
    if (stride_a < 0 || stride_b < 0 || stride_d < 0) return B2SP_ERR_INVALID_ARG;
    if (M > 0 && N > 0 && (!O || ldo < N || (batch > 1 && stride_o < (long long)(M - 1) * ldo + N))) return B2SP_ERR_INVALID_ARG;
    if (nnz_stride > 0 && N > 0 && (!D || ldd < N)) return B2SP_ERR_INVALID_ARG;
    if (nnz_stride > 0 && N > 0 && Kd > 0 && (!A || !B || lda < Kd || ldb < Kd)) return B2SP_ERR_INVALID_ARG;
    const size_t row_bytes = row_workspace_bytes(M);
    b2sp_status rc = check_workspace(workspace, workspace_bytes, row_bytes);
    if (rc != B2SP_OK) return rc;
    FusedPlan plan;
    // (the family is chosen from nnz_stride, an upper bound of every problem's entry count)
    if (algo == B2SP_ALGO_TILE ||
        (algo == B2SP_ALGO_AUTO && tile_profitable(B2SP_OP_FUSEDMM, M, K, Kd < N ? Kd : N, nnz_stride)))
        plan = plan_batched(batch, M, K, Kd, N, nnz_stride);
    int use = B2SP_ALGO_ROW_NAT;   // the row family takes the problems' rows in natural order
    if (plan.feasible && workspace_bytes >= plan.bytes) use = B2SP_ALGO_TILE;
    else if (algo == B2SP_ALGO_TILE) return plan.feasible ? B2SP_ERR_WORKSPACE : B2SP_ERR_UNSUPPORTED;
    g_last_algo[B2SP_OP_FUSEDMM] = use;
    int launches = 0;
    g_last_launches[B2SP_OP_FUSEDMM] = 0;
    if (M == 0 || N == 0) return B2SP_OK;
    if (nnz_stride == 0 || Kd == 0) {   // empty patterns or empty dot products: zero outputs
        for (int b = 0; b < batch; ++b) {
            rc = zero_rows(O + (long long)b * stride_o, ldo, M, N, st);
            if (rc != B2SP_OK) return rc;
        }
        return B2SP_OK;
    }
    const long long nz_step = row_ptr_stride == 0 ? 0 : nnz_stride;   // a shared pattern shares its arrays
    const RowBatch rb{row_ptr_stride, nz_step, stride_a, stride_b, stride_d, stride_o};
    if (use == B2SP_ALGO_TILE) {
        BatchDesc bd;
        bd.count = batch; bd.rp = row_ptr_stride; bd.nz = nz_step;
        bd.A = stride_a; bd.B = stride_b; bd.D = stride_d; bd.O = stride_o;
        rc = fused_tile(plan, prepared, 1, M, K, Kd, N, nnz_stride, row_ptr, col_idx, s_values, A, lda, B, ldb, D, ldd,
                        O, ldo, workspace, st, &launches, false, bd, dense_dtype<DT>());
        if (rc != B2SP_OK) return rc;
        int *gate = reinterpret_cast<int *>(static_cast<char *>(workspace) + kWsTileFlagsOffset);
        rc = fused_rows(M, Kd, N, nnz_stride, row_ptr, col_idx, s_values, A, lda, B, ldb, D, ldd, O, ldo, nullptr, gate, nullptr, st,
                        batch, rb);
        g_last_launches[B2SP_OP_FUSEDMM] = launches + 1;
        return rc;
    }
    int *clear = reinterpret_cast<int *>(static_cast<char *>(workspace) + kWsStatusOffset);
    rc = fused_rows(M, Kd, N, nnz_stride, row_ptr, col_idx, s_values, A, lda, B, ldb, D, ldd, O, ldo, nullptr, nullptr, clear, st,
                    batch, rb);
    g_last_launches[B2SP_OP_FUSEDMM] = 1;
    return rc;
}

extern "C" b2sp_status b2sp_fusedmm_batched(int batch, int M, int K, int Kd, int N, long long nnz_stride,
                                            const int *row_ptr, long long row_ptr_stride, const int *col_idx,
                                            const float *s_values, const float *A, long long lda, long long stride_a,
                                            const float *B, long long ldb, long long stride_b, const float *D,
                                            long long ldd, long long stride_d, float *O, long long ldo,
                                            long long stride_o, void *workspace, size_t workspace_bytes, int algo,
                                            void *stream)
{
    return fusedmm_batched_impl<float>(batch, M, K, Kd, N, nnz_stride, row_ptr, row_ptr_stride, col_idx, s_values, A, lda,
                                       stride_a, B, ldb, stride_b, D, ldd, stride_d, O, ldo, stride_o, workspace,
                                       workspace_bytes, algo, stream);
}
extern "C" b2sp_status b2sp_fusedmm_batched_bf16(int batch, int M, int K, int Kd, int N, long long nnz_stride,
                                                 const int *row_ptr, long long row_ptr_stride, const int *col_idx,
                                                 const float *s_values, const void *A, long long lda, long long stride_a,
                                                 const void *B, long long ldb, long long stride_b, const void *D,
                                                 long long ldd, long long stride_d, float *O, long long ldo,
                                                 long long stride_o, void *workspace, size_t workspace_bytes, int algo,
                                                 void *stream)
{
    return fusedmm_batched_impl<bf16_t>(batch, M, K, Kd, N, nnz_stride, row_ptr, row_ptr_stride, col_idx, s_values,
                                        static_cast<const bf16_t *>(A), lda, stride_a, static_cast<const bf16_t *>(B), ldb,
                                        stride_b, static_cast<const bf16_t *>(D), ldd, stride_d, O, ldo, stride_o,
                                        workspace, workspace_bytes, algo, stream);
}

extern "C" b2sp_status b2sp_prepare_pattern(int M, int K, long long nnz, const int *row_ptr, const int *col_idx,
                                 void *workspace, size_t workspace_bytes, void *stream)
{
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (bad_csr_args(M, K, nnz, row_ptr, col_idx) || M == 0 || K == 0 || nnz == 0) return B2SP_ERR_INVALID_ARG;
    const size_t need = pattern_table_offset(M) + pattern_table_bytes(M, K);
    b2sp_status rc = check_workspace(workspace, workspace_bytes, need);
    if (rc != B2SP_OK) return rc;
    int launches = 0;
    return pattern_pass(false, M, K, nnz, row_ptr, col_idx, workspace, st, &launches);
}

extern "C" b2sp_status b2sp_validate_csr(int M, int K, long long nnz, const int *row_ptr, const int *col_idx,
                              void *workspace, size_t workspace_bytes, void *stream)
{
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (M < 0 || K < 0 || nnz < 0 || nnz > (long long)INT_MAX || !row_ptr || (nnz > 0 && !col_idx))
        return B2SP_ERR_INVALID_ARG;
    b2sp_status rc = check_workspace(workspace, workspace_bytes, 256);
    if (rc != B2SP_OK) return rc;
    int *flag = static_cast<int *>(workspace);
    if (cudaMemsetAsync(flag, 0, sizeof(int), st) != cudaSuccess) return B2SP_ERR_CUDA;
    long long work = nnz > M ? nnz : M;
    int blocks = (int)((work + 255) / 256);
    if (blocks < 1) blocks = 1;
    if (blocks > 148 * 16) blocks = 148 * 16;
    validate_csr_kernel<<<blocks, 256, 0, st>>>(M, K, nnz, row_ptr, col_idx, flag);
    if (cudaGetLastError() != cudaSuccess) return B2SP_ERR_CUDA;
    int h = 0;
    if (cudaMemcpyAsync(&h, flag, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return B2SP_ERR_CUDA;
    return h ? B2SP_ERR_BAD_CSR : B2SP_OK;
}

extern "C" b2sp_status b2sp_device_status(const void *workspace, void *stream)
{
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (!workspace) return B2SP_ERR_WORKSPACE;
    int h = 0;
    const int *status = reinterpret_cast<const int *>(static_cast<const char *>(workspace) + 256);
    if (cudaMemcpyAsync(&h, status, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return B2SP_ERR_CUDA;
    return h == 0 ? B2SP_OK : B2SP_ERR_TIMEOUT;
}


// ---- host-buffer forms ------------------------------------------------------------------------
namespace {

// Device memory of one host-buffer call.  It comes from a stream-ordered pool that the library owns (one
// per device, created at first use, release threshold "never": freed blocks stay in it across calls, so a
// call does not pay for fresh allocations).  The process's default pool is left as it is.
cudaMemPool_t library_pool()
{
    constexpr int kMaxDevices = 64;
    static std::mutex mu;
    static cudaMemPool_t pools[kMaxDevices] = {};
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
    std::lock_guard<std::mutex> lock(mu);
    if (!pools[dev]) {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.handleTypes = cudaMemHandleTypeNone;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t pool = nullptr;
        if (cudaMemPoolCreate(&pool, &props) != cudaSuccess) { cudaGetLastError(); return nullptr; }
        unsigned long long keep = ~0ull;
        cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
        pools[dev] = pool;
    }
    return pools[dev];
}

struct DevArena {
    cudaStream_t st;
    cudaMemPool_t pool;
    void *ptrs[16];
    int n = 0;
    bool ok = true;
    int device_word = 0;   // the workspace's status word, copied back with the result
    explicit DevArena(cudaStream_t s) : st(s), pool(library_pool()) { ok = pool != nullptr; }
    void *alloc(size_t bytes)
    {
        void *p = nullptr;
        if (bytes == 0) bytes = 16;
        if (!ok || cudaMallocFromPoolAsync(&p, bytes, pool, st) != cudaSuccess) { ok = false; return nullptr; }
        ptrs[n++] = p;
        return p;
    }
    template <typename T> T *upload(const T *host, size_t count)
    {
        T *d = static_cast<T *>(alloc(sizeof(T) * count));
        if (d && host && count &&
            cudaMemcpyAsync(d, host, sizeof(T) * count, cudaMemcpyHostToDevice, st) != cudaSuccess)
            ok = false;
        return d;
    }
    // Queues the read-back of the status word that device code left in `ws` (a bounded wait that gave up).
    void fetch_status(const void *ws)
    {
        if (ok && ws &&
            cudaMemcpyAsync(&device_word, static_cast<const char *>(ws) + b2sp::kWsStatusOffset, sizeof(int),
                            cudaMemcpyDeviceToHost, st) != cudaSuccess)
            ok = false;
    }
    b2sp_status finish(b2sp_status rc)
    {
        for (int i = 0; i < n; ++i) cudaFreeAsync(ptrs[i], st);
        if (cudaStreamSynchronize(st) != cudaSuccess && rc == B2SP_OK) rc = B2SP_ERR_CUDA;
        if (!ok && rc == B2SP_OK) rc = B2SP_ERR_CUDA;
        if (rc == B2SP_OK && device_word != 0) rc = B2SP_ERR_TIMEOUT;   // the outputs are undefined
        return rc;
    }
};

}  // namespace

extern "C" b2sp_status b2sp_spmm_host(int M, int K, int N, long long nnz, const int *row_ptr,
                           const int *col_idx, const float *values, const float *D, float *O,
                           void *stream)
{
    if (bad_csr_args(M, K, nnz, row_ptr, col_idx) || N < 0) return B2SP_ERR_INVALID_ARG;
    if ((M > 0 && N > 0 && !O) || (nnz > 0 && N > 0 && (!values || !D))) return B2SP_ERR_INVALID_ARG;
    DevArena a(static_cast<cudaStream_t>(stream));
    int *d_rp = a.upload(row_ptr, (size_t)M + 1);
    int *d_ci = a.upload(col_idx, (size_t)nnz);
    float *d_v = a.upload(values, (size_t)nnz);
    float *d_D = a.upload(D, (size_t)K * N);
    float *d_O = static_cast<float *>(a.alloc(sizeof(float) * (size_t)M * N));
    size_t wsb = b2sp_workspace_bytes_algo(B2SP_OP_SPMM, B2SP_ALGO_AUTO, M, K, 0, N, nnz);
    void *ws = a.alloc(wsb);
    b2sp_status rc = B2SP_ERR_CUDA;
    const bool launched_work = M > 0 && N > 0 && nnz > 0;   // otherwise no kernel ran and the status word is unset
    if (a.ok) {
        rc = b2sp_spmm(M, K, N, nnz, d_rp, d_ci, d_v, d_D, N, d_O, N, ws, wsb, B2SP_ALGO_AUTO, stream);
        if (rc == B2SP_OK && (size_t)M * N > 0 &&
            cudaMemcpyAsync(O, d_O, sizeof(float) * (size_t)M * N, cudaMemcpyDeviceToHost, a.st) != cudaSuccess)
            rc = B2SP_ERR_CUDA;
        if (rc == B2SP_OK && launched_work) a.fetch_status(ws);
    }
    return a.finish(rc);
}

extern "C" b2sp_status b2sp_sddmm_host(int M, int K, int Kd, long long nnz, const int *row_ptr,
                            const int *col_idx, const float *s_values, const float *A,
                            const float *B, float *out_values, void *stream)
{
    if (bad_csr_args(M, K, nnz, row_ptr, col_idx) || Kd < 0) return B2SP_ERR_INVALID_ARG;
    if (nnz > 0 && (!out_values || (Kd > 0 && (!A || !B)))) return B2SP_ERR_INVALID_ARG;
    DevArena a(static_cast<cudaStream_t>(stream));
    int *d_rp = a.upload(row_ptr, (size_t)M + 1);
    int *d_ci = a.upload(col_idx, (size_t)nnz);
    float *d_v = s_values ? a.upload(s_values, (size_t)nnz) : nullptr;
    float *d_A = a.upload(A, (size_t)M * Kd);
    float *d_B = a.upload(B, (size_t)K * Kd);
    float *d_C = static_cast<float *>(a.alloc(sizeof(float) * (size_t)nnz));
    size_t wsb = b2sp_workspace_bytes_algo(B2SP_OP_SDDMM, B2SP_ALGO_AUTO, M, K, Kd, 0, nnz);
    void *ws = a.alloc(wsb);
    b2sp_status rc = B2SP_ERR_CUDA;
    const bool launched_work = M > 0 && Kd > 0 && nnz > 0;
    if (a.ok) {
        rc = b2sp_sddmm(M, K, Kd, nnz, d_rp, d_ci, d_v, d_A, Kd, d_B, Kd, d_C, ws, wsb, B2SP_ALGO_AUTO, stream);
        if (rc == B2SP_OK && nnz > 0 &&
            cudaMemcpyAsync(out_values, d_C, sizeof(float) * (size_t)nnz, cudaMemcpyDeviceToHost, a.st) != cudaSuccess)
            rc = B2SP_ERR_CUDA;
        if (rc == B2SP_OK && launched_work) a.fetch_status(ws);
    }
    return a.finish(rc);
}

extern "C" b2sp_status b2sp_fusedmm_host(int M, int K, int Kd, int N, long long nnz, const int *row_ptr,
                              const int *col_idx, const float *s_values, const float *A,
                              const float *B, const float *D, float *O, void *stream)
{
    if (bad_csr_args(M, K, nnz, row_ptr, col_idx) || Kd < 0 || N < 0) return B2SP_ERR_INVALID_ARG;
    if ((M > 0 && N > 0 && !O) || (nnz > 0 && N > 0 && (!D || (Kd > 0 && (!A || !B)))))
        return B2SP_ERR_INVALID_ARG;
    DevArena a(static_cast<cudaStream_t>(stream));
    int *d_rp = a.upload(row_ptr, (size_t)M + 1);
    int *d_ci = a.upload(col_idx, (size_t)nnz);
    float *d_v = s_values ? a.upload(s_values, (size_t)nnz) : nullptr;
    float *d_A = a.upload(A, (size_t)M * Kd);
    float *d_B = a.upload(B, (size_t)K * Kd);
    float *d_D = a.upload(D, (size_t)K * N);
    float *d_O = static_cast<float *>(a.alloc(sizeof(float) * (size_t)M * N));
    size_t wsb = b2sp_workspace_bytes_algo(B2SP_OP_FUSEDMM, B2SP_ALGO_AUTO, M, K, Kd, N, nnz);
    void *ws = a.alloc(wsb);
    b2sp_status rc = B2SP_ERR_CUDA;
    const bool launched_work = M > 0 && N > 0 && Kd > 0 && nnz > 0;
    if (a.ok) {
        rc = b2sp_fusedmm(M, K, Kd, N, nnz, d_rp, d_ci, d_v, d_A, Kd, d_B, Kd, d_D, N, d_O, N, ws, wsb,
                          B2SP_ALGO_AUTO, stream);
        if (rc == B2SP_OK && (size_t)M * N > 0 &&
            cudaMemcpyAsync(O, d_O, sizeof(float) * (size_t)M * N, cudaMemcpyDeviceToHost, a.st) != cudaSuccess)
            rc = B2SP_ERR_CUDA;
        if (rc == B2SP_OK && launched_work) a.fetch_status(ws);
    }
    return a.finish(rc);
}

