"""The dense-tile kernels when an operand chunk never arrives.  b2sp_debug_inject_wait_timeout makes the TMA producer of every CTA
leave one chunk out and shortens the limit of the bounded waits to 2 ms; the call reports B2SP_ERR_TIMEOUT (6) through the status
word, and nothing computed from the incomplete operands reaches the output."""
import pytest
import torch

from paper_2311_00368_b200 import workloads as W

pytestmark = pytest.mark.gpu

TILE, TIMEOUT = 3, 6
LIMIT_NS = 2_000_000


@pytest.fixture(scope="module")
def b():
    assert torch.cuda.is_available()
    from paper_2311_00368_b200 import binding
    return binding


@pytest.mark.parametrize("op,dtype,values", [
    ("sddmm", torch.float32, True),
    ("sddmm", torch.bfloat16, True),
    ("fusedmm", torch.bfloat16, True),
    ("fusedmm", torch.bfloat16, False),
])
def test_an_incomplete_dot_product_is_never_stored(b, op, dtype, values):
    """The first B chunk of the second of two blocks is withheld.  The ring has room for all the other chunks, so every other wait
    can be met, and only GEMM1's own check keeps its incomplete sums from the processors.  148 CTAs, in each of which GEMM1's wait and
    those of the processors run out in whatever order: none may write an output of the second block."""
    M, K, Kd, N = 148 * 128, 256, 64, 64   # a CTA per 128 rows, two blocks each
    p = W.small_random(4700, M, K, 0.1, Kd, N)
    dev = lambda x, dt=None: torch.from_numpy(x).cuda().to(dt) if dt else torch.from_numpy(x).cuda()
    rp, ci, v = dev(p.row_ptr), dev(p.col_idx), dev(p.values) if values else None
    A, B, D = (dev(x, dtype) for x in (p.A, p.B, p.D))
    sddmm = op == "sddmm"
    code = b.OP_SDDMM if sddmm else b.OP_FUSEDMM
    ws = torch.empty(b.workspace_bytes(code, M, K, Kd, N, p.nnz), dtype=torch.uint8, device="cuda")
    untouched = 1234.5
    out = torch.full((p.nnz,) if sddmm else (M, N), untouched, device="cuda")
    second = ci >= 128 if sddmm else torch.ones_like(out, dtype=torch.bool)   # (FusedMM adds the blocks up before it writes)

    def call():
        if sddmm:
            b.sddmm(rp, ci, v, A, B, out=out, workspace=ws, algo=TILE, dtype=dtype)
        else:
            b.fusedmm(rp, ci, v, A, B, D, out=out, workspace=ws, algo=TILE, dtype=dtype)
        assert b.last_algo(code) == TILE
        return b.device_status(ws)

    # order of the chunks: B(0) twice; FusedMM: D(0,0) D(0,1); B(1) twice; ...
    b.debug_inject_wait_timeout(2 if sddmm else 4, LIMIT_NS)
    try:
        assert call() == TIMEOUT
        assert bool((out[second] == untouched).all()), "results of an incomplete sum were written"
    finally:
        b.debug_inject_wait_timeout(-1)
    assert call() == 0
    assert not bool((out == untouched).any())


def _chunk_of(kind, block, which, dtype, nblk):
    """The number of a chunk of FusedMM at Kd = 64: two B chunks of block 0; then, block by block, D of its windows 0 and 1, the two B
    chunks of the next block, D of its windows 2 and 3 -- with fp32 operands B comes after all four D at every fourth block."""
    order = [("B", 0, 0), ("B", 0, 1)]
    for b in range(nblk):
        last = dtype == torch.float32 and b % 4 == 3
        nxt = [("B", b + 1, 0), ("B", b + 1, 1)] if b + 1 < nblk else []
        order += [("D", b, 0), ("D", b, 1)] + (nxt if not last else []) + [("D", b, 2), ("D", b, 3)] + (nxt if last else [])
    return order.index((kind, block, which))


@pytest.mark.parametrize("values", [True, False])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("M,K,partition,chunks", [
    # a CTA per 128 rows, ten blocks each; the first four blocks are added up before anything is written.  The last two chunks come when
    # every slot of the ring has been used several times.
    (148 * 128, 1280, 1, [("D", 0, 0), ("D", 2, 3), ("D", 5, 1), ("D", 9, 3), ("B", 9, 0)]),
    # 200 row tiles of four blocks on 148 CTAs: every third CTA goes on into a second row tile (blocks 4 to 7), for which the chunk is missing
    (200 * 128, 512, 2, [("D", 3, 3), ("B", 4, 1), ("D", 4, 0), ("D", 7, 2)]),
])
def test_a_missing_chunk_of_fusedmm_is_reported(b, M, K, partition, chunks, dtype, values):
    """FusedMM with one chunk of D (GEMM2's own barriers) or a late one of B withheld, on either partition, with helper warps (stored
    values) and without: the status word says so, sums that lack a window of D are not written, and the next call on the same
    workspace gives what the call before did, to the bit."""
    Kd = N = 64
    p = W.small_random(4710 + K, M, K, 0.05, Kd, N)
    dev = lambda x, dt=None: torch.from_numpy(x).cuda().to(dt) if dt else torch.from_numpy(x).cuda()
    rp, ci, v = dev(p.row_ptr), dev(p.col_idx), dev(p.values) if values else None
    A, B, D = (dev(x, dtype) for x in (p.A, p.B, p.D))
    untouched = 1234.5
    b.debug_force_partition(partition)
    try:
        ws = torch.empty(b.workspace_bytes(b.OP_FUSEDMM, M, K, Kd, N, p.nnz, algo=TILE), dtype=torch.uint8, device="cuda")

        def call():
            out = torch.full((M, N), untouched, device="cuda")
            b.fusedmm(rp, ci, v, A, B, D, out=out, workspace=ws, algo=TILE, dtype=dtype)
            assert b.last_algo(b.OP_FUSEDMM) == TILE
            return out, b.device_status(ws)

        before, status = call()
        assert status == 0 and not bool((before == untouched).any())
        for kind, block, which in chunks:
            # (blocks of a CTA: ten, or the two row tiles' eight)
            b.debug_inject_wait_timeout(_chunk_of(kind, block, which, dtype, 10 if partition == 1 else 8), LIMIT_NS)
            try:
                out, status = call()
            finally:
                b.debug_inject_wait_timeout(-1)
            what = f"{kind} chunk {which} of block {block}"
            assert status == TIMEOUT, f"{what}: status {status}"
            if partition == 1 and block < 4:
                assert bool((out == untouched).all()), f"{what}: an incomplete sum was written"
            out, status = call()
            assert status == 0 and torch.equal(out, before), f"after {what}: the next call differs"
    finally:
        b.debug_force_partition(0)
