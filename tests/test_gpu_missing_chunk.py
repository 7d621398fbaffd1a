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
