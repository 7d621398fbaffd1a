"""FusedMM where a CTA of the dense-tile family goes from one row tile, and one problem, into the next: B and D are read a segment
apart, and without stored values the processors read the next segment's occupancy masks ahead.  Against the CPU oracle on the operands
as rounded (gate |gpu - ref| <= 1e-5 * T + 1e-6)."""
import pytest
import torch

import oracle
from paper_2311_00368_b200 import workloads as W
from tests.test_gpu_batched import TILE, Stacked

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    assert torch.cuda.is_available()
    from paper_2311_00368_b200 import binding
    return binding


# (a granule is a run of four 128-column blocks)
@pytest.mark.parametrize("nb,M,K,Kd,N", [
    (5, 4100, 1024, 64, 64),     # 165 row tiles of two granules on 148 CTAs: two or three each, of one or two row tiles
    (5, 8200, 512, 64, 64),      # 325 row tiles of one granule: two or three each, every one a segment
    (5, 4500, 512, 128, 128),    # 180 row tiles of one granule
    (4, 5000, 500, 128, 40),     # 160 of them, a last window of 20 columns
    (7, 2000, 512, 32, 130),     # two column tiles: 74 groups of CTAs for 112 row tiles
])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("values", [False, True])
def test_fusedmm_over_several_segments(b, nb, M, K, Kd, N, dtype, values):
    rounded = []
    for i, density in zip(range(nb), (0.05, 0.03, 0.08, 0.04, 0.06, 0.03, 0.05)):
        p = W.small_random(5800 + 7 * i + M, M, K, density, Kd, N)
        A, B, D = (torch.from_numpy(x).to(dtype).float().numpy() for x in (p.A, p.B, p.D))
        rounded.append(W.Problem(p.name, M, K, p.row_ptr, p.col_idx, p.values, Kd, N, A, B, D))
    s = Stacked(rounded)
    refs = s.refs if values else [oracle.fusedmm(p.row_ptr, p.col_idx, None, p.A, p.B, p.D) for p in rounded]
    A, B, D = (x.to(dtype) for x in (s.A, s.B, s.D))
    for partition in (2, 1):
        b.debug_force_partition(partition)
        try:
            ws = s.workspace(b)
            outs = []
            for _ in range(2):
                out = torch.full((nb, M, N), float("nan"), device="cuda")
                b.fusedmm_batched(s.row_ptr, s.col_idx, s.values if values else None, A, B, D, out=out, workspace=ws, algo=TILE, dtype=dtype)
                assert b.last_algo(b.OP_FUSEDMM) == TILE and b.device_status(ws) == 0
                outs.append(out)
            assert torch.equal(outs[0], outs[1]), f"partition {partition}: two runs differ"
            s.check(outs[0], f"partition {partition}", refs)
        finally:
            b.debug_force_partition(0)
