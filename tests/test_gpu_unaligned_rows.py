"""The row family on dense operands whose rows are not aligned groups of four: widths, leading dimensions and first addresses
that are a multiple of nothing or of two, both types, every width class of the kernels, against the oracle on every element.
Guard words around the outputs must survive."""
import numpy as np
import pytest
import torch

import oracle
from paper_2311_00368_b200 import workloads as W
from tests.test_gpu_parity import gate

pytestmark = pytest.mark.gpu

ROW, ROW_NAT = 1, 2


@pytest.fixture(scope="module")
def b():
    assert torch.cuda.is_available()
    from paper_2311_00368_b200 import binding
    return binding


def strided(x, dtype, pad, shift):
    """x on the GPU with `pad` elements between its rows and its first one `shift` elements into an aligned buffer; NaN around it."""
    r, c = x.shape
    buf = torch.full((shift + r * (c + pad) + 8,), float("nan"), dtype=dtype, device="cuda")
    view = buf[shift:shift + r * (c + pad)].view(r, c + pad)[:, :c]
    view.copy_(torch.from_numpy(x))
    return view


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("Kd,N,pad,shift", [
    (1, 1, 0, 0), (2, 3, 1, 0), (3, 5, 0, 1), (5, 31, 2, 0), (31, 33, 0, 0), (33, 63, 1, 2), (50, 70, 0, 0), (62, 66, 0, 2),
    (63, 65, 1, 1), (65, 127, 0, 3), (127, 129, 1, 0), (130, 131, 0, 0), (64, 64, 1, 0), (64, 128, 0, 1), (128, 128, 2, 2),
    (255, 255, 0, 0), (257, 257, 1, 0), (258, 300, 0, 0), (301, 515, 0, 1),
])
def test_row_kernels_at_any_alignment(b, dtype, Kd, N, pad, shift):
    p = W.small_random(7000 + Kd + N, 37, 300, 0.2, Kd, N, kind="powerlaw")
    A, B, D = (torch.from_numpy(x).to(dtype).float().numpy() for x in (p.A, p.B, p.D))
    rp, ci, v = (torch.from_numpy(x).cuda() for x in (p.row_ptr, p.col_idx, p.values))
    dA, dB, dD = (strided(x, dtype, pad, shift) for x in (A, B, D))
    for algo in (ROW, ROW_NAT):
        for op in ("spmm", "fusedmm"):
            out = strided(np.zeros((p.M, N), np.float32), torch.float32, 3, shift)
            whole = torch.as_strided(out, (p.M, N + 3), (N + 3, 1))
            whole.fill_(-7.0)
            if op == "spmm":
                ref = oracle.spmm(p.row_ptr, p.col_idx, p.values, D)
                b.spmm(rp, ci, v, dD, out=out, algo=algo, dtype=dtype)
            else:
                ref = oracle.fusedmm(p.row_ptr, p.col_idx, p.values, A, B, D)
                b.fusedmm(rp, ci, v, dA, dB, dD, out=out, algo=algo, dtype=dtype)
            gate(out, *ref, f"{op} algo={algo}")
            assert bool((whole[:, N:] == -7.0).all()), "columns beyond N were written"
        out = torch.full((p.nnz + 1,), -7.0, device="cuda")
        b.sddmm(rp, ci, v, dA, dB, out=out[:p.nnz], algo=algo, dtype=dtype)
        gate(out[:p.nnz], *oracle.sddmm(p.row_ptr, p.col_idx, p.values, A, B), f"sddmm algo={algo}")
        assert out[p.nnz].item() == -7.0


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("Kd,N", [(17, 30), (50, 71), (129, 33), (300, 130)])
def test_batched_row_kernels_at_any_alignment(b, dtype, Kd, N):
    nb, M, K = 3, 29, 200
    probs = [W.small_random(7100 + i, M, K, 0.2, Kd, N) for i in range(nb)]
    most = max(p.nnz for p in probs)
    pad = lambda x: np.pad(x, (0, most - x.size))
    rp = torch.from_numpy(np.stack([p.row_ptr for p in probs])).cuda()
    ci = torch.from_numpy(np.stack([pad(p.col_idx) for p in probs])).cuda()
    v = torch.from_numpy(np.stack([pad(p.values) for p in probs])).cuda()
    host = [[torch.from_numpy(x).to(dtype) for x in (p.A, p.B, p.D)] for p in probs]
    A, B, D = (torch.stack([h[i] for h in host]).cuda() for i in range(3))
    out = b.fusedmm_batched(rp, ci, v, A, B, D, algo=ROW, dtype=dtype)
    for i, p in enumerate(probs):
        hA, hB, hD = (t.float().numpy() for t in host[i])
        gate(out[i], *oracle.fusedmm(p.row_ptr, p.col_idx, p.values, hA, hB, hD), f"problem {i}")


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("Kd,N,pad,shift", [
    (12289, 5, 0, 0), (12290, 6, 0, 0), (12292, 8, 0, 0), (13001, 33, 0, 0),   # more than 48 KB of shared memory for A_i
    (16384, 5, 1, 0), (16383, 6, 0, 1), (24576, 6, 0, 2), (40960, 8, 0, 0),     # the longest that are staged there
    (16385, 5, 0, 0), (16388, 6, 1, 0), (24578, 130, 0, 0), (24580, 6, 2, 2),   # a lane per dot product
    (40961, 5, 0, 0), (40964, 132, 0, 0),
])
def test_long_dot_products(b, dtype, Kd, N, pad, shift):
    nb, M, K = 2, 9, 40
    probs = [W.small_random(7200 + Kd % 97 + i, M, K, 0.3, Kd, N) for i in range(nb)]
    most = max(p.nnz for p in probs)
    fill = lambda x: np.pad(x, (0, most - x.size))
    rp = torch.from_numpy(np.stack([p.row_ptr for p in probs])).cuda()
    ci, v = (torch.from_numpy(np.stack([fill(x) for x in xs])).cuda() for xs in ([p.col_idx for p in probs], [p.values for p in probs]))
    host = [[torch.from_numpy(x).to(dtype).float().numpy() for x in (p.A, p.B, p.D)] for p in probs]
    refs = [oracle.fusedmm(p.row_ptr, p.col_idx, p.values, *h) for p, h in zip(probs, host)]
    for i, (p, h) in enumerate(zip(probs, host)):
        dA, dB, dD = (strided(x, dtype, pad, shift) for x in h)
        sd = oracle.sddmm(p.row_ptr, p.col_idx, p.values, h[0], h[1])
        for algo in (ROW, ROW_NAT):
            gate(b.fusedmm(rp[i], ci[i, :p.nnz], v[i, :p.nnz], dA, dB, dD, algo=algo, dtype=dtype), *refs[i], f"fusedmm algo={algo}")
            gate(b.sddmm(rp[i], ci[i, :p.nnz], v[i, :p.nnz], dA, dB, algo=algo, dtype=dtype), *sd, f"sddmm algo={algo}")
    A, B, D = (torch.stack([torch.from_numpy(h[j]).to(dtype) for h in host]).cuda() for j in range(3))
    out = b.fusedmm_batched(rp, ci, v, A, B, D, algo=ROW, dtype=dtype)
    for i in range(nb):
        gate(out[i], *refs[i], f"problem {i}")
