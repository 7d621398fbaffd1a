"""The row kernels on both sides of the average row length at which the form for long rows takes over, at every width that has
both, against the oracle on every element."""
import numpy as np
import pytest
import torch

import oracle
from tests.test_gpu_parity import gate

pytestmark = pytest.mark.gpu

ROW, ROW_NAT = 1, 2


@pytest.fixture(scope="module")
def b():
    assert torch.cuda.is_available()
    from paper_2311_00368_b200 import binding
    return binding


def pattern(rng, M, K, line, extra):
    """Rows of every remainder of the kernels' chunks, line * M + extra entries in all."""
    lens = np.resize(np.array([0, 1, 4, 31, 32, 33, 64, 65, 127, 128, 129, 160, 161, 255]), M)
    target = line * M + extra
    while lens.sum() != target:
        step = 1 if lens.sum() < target else -1
        i = rng.integers(0, M, min(M // 2, abs(int(lens.sum()) - target)))
        i = np.unique(i)
        lens[i] = np.clip(lens[i] + step, 0, K)
    rp = np.zeros(M + 1, np.int32)
    rp[1:] = np.cumsum(lens)
    ci = np.concatenate([np.sort(rng.choice(K, n, replace=False)) for n in lens]).astype(np.int32)
    return rp, ci, rng.uniform(-1, 1, rp[-1]).astype(np.float32)


def operand(rng, rows, cols, dtype):
    """On the GPU, and the values it holds as fp32."""
    t = torch.from_numpy(rng.standard_normal((rows, cols), dtype=np.float32)).to(dtype)
    return t.cuda(), t.float().numpy()


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("extra", [0, 1])
@pytest.mark.parametrize("line,M,N", [(144, 60, 40), (144, 60, 64), (144, 1480, 132), (144, 1480, 256), (72, 60, 260), (72, 60, 512), (72, 60, 516)])
def test_spmm(b, line, M, N, extra, dtype):
    rng = np.random.default_rng(N + extra)
    rp, ci, v = pattern(rng, M, 300, line, extra)
    dD, D = operand(rng, 300, N, dtype)
    ref = oracle.spmm(rp, ci, v, D)
    for algo in (ROW, ROW_NAT):
        out = b.spmm(torch.from_numpy(rp).cuda(), torch.from_numpy(ci).cuda(), torch.from_numpy(v).cuda(), dD, algo=algo, dtype=dtype)
        gate(out, *ref, f"algo={algo}")


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("extra", [0, 1])
@pytest.mark.parametrize("Kd", [4, 32, 64, 132, 256, 257, 258, 260, 516])
def test_sddmm(b, Kd, extra, dtype):
    rng = np.random.default_rng(Kd + extra)
    rp, ci, v = pattern(rng, 60, 300, 128, extra)
    (dA, A), (dB, B) = operand(rng, 60, Kd, dtype), operand(rng, 300, Kd, dtype)
    ref = oracle.sddmm(rp, ci, v, A, B)
    for algo in (ROW, ROW_NAT):
        out = b.sddmm(torch.from_numpy(rp).cuda(), torch.from_numpy(ci).cuda(), torch.from_numpy(v).cuda(), dA, dB, algo=algo, dtype=dtype)
        gate(out, *ref, f"algo={algo}")


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("extra", [0, 1])
@pytest.mark.parametrize("Kd,N", [(64, 32), (60, 64), (64, 100), (64, 256), (128, 128), (128, 256), (128, 512), (100, 516), (256, 256), (160, 132), (260, 64), (301, 33)])
def test_fusedmm(b, Kd, N, extra, dtype):
    rng = np.random.default_rng(Kd + N + extra)
    line = 72 if N * dtype.itemsize <= 128 else 144
    probs = [pattern(rng, 60, 300, line, extra) for _ in range(2)]
    dense = [[operand(rng, r, c, dtype) for r, c in ((60, Kd), (300, Kd), (300, N))] for _ in probs]
    refs = [oracle.fusedmm(*p, *(x for _, x in d)) for p, d in zip(probs, dense)]
    cuda = lambda x: torch.from_numpy(x).cuda()
    for p, d, ref in zip(probs, dense, refs):
        for algo in (ROW, ROW_NAT):
            gate(b.fusedmm(*map(cuda, p), *(t for t, _ in d), algo=algo, dtype=dtype), *ref, f"algo={algo}")
    stack = lambda i: torch.stack([cuda(p[i]) for p in probs])
    out = b.fusedmm_batched(stack(0), stack(1), stack(2), *(torch.stack([d[i][0] for d in dense]) for i in range(3)), algo=ROW, dtype=dtype)
    for o, ref in zip(out, refs):
        gate(o, *ref, "batched")
