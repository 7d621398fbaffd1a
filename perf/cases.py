"""The calls that the library's speed is judged on.

The library does three things over a CSR pattern S: SPMM (O = S D), SDDMM (C = S .* (A B^T), on S's entries) and FusedMM
(O = (S .* (A B^T)) D).  The listed cases are what its users have it do, through ``paper_2311_00368_b200.binding``: the
named workloads of ``workloads.py`` and ``bench.py``, points of the paper's grid from the smallest to the largest, sizes
that are a multiple of nothing, both operand types, and each way to call it:

  plain     the op by itself, everything left to the library (the pattern is new, so its analysis belongs to the call)
  prepared  the pattern was analysed once, before: a training loop over a fixed mask
  step      the pattern is analysed, then all three ops run on it: one step of a model whose mask changes
  batched   FusedMM on (batch x heads) problems of sparse attention
  host      arrays in host memory, result in host memory

A case holds: call, op, M, K (S is M x K), Kd (length of the sampled dot products), N (width of D and O), density,
pattern ("uniform"; "powerlaw": Zipf row lengths, exponent 1.1; "band": a 128-wide diagonal band and uniform extras),
values ("uniform": U(-1, 1); "ones": no stored values, an all-ones mask), dtype of A, B and D, batch.
"""
import math

import torch

from paper_2311_00368_b200 import workloads

_BAND = 128
_CELLS_MOST = 32768 * 8192   # M * K of the paper's largest matrices


def _case(name, call, op, M, K, Kd, N, density, pattern="uniform", values="uniform", dtype="fp32", batch=1):
    c = dict(call=call, op=op, M=M, K=K, Kd=Kd, N=N, density=density, pattern=pattern, values=values, dtype=dtype, batch=batch)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest workload: what a call costs when there is next to nothing to compute
        _case("tiny_fusedmm", "plain", "fusedmm", 256, 256, 64, 64, 0.10),
        # a pruned layer of a small model on a narrow batch (3k/1k/32/90% of the paper's grid): short, latency-bound
        _case("narrow_spmm_3k_1k", "plain", "spmm", 3072, 1024, 0, 32, 0.10),
        # a pruned weight matrix times activations
        _case("spmm_2048_n256", "plain", "spmm", 2048, 2048, 0, 256, 0.20),
        # sampled similarities: the gradient of a sparse weight, or attention scores on a mask
        _case("sddmm_4096_k128", "plain", "sddmm", 4096, 4096, 128, 0, 0.10, values="ones"),
        # a graph layer on features whose widths and counts are a multiple of nothing
        _case("ragged_fusedmm", "plain", "fusedmm", 1501, 2903, 50, 70, 0.12),
        # sparse attention, batch x heads = 8, in fp32 and on bfloat16 Q, K, V
        _case("attention_8x4096", "batched", "fusedmm", 4096, 4096, 64, 64, 0.20, "band", "ones", batch=8),
        _case("attention_8x4096_bf16", "batched", "fusedmm", 4096, 4096, 64, 64, 0.20, "band", "ones", "bf16", batch=8),
        # skewed rows, the headline sizes (8k/8k/128/70%): FusedMM by itself, and all three ops on a pattern analysed once
        _case("powerlaw_fusedmm_8k", "plain", "fusedmm", 8192, 8192, 128, 128, 0.30, "powerlaw"),
        _case("powerlaw_step_8k", "step", "all", 8192, 8192, 128, 128, 0.30, "powerlaw"),
        # a wide activation matrix against a fixed, sparser mask, step after step
        _case("prepared_spmm_8k_n512", "prepared", "spmm", 8192, 8192, 0, 512, 0.10, "powerlaw"),
        # one attention head whose arrays live in host memory
        _case("host_fusedmm_4096", "host", "fusedmm", 4096, 4096, 64, 64, 0.20, "band"),
        # the largest matrix of the paper's grid (32k/8k/128/80%)
        _case("fusedmm_32k_8k", "plain", "fusedmm", 32768, 8192, 128, 128, 0.20),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: sizes over the whole range, odd ones among them, every op, way to call, pattern and type."""
    call = rng.choice(["plain", "plain", "plain", "prepared", "step", "batched", "host"])
    M = _log_uniform(rng, 256, 32768)
    K = _log_uniform(rng, 256, 8192)
    if rng.random() < 0.5:   # half of the sizes are round, half are whatever they come out as
        M, K = max(256, M // 256 * 256), max(256, K // 256 * 256)
    density = round(rng.uniform(0.05, 0.30), 3)
    width = lambda hi: rng.choice([32, 64, 128, 128, _log_uniform(rng, 16, hi)])
    Kd, N = width(128), rng.choice([width(256), width(256), 256])
    op = "all" if call == "step" else rng.choice(["spmm", "sddmm", "fusedmm", "fusedmm"])
    batch = 1
    if call == "batched":
        op = "fusedmm"
        batch = rng.randint(2, 16)
        M = min(M, 4096)
        K = M if rng.random() < 0.7 else min(K, 4096)
        N = min(N, 128)
        while batch * M * K > _CELLS_MOST // 2:
            batch -= 1
    if call in ("host", "step"):
        while M * K > _CELLS_MOST // 8:
            M //= 2
    while M * K * max(Kd + N, 128) > _CELLS_MOST * 256:
        M //= 2
    pattern = rng.choice(["uniform", "uniform", "powerlaw", "band"])
    if pattern == "band" and density * K < 2 * _BAND:
        pattern = "uniform"
    values = rng.choice(["uniform", "uniform", "ones"]) if op in ("sddmm", "fusedmm") else "uniform"
    dtype = rng.choice(["fp32", "fp32", "bf16"]) if call in ("plain", "batched") else "fp32"
    if op == "spmm":
        Kd = 0
    if op == "sddmm":
        N = 0
    return _case(None, call, op, M, K, Kd, N, density, pattern, values, dtype, batch)


def _pattern(case, gen):
    """row_ptr [M + 1], col_idx [nnz], nnz = density * M * K: every entry is drawn on its own, with the density that its
    place has, from a pattern that is a little denser, and as many of the entries as there are too many are left out."""
    M, K, density = case["M"], case["K"], case["density"]
    nnz = int(density * M * K)
    if case["pattern"] == "powerlaw":
        lens = torch.from_numpy(workloads.powerlaw_row_lengths(M, K, density)).to("cuda", torch.float32)
        p_row = (lens / K)[torch.randperm(M, generator=gen, device="cuda")]
    elif case["pattern"] == "band":
        nband = workloads.band_entry_count(M, K, _BAND // 2)
        p_extra = (density * M * K - nband) / float(M * K - nband)
    block = max(1, (1 << 26) // K)
    j = torch.arange(K, device="cuda")
    denser = 1.0 + 6.0 / math.sqrt(nnz)
    while True:
        at = []
        for r0 in range(0, M, block):
            r1 = min(M, r0 + block)
            u = torch.rand((r1 - r0, K), generator=gen, device="cuda")
            if case["pattern"] == "powerlaw":
                mask = u < denser * p_row[r0:r1, None]
            elif case["pattern"] == "band":
                off = j[None, :] - torch.arange(r0, r1, device="cuda")[:, None]
                mask = (u < denser * p_extra) | ((off >= -(_BAND // 2)) & (off < _BAND // 2))
            else:
                mask = u < denser * density
            at.append(mask.view(-1).nonzero().view(-1) + r0 * K)
        at = torch.cat(at)
        if at.numel() >= nnz:
            break
        denser *= 1.05
    if at.numel() > nnz:
        keep = torch.ones(at.numel(), dtype=torch.bool, device="cuda")
        keep[torch.randperm(at.numel(), generator=gen, device="cuda")[:at.numel() - nnz]] = False
        at = at[keep]
    row_ptr = torch.searchsorted(at, torch.arange(M + 1, device="cuda") * K).to(torch.int32)
    return row_ptr, (at % K).to(torch.int32)


def _inputs(case, seed):
    """The arrays of a case, on the GPU; of a batch, stacked."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    nb, M, K, Kd, N = case["batch"], case["M"], case["K"], case["Kd"], case["N"]
    patterns = [_pattern(case, gen) for _ in range(nb)]
    nnz = patterns[0][1].numel()
    dtype = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    dense = lambda rows, cols: torch.randn((nb, rows, cols), generator=gen, device="cuda").to(dtype) if cols else None
    values = None
    if case["values"] == "uniform":
        values = torch.rand((nb, nnz), generator=gen, device="cuda") * 2 - 1
    x = dict(row_ptr=torch.stack([rp for rp, _ in patterns]),
             col_idx=torch.stack([ci for _, ci in patterns]),
             values=values, A=dense(M, Kd), B=dense(K, Kd), D=dense(K, N))
    if case["call"] != "batched":
        x = {k: None if v is None else v[0] for k, v in x.items()}
    return x


def prepare(case, seed):
    from paper_2311_00368_b200 import binding
    x = _inputs(case, seed)
    x.update(case=case, binding=binding, dtype=torch.bfloat16 if case["dtype"] == "bf16" else torch.float32)
    M, K, Kd, N = case["M"], case["K"], case["Kd"], case["N"]
    nnz = x["col_idx"].shape[-1]
    if case["call"] == "host":   # pinned arrays in host memory, the result's too
        for k in ("row_ptr", "col_idx", "values", "A", "B", "D"):
            if x[k] is not None:
                x[k] = x[k].cpu().pin_memory()
        shape = (nnz,) if case["op"] == "sddmm" else (M, N)
        x["out"] = torch.empty(shape, dtype=torch.float32).pin_memory()
    elif case["call"] in ("prepared", "step"):   # one workspace for all calls on this pattern
        ops = {"spmm": (binding.OP_SPMM, 0, N), "sddmm": (binding.OP_SDDMM, Kd, 0), "fusedmm": (binding.OP_FUSEDMM, Kd, N)}
        need = [binding.workspace_bytes(op, M, K, kd, n, nnz) for name, (op, kd, n) in ops.items() if case["op"] in (name, "all")]
        x["workspace"] = torch.empty(max(need), dtype=torch.uint8, device="cuda")
        if case["call"] == "prepared":
            binding.prepare_pattern(x["row_ptr"], x["col_idx"], K, x["workspace"])
    return x


def run(s):
    case, b = s["case"], s["binding"]
    call, op = case["call"], case["op"]
    rp, ci, v, A, B, D = (s[k] for k in ("row_ptr", "col_idx", "values", "A", "B", "D"))
    if call == "batched":
        return b.fusedmm_batched(rp, ci, v, A, B, D, dtype=s["dtype"])
    if call == "host":
        if op == "spmm":
            return b.spmm_host(rp, ci, v, D, s["out"])
        if op == "sddmm":
            return b.sddmm_host(rp, ci, v, A, B, s["out"])
        return b.fusedmm_host(rp, ci, v, A, B, D, s["out"])
    kw = dict(dtype=s["dtype"])
    if call in ("prepared", "step"):
        kw.update(workspace=s["workspace"], algo=b.ALGO_TILE_PREPARED)
    if call == "step":
        b.prepare_pattern(rp, ci, case["K"], s["workspace"])
        return (b.spmm(rp, ci, v, D, **kw), b.sddmm(rp, ci, v, A, B, **kw), b.fusedmm(rp, ci, v, A, B, D, **kw))
    if op == "spmm":
        return b.spmm(rp, ci, v, D, **kw)
    if op == "sddmm":
        return b.sddmm(rp, ci, v, A, B, **kw)
    return b.fusedmm(rp, ci, v, A, B, D, **kw)


def work(case):
    M, K, Kd, N, nb = case["M"], case["K"], case["Kd"], case["N"], case["batch"]
    nnz = int(case["density"] * M * K)
    e = 2 if case["dtype"] == "bf16" else 4
    has_values = case["values"] == "uniform"
    csr = 4 * (M + 1) + 4 * nnz + (4 * nnz if has_values else 0)
    a, b, d, o, c = e * M * Kd, e * K * Kd, e * K * N, 4 * M * N, 4 * nnz
    per_op = {"spmm": csr + d + o, "sddmm": csr + a + b + c, "fusedmm": csr + a + b + d + o}
    per_op["all"] = csr + a + b + d + 2 * o + c   # each input read once, the three results written once
    if case["op"] == "all":
        flops = sum(workloads.flops(op, nnz, Kd, N) for op in ("spmm", "sddmm", "fusedmm"))
    else:
        flops = workloads.flops(case["op"], nnz, Kd, N)
    return {"bytes": nb * per_op[case["op"]], "flops": nb * flops}


def tolerance(case):
    # fp32 sums of up to a few thousand terms; measured against float64: 1e-7 on the CUDA cores, up to 4e-6 on the tensor
    # cores (which add into their fp32 accumulators with truncation)
    return {"rel": 1.6e-5}


def exact(case, seed):
    x = _inputs(case, seed)
    single = case["call"] != "batched"
    outs = []
    for p in range(case["batch"]):
        at = lambda k: x[k] if single or x[k] is None else x[k][p]
        outs.append(_exact_one(case, *(at(k) for k in ("row_ptr", "col_idx", "values", "A", "B", "D"))))
    if single:
        return outs[0]
    return torch.stack(outs)


def _exact_one(case, row_ptr, col_idx, values, A, B, D):
    M, K, op = case["M"], case["K"], case["op"]
    A, B, D = (None if t is None else t.double() for t in (A, B, D))
    rp = row_ptr.long()
    o_spmm, c_all, o_fused = [], [], []
    block = max(1, (1 << 24) // K)
    for r0 in range(0, M, block):
        r1 = min(M, r0 + block)
        p0, p1 = int(rp[r0]), int(rp[r1])
        rows = torch.repeat_interleave(torch.arange(r1 - r0, device="cuda"), rp[r0 + 1:r1 + 1] - rp[r0:r1])
        cols = col_idx[p0:p1].long()
        v = torch.ones(p1 - p0, dtype=torch.float64, device="cuda") if values is None else values[p0:p1].double()
        if op in ("spmm", "all"):
            S = torch.zeros((r1 - r0, K), dtype=torch.float64, device="cuda")
            S[rows, cols] = v
            o_spmm.append(S @ D)
        if op in ("sddmm", "fusedmm", "all"):
            c = v * (A[r0:r1] @ B.T)[rows, cols]
            c_all.append(c)
            if op in ("fusedmm", "all"):
                S = torch.zeros((r1 - r0, K), dtype=torch.float64, device="cuda")
                S[rows, cols] = c
                o_fused.append(S @ D)
    if op == "spmm":
        return torch.cat(o_spmm)
    if op == "sddmm":
        return torch.cat(c_all)
    if op == "fusedmm":
        return torch.cat(o_fused)
    return torch.cat(o_spmm), torch.cat(c_all), torch.cat(o_fused)
