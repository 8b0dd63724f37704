"""The workloads this engine is timed on: all-mode sweeps, single-mode products, CP-ALS and the CP loss.

Every case is one sparse COO tensor (synthetic: distinct random coordinates, uniform or
Zipf-skewed per mode) with dense factors, run through the package's public entry points.
Sizes follow the repository's benchmark and tests: the shapes of its workloads, some with
fewer nonzeros so that a tensor is drawn quickly, and generic odd sizes.
"""
import math

import numpy as np
import torch

from paper_2405_08470_gb300 import Plan
from paper_2405_08470_gb300.cp import cp_als, cp_loss


def listed():
    return [
        # The smallest calls: one sweep of a tensor that fits any cache, where launches count.
        _case("sweep_small", "sweep", "200x150x100", 50_000, "0x0x0", 16, "f32"),
        # The same tensor decomposed: a few ALS iterations, each with its fit read back.
        _case("als_small", "als", "200x150x100", 50_000, "0x0x0", 16, "f32", iters=3),
        # An ordinary tensor of odd sizes at a rank that is no multiple of four.
        _case("sweep_odd_rank", "sweep", "10007x30011x1009", 3_000_017, "1.1x1.1x0", 25, "f32"),
        # One mode's product again and again with new factors (a user's own update loop), even rank.
        _case("mode_repeat", "mode", "50021x4001x20011", 5_000_011, "0x1.1x1.1", 50, "f32", mode=1),
        # The benchmark's sweep: three long skewed modes, one of them with short rows.
        _case("sweep_3mode", "sweep", "120000x90000x2000000", 100_000_000, "1.1x1.1x1.1", 32, "f32"),
        # The same shape with BF16 factors (half the gathered bytes), as an inner step of a user's solver.
        _case("sweep_3mode_bf16", "sweep", "120000x90000x2000000", 30_000_000, "1.1x1.1x1.1", 32, "bf16"),
        # Four modes, two skewed and two short uniform ones, wide rows.
        _case("sweep_4mode", "sweep", "1000000x20000x2000x500", 40_000_000, "1.2x1.2x0x0", 64, "bf16"),
        # One ALS iteration on a five-mode tensor.
        _case("als_5mode", "als_run", "500000x50000x5000x1000x200", 20_000_000,
              "1.1x1.1x1.1x1.1x1.1", 32, "f32", iters=1),
        # Six modes at a small rank: the index stream outweighs the factor rows.
        _case("sweep_6mode", "sweep", "100000x20000x2000x500x100x50", 20_000_000,
              "1.1x1.1x1.1x1.1x1.1x1.1", 16, "f32"),
        # A completion step: loss of the observed entries and all gradients, two long modes.
        _case("loss_3mode", "loss", "2000000x2000000x100000", 50_000_000, "1.1x1.1x1.1", 64, "f32"),
        # The same step in BF16 on a smaller tensor, as an optimiser's inner step.
        _case("loss_3mode_bf16", "loss", "120000x90000x200000", 8_000_009, "1.1x1.1x1.1", 32, "bf16"),
        # Loss and gradients with four modes (separate forward pass).
        _case("loss_4mode", "loss", "100003x20011x2003x503", 10_000_019, "1.2x1.2x0x0", 16, "f32"),
    ]


def _case(name, kind, dims, nnz, skew, rank, dtype, mode=0, iters=1):
    return {"name": name, "kind": kind, "dims": dims, "nnz": nnz, "skew": skew, "rank": rank,
            "dtype": dtype, "mode": mode, "iters": iters}


def draw(rng):
    """A tensor of 3 to 6 modes, 20 thousand to 25 million nonzeros, rank 8 to 64."""
    kind = rng.choice(["sweep", "sweep", "sweep", "mode", "als", "als_run", "loss", "loss"])
    n = rng.choice([3, 3, 3, 4, 5, 6])
    rank = rng.choice([8, 10, 16, 16, 20, 25, 32, 32, 32, 48, 50, 64])
    iters = rng.randint(1, 2) if kind.startswith("als") else 1
    # up to the largest listed case's work, and less where rows are no whole 16-byte vectors
    most = 100e6 * 3 * 32 / (n * max(rank, 32) * iters * (4 if rank % 4 == 0 else 8))
    nnz = int(math.exp(rng.uniform(math.log(2e4), math.log(most))))
    top = 6.3 if n == 3 else 5.5 if n == 4 else 4.5
    while True:
        dims = [max(2, int(10 ** rng.uniform(2, top))) for _ in range(n)]
        if 5e3 * nnz < math.prod(dims) < 2 ** 62:
            break
    skew = [rng.choice([0, 1.05, 1.1, 1.1]) for _ in range(n)]
    if all(skew):  # leave room for distinct coordinates
        skew[dims.index(max(dims))] = 0
    dtype = "f32" if kind.startswith("als") else rng.choice(["f32", "f32", "bf16"])
    c = _case("", kind, "x".join(map(str, dims)), nnz, "x".join(map(str, skew)), rank, dtype,
              mode=rng.randrange(n) if kind == "mode" else 0,
              iters=iters)
    del c["name"]
    return c


def _dims(case):
    return [int(d) for d in case["dims"].split("x")]


def _index(g, count, dim, skew):
    """Indices of one mode: uniform, or Zipf(skew) over a random order of the rows."""
    if skew <= 0:
        return torch.randint(dim, (count,), generator=g, device="cuda")
    # summed on the host, in order: a scan on the GPU may round otherwise the next time
    cdf = torch.from_numpy(np.cumsum(np.arange(1, dim + 1, dtype=np.float64) ** -skew)).cuda()
    u = torch.rand(count, generator=g, device="cuda", dtype=torch.float64) * cdf[-1]
    rank = torch.searchsorted(cdf, u).clamp_(max=dim - 1)
    return torch.randperm(dim, generator=g, device="cuda")[rank]


def _inputs(case, seed):
    """Coordinates [nnz, N] int64 in random order, values, and factors, from the seed alone."""
    dims, nnz = _dims(case), case["nnz"]
    skew = [float(s) for s in case["skew"].split("x")]
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    count = int(1.3 * nnz) + 1024
    keys = torch.zeros(count, dtype=torch.int64, device="cuda")
    for d, s in zip(dims, skew):
        keys.mul_(d).add_(_index(g, count, d, s))
    keys = torch.unique(keys)
    while keys.numel() < nnz:  # heavy rows repeat coordinates: top up with uniform ones
        more = torch.zeros(nnz - keys.numel() + 1024, dtype=torch.int64, device="cuda")
        for d in dims:
            more.mul_(d).add_(_index(g, more.numel(), d, 0))
        keys = torch.unique(torch.cat([keys, more]))
    keys = keys[torch.randperm(keys.numel(), generator=g, device="cuda")[:nnz]]
    coo = torch.empty(nnz, len(dims), dtype=torch.int64, device="cuda")
    for k in reversed(range(len(dims))):
        coo[:, k] = keys % dims[k]
        keys = torch.div(keys, dims[k], rounding_mode="floor")
    vals = torch.rand(nnz, generator=g, device="cuda")
    scale = 0.3 if case["kind"] == "loss" else 1.0
    dtype = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    factors = [(torch.randn(d, case["rank"], generator=g, device="cuda") * scale).to(dtype)
               for d in dims]
    return coo, vals, factors


def prepare(case, seed):
    dims = _dims(case)
    coo, vals, factors = _inputs(case, seed)
    plan = Plan(coo, vals, dims, case["rank"], dtype=case["dtype"])
    del coo, vals
    torch.cuda.empty_cache()
    state = {"kind": case["kind"], "mode": case["mode"], "iters": case["iters"], "plan": plan,
             "factors": factors}
    if case["kind"] == "sweep":
        state["outs"] = [torch.empty(d, case["rank"], device="cuda") for d in dims]
    elif case["kind"] == "mode":
        state["outs"] = [torch.empty(dims[case["mode"]], case["rank"], device="cuda")]
    elif case["kind"] == "loss":
        state["factors"] = [f.requires_grad_(True) for f in factors]
    else:  # ALS updates factors in place: a copy to work on, started anew by every pass
        state["work"] = [f.clone() for f in factors]
        state["lam"] = torch.empty(case["rank"], device="cuda")
    return state


def run(state):
    plan, factors, kind = state["plan"], state["factors"], state["kind"]
    if kind == "sweep":
        plan.sweep(factors, state["outs"])
        return state["outs"]
    if kind == "mode":
        plan.compute(state["mode"], factors, state["outs"][0], keep_order=True)
        return state["outs"]
    if kind == "loss":
        loss = cp_loss(plan, factors)
        return [loss.detach(), *torch.autograd.grad(loss, factors)]
    for w, f in zip(state["work"], factors):
        w.copy_(f)
    if kind == "als":
        lam, fits = cp_als(plan, state["work"], state["iters"])
    else:
        lam = state["lam"]
        fits = plan.als_run(state["work"], lam, state["iters"])
    # the residual |X - Y| / |X| of every iteration, which is what a solver watches
    return [*state["work"], lam, *[1.0 - f for f in fits]]


def work(case):
    """Each pass streams the stored nonzeros (N indices and a value) once and writes them once
    in the next mode's order; each factor row that can be touched is read once and the result
    written once.  A mode repeated in place writes no reordered copy."""
    dims, nnz, rank = _dims(case), case["nnz"], case["rank"]
    n, size = len(dims), 2 if case["dtype"] == "bf16" else 4
    element = 4 * n + 4
    rows = [min(d, nnz) for d in dims]

    def one(k, copies):
        read = sum(rows[j] for j in range(n) if j != k) * rank * size
        return copies * nnz * element + read + dims[k] * rank * 4

    flops = nnz * rank * n  # a mode: N - 1 products and one sum per rank entry
    if case["kind"] == "mode":
        return {"bytes": one(case["mode"], 1), "flops": flops}
    bytes_, flops = sum(one(k, 2) for k in range(n)), n * flops
    if case["kind"] == "loss":  # the model value of every nonzero, and one copy less to order
        bytes_ += rows[0] * rank * size - nnz * element
        flops += nnz * rank * 2
    elif case["kind"] != "sweep":  # Gram matrices and solves
        bytes_ = case["iters"] * (bytes_ + sum(dims) * rank * 8)
        flops = case["iters"] * (flops + sum(dims) * rank * rank * 4)
    return {"bytes": bytes_, "flops": flops}


def _mttkrp64(coo, vals, factors, k):
    """sum over nonzeros of val * the product of the other modes' rows, in 64 bits."""
    out = torch.zeros(factors[k].shape, dtype=torch.float64, device="cuda")
    step = max(1, (1 << 26) // out.shape[1])
    for a in range(0, coo.shape[0], step):
        ix = coo[a:a + step]
        p = vals[a:a + step, None].double().expand(-1, out.shape[1]).clone()
        for j, f in enumerate(factors):
            if j != k:
                p *= f[ix[:, j]]
        out.index_add_(0, ix[:, k], p)
    return out


def _residual64(coo, vals, factors):
    out = torch.empty(coo.shape[0], dtype=torch.float64, device="cuda")
    step = max(1, (1 << 26) // factors[0].shape[1])
    for a in range(0, coo.shape[0], step):
        ix = coo[a:a + step]
        p = factors[0][ix[:, 0]]
        for j in range(1, len(factors)):
            p = p * factors[j][ix[:, j]]
        out[a:a + step] = p.sum(1) - vals[a:a + step]
    return out


def exact(case, seed):
    coo, vals, factors = _inputs(case, seed)
    factors = [f.double() for f in factors]
    n = len(factors)
    if case["kind"] == "sweep":
        return [_mttkrp64(coo, vals, factors, k) for k in range(n)]
    if case["kind"] == "mode":
        return [_mttkrp64(coo, vals, factors, case["mode"])]
    if case["kind"] == "loss":
        r = _residual64(coo, vals, factors)
        return [0.5 * (r * r).sum(), *[_mttkrp64(coo, r, factors, k) for k in range(n)]]
    norm2, residuals = vals.double().square().sum(), []
    for _ in range(case["iters"]):
        for k in range(n):
            m = _mttkrp64(coo, vals, factors, k)
            v = torch.ones(m.shape[1], m.shape[1], dtype=torch.float64, device="cuda")
            for j in range(n):
                if j != k:
                    v *= factors[j].T @ factors[j]
            u = torch.cholesky_solve(m.T, torch.linalg.cholesky(v)).T
            lam = u.norm(dim=0)
            factors[k] = u / lam
        v *= factors[n - 1].T @ factors[n - 1]
        inner = (m * factors[n - 1] * lam).sum()
        residuals.append(((norm2 + lam @ v @ lam - 2 * inner).clamp(min=0) / norm2).sqrt().item())
    return [*factors, lam, *residuals]
