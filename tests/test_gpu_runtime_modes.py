"""The runtime-modes kernel (2 modes, 7 and more, packed nonzeros at odd ranks, ranks above 64
that are no multiple of four) where its chunks end early, against the FP64 oracle: short
blocks, rows that change inside a chunk, and every piece count of a lane.  FP32 sums of a
few hundred products: normwise 1e-5, the bar of the other parity tests."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_2405_08470_gb300 import Plan

pytestmark = pytest.mark.gpu

DIMS = (40, 30, 12, 9, 7, 6, 5, 4, 4, 3, 3, 3, 2, 2, 2, 2)


@pytest.mark.parametrize("N,element_bytes,R,dtype", [
    (2, 0, 4, "f32"), (2, 0, 25, "f32"), (2, 0, 32, "bf16"), (2, 0, 64, "f32"), (2, 16, 16, "f32"),
    (7, 0, 10, "f32"), (7, 0, 25, "bf16"), (8, 0, 1, "f32"), (9, 0, 32, "f32"), (16, 0, 4, "f32"),
    (16, 0, 25, "f32"), (16, 0, 64, "bf16"), (4, 16, 25, "f32"), (5, 16, 50, "f32"),
    (6, 16, 33, "bf16"), (3, 0, 66, "f32"), (3, 0, 130, "f32"), (3, 0, 255, "bf16")])
@pytest.mark.parametrize("nnz", [1, 3, 4, 5, 31, 33, 127, 401])
def test_chunk_ends(nnz, N, element_bytes, R, dtype):
    dims = DIMS[:N]
    coo, vals = synth.make_coo(dims, nnz, (1.1,) + (0.0,) * (N - 1), seed=nnz + N)
    c, v = coo.numpy(), vals.numpy()
    td = torch.bfloat16 if dtype == "bf16" else torch.float32
    F = [f.to(td) for f in synth.make_factors(dims, R, seed=3)]
    Fd = [f.cuda() for f in F]
    for nblk in (1, 3):
        p = Plan(c, v, dims, R, dtype=dtype, nblk=nblk, checks=True, element_bytes=element_bytes)
        outs = [torch.full((d, R), float("nan"), device="cuda") for d in dims]
        p.sweep(Fd, outs)
        for n in range(N):
            want = oracle.mttkrp(c, v, dims, [f.double().numpy() for f in F], n)
            assert oracle.relerr(outs[n].cpu().numpy(), want) <= 1e-5, (nblk, n)
        assert np.array_equal(p.elements()[0], oracle.elements_in_order(c, v, 0)[0])
        p.close()
