"""Every ring depth and tile of the warp-block kernel at the ranks whose lane groups are one
lane (32 nonzeros a step, so a tile holds at least 32 U of them), against the FP64 oracle:
the plan's tile has to fit shared memory for each of them.  FP32 sums of at most a few
thousand products: normwise 1e-5, the bar of the other parity tests."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_2405_08470_gb300 import Plan

pytestmark = pytest.mark.gpu

DIMS = (40, 30, 12, 9, 7, 6, 5, 4, 4, 3, 3, 3, 2, 2, 2, 2)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("R", [1, 2, 4])
@pytest.mark.parametrize("N,element_bytes", [(2, 0), (3, 0), (3, 16), (4, 0), (4, 16), (5, 0), (6, 0),
                                             (7, 0), (8, 0), (11, 0), (12, 0), (15, 0), (16, 0)])
def test_rings_of_one_lane_groups(N, element_bytes, R, dtype):
    dims = DIMS[:N]
    coo, vals = synth.make_coo(dims, 900 if N == 2 else 3001, (1.1,) + (0.0,) * (N - 1),
                               seed=10 * N + R)
    c, v = coo.numpy(), vals.numpy()
    td = torch.bfloat16 if dtype == "bf16" else torch.float32
    F = [f.to(td) for f in synth.make_factors(dims, R, seed=3)]
    Fd = [f.cuda() for f in F]
    want = [oracle.mttkrp(c, v, dims, [f.double().numpy() for f in F], n) for n in range(N)]
    for stages in (0, 2, 3, 4):
        for tile in (0, 256):
            p = Plan(c, v, dims, R, dtype=dtype, stages=stages, tile=tile, nblk=5, checks=True,
                     element_bytes=element_bytes)
            outs = [torch.full((d, R), float("nan"), device="cuda") for d in dims]
            p.sweep(Fd, outs)
            for n in range(N):
                err = oracle.relerr(outs[n].cpu().numpy(), want[n])
                assert err <= 1e-5, (stages, tile, n, err)
            idx, _ = p.elements()
            assert np.array_equal(idx, oracle.elements_in_order(c, v, 0)[0])
            p.close()
