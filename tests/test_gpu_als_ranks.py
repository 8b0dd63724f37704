"""The Gram Hadamard's inverse at ranks around the edges of its 16 x 16 blocks, through one
CP-ALS iteration against the FP64 oracle.  The factors are normal with more than 3 R rows,
so every V is well conditioned and the FP32 bar of the other ALS tests (1e-5) holds; the
zero column makes V singular at its last, first or a middle pivot, which is a status."""
import numpy as np
import pytest
import torch

import oracle as O
import synth
from paper_2405_08470_gb300 import Plan, SpmError

pytestmark = pytest.mark.gpu

DIMS = (300, 260, 220)


@pytest.mark.parametrize("R", [1, 2, 15, 16, 17, 31, 32, 33, 47, 48, 49, 63, 64, 65])
def test_als_iteration_at_block_edges(R):
    coo, vals = synth.make_coo(DIMS, 30_000, (0.0,) * 3, seed=R)
    c, v = coo.numpy(), vals.numpy()
    F0 = synth.make_factors(DIMS, R, seed=100 + R)
    p = Plan(c, v, DIMS, R)
    F = [f.cuda() for f in F0]
    lam = torch.empty(R, device="cuda")
    fit = p.als_iter(F, lam)
    Fo, lo, fo = O.cp_als_iter(c, v, DIMS, [f.numpy().astype(np.float64) for f in F0])
    assert abs(fit - fo) <= 1e-5
    assert O.relerr(lam.cpu().numpy(), lo) <= 1e-5
    for k in range(3):
        assert O.relerr(F[k].cpu().numpy(), Fo[k]) <= 1e-5, k
    p.close()


@pytest.mark.parametrize("R,col", [(16, 15), (16, 0), (17, 16), (32, 31), (33, 32), (48, 20), (64, 63)])
def test_singular_gram_hadamard_is_a_status(R, col):
    coo, vals = synth.make_coo(DIMS, 30_000, (0.0,) * 3, seed=R)
    p = Plan(coo.numpy(), vals.numpy(), DIMS, R)
    F = [f.cuda() for f in synth.make_factors(DIMS, R, seed=100 + R)]
    for f in F[1:]:
        f[:, col] = 0.0
    with pytest.raises(SpmError) as ei:
        p.als_iter(F, torch.empty(R, device="cuda"))
    assert "SPD" in str(ei.value)
    p.close()
