"""Plans whose blocks are cut again after work has been captured on them: a re-cut frees the
block tables, the partials and the lists of empty rows that captured graphs point at."""
import numpy as np
import pytest
import torch

import oracle as O
import synth
from paper_2405_08470_gb300 import Plan

pytestmark = pytest.mark.gpu


def test_als_loop_after_a_recut_uses_the_new_tables():
    """cp_als_run, autotune (which re-cuts for every candidate), the same cp_als_run: the
    second loop must not replay the first one's graph.  FP32 bar of the other ALS tests."""
    dims, R = (200, 150, 100), 16
    coo, vals = synth.make_coo(dims, 50_000, (0.0,) * 3, seed=5)
    c, v = coo.numpy(), vals.numpy()
    F0 = [f.cuda() for f in synth.make_factors(dims, R, seed=6)]
    F = [f.clone() for f in F0]
    lam = torch.empty(R, device="cuda")
    scratch = [torch.empty(d, R, device="cuda") for d in dims]
    p = Plan(c, v, dims, R, nblk=37)
    fits = []
    for _ in range(2):
        for a, b in zip(F, F0):
            a.copy_(b)
        fits.append(p.als_run(F, lam, 3))
        p.autotune(scratch, [torch.empty_like(s) for s in scratch], ignore_cache=True)
        assert p.info()["nblk"] != 37
    Fo = [f.cpu().numpy().astype(np.float64) for f in F0]
    for it in range(3):
        Fo, lo, fo = O.cp_als_iter(c, v, dims, Fo)
        assert abs(fits[0][it] - fo) <= 1e-5 and abs(fits[1][it] - fo) <= 1e-5, it
    assert O.relerr(lam.cpu().numpy(), lo) <= 1e-5
    for k in range(3):
        assert O.relerr(F[k].cpu().numpy(), Fo[k]) <= 1e-5, k
    p.close()
