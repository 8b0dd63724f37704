"""Plans whose blocks are cut again after work has been captured on them: a re-cut frees the
block tables, the partials and the lists of empty rows that captured graphs point at."""
import numpy as np
import pytest
import torch

import oracle as O
import synth
from paper_2405_08470_gb300 import Plan, SpmError

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


@pytest.mark.parametrize("dims,skew", [((300, 200, 100), (1.1, 1.1, 0.0)),
                                       ((3000, 40, 20, 10), (0.0, 1.1, 0.0, 0.0))])
def test_recut_that_does_not_fit_leaves_the_plan_as_it_was(dims, skew):
    """A plan at its memory cap: the autotuner's larger block counts need larger tables and
    partials than the cap allows, which is a status; the plan keeps the blocks it had and
    computes with them (FP32 bar of the other parity tests)."""
    R, N = 32, len(dims)
    coo, vals = synth.make_coo(dims, 20_000, skew, seed=N)
    c, v = coo.numpy(), vals.numpy()
    probe = Plan(c, v, dims, R, max_bytes=1 << 30)
    need = probe.info()["device_bytes"]
    probe.close()
    p = Plan(c, v, dims, R, max_bytes=need + (64 << 10))
    before = [p.info(n)["nblk"] for n in range(N)]
    F = [f.cuda() for f in synth.make_factors(dims, R, seed=7)]
    outs = [torch.empty(d, R, device="cuda") for d in dims]
    p.sweep(F, outs, graph=True)
    with pytest.raises(SpmError) as ei:
        p.autotune(F, outs, ignore_cache=True)
    assert ei.value.status == -4
    assert [p.info(n)["nblk"] for n in range(N)] == before
    assert p.info()["device_bytes"] <= need + (64 << 10)
    for graph in (False, True):
        for o in outs:
            o.fill_(float("nan"))
        p.sweep(F, outs, graph=graph)
        p.device_status()
        for n in range(N):
            want = O.mttkrp(c, v, dims, [f.cpu().numpy() for f in F], n)
            assert O.relerr(outs[n].cpu().numpy(), want) <= 1e-5, (graph, n)
    p.close()
