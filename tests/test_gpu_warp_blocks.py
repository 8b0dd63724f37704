"""The warp-block kernel at the sizes where its tiling can go wrong, against the FP64
oracle: ranks on every lane width (1, 2, 4 and 8 values a lane), factors aligned to less
than 16 bytes, block lengths around its chunks and tiles, rows of one nonzero, gaps of
empty rows, and more blocks than the resident warps hold (claimed from the counter).
FP32 sums of at most a few thousand products: normwise 1e-5, the bar of the other
parity tests."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_2405_08470_gb300 import Plan

pytestmark = pytest.mark.gpu


def check(coo, vals, dims, R, dtype="f32", offset=0, keep_order=False, **kw):
    c, v = coo.numpy(), vals.numpy()
    td = torch.bfloat16 if dtype == "bf16" else torch.float32
    F = [f.to(td) for f in synth.make_factors(dims, R, seed=3)]
    Fd = []
    for f in F:  # factors that start `offset` elements into their storage
        buf = torch.empty(f.numel() + offset, dtype=td, device="cuda")
        g = buf[offset:].view(f.shape)
        g.copy_(f)
        Fd.append(g)
    p = Plan(c, v, dims, R, dtype=dtype, checks=True, **kw)
    want = [oracle.mttkrp(c, v, dims, [f.double().numpy() for f in F], n) for n in range(len(dims))]
    for n in range(len(dims)):
        out = torch.full((dims[n], R), float("nan"), device="cuda")
        again = torch.full((dims[n], R), float("nan"), device="cuda")
        p.remap(n)
        p.compute(n, Fd, out, keep_order=True)
        p.compute(n, Fd, again)  # with the remap: the same sums
        assert oracle.relerr(out.cpu().numpy(), want[n]) <= 1e-5, n
        assert torch.equal(out, again), n
    idx, val = p.elements()
    want_idx, want_val = oracle.elements_in_order(c, v, 0)
    assert np.array_equal(idx, want_idx) and np.array_equal(val, want_val)
    p.close()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("N,R", [(3, 1), (3, 2), (3, 5), (3, 10), (3, 25), (3, 33), (3, 50), (3, 63),
                                 (3, 66), (3, 36), (4, 10), (4, 25), (4, 33), (5, 6), (5, 25), (5, 50),
                                 (6, 10), (6, 21), (6, 34), (6, 64), (2, 25), (7, 10)])
def test_lane_widths(N, R, dtype):
    dims = (60, 45, 30, 20, 11, 7, 5)[:N]
    coo, vals = synth.make_coo(dims, 2500 if N == 2 else 5003, (1.1,) * N, seed=N * 100 + R)
    check(coo[:2500] if N == 2 else coo, vals[:2500] if N == 2 else vals, dims, R, dtype=dtype, nblk=11)


@pytest.mark.parametrize("R,dtype,offset", [(32, "f32", 1), (32, "f32", 2), (32, "bf16", 1),
                                            (32, "bf16", 2), (32, "bf16", 4), (64, "bf16", 4),
                                            (50, "f32", 1), (64, "f32", 2)])
def test_factors_aligned_to_less(R, dtype, offset):
    dims = (60, 45, 30)
    coo, vals = synth.make_coo(dims, 5003, (1.1, 0.0, 1.1), seed=R + offset)
    check(coo, vals, dims, R, dtype=dtype, offset=offset, nblk=11)


@pytest.mark.parametrize("R", [8, 16, 32, 64, 25])
@pytest.mark.parametrize("nnz", [1, 7, 8, 9, 31, 32, 33, 63, 64, 65, 127, 128, 129, 257])
def test_chunk_and_tile_edges(nnz, R):
    dims = (300, 40, 700)
    coo, vals = synth.make_coo(dims, nnz, (0.0, 1.1, 0.0), seed=nnz)
    check(coo, vals, dims, R, nblk=1)
    check(coo, vals, dims, R, nblk=3, stages=3, tile=32)


@pytest.mark.parametrize("R,dtype", [(32, "f32"), (16, "f32"), (64, "bf16"), (25, "f32"), (4, "f32")])
def test_rows_of_one_nonzero_and_gaps(R, dtype):
    dims = (90001, 5, 200003)  # mode 0: mostly single nonzeros; mode 2: gaps between them
    coo, vals = synth.make_coo(dims, 30011, (0.0, 0.0, 0.0), seed=R)
    check(coo, vals, dims, R, dtype=dtype)


@pytest.mark.parametrize("R,N", [(32, 3), (16, 4), (25, 3)])
def test_claimed_blocks(R, N):
    dims = (700, 300, 50, 20)[:N]
    coo, vals = synth.make_coo(dims, 60000, (1.1, 1.1, 0.0, 0.0)[:N], seed=R)
    check(coo, vals, dims, R, nblk=20011)  # far more than two per resident warp


@pytest.mark.parametrize("variant", [0, 1, 2, 3])
@pytest.mark.parametrize("R,max_bytes", [(32, 0), (25, 0), (16, 0), (32, 1 << 30)])
def test_long_runs_of_empty_rows(R, max_bytes, variant):
    # runs of 31 to 34 empty rows (the line between the two ways), runs of thousands
    # before, between and after the nonempty rows, and a split row behind one; a plan with
    # a memory cap keeps no list of them
    rows = np.concatenate([[5000], 5001 + np.cumsum([32, 33, 34, 35, 1, 64, 65, 66, 5000, 1])])
    dims, r = (int(rows[-1]) + 3000, 40, 11), np.random.default_rng(1)
    c = np.unique(np.stack([np.concatenate([r.choice(rows, 300), np.full(300, rows[-2])]),
                            r.integers(0, 40, 600), r.integers(0, 11, 600)], 1), axis=0)
    assert len(np.unique(c[:, 0])) == len(rows)
    v = r.random(len(c)).astype(np.float32)
    check(torch.from_numpy(c), torch.from_numpy(v), dims, R, nblk=7, variant=variant,
          max_bytes=max_bytes)
