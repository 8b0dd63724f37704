"""Default block counts of plans under a memory cap: every block costs 2 R floats of split-row
partials, so a capped plan is cut into blocks of 256 nonzeros at least, at most 384 per SM
and at most 4096 nonzeros each, whatever an uncapped one would take."""
import numpy as np
import pytest

from paper_2405_08470_gb300 import Plan


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("nnz", [1, 63, 64, 255, 256, 257, 1000, 50_000, 77_800, 311_000])
def test_capped_plans_take_no_smaller_blocks(nnz):
    dims = (1000, 997, 50)
    k = np.arange(nnz, dtype=np.int64)
    coo = np.stack([k % 1000, (k * 7 + k // 1000) % 997, k // 997 % 50], 1)
    v = np.ones(nnz, np.float32)
    p = Plan(coo, v, dims, 8, host_only=True, max_bytes=1 << 40)
    sms = p.info()["num_sms"]
    want = max(min(sms * 384, -(-nnz // 256)), -(-nnz // 4096))
    for n in range(3):
        assert p.info(n)["nblk"] == want, n
    p.close()
