"""Default block counts.  Every block costs 2 R floats of split-row partials, so a plan under a
memory cap is cut into blocks of 256 nonzeros at least, at most 384 per SM and at most 4096
nonzeros each, whatever an uncapped one would take."""
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


@pytest.mark.parametrize("nnz", [11_000_001, 14_600_000])
def test_blocks_hold_256_nonzeros_while_they_are_few(nnz):
    """A block's lane groups each add their share of its nonzeros in FP32, so longer blocks
    round more: up to 384 blocks per SM they hold 256."""
    dims = (5000, 4001)
    k = np.arange(nnz, dtype=np.int64)
    p = Plan(np.stack([k // 4001, k % 4001], 1), np.ones(nnz, np.float32), dims, 8, host_only=True)
    sms = p.info()["num_sms"]
    want = max(min(sms * 384, -(-nnz // 256)), min(sms * 1024, -(-nnz // 512)))
    for n in range(2):
        assert p.info(n)["nblk"] == want
        assert np.diff(p.bounds(n)).max() <= 257
    p.close()


@pytest.mark.parametrize("R,dtype,variant,lanes", [
    (10, "f32", 0, 8), (10, "f32", 3, 8), (25, "f32", 0, 32), (32, "f32", 0, 8), (50, "f32", 0, 32),
    (32, "bf16", 0, 8), (64, "bf16", 0, 8), (36, "bf16", 0, 16), (10, "f32", 1, 16),
    (32, "bf16", 1, 4), (32, "f32", 2, 8)])
def test_plan_reports_the_lanes_of_its_kernel_form(R, dtype, variant, lanes):
    # forms 0 and 3: the widest piece of at most 16 bytes (8 for BF16 rows of at most 32
    # values) that divides the rank, lanes rounded up to a power of two; forms 1 and 2:
    # 16-byte pieces or single values
    coo = np.stack([np.arange(50), np.arange(50) % 7, np.arange(50) % 5], 1).astype(np.int64)
    p = Plan(coo, np.ones(50, np.float32), (50, 7, 5), R, dtype=dtype, variant=variant, host_only=True)
    assert p.info()["lanes"] == lanes
    p.close()


@pytest.mark.parametrize("N,R,dtype,unroll,element_bytes,steps", [
    (3, 32, "f32", 0, 0, 8), (3, 32, "f32", 4, 0, 4), (3, 32, "f32", 8, 16, 8), (3, 4, "f32", 8, 0, 4),
    (3, 25, "f32", 4, 0, 8), (3, 32, "bf16", 4, 0, 8), (3, 64, "bf16", 8, 0, 4), (3, 2, "f32", 0, 0, 4),
    (4, 32, "f32", 8, 0, 4), (5, 50, "f32", 0, 0, 4), (6, 32, "f32", 0, 0, 2), (6, 32, "bf16", 0, 0, 4),
    (7, 1, "f32", 0, 0, 4), (8, 1, "f32", 0, 0, 2), (2, 32, "f32", 0, 0, 4)])
def test_plan_reports_its_steps_in_flight(N, R, dtype, unroll, element_bytes, steps):
    # the unroll option is for FP32 with 3 modes and 16-byte lanes; elsewhere it is fixed
    coo = np.stack([np.arange(50) % (50 - n) for n in range(N)], 1).astype(np.int64)
    p = Plan(coo, np.ones(50, np.float32), [50 - n for n in range(N)], R, dtype=dtype,
             unroll=unroll, element_bytes=element_bytes, host_only=True)
    assert p.info()["steps"] == steps
    assert p.info()["hot_rows"] == 0 and p.info()["host_only"] == 1
    p.close()
