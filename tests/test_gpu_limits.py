"""What a check does at its limits: clocks at the edge of the compact packing and the largest
retry cap."""
import numpy as np
import pytest

from paper_2401_04701_gb300 import tracegen as tg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hr():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2401_04701_gb300 import hirace
    return hirace


def to_dev(trace):
    import torch
    return torch.from_numpy(np.ascontiguousarray(trace).view(np.uint8)).cuda()


@pytest.mark.parametrize("how", [None, 0, 1, 2, 3, 4, 5, 6, "plain", "batch"])
@pytest.mark.parametrize("tid_bits", [4, 5, 6, 7])
def test_compact_warp_clock_limit(hr, tid_bits, how):
    """The 8-byte value that the FSM works on holds 8 bits of wc, whatever the compact form has
    room for: two writes of one wave race up to wc 255, and beyond it the check reports the overflow."""
    for wcs, status, n in (([255, 255], "HR_OK", 1), ([254, 255], "HR_OK", 0), ([256, 256], "HR_ERR_CLOCK_OVERFLOW", 0),
                           ([300, 300], "HR_ERR_CLOCK_OVERFLOW", 0), ([44, 300], "HR_ERR_CLOCK_OVERFLOW", 0)):
        rec = np.zeros(2, tg.RECORD)
        rec["word"], rec["tid"], rec["wc"], rec["op"] = 1, [0, 1], wcs, tg.OP_W
        reg = dict(n_words=4, block_dim=16, warp_size=4, shadow_bytes=4, tid_bits=tid_bits)
        with hr.Checker([reg] * 2) as ck:
            if isinstance(how, int):
                ck.set_variant(how)
            if how == "batch":
                ck.check_batch([(0, to_dev(rec)), (1, to_dev(rec))])
            else:
                ck.check_trace(0, to_dev(rec), aggregate=how != "plain")
            _, got, races, _ = ck.report(0)
        assert (hr.STATUS[got], races) == (status, n), wcs


@pytest.mark.parametrize("variant", [0, 1, 2, 3])
@pytest.mark.parametrize("cap", [0xFFFFFFFF, 0xFFFFFFFE, 1 << 20])
def test_largest_retry_cap(oracle_mod, hr, variant, cap):
    """A retry cap near the top of its range is no limit: hot words, which every CTA has CASes out
    for at once, give the oracle's races and no contention."""
    rng = np.random.default_rng(variant)
    rec = np.zeros(1 << 16, tg.RECORD)
    rec["word"] = rng.integers(0, 4, len(rec))
    rec["tid"] = rng.integers(0, 4096, len(rec))
    rec["kernel"] = np.arange(len(rec)) * 4 // len(rec)
    rec["op"] = rng.choice([tg.OP_R, tg.OP_A], len(rec))
    want = oracle_mod.race_keys(oracle_mod.bruteforce_parallel(rec, 64, 4))
    with hr.Checker([dict(n_words=4, block_dim=64)]) as ck:
        ck.set_variant(variant)
        ck.set_limits(cas_retry_cap=cap)
        ck.check_trace(0, to_dev(rec))
        races, status, n, _ = ck.report(0)
        assert ck.counters(0)["accesses"] == len(rec)
    assert hr.STATUS[status] == "HR_OK" and n == len(want) and hr.race_keys(races) == want
