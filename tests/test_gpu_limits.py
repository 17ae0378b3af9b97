"""What a check does at its limits: clocks at the edge of the compact packing, the largest retry
cap, a stage wait that runs out, and the alignment of a shadow handed in."""
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


@pytest.mark.parametrize("how", ["first", "every"])
def test_no_access_passes_a_wait_that_ran_out(hr, how):
    """A stage wait that runs out ends the check there: the items that waited are not counted as
    done, so no later wave is applied (the hook holds the second stage; the races are in the third)."""
    lengths = [64, 1, 60_000]
    rec = np.zeros(sum(lengths), tg.RECORD)
    rec["bc"] = np.repeat(np.arange(3), lengths)
    rec["word"] = np.arange(len(rec))
    rec["tid"] = np.arange(len(rec))
    rec["op"] = tg.OP_W
    rec["word"][65:] = np.arange(60_000) // 2    # each word written by two threads of two blocks
    rec["tid"][65:] = (np.arange(60_000) % 2) * 64
    for variant in range(4) if how == "first" else [3]:
        reg = dict(n_words=len(rec), block_dim=64, report_mode=hr.REPORT_EVERY_EPOCH if how == "every" else 0)
        with hr.Checker([reg]) as ck:
            ck.set_variant(variant)
            ck.check_trace(0, to_dev(rec))
            assert ck.report(0, cap=0)[1:3] == (hr.HR_OK, 30_000)
            ck.reset(0)
            ck.set_limits(wait_ns=100_000_000, test_flags=1)
            ck.check_trace(0, to_dev(rec))
            _, status, n, _ = ck.report(0, cap=0)
        assert (hr.STATUS[status], n) == ("HR_ERR_TIMEOUT", 0), variant


@pytest.mark.parametrize("offset", [0, 1, 2, 3])
@pytest.mark.parametrize("words", [1, 2, 8191, 16384, 40_001])
def test_noalloc_shadow_at_any_multiple_of_8(oracle_mod, hr, words, offset):
    """The allocation-free check clears exactly its n_words values wherever an 8-byte shadow lies,
    and refuses one that no 64-bit atomic could work on."""
    import ctypes
    import torch
    rng = np.random.default_rng(words)
    rec = np.zeros(5000, tg.RECORD)
    rec["word"], rec["tid"] = rng.integers(0, words, len(rec)), rng.integers(0, 512, len(rec))
    rec["op"] = rng.integers(0, 2, len(rec))
    rec["kernel"] = np.arange(len(rec)) * 20 // len(rec)      # (clears between the tag groups, too)
    want = oracle_mod.race_keys(oracle_mod.bruteforce_parallel(rec, 64, words))
    d, buf = to_dev(rec), torch.full((words + 8,), -7, dtype=torch.int64, device="cuda")
    races = torch.zeros(1 << 20, dtype=torch.uint8, device="cuda")
    result = torch.zeros(2, dtype=torch.int64, device="cuda")
    fn = hr.load_library().hr_check_trace_noalloc
    P, u32, u64 = ctypes.c_void_p, ctypes.c_uint32, ctypes.c_uint64
    fn.argtypes, fn.restype = [P, u64, P, u64, u32, u32, P, u64, P, P], ctypes.c_int

    def call(shadow):
        return fn(d.data_ptr(), len(rec), shadow, words, 64, 32, races.data_ptr(), 1 << 16, result.data_ptr(),
                  torch.cuda.current_stream().cuda_stream)

    assert call(buf.data_ptr() + 8 * offset + 4) == 1           # HR_ERR_INVALID, before any launch
    assert call(buf.data_ptr() + 8 * offset) == 0
    torch.cuda.synchronize()
    n = int(result[0])
    assert int(result[1]) == 0 and n == len(want)
    assert hr.race_keys(races.cpu().numpy().view(hr.RACE_DTYPE)[:n]) == want
    assert (buf[:offset] == -7).all() and (buf[offset + words:] == -7).all()
    assert (buf[offset:offset + words] != -7).all()
