"""Traces in host memory on a context with the binned variant chosen: cut into equal pieces of each
2^24 records, they give what one check from device memory gives, and the limit of waves per call
holds for the pieces of 2^24 records together."""
import numpy as np
import pytest

from tests.test_gpu_route import trace_of

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


@pytest.mark.parametrize("n", [(1 << 21) - 1, (1 << 22) + 99, (1 << 24) + 4_500_001])
def test_pieces_equal_one_check(hr, n):
    import torch
    words = (1 << 22) + 5
    trace = torch.from_numpy(trace_of(n % 97, n=n, words=words).view(np.uint8)).pin_memory()
    told = []
    for host in (False, True):
        shadow = torch.zeros(words, dtype=torch.int64, device="cuda")
        with hr.Checker([dict(n_words=words, block_dim=64)], report_capacity=1 << 22, buffers=[shadow]) as ck:
            ck.set_variant(hr.binned_variant() if host else 3)
            if host:
                ck.check_trace_host(0, trace)
            else:
                ck.check_trace(0, trace.cuda())
            races, status, total, _ = ck.report(0)
            told.append((status, total, hr.race_keys(races), ck.counters(0)["accesses"]))
        told[-1] += (shadow.cpu().numpy().tobytes(),)
    assert told[0][0] == hr.HR_OK and told[0][1] == len(told[0][2]) > 100
    assert told[1] == told[0]


def test_wave_limit_counts_over_pieces(hr, monkeypatch):
    import torch
    monkeypatch.setenv("HR_MAX_WAVES", "8")
    for waves, status in ((8, "HR_OK"), (9, "HR_ERR_CAPACITY")):
        trace = trace_of(waves, n=(1 << 22) + 99, words=1 << 20, waves=waves)   # two pieces, at most 5 waves each
        with hr.Checker([dict(n_words=1 << 20, block_dim=64)]) as ck:
            ck.set_variant(hr.binned_variant())
            ck.check_trace_host(0, torch.from_numpy(trace.view(np.uint8)).pin_memory())
            assert hr.STATUS[ck.report(0, cap=0)[1]] == status
