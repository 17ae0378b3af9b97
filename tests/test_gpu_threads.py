"""Two host threads that check different regions of one context at once, each on its own stream,
get what one thread gets: with the library's choice of checker, which allocates scratch on first
use, and with chosen ones."""
import threading

import numpy as np
import pytest

from tests.test_gpu_route import N, WORDS, trace_of

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


@pytest.mark.parametrize("variant", [None, 1, 3, 5, 6])
def test_two_regions_from_two_threads(hr, variant):
    import torch
    traces = [trace_of(1, n=N), trace_of(2, n=2 * N, waves=11)]
    dev = [torch.from_numpy(t.view(np.uint8)).cuda() for t in traces]
    regs = [dict(n_words=WORDS, block_dim=64), dict(n_words=WORDS, block_dim=96)]
    want = []
    for d, reg in zip(dev, regs):
        with hr.Checker([reg]) as ck:
            ck.set_variant(3)
            ck.check_trace(0, d)
            want.append(hr.race_keys(ck.report(0)[0]))
    assert all(len(w) > 100 for w in want)
    torch.cuda.synchronize()
    with hr.Checker(regs) as ck:
        if variant is not None:
            ck.set_variant(variant)
        start, got = threading.Barrier(2), [[], []]

        def work(i):
            stream = torch.cuda.Stream()
            start.wait()
            for _ in range(4):
                ck.reset(i, stream=stream)
                ck.check_trace(i, dev[i], stream=stream)
                races, status, n, _ = ck.report(i)
                got[i].append((status, n, hr.race_keys(races)))

        threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
    for i in range(2):
        assert got[i] == [(hr.HR_OK, len(want[i]), want[i])] * 4
