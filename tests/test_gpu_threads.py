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


def test_first_checks_while_another_thread_captures(hr):
    """A check that allocates its scratch, and one that outgrows it, queued by one thread while another
    captures a graph in the strictest mode: the capture stays valid and the checks are right."""
    import torch
    traces = [trace_of(7), trace_of(8, n=6 * N)]
    dev = [torch.from_numpy(t.view(np.uint8)).cuda() for t in traces]
    x, other, side = torch.zeros(1000, device="cuda"), torch.cuda.Stream(), torch.cuda.Stream()
    reg = dict(n_words=WORDS, block_dim=64)
    with hr.Checker([reg] * 4) as ck:
        ck.set_variant(3)
        for i, d in enumerate(dev):
            ck.check_trace(2 + i, d)
        want = [hr.race_keys(ck.report(2 + i)[0]) for i in range(2)]
    with hr.Checker([reg]) as ck:
        torch.cuda.synchronize()
        failed = []

        def work():
            try:
                for d in dev:
                    ck.reset(0, stream=other)
                    ck.check_trace(0, d, stream=other)
            except Exception as e:   # noqa: BLE001 (told by the main thread)
                failed.append(e)

        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side, capture_error_mode="global"):
            x.add_(1.0)
            t = threading.Thread(target=work)
            t.start()
            t.join()
        assert not failed
        graph.replay()
        torch.cuda.synchronize()
        assert float(x.sum()) == 1000.0
        races, status, n, _ = ck.report(0)
        assert (status, n, hr.race_keys(races)) == (hr.HR_OK, len(want[1]), want[1])
        ck.reset(0)
        ck.check_trace(0, dev[0])
        assert hr.race_keys(ck.report(0)[0]) == want[0]
