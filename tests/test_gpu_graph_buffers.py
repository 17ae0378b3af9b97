"""Scratch that a captured graph works in stays its own: later calls that need more of it get a larger
buffer beside it, and the graph's replays still give what they gave."""
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


def dev(trace):
    import torch
    return torch.from_numpy(trace.view(np.uint8)).cuda()


def keys(hr, ck, region):
    races, status, n, _ = ck.report(region)
    assert status == hr.HR_OK and n == len(races)
    return hr.race_keys(races)


def capture(queue):
    import torch
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=side):
        queue(side)
    return graph


@pytest.mark.parametrize("variant", [None, 6])
def test_binned_buffer_grows_beside_a_graph(hr, variant):
    import torch
    small, large = dev(trace_of(21)), dev(trace_of(22, n=8 * N))
    with hr.Checker([dict(n_words=WORDS, block_dim=64)]) as ck:
        if variant is not None:
            ck.set_variant(variant)
        ck.check_trace(0, small)
        want = keys(hr, ck, 0)
        assert len(want) > 100

        def queue(side):
            ck.reset(0, stream=side)
            ck.check_trace(0, small, stream=side)
        graph = capture(queue)
        for _ in range(2):
            graph.replay()
            torch.cuda.synchronize()
            assert keys(hr, ck, 0) == want
            ck.reset(0)
            ck.check_trace(0, large)     # outgrows the buffer the graph was captured with
            assert len(keys(hr, ck, 0)) > 100


def test_batch_scratch_grows_beside_a_graph(hr):
    import torch
    traces = [dev(trace_of(30 + i, n=20_000 + i, words=1 << 14, threads=512)) for i in range(5)]
    with hr.Checker([dict(n_words=1 << 14, block_dim=64)] * 5) as ck:
        ck.check_batch([(i, traces[i]) for i in range(2)])
        want = [keys(hr, ck, i) for i in range(2)]
        assert all(len(w) > 100 for w in want)

        def queue(side):
            for i in range(2):
                ck.reset(i, stream=side)
            ck.check_batch([(i, traces[i]) for i in range(2)], stream=side)
        graph = capture(queue)
        for _ in range(2):
            graph.replay()
            torch.cuda.synchronize()
            assert [keys(hr, ck, i) for i in range(2)] == want
            for i in range(5):
                ck.reset(i)
            ck.check_batch([(i, traces[i]) for i in range(5)])   # more jobs than the scratch was sized for
            ck.batch_reserve(64, 1 << 19)
            assert keys(hr, ck, 4)
