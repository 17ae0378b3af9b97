"""Checks for which no variant was chosen, at sizes where the library picks the checker itself:
the same status, races and shadow as the per-wave checker, whichever way the choice falls (waves,
skew, filters, packings, errors, calls that continue a kernel, stream capture), and for both
cluster sizes of the binned checker's scatter."""
import numpy as np
import pytest

from paper_2401_04701_gb300 import tracegen as tg

pytestmark = pytest.mark.gpu

N, WORDS = (1 << 18) + 777, (1 << 20) + 333     # just above the smallest records and segments


@pytest.fixture(scope="module")
def hr():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2401_04701_gb300 import hirace
    return hirace


def trace_of(seed, n=N, words=WORDS, waves=30, kernels=1, threads=1 << 14, hot=0.0, tid_base=0):
    rng = np.random.default_rng(seed)
    r = np.zeros(n, tg.RECORD)
    # half the accesses meet their words from one thread only, half from anywhere
    r["tid"] = rng.integers(0, threads, n)
    own = rng.random(n) < 0.5
    r["word"] = np.where(own, r["tid"].astype(np.int64) * (words // threads), rng.integers(0, words, n))
    r["word"][rng.random(n) < hot] = rng.integers(0, 64)
    r["tid"] += tid_base
    r["op"] = np.where(own, rng.choice([0, 1], n), rng.choice([0, 2], n, p=[0.9, 0.1]))
    at = np.sort(rng.integers(0, waves * kernels, n))
    at[:1], at[-1:] = 0, waves * kernels - 1
    r["bc"], r["kernel"] = at % waves, at // waves
    return r


# name -> (trace arguments, region arguments, filter, calls (0: one per kernel))
CASES = {
    "taken": (dict(), dict(), {}, 1),
    "block of 96": (dict(), dict(block_dim=96), {}, 1),
    "few waves": (dict(waves=2), dict(), {}, 1),
    "more waves than the binned checker takes": (dict(waves=300), dict(), {}, 1),
    "hub word": (dict(hot=0.4), dict(), {}, 1),
    "kernels, clears": (dict(waves=3, kernels=17), dict(), {}, 1),
    "three calls": (dict(waves=60, n=3 * N), dict(), {}, 3),
    "a call per kernel": (dict(waves=20, kernels=3, n=3 * N), dict(), {}, 0),
    "compact": (dict(waves=9), dict(shadow_bytes=4, tid_bits=14), {}, 1),
    "wide tids": (dict(tid_base=1 << 22), dict(), {}, 1),
    "window": (dict(words=2 * WORDS), dict(), dict(word_lo=1000, word_hi=1000 + WORDS), 1),
    "lanes and symmetric blocks": (dict(), dict(), dict(lane_mask=0x7FFF00FF, sym_lo=1, sym_hi=9, sym_stride=256), 1),
    "more segments": (dict(words=1 << 24, n=1 << 20), dict(), {}, 1),
}


def check(hr, trace, reg, filt, calls, variant, capture=False):
    import torch
    d = torch.from_numpy(trace.view(np.uint8)).cuda()
    cuts = [16 * (len(trace) * i // calls) for i in range(calls)] if calls else \
        [16 * int(i) for i in np.unique(trace["kernel"], return_index=True)[1]]
    cuts.append(d.numel())
    shadow = torch.full((reg["n_words"],), -1, dtype=torch.int64, device="cuda")
    with hr.Checker([reg], report_capacity=1 << 20, buffers=[shadow]) as ck:
        if filt:
            ck.set_filter(0, **filt)
        if variant is not None:
            ck.set_variant(variant)
        for a, b in zip(cuts[:-1], cuts[1:]):
            ck.check_trace(0, d[a:b])
        if capture:  # the same again from a graph, queued after an eager check
            torch.cuda.synchronize()
            graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
            with torch.cuda.graph(graph, stream=side):
                ck.reset(0, stream=side)
                ck.check_trace(0, d, stream=side)
            graph.replay()
            torch.cuda.synchronize()
        races, status, n, _ = ck.report(0)
        return status, n, hr.race_keys(races), shadow.cpu().numpy().tobytes(), ck.counters(0)["accesses"]


@pytest.mark.parametrize("name", CASES)
def test_default_equals_per_wave(hr, name):
    t, reg, filt, calls = CASES[name]
    trace = trace_of(len(name), **t)
    reg = dict(dict(n_words=WORDS if filt else t.get("words", WORDS), block_dim=64), **reg)
    want = check(hr, trace, reg, filt, calls, 3)
    assert want[0] == hr.HR_OK and want[1] == len(want[2]) > 100
    assert check(hr, trace, reg, filt, calls, None) == want
    got = check(hr, trace, reg, filt, calls, hr.binned_variant())
    assert got[:3] == want[:3] and (calls == 0 or got == want)   # (0: drops an older kernel's values)


@pytest.mark.parametrize("variant", [None, 3, 5, 6])
def test_capture(hr, variant):
    trace = trace_of(5)
    reg = dict(n_words=WORDS, block_dim=64)
    assert check(hr, trace, reg, {}, 1, variant, capture=True) == check(hr, trace, reg, {}, 1, 3)


@pytest.mark.parametrize("what", ["order", "range", "unsupported"])
def test_errors_as_the_per_wave_checker_has_them(hr, what):
    """The accesses before an error are still checked: the default route reports their races too."""
    trace = trace_of(6)
    if what == "order":
        trace["bc"][-5] = 0
    elif what == "range":
        trace["word"][-5] = WORDS
    else:
        trace["op"][-5] = 9
    reg = dict(n_words=WORDS, block_dim=64)
    want, got = check(hr, trace, reg, {}, 1, 3), check(hr, trace, reg, {}, 1, None)
    assert hr.STATUS[got[0]] == hr.STATUS[want[0]] == "HR_ERR_" + what.upper()
    clean = check(hr, trace_of(6), reg, {}, 1, 3)
    assert 0.9 * clean[1] < got[1] <= clean[1]


def test_host_trace_wave_limit_counts_over_pieces(hr, monkeypatch):
    """By default a host trace travels in pieces of 2^21 records; the limit of waves per call still
    holds for each 2^24 records together."""
    import torch
    monkeypatch.setenv("HR_MAX_WAVES", "8")
    for waves, status in ((8, "HR_OK"), (9, "HR_ERR_CAPACITY")):
        trace = trace_of(waves, n=(1 << 22) + 99, waves=waves)   # three pieces, at most 5 waves each
        with hr.Checker([dict(n_words=WORDS, block_dim=64)]) as ck:
            ck.check_trace_host(0, torch.from_numpy(trace.view(np.uint8)).pin_memory())
            assert hr.STATUS[ck.report(0, cap=0)[1]] == status


EVERY = ["taken", "block of 96", "few waves", "hub word", "kernels, clears", "three calls", "a call per kernel",
         "wide tids", "window", "more segments"]


@pytest.mark.parametrize("name", EVERY)
def test_every_epoch_equals_per_wave(hr, name):
    """Every-epoch regions: the default against the plain entry point, which is always per-wave."""
    import torch
    t, reg, filt, calls = CASES[name]
    trace = trace_of(len(name) + 100, **t)
    n_words = WORDS if filt else t.get("words", WORDS)
    reg = dict(dict(n_words=n_words, block_dim=64, report_mode=hr.REPORT_EVERY_EPOCH), **reg)
    d = torch.from_numpy(trace.view(np.uint8)).cuda()
    cuts = [16 * (len(trace) * i // calls) for i in range(calls)] if calls else \
        [16 * int(i) for i in np.unique(trace["kernel"], return_index=True)[1]]
    cuts.append(d.numel())
    told = []
    for aggregate in (False, True):
        shadow = torch.full((3 * n_words,), -1, dtype=torch.int64, device="cuda")
        with hr.Checker([reg], report_capacity=1 << 22, buffers=[shadow]) as ck:
            if filt:
                ck.set_filter(0, **filt)
            for a, b in zip(cuts[:-1], cuts[1:]):
                ck.check_trace(0, d[a:b], aggregate=aggregate)
            races, status, n, _ = ck.report(0)
            told.append((status, n, hr.race_keys(races), ck.counters(0)["accesses"], shadow.cpu().numpy().tobytes()))
    assert told[0][0] == hr.HR_OK and told[0][1] == len(told[0][2]) > 100
    assert told[1] == told[0]
