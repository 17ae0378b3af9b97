"""The per-wave checker of single traces (csrc/hr_runs.cu: variants 0 to 3 and every-epoch regions)
== CPU oracle where its own structure could go wrong: waves around the 32-, 64- and 128-record
steps, words every thread meets (the table of absorbed accesses, with words that share its slots,
over several kernels), and queues that fill within one wave."""
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


def trace_of(rng, lengths, words, n_threads, ops, kernels=1):
    """One wave per length: random accesses of `words`, a block clock per wave."""
    parts = []
    for k in range(kernels):
        for bc, n in enumerate(lengths):
            r = np.zeros(n, tg.RECORD)
            r["word"] = rng.choice(words, n)
            r["tid"] = rng.integers(0, n_threads, n)
            r["bc"], r["kernel"] = bc, k
            r["op"] = rng.choice(ops, n)
            parts.append(r)
    return np.concatenate(parts)


CASES = {
    "step edges": dict(lengths=[1, 31, 32, 33, 63, 64, 65, 127, 128, 129, 1023, 1024, 1025, 1], words=np.arange(700),
                       n_threads=512, ops=[0, 1, 2], kernels=2),
    "one word": dict(lengths=[3000, 1, 3000], words=np.array([5]), n_threads=4096, ops=[2], kernels=9),
    "hot words, shared slots": dict(lengths=[20000, 20000], words=np.array([1, 2049, 4097, 7, 2055]), n_threads=9000,
                                    ops=[0] * 60 + [1], kernels=3),
    "reads, then atomics": dict(lengths=[40000], words=np.arange(64), n_threads=70000, ops=[0, 0, 0, 2], kernels=10),
    "all change": dict(lengths=[9000], words=np.arange(6000), n_threads=64, ops=[1], kernels=1),
}


@pytest.mark.parametrize("name", CASES)
@pytest.mark.parametrize("block_dim", [64, 96])
def test_variants_equal_oracle(oracle_mod, hr, name, block_dim):
    import torch
    rng = np.random.default_rng(len(name) + block_dim)
    tr = trace_of(rng, **CASES[name])
    n_words = int(tr["word"].max()) + 1
    d = torch.from_numpy(tr.view(np.uint8)).cuda()
    # (the form that does not recompute clocks: these traces leave the barrier records out)
    want = oracle_mod.race_keys(oracle_mod.bruteforce_parallel(tr, block_dim, n_words))
    shadows = set()
    for variant in range(6):  # (4 and 5: the other per-wave checker, the same shadow)
        shadow = torch.zeros(n_words, dtype=torch.int64, device="cuda")
        with hr.Checker([dict(n_words=n_words, block_dim=block_dim)], buffers=[shadow]) as ck:
            ck.set_variant(variant)
            ck.check_trace(0, d)
            races, status, n, _ = ck.report(0)
            assert status == hr.HR_OK and n == len(want) and hr.race_keys(races) == want, variant
            assert ck.counters(0)["accesses"] == len(tr)
            shadows.add(shadow.cpu().numpy().tobytes())
    assert len(shadows) == 1
    # every-epoch regions: the same races as in a batch, which the other checker takes
    reg = dict(n_words=n_words, block_dim=block_dim, report_mode=hr.REPORT_EVERY_EPOCH)
    with hr.Checker([reg] * 3) as ck:
        ck.check_trace(0, d)
        ck.check_batch([(1, d), (2, d)])
        told = [ck.report(i) for i in range(3)]
    assert [t[1] for t in told] == [hr.HR_OK] * 3
    keys = [hr.race_keys(t[0]) for t in told]
    assert keys[0] == keys[1] == keys[2] and want <= keys[0] and told[0][2] == len(keys[0])
