"""Single traces that one of two per-wave checkers takes by their waves: the same races, counts and
shadow on both sides of each line as the checker of the other shape gives."""
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


def told(ck, region, hr, shadow):
    races, status, n, _ = ck.report(region)
    assert status == hr.HR_OK and n > 100
    return n, hr.race_keys(races), ck.counters(region)["accesses"], shadow.cpu().numpy().tobytes()


# records, waves, kernels: below the least size, waves too short, in range (with clears), waves too long
@pytest.mark.parametrize("n,waves,kernels", [((1 << 21) - 1, 4, 1), ((1 << 21) + 1, 30, 1), ((1 << 21) + 1, 4, 1),
                                             (1 << 22, 1, 17), (2_600_000, 2, 1), (2_600_000, 1, 1)])
def test_every_epoch_shapes(hr, n, waves, kernels):
    """One trace against a batch, which hr_check_kernel takes; then the same as a later kernel."""
    import torch
    words = (1 << 19) + 3
    d = torch.from_numpy(trace_of(n % 89, n=n, words=words, waves=waves, kernels=kernels).view(np.uint8)).cuda()
    reg = dict(n_words=words, block_dim=64, report_mode=hr.REPORT_EVERY_EPOCH)
    small = torch.from_numpy(trace_of(3, n=5000, words=words).view(np.uint8)).cuda()
    shadows = [torch.zeros(3 * words, dtype=torch.int64, device="cuda") for _ in range(3)]
    with hr.Checker([reg] * 3, report_capacity=1 << 22, buffers=shadows) as ck:
        for later in range(2):
            if later:
                ck.check_trace(0, d, kernel_base=kernels)
            else:
                ck.check_trace(0, d)
                ck.check_batch([(1, d), (2, small)])
                assert told(ck, 0, hr, shadows[0]) == told(ck, 1, hr, shadows[1])
        first = len(ck.report(1)[0])
        assert ck.report(0, cap=0)[1:3] == (hr.HR_OK, 2 * first)


@pytest.mark.parametrize("variant", [None, 0, 1, 2, 3])
@pytest.mark.parametrize("n,block_dim,waves,words",
                         [((1 << 19) - 1, 96, 9, 1 << 14), (1 << 19, 96, 4, 1 << 14), (1 << 19, 96, 5, 1 << 14),
                          (1 << 19, 96, 5, (1 << 14) + 1), (512 * 1536, 96, 9, 512), (512 * 1536 + 1, 96, 9, 512),
                          ((1 << 18) - 1, 64, 9, 1 << 14), (1 << 18, 64, 9, 1 << 14), ((1 << 23) - 1, 64, 5, 1 << 14),
                          (1 << 23, 64, 5, 1 << 14), ((1 << 23) - 1, 96, 30, 1 << 14), (1 << 23, 96, 30, 1 << 14)])
def test_small_region_shapes(hr, variant, n, block_dim, waves, words):
    """Regions of a shared array's size: variants 0 to 3 against variant 5, on and beside each line."""
    import torch
    d = torch.from_numpy(trace_of(n % 83, n=n, words=words, waves=waves, kernels=2, threads=512).view(np.uint8)).cuda()
    shadows = [torch.zeros(words, dtype=torch.int64, device="cuda") for _ in range(2)]
    with hr.Checker([dict(n_words=words, block_dim=block_dim)] * 2, buffers=shadows) as ck:
        if variant is not None:
            ck.set_variant(variant)
        ck.check_trace(0, d)
        ck.set_variant(5)
        ck.check_trace(1, d)
        assert told(ck, 0, hr, shadows[0]) == told(ck, 1, hr, shadows[1])
