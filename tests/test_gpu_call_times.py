"""Times that two forms of one call must not be apart by: ratios of device times
on the same GPU, minimum of several runs, with wide margins."""
import pytest

from gpu_util import cuda_or_skip

pytestmark = pytest.mark.gpu


def _us(torch, call, reps=20, runs=7):
    for _ in range(3):
        call()
    best = float("inf")
    for _ in range(runs):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        for _ in range(reps):
            call()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3 / reps)
    return best


def _written(torch, ci, S, n, offset=0, segments=None, **kw):
    st = ci.States(S, seed=1, **kw)
    out = torch.empty(S * n + offset, dtype=torch.int32, device="cuda")[offset:].view(S, n)
    if segments is None:
        return _us(torch, lambda: st.generate(n, out=out))
    return _us(torch, lambda: st.generate_split(n, out=out, segments=segments))


def test_a_warp_per_scheduler_costs_as_much_as_a_warp_per_sm():
    """Algorithm 5 as printed, three and one warp groups per SM: no scheduler has two of
    them while another has none."""
    torch, ci = cuda_or_skip()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    one = _written(torch, ci, 32 * sms, 1024, segments=1, variant="bbs16")
    two = _written(torch, ci, 32 * 3 * sms, 1024, segments=1, variant="bbs16")
    assert two < 1.25 * one, (one, two)


@pytest.mark.parametrize("S,n", [(1 << 17, 64), (1 << 17, 24), (1 << 15, 1024)])
def test_rows_off_a_16_byte_boundary(S, n):
    """Rows of a multiple of eight words from the second word of a buffer on,
    against rows one word longer: no bank conflicts between the rows of a warp."""
    torch, ci = cuda_or_skip()
    even, odd = (_written(torch, ci, S, k, offset=1, segments=1) for k in (n, n + 1))
    assert even < 1.5 * odd, (even, odd)


@pytest.mark.parametrize("variant,S,n", [("bbs16", 64, 130), ("bbs16", 64, 500), ("bbs16", 4800, 512),
                                         ("bbs", 30000, 130), ("bbs", 20000, 200), ("bbs", 10000, 130)])
def test_a_call_is_not_slower_than_whole(variant, S, n):
    """Calls that choose segments themselves, against one segment."""
    torch, ci = cuda_or_skip()
    chosen, whole = (_written(torch, ci, S, n, segments=k, variant=variant) for k in (None, 1))
    assert chosen < 1.25 * whole, (chosen, whole)


def test_digesting_is_not_slower_than_writing():
    """xor128, one warp per SM: the digest stores nothing."""
    torch, ci = cuda_or_skip()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    S, n = 32 * sms, 2048
    st = ci.States(S, seed=1)
    d = torch.zeros(S, dtype=torch.int64, device="cuda")
    digest = _us(torch, lambda: st.generate_split(n, sink="digest", out=d, segments=1))
    written = _written(torch, ci, S, n, segments=1)
    assert digest < written, (digest, written)
