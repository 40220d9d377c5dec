"""The carry scan of split calls at the edges of its warps (up to 32, each with
ceil((K - 1) / 32) segments, eight loaded at a time), and the segment jumps,
against the oracle: outputs, digests and the state the call leaves."""
import numpy as np
import pytest

from gpu_util import cuda_or_skip, digest_rows, oracle_gen, u32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", ["xor", "bbs", "bbs16"])
@pytest.mark.parametrize("C", [2, 32])
@pytest.mark.parametrize("K", [2, 3, 9, 32, 33, 34, 65, 258, 300])
def test_segment_counts_equal_the_oracle(variant, C, K):
    torch, ci = cuda_or_skip()
    S, L, more = 40, 32 * K - 12, 20
    ref = oracle_gen(variant, "xor128", C, 6, 0, S)
    first, then = ref.streams(L), ref.streams(more)
    st = ci.States(S, variant=variant, comb_size=C, seed=6)
    assert np.array_equal(u32(st.generate_split(L, segments=K)), first)
    assert np.array_equal(u32(st.generate_split(more, segments=1)), then)
    st = ci.States(S, variant=variant, comb_size=C, seed=6)
    d = st.generate_split(L, sink="digest", segments=K).cpu().numpy().view(np.uint64)
    assert np.array_equal(d, digest_rows(first))
    assert np.array_equal(u32(st.generate_split(more, segments=1)), then)


def test_workspaces_are_given_back():
    """Two streams and threads share the workspace pool; when the last handle is
    freed the pool keeps nothing (the handles of earlier tests are collected
    first)."""
    torch, ci = cuda_or_skip()
    import gc
    import threading

    gc.collect()
    ref = oracle_gen("bbs", "xor128", 32, 9, 0, 64).streams(2048)
    out = {}

    def work(i):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            st = ci.States(64, variant="bbs", seed=9, stream=s)
            for _ in range(3):
                st.import_state(st.export_state(stream=s), stream=s)
            out[i] = st.generate(2048, stream=s)
            s.synchronize()
            st.free()

    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for i in range(4):
        assert np.array_equal(u32(out[i]), ref)
