"""Narrow xor-like calls in one launch of clusters: lengths at the edges of the
32 segments, ragged states, every sink and alignment, against the oracle, the
state left behind included."""
import numpy as np
import pytest

from gpu_util import cuda_or_skip, digest_rows, oracle_gen, u32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("xl", ["xor128", "xorshift32", "xor64"])
@pytest.mark.parametrize("S,C", [(1, 32), (33, 8), (200, 32)])
@pytest.mark.parametrize("n", [447, 448, 449, 1000, 1023, 1024, 1025, 1056, 2049, 4100])
def test_lengths_and_sinks_equal_the_oracle(xl, S, C, n):
    torch, ci = cuda_or_skip()
    orc = oracle_gen("xor", xl, C, 12, 0, S)
    ref, then = orc.streams(n), orc.streams(8)
    for off in (0, 1):
        st = ci.States(S, xl=xl, comb_size=C, seed=12)
        buf = torch.full((S * n + 64,), 777, dtype=torch.int32, device="cuda")
        st.generate(n, out=buf[16 + off:16 + off + S * n].view(S, n))
        got = u32(buf)
        assert np.array_equal(got[16 + off:16 + off + S * n].reshape(S, n), ref)
        assert np.all(got[:16 + off] == 777) and np.all(got[16 + off + S * n:] == 777)
        assert np.array_equal(u32(st.generate(8)), then)
    st = ci.States(S, xl=xl, comb_size=C, seed=12)
    assert np.array_equal(st.generate_digest(n).cpu().numpy().view(np.uint64), digest_rows(ref))
    assert np.array_equal(u32(st.generate(8)), then)
    if n % 2 == 0:
        st = ci.States(S, xl=xl, comb_size=C, seed=12)
        counts = torch.full((S,), 5, dtype=torch.int64, device="cuda")
        st.generate_fused_qc(n, counts=counts)
        a, b = (ref[:, k::2].astype(np.uint64) >> np.uint64(8) for k in (0, 1))
        assert np.array_equal(counts.cpu().numpy() - 5, ((a * a + b * b) < (1 << 48)).sum(axis=1))
        assert np.array_equal(u32(st.generate(8)), then)


@pytest.mark.parametrize("variant,n", [("xor", 1024), ("xor", 300), ("bbs", 200), ("bbs16", 200)])
def test_a_captured_call_replays(variant, n):
    """Captured into a graph, a short call of a narrow state is plain kernels;
    each replay goes on from the state the last one left."""
    torch, ci = cuda_or_skip()
    orc = oracle_gen(variant, "xor128", 32, 3, 0, 64)
    st = ci.States(64, variant=variant, seed=3)
    out = torch.empty((64, n), dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        st.generate(n, out=out)
    for _ in range(3):
        graph.replay()
        assert np.array_equal(u32(out), orc.streams(n))
