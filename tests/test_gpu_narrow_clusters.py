"""Narrow xor-like calls in clusters of one, two and four blocks (about 50 warp
groups up to two per SM), and the automatic segments of calls too long for that
form: the first, a middle and the last group against the oracle."""
import numpy as np
import pytest

from gpu_util import cuda_or_skip, digest_rows, oracle_gen, u32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S,n", [(1601, 1000), (1601, 1026), (1601, 2047), (5000, 1024), (5000, 2100), (9001, 1025),
                                 (9001, 2050), (40, 16386), (300, 20001), (1601, 17000)])
@pytest.mark.parametrize("xl", ["xor128", "xorshift32", "xor64"])
def test_wider_states_equal_the_oracle(xl, S, n):
    torch, ci = cuda_or_skip()
    P = (S + 31) // 32 * 32
    rows = {}
    for lane0 in sorted({0, P // 64 * 32, P - 32}):
        g = oracle_gen("xor", xl, 32, 31, 0, S, lane0=lane0, n_lanes=32)
        rows[lane0] = (g.generate(n)[:min(32, S - lane0)], g.generate(8)[:min(32, S - lane0)])

    def check(got, ref, what):
        for lane0, (first, then) in rows.items():
            want = ref(first, then)
            assert np.array_equal(got[lane0:lane0 + len(want)], want), (what, lane0)

    for off in (0, 1):
        st = ci.States(S, xl=xl, seed=31)
        buf = torch.full((S * n + 64,), 777, dtype=torch.int32, device="cuda")
        st.generate(n, out=buf[16 + off:16 + off + S * n].view(S, n))
        got = u32(buf)
        check(got[16 + off:16 + off + S * n].reshape(S, n), lambda a, b: a, off)
        assert np.all(got[:16 + off] == 777) and np.all(got[16 + off + S * n:] == 777)
        check(u32(st.generate(8)), lambda a, b: b, "state")
        st.free()
    st = ci.States(S, xl=xl, seed=31)
    check(st.generate_digest(n).cpu().numpy().view(np.uint64), lambda a, b: digest_rows(a), "digest")
    check(u32(st.generate(8)), lambda a, b: b, "state after the digest")
    if n % 2 == 0:
        st = ci.States(S, xl=xl, seed=31)

        def hits(a, b):
            x, y = (a[:, k::2].astype(np.uint64) >> np.uint64(8) for k in (0, 1))
            return ((x * x + y * y) < (1 << 48)).sum(axis=1)

        check(st.generate_fused_qc(n).cpu().numpy(), hits, "counts")
        check(u32(st.generate(8)), lambda a, b: b, "state after the counts")
