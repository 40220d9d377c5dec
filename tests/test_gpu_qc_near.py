"""Quarter-circle counts of pairs close to the circle: the consumer's quick
test decides all but the nearest pairs and hands their blocks to the exact one.
Pairs are planted through imported states: C = 1 reduces the mixing to x ^= own
(two equal partners cancel), so a state's x and xorshift word place its first
pair anywhere."""
import numpy as np
import pytest

from gpu_util import cuda_or_skip, oracle_gen

pytestmark = pytest.mark.gpu


def _xorshift32(z):
    z ^= (z << 13) & 0xFFFFFFFF
    z ^= z >> 17
    return z ^ ((z << 5) & 0xFFFFFFFF)


@pytest.mark.parametrize("S", [64, 200])
def test_planted_pairs_near_the_circle(S):
    torch, ci = cuda_or_skip()
    rng = np.random.default_rng(S)
    st = ci.States(S, xl="xorshift32", comb_size=1, seed=4)
    buf = st.export_state().copy()
    P = int(st.query().n_lanes)
    u32 = buf[512:512 + 36 * P].view(np.uint32).reshape(9, P)
    want = np.zeros(S, dtype=np.int64)
    for l in range(S):
        # o0 = x ^ own(1) and o1 = o0 ^ own(2) (array entries equal: partners cancel);
        # choose the source word, then x so that a^2 + b^2 comes close to 2^48
        best = None
        for _ in range(400):
            z0 = int(rng.integers(1, 1 << 32))
            w1 = _xorshift32(z0)
            w2 = _xorshift32(w1)
            o0 = int(rng.integers(0, 1 << 32))
            o1 = o0 ^ w2
            d = abs((o0 >> 8) ** 2 + (o1 >> 8) ** 2 - (1 << 48))
            if best is None or d < best[0]:
                best = (d, z0, o0 ^ w1, o0, o1)
        _, z0, x, o0, o1 = best
        # move o0 and o1 together through x's bits until the pair crosses the circle
        for bit in range(31, -1, -1):
            a, b = (o0 ^ (1 << bit)), (o1 ^ (1 << bit))
            d = abs((a >> 8) ** 2 + (b >> 8) ** 2 - (1 << 48))
            if d < best[0]:
                best = (d,) + best[1:]
                o0, o1, x = a, b, x ^ (1 << bit)
        u32[0, l], u32[4, l], u32[5, l] = z0, x, 0
        want[l] = (o0 >> 8) ** 2 + (o1 >> 8) ** 2 < (1 << 48)
    st.import_state(buf)
    first = st.generate_split(2, sink="qc", segments=1).cpu().numpy()  # the plain test: under a block
    assert np.array_equal(first, want)
    st.import_state(buf)
    out = st.generate_split(32, segments=1).cpu().numpy().view(np.uint32).astype(np.uint64) >> np.uint64(8)
    exact = (out[:, 0::2] ** 2 + out[:, 1::2] ** 2 < (1 << 48)).sum(axis=1)
    st.import_state(buf)
    assert np.array_equal(st.generate_split(32, sink="qc", segments=1).cpu().numpy(), exact)


@pytest.mark.parametrize("xl", ["xor128", "xorshift32", "xor64"])
def test_counts_over_many_pairs(xl):
    """2^24 pairs a source: a few of them fall into the exact test's zone."""
    torch, ci = cuda_or_skip()
    S, n = 1 << 14, 2048
    out = ci.States(S, xl=xl, seed=8).generate_split(n, segments=1)
    v = (out.long() & 0xFFFFFFFF) >> 8
    want = (v[:, 0::2] ** 2 + v[:, 1::2] ** 2 < (1 << 48)).sum(dim=1)
    got = ci.States(S, xl=xl, seed=8).generate_split(n, sink="qc", segments=1)
    assert torch.equal(got, want)
