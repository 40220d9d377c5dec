"""Written rows of every length class and alignment (whole-group spans, TMA
tiles with a clipped last tile, line-staged rows), with guard words around the
output, against the oracle."""
import numpy as np
import pytest

from gpu_util import cuda_or_skip, oracle_gen, u32

pytestmark = pytest.mark.gpu

LENGTHS = (1, 3, 8, 16, 31, 32, 33, 36, 63, 64, 65, 100, 104, 279, 280, 281, 282, 284, 300, 301, 320, 333)
GUARD = 0x5A5A5A5A


@pytest.mark.parametrize("source", ["xor128", "xorshift32", "xor64", "bbs", "bbs16"])
@pytest.mark.parametrize("S", [1, 33, 96])
def test_rows_of_every_length_and_offset(source, S):
    torch, ci = cuda_or_skip()
    variant = source if source.startswith("bbs") else "xor"
    xl = "xor128" if variant != "xor" else source
    ref = oracle_gen(variant, xl, 32, 17, 0, S).streams(max(LENGTHS))
    for n in LENGTHS:
        for off in (0, 1, 2, 3):
            st = ci.States(S, variant=variant, xl=xl, seed=17)
            buf = torch.full((S * n + 64,), GUARD, dtype=torch.int32, device="cuda")
            st.generate_split(n, out=buf[16 + off:16 + off + S * n].view(S, n), segments=1)
            got = u32(buf)
            assert np.array_equal(got[16 + off:16 + off + S * n].reshape(S, n), ref[:, :n]), (n, off)
            assert np.all(got[:16 + off] == GUARD) and np.all(got[16 + off + S * n:] == GUARD), (n, off)
            st.free()


@pytest.mark.parametrize("n", [8, 100, 256, 777])
def test_more_groups_than_resident_warps(n):
    """States of more warp groups than fit the GPU at once (blocks of
    consecutive groups), ragged last group: the first, a middle and the last
    group against the oracle, written and consumed."""
    torch, ci = cuda_or_skip()
    S = 400_003
    out = u32(ci.States(S, seed=23).generate(n))
    counts = ci.States(S, seed=23).generate_fused_qc(n - n % 2).cpu().numpy() if n > 1 else None
    for lane0 in (0, 199_968, 399_968):
        rows = min(32, S - lane0)
        g = oracle_gen("xor", "xor128", 32, 23, 0, S, lane0=lane0, n_lanes=32)
        ref = g.generate(n)[:rows]
        assert np.array_equal(out[lane0:lane0 + rows], ref), lane0
        a, b = (ref[:, k:n - n % 2:2].astype(np.uint64) >> np.uint64(8) for k in (0, 1))
        assert np.array_equal(counts[lane0:lane0 + rows], ((a * a + b * b) < (1 << 48)).sum(axis=1)), lane0
