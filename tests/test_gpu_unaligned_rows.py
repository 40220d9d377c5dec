"""Written rows whose stride is a multiple of four words in buffers that are not
16-byte aligned, by every source and entry point that takes them: around the
lengths of a tile, ragged states, segments between other columns."""
import numpy as np
import pytest

from gpu_util import cuda_or_skip, oracle_gen, u32

pytestmark = pytest.mark.gpu
GUARD = 0x5A5A5A5A
LENGTHS = (4, 12, 28, 32, 36, 40, 60, 64, 68, 96, 100, 128, 132, 256, 260, 292, 296, 324)


def _check(buf, at, S, n, ref, what):
    got = u32(buf)
    assert np.array_equal(got[at:at + S * n].reshape(S, n), ref), what
    assert np.all(got[:at] == GUARD) and np.all(got[at + S * n:] == GUARD), what


@pytest.mark.parametrize("source", ["xor128", "xorshift32", "xor64", "bbs", "bbs16"])
@pytest.mark.parametrize("S", [1, 31, 64, 70])
def test_single_and_batched_calls(source, S):
    torch, ci = cuda_or_skip()
    variant = source if source.startswith("bbs") else "xor"
    xl = "xor128" if variant != "xor" else source
    ref = oracle_gen(variant, xl, 32, 19, 0, S).streams(max(LENGTHS))
    batch = ci.Batch(1)
    for n in LENGTHS:
        for off in (1, 2, 3, 29, 31):
            for form in ("call", "batch"):
                st = ci.States(S, variant=variant, xl=xl, seed=19)
                buf = torch.full((S * n + 96,), GUARD, dtype=torch.int32, device="cuda")
                out = buf[32 + off:32 + off + S * n].view(S, n)
                if form == "call":
                    st.generate_split(n, out=out, segments=1)
                else:
                    batch.run([(st, n, "written", out)])
                _check(buf, 32 + off, S, n, ref[:, :n], (n, off, form))
                st.free()


@pytest.mark.parametrize("variant", ["xor", "bbs", "bbs16"])
@pytest.mark.parametrize("n,segments", [(128, 3), (1000, 7), (1024, 0), (2048, 5), (20000, 0)])
def test_split_calls(variant, n, segments):
    torch, ci = cuda_or_skip()
    S = 70
    ref = oracle_gen(variant, "xor128", 32, 20, 0, S).streams(n)
    for off in (1, 2, 31):
        st = ci.States(S, variant=variant, seed=20)
        buf = torch.full((S * n + 96,), GUARD, dtype=torch.int32, device="cuda")
        out = buf[32 + off:32 + off + S * n].view(S, n)
        st.generate_split(n, out=out, segments=segments) if segments else st.generate(n, out=out)
        _check(buf, 32 + off, S, n, ref, off)
        st.free()


@pytest.mark.parametrize("S", [31, 70])
def test_naive(S):
    import oracle

    torch, ci = cuda_or_skip()
    for n in LENGTHS:
        ref = oracle.naive_run(oracle.naive_init_lanes(3, 0, S), n)
        for off in (1, 2, 3, 31):
            ns = ci.NaiveStates(S, seed=3)
            buf = torch.full((S * n + 96,), GUARD, dtype=torch.int32, device="cuda")
            ns.generate(n, out=buf[32 + off:32 + off + S * n].view(S, n))
            _check(buf, 32 + off, S, n, ref, (n, off))
