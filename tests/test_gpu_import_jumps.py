"""Time-split calls on imported states whose moduli are not the product of two
distinct primes, or whose BBS state is no unit: what ci_import_state accepts,
every call form must advance as the oracle does."""
import numpy as np
import pytest

import oracle
from gpu_util import cuda_or_skip, digest_rows, u32
from test_gpu_bbs_import import P, S, SEED, _apply, _views

pytestmark = pytest.mark.gpu

C = 32
LOW, Q31 = (1 << 30) + 3, (1 << 31) - 1                 # primes
COMPOSITE = 1500000003                                  # 3^2 43 983 3943, in (2^30, 2^31)
FACTORS = {
    "composite": [(LOW, COMPOSITE), (COMPOSITE, Q31), (COMPOSITE, COMPOSITE + 2)],
    "equal": [(LOW, LOW), (Q31, Q31), (65537, 65537), (65539, 65539)],
    "short_composite": [(3 ** 10, 3 ** 11), (3 ** 10, 131071), (255 * 257, 65537 * 3), (5, 4000000005)],
    "not_units": [(LOW, Q31), (65539, 131071)],
}


def _state(kind):
    """Edited lanes 32..63 for the import, and the oracle's lanes edited the same way."""
    lanes = oracle.init_lanes(oracle.VAR_BBS, oracle.XL_XOR128, SEED, 0, P)
    edits = {}
    for l in range(32, 64):
        p, q = FACTORS[kind][l % len(FACTORS[kind])]
        M = p * q
        assert 33 <= M.bit_length() <= 62
        y = int(lanes[l]["y"]) % M
        if kind == "not_units":
            y = [p * (y % q), q * (y % p), 0, 1, p][l % 5]
        edits[l] = (p, q, M, y)
        lanes[l]["p"], lanes[l]["q"], lanes[l]["M"], lanes[l]["y"] = p, q, M, y
    return edits, lanes


@pytest.mark.parametrize("kind", list(FACTORS))
@pytest.mark.parametrize("L,segments", [(100, 0), (128, 0), (300, 0), (1024, 0), (100, 2), (1024, 5)])
def test_bbs_moduli_equal_the_oracle(kind, L, segments):
    torch, ci = cuda_or_skip()
    edits, lanes = _state(kind)
    ref, _ = oracle.run(oracle.VAR_BBS, oracle.XL_XOR128, C, oracle.comb_arrays(oracle.VAR_BBS, C, 0), lanes, L)
    for sink in ("written", "digest"):
        st = ci.States(S, variant="bbs", comb_size=C, seed=SEED)
        st.import_state(_apply(st.export_state().copy(), edits))
        if segments:
            got = st.generate_split(L, sink=sink, segments=segments)
        else:
            got = st.generate(L) if sink == "written" else st.generate_digest(L)
        if sink == "written":
            assert np.array_equal(u32(got), ref[:S])
        else:
            assert np.array_equal(got.cpu().numpy().view(np.uint64), digest_rows(ref[:S]))
        u32v, u64v = _views(st.export_state())
        assert np.array_equal(u64v[:P], lanes["y"])
        assert np.array_equal(u32v[4 * P:5 * P], lanes["x"])
        assert np.array_equal(u32v[5 * P:6 * P], lanes["tprev"])
        st.free()


MODULI16 = [585, 8, 24, 3, 15, 255, 19683, 6561, 65535, 65534, 32768, 4, 65521, 257, 289, 143 * 143, 46341, 51 * 257]


@pytest.mark.parametrize("L,segments", [(100, 0), (128, 0), (300, 0), (1500, 0), (100, 2), (1024, 5)])
def test_bbs16_moduli_equal_the_oracle(L, segments):
    """Prime powers, even moduli, one prime, more than two; units and not."""
    torch, ci = cuda_or_skip()
    st = ci.States(S, variant="bbs16", comb_size=C, seed=SEED)
    buf = st.export_state().copy()
    f = buf[512:].view(np.uint32).reshape(25, P)
    lanes = oracle.init_lanes(oracle.VAR_BBS16, oracle.XL_XOR128, SEED, 0, P)
    for l in range(32, 64):
        for g in range(8):
            M = MODULI16[(3 * l + g) % len(MODULI16)]
            y = [0, 2 % M, 3 % M, M - 1, 51 % M, (12345 * l + g) % M][(l + g) % 6]
            f[9 + g, l], f[17 + g, l] = y, M
            lanes[l]["y16"][g], lanes[l]["m16"][g] = y, M
    ref, _ = oracle.run(oracle.VAR_BBS16, oracle.XL_XOR128, C, oracle.comb_arrays(oracle.VAR_BBS16, C, 0), lanes, L)
    for sink in ("written", "digest"):
        st.import_state(buf)
        if segments:
            got = st.generate_split(L, sink=sink, segments=segments)
        else:
            got = st.generate(L) if sink == "written" else st.generate_digest(L)
        if sink == "written":
            assert np.array_equal(u32(got), ref[:S])
        else:
            assert np.array_equal(got.cpu().numpy().view(np.uint64), digest_rows(ref[:S]))
        f2 = st.export_state()[512:].view(np.uint32).reshape(25, P)
        assert np.array_equal(f2[9:17].T, lanes["y16"]) and np.array_equal(f2[17:25].T, lanes["m16"])
        assert np.array_equal(f2[4], lanes["x"]) and np.array_equal(f2[5], lanes["tprev"])


@pytest.mark.parametrize("variant", ["xor", "bbs", "bbs16"])
def test_partner_tables_count_modulo_the_warp(variant):
    """An imported table whose bytes name the same lanes above 31: the plain
    loop's shuffles take them modulo 32, and so do calls in segments."""
    torch, ci = cuda_or_skip()
    st = ci.States(S, variant=variant, comb_size=C, seed=SEED)
    good = st.export_state().copy()
    high = good.copy()
    high[:512] += (np.arange(512) % 8 * 32).astype(np.uint8)
    for L, segments in ((100, 1), (600, 0), (3000, 0), (20000, 0), (300, 3)):
        out = []
        for buf in (good, high):
            st.import_state(buf)
            out.append(u32(st.generate_split(L, segments=segments) if segments else st.generate(L)))
        assert np.array_equal(out[0], out[1]), (L, segments)
