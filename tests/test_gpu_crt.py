"""BBS squaring on the residues of the two factors: which lengths, factors and
warps take it, against the oracle."""
import numpy as np
import pytest

import oracle
from gpu_util import cuda_or_skip, u32
from test_gpu_bbs_import import _apply, _barrett_mu, _views  # noqa: F401
from paper_1112_5239_gb300 import workloads as W

pytestmark = pytest.mark.gpu

S = P = 96
C, SEED = 32, 21


def _prime_from(c, step):
    while c % 4 != 3 or not oracle.is_prime(c):
        c += step
    return c


LOW = _prime_from((1 << 30) + 1, 1)       # the smallest Blum prime the residue form takes
HIGH = _prime_from((1 << 31) - 1, -1)     # the largest
BELOW = _prime_from((1 << 30) - 1, -1)    # just too short
MIDDLE = _prime_from(1518500249, 1)


def _edits(kind, lanes):
    """Factor pairs by lane; warp 1 holds the special ones, warps 0 and 2 seeded lanes."""
    pairs = {"ends": [(LOW, HIGH), (HIGH, LOW), (LOW, MIDDLE), (MIDDLE, HIGH)],
             "one_short": [(LOW, HIGH), (BELOW, HIGH), (HIGH, MIDDLE), (HIGH, BELOW)],
             "multiple": [(LOW, HIGH), (HIGH, MIDDLE)]}[kind]
    out = {}
    for l in range(32, 64):
        p, q = pairs[l % len(pairs)]
        M = p * q
        y = int(lanes[l]["y"]) % M
        if kind == "multiple":  # not units: a multiple of one factor, 0 and 1
            y = [p * (y % q), q * (y % p), 0, 1, M - 1][l % 5]
        out[l] = (p, q, M, y)
        lanes[l]["p"], lanes[l]["q"], lanes[l]["M"], lanes[l]["y"] = p, q, M, y
    return out


@pytest.mark.parametrize("kind", ["seeded", "ends", "one_short", "multiple"])
@pytest.mark.parametrize("L,segments", [(1, 0), (11, 0), (12, 0), (13, 0), (33, 0), (100, 2), (512, 5)])
def test_lengths_and_factors_equal_the_oracle(kind, L, segments):
    torch, ci = cuda_or_skip()
    if kind == "multiple" and segments:
        pytest.skip("the jump of a split call takes units")
    lanes = oracle.init_lanes(oracle.VAR_BBS, oracle.XL_XOR128, SEED, 0, P)
    st = ci.States(S, variant="bbs", comb_size=C, seed=SEED)
    if kind != "seeded":
        st.import_state(_apply(st.export_state().copy(), _edits(kind, lanes)))
    out = u32(st.generate_split(L, segments=segments) if segments else st.generate(L))
    ref, _ = oracle.run(oracle.VAR_BBS, oracle.XL_XOR128, C, oracle.comb_arrays(oracle.VAR_BBS, C, 0), lanes, L)
    assert np.array_equal(out, ref[:S])
    u32v, u64v = _views(st.export_state())
    assert np.array_equal(u64v[:P], lanes["y"])
    assert np.array_equal(u32v[4 * P:5 * P], lanes["x"])
    assert np.array_equal(u32v[5 * P:6 * P], lanes["tprev"])
    st.free()


@pytest.mark.parametrize("L", [1, 32, 45])
def test_decryption_with_factors_at_the_ends(L):
    """Warp 0: factors at both ends of the range, one rejected key; warp 1: one
    factor just below it (the 62-bit form); a ragged third warp."""
    torch, ci = cuda_or_skip()
    n = 70
    b = W.bg_batch(5, n, n_keys=8)
    for i, (p, q) in ((0, (LOW, HIGH)), (1, (HIGH, LOW)), (2, (MIDDLE, HIGH)), (40, (BELOW, HIGH)), (69, (HIGH, MIDDLE))):
        b["p"][i], b["q"][i], b["N"][i] = p, q, p * q
        b["r"][i] = int(b["r"][i]) % (p * q - 3) + 2
    m = W.bg_messages(6, n, L)
    dev = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in b.items()}
    c, y = ci.bg_encrypt(dev["N"], dev["S0"], dev["r"], torch.from_numpy(m).cuda())
    dev["p"][7] = 1 << 30  # not a prime: rejected
    rej = torch.zeros(1, dtype=torch.int32, device="cuda")
    got = ci.bg_decrypt(dev["p"], dev["q"], dev["S0"], y, c, rejected=rej).cpu().numpy()
    assert int(rej.item()) == 1
    m[7] = 0
    assert np.array_equal(got, m)
