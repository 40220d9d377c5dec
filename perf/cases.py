"""The work that this library is used for, as measurable cases.

A case is a dict of plain values.  ``listed()`` holds the fixed ones,
``draw(rng)`` makes more of the same ranges, ``prepare(case, seed)`` builds
what a user's program has in hand before the call, ``run(state)`` is one pass
through the public entry points, ``work(case)`` is what the pass cannot do
without, and ``exact(case, seed)`` recomputes its outputs in 64-bit torch and
numpy arithmetic without this package.

Kinds:
  generate   one ``States`` object of S streams advanced by n outputs each:
             written (``States.generate``), counted (``generate_fused_qc``) or
             digested (``generate_digest``)
  batch      many requests of uneven size in one ``Batch.run``
  bg         chaotic Blum-Goldwasser encryption or decryption of a batch of
             messages

Every output is a whole number, so two implementations agree only if they are
equal bit for bit.  The generators' own state after the pass is among the
outputs.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

import paper_1112_5239_gb300 as ci
from paper_1112_5239_gb300 import _lib, workloads

MASK32 = 0xFFFFFFFF


# ------------------------------------------------------------------ cases
def listed() -> list[dict]:
    return [
        # a small draw, as a program makes between other work: about 100
        # numbers per stream (the paper's shape), latency counts
        _gen("xor128_small", "xor", "xor128", 1000, 100),
        # the library's plain parity workload: 4 Mi numbers
        _gen("xor128_plain", "xor", "xor128", 4096, 1024),
        # the paper's own use: very many threads, 100 numbers each
        _gen("xor128_threads", "xor", "xor128", 1000000, 100),
        # the benchmark's headline: one 1 GiB time chunk of 2^20 streams
        _gen("xor128_chunk", "xor", "xor128", 1 << 20, 256),
        # ragged rows: odd length and a stream count that fills no warp
        _gen("xorshift32_odd", "xor", "xorshift32", 50001, 1001, comb_size=8),
        # Sec. 7: numbers consumed in the kernel, nothing stored
        _gen("xor128_consumed", "xor", "xor128", 1 << 20, 1024, sink="qc"),
        # the secure variant, many streams
        _gen("bbs_wide", "bbs", "xor128", 1 << 16, 4096),
        # the secure variant, one long call for a few streams
        _gen("bbs_narrow", "bbs", "xor128", 32, 1 << 16),
        # Algorithm 5 as printed, many streams
        _gen("bbs16_wide", "bbs16", "xor128", 1 << 16, 1024),
        # uneven requests of many users in one launch
        {"name": "batch_uneven", "kind": "batch", "requests": 300, "mix": 4, "max_len_log2": 12},
        # many short secret messages to few recipients, each direction
        _bg("bg_encrypt", "encrypt", 1 << 18, 1024),
        _bg("bg_decrypt", "decrypt", 1 << 18, 1024),
    ]


def _gen(name, variant, xl, streams, length, comb_size=32, sink="written") -> dict:
    return {"name": name, "kind": "generate", "variant": variant, "xl": xl, "comb_size": comb_size,
            "streams": streams, "length": length, "sink": sink}


def _bg(name, direction, messages, chunks) -> dict:
    return {"name": name, "kind": "bg", "direction": direction, "messages": messages, "chunks": chunks}


def _log_int(rng, lo, hi) -> int:
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng) -> dict:
    """One more case: kinds and options as listed, sizes log-uniform over the
    listed ranges; no more outputs than the largest listed case of its kind."""
    kind = rng.choice(["xor", "xor", "xor", "bbs", "bbs", "bbs16", "batch", "bg"])
    if kind == "batch":
        return {"kind": "batch", "requests": _log_int(rng, 20, 300), "mix": rng.randrange(1 << 20),
                "max_len_log2": rng.choice([9, 10, 11])}
    if kind == "bg":
        messages = _log_int(rng, 1 << 10, 1 << 18)
        c = _bg("", rng.choice(["encrypt", "decrypt"]), messages, _log_int(rng, 32, 1024))
    else:
        cap = {"xor": 1 << 28, "bbs": 1 << 27, "bbs16": 1 << 26}[kind]
        streams = _log_int(rng, 32, 1 << 20) if kind == "xor" else _log_int(rng, 32, 1 << 16)
        longest = min(1 << 16, cap // streams)
        length = _log_int(rng, min(100, longest), longest)
        sink = rng.choice(["written", "written", "written", "qc", "digest"])
        if sink == "qc" or rng.random() < 0.5:
            length += length & 1
        c = _gen("", kind, rng.choice(["xor128", "xor128", "xorshift32", "xor64"]) if kind == "xor" else "xor128",
                 streams, length, rng.choice([32, 32, 16, 8, 4, 2]), sink)
    del c["name"]
    return c


# ---------------------------------------------------------------- prepare
def _states(streams, variant, xl, comb_size, seed):
    """A ``States`` whose state lies in a torch tensor, and that state as a
    uint8 tensor (what a checkpoint would hold)."""
    st = ci.States(streams, variant=variant, xl=xl, comb_size=comb_size, seed=seed, comb_seed=seed + 1,
                   memory="torch")
    d = st.query()
    off = int(d.state_dev) - st._buf.data_ptr()
    return st, st._buf[off:off + int(d.state_bytes)]


def _requests(case) -> list:
    """The requests of a batch case (sizes from the case alone)."""
    return workloads.batched_requests(case["mix"], case["requests"], case["max_len_log2"])


def _sink_of(r) -> str:
    """Small results are stored; large ones are counted or digested in the kernel."""
    if r.n_streams * r.n_per_stream <= 1 << 20:
        return "written"
    return "qc" if r.n_per_stream % 2 == 0 else "digest"


class _Requests:
    """A batch's requests over memory of the caller's own: the states in one
    arena, the written outputs in one buffer (every request on a 16-byte
    boundary, as an allocator gives), counts and digests in another."""

    def __init__(self, requests, seed):
        self.handles = []
        params, places, arena, words, sums = [], [], 0, 0, 0
        for i, r in enumerate(requests):
            p, _ = ci.make_params(r.variant, "xor128", 32, seed * 100003 + i, seed + 1)
            n = ctypes.c_uint64()
            _lib.call("ci_state_bytes", ctypes.byref(p), r.n_streams, ctypes.byref(n))
            params.append((p, int(n.value)))
            places.append((arena, words, sums))
            arena += -(-int(n.value) // 256) * 256
            if _sink_of(r) == "written":
                words += -(-r.n_streams * r.n_per_stream // 4) * 4
            else:
                sums += r.n_streams
        self.arena = torch.zeros(arena, dtype=torch.uint8, device="cuda")
        self.written = torch.zeros(words, dtype=torch.int32, device="cuda")
        self.sums = torch.zeros(sums, dtype=torch.int64, device="cuda")
        self.items = []
        for r, (p, n), (a, w, s) in zip(requests, params, places):
            h = ctypes.c_void_p()
            _lib.call("ci_init_states_at", ctypes.byref(p), r.n_streams, self.arena.data_ptr() + a, n,
                      ci.stream_ptr(), ctypes.byref(h))
            self.handles.append(h)
            sink = _sink_of(r)
            out = (self.written[w:w + r.n_streams * r.n_per_stream] if sink == "written"
                   else self.sums[s:s + r.n_streams])
            self.items.append((h, r.n_per_stream, sink, out))
        self.batch = ci.Batch(len(self.items))

    def __del__(self):
        for h in self.handles:
            _lib.call("ci_free_states", h)


def _bg_inputs(case, seed):
    keys = workloads.bg_batch(seed, case["messages"], n_keys=64)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    text = torch.randint(0, 32, (case["messages"], case["chunks"]), dtype=torch.uint8, device="cuda", generator=g)
    return {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in keys.items()}, text


def prepare(case, seed):
    if case["kind"] == "generate":
        S, n = case["streams"], case["length"]
        st, view = _states(S, case["variant"], case["xl"], case["comb_size"], seed)
        if case["sink"] == "written":
            out = torch.empty((S, n), dtype=torch.int32, device="cuda")
        else:
            out = torch.zeros(S, dtype=torch.int64, device="cuda")
        return {"kind": "generate", "sink": case["sink"], "st": st, "view": view, "n": n, "out": out}
    if case["kind"] == "batch":
        return {"kind": "batch", "work": _Requests(_requests(case), seed)}
    keys, text = _bg_inputs(case, seed)
    state = {"kind": "bg", "direction": case["direction"], "keys": keys, "out": torch.empty_like(text)}
    if case["direction"] == "encrypt":
        state["text"] = text
        state["y"] = torch.empty(case["messages"], dtype=torch.int64, device="cuda")
    else:
        state["text"], state["y"] = ci.bg_encrypt(keys["N"], keys["S0"], keys["r"], text)
    return state


# -------------------------------------------------------------------- run
def run(state):
    if state["kind"] == "generate":
        st, n, out = state["st"], state["n"], state["out"]
        if state["sink"] == "written":
            st.generate(n, out=out)
        elif state["sink"] == "qc":
            st.generate_fused_qc(n, counts=out)
        else:
            st.generate_digest(n, digest=out)
        return [out, state["view"]]
    if state["kind"] == "batch":
        w = state["work"]
        w.batch.run(w.items)
        return [w.written, w.sums, w.arena]
    k = state["keys"]
    if state["direction"] == "encrypt":
        return list(ci.bg_encrypt(k["N"], k["S0"], k["r"], state["text"], out=state["out"], y=state["y"]))
    return [ci.bg_decrypt(k["p"], k["q"], k["S0"], state["y"], state["text"], out=state["out"])]


# ------------------------------------------------------------------- work
# Integer operations per output, by the definitions: the xor-like's shifts
# and XORs (xor128: 3 + 4; XORshift: 3 + 3; xor64, two words: 2 x (3 + 3)),
# two XORs of partners and one of the state; a modular squaring as one
# product, one quotient product, one product back and two additions, a chunk
# as a mask, a shift and an OR.
_XL_OPS = {"xor128": 7, "xorshift32": 6, "xor64": 12}
_SQUARING = 5


def _per_output(variant, xl) -> int:
    if variant == "xor":
        return _XL_OPS[xl] + 3
    if variant == "bbs":
        return 11 * _SQUARING + 7 * 3 + 2 * 5 + 3
    return 12 * _SQUARING + 8 * 3 + 2 * 5 + 3


def _gen_work(variant, xl, S, n, sink):
    lanes = -(-S // 32) * 32
    words = {"xor": {"xor128": 4, "xorshift32": 1, "xor64": 2}[xl], "bbs": 2, "bbs16": 8}[variant]
    fixed = {"xor": 0, "bbs": 5, "bbs16": 8}[variant]  # moduli, reciprocals, array choice
    state = lanes * 4 * (2 * (words + 2) + fixed)
    out = 4 * S * n if sink == "written" else (16 if sink == "qc" else 8) * S
    ops = S * n * _per_output(variant, xl)
    if sink != "written":
        ops += S * n * 3
    return state + out, ops


def work(case) -> dict:
    if case["kind"] == "generate":
        b, f = _gen_work(case["variant"], case["xl"], case["streams"], case["length"], case["sink"])
    elif case["kind"] == "batch":
        b = f = 0
        for r in _requests(case):
            rb, rf = _gen_work(r.variant, "xor128", r.n_streams, r.n_per_stream, _sink_of(r))
            b, f = b + rb, f + rf
    else:
        cells = case["messages"] * case["chunks"]
        per_key = 25 if case["direction"] == "encrypt" else 33
        b = 2 * cells + case["messages"] * per_key
        f = cells * (_SQUARING + 3)
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ exact
def exact(case, seed):
    """The outputs of one pass from freshly prepared inputs, in the layout of
    ``run``; None for the state (bytes) and for cases that take too long."""
    if case["kind"] == "bg":
        return _exact_bg(case, seed)
    if case["kind"] != "generate":
        return None
    S, n, variant = case["streams"], case["length"], case["variant"]
    steps = {"xor": n, "bbs": 60 * n, "bbs16": 15 * n}[variant]
    if steps > 250000 or steps * S > 1 << 34:
        return None
    lanes = -(-S // 32) * 32
    with np.errstate(over="ignore"):
        draws = _Draws(seed, lanes)
        source, x, slot, arrays = _SOURCES[variant](case, draws)
    comb = _combination(variant, case["comb_size"], seed + 1)
    lane = torch.arange(lanes, device="cuda")
    base = lane - lane % case["comb_size"]
    o1, o2 = (base + comb[a, lane % case["comb_size"]] for a in arrays)
    sink = case["sink"]
    out = torch.zeros((S, n) if sink == "written" else S, dtype=torch.int32 if sink == "written" else torch.int64,
                      device="cuda")
    last = None
    for i in range(n):
        slot = source() ^ slot[o1] ^ slot[o2]
        x = x ^ slot
        if sink == "written":
            out[:, i] = x[:S].to(torch.int32)
        elif sink == "digest":
            out = out * (ci.DIGEST_MUL - (1 << 64)) + x[:S]
        elif i % 2 == 0:
            last = x >> 8
        else:
            b = x >> 8
            out += (last * last + b * b < 1 << 48)[:S].long()
    return [out, None]


_GAMMA = 0x9E3779B97F4A7C15


def _splitmix(counter):
    """splitmix64's output function on numpy uint64 counters (seed + i gamma)."""
    z = counter.astype(np.uint64)
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


class _Draws:
    """Draw k of lane l is output l 2^32 + k + 1 of splitmix64 from ``seed``;
    each lane keeps its own count of draws taken."""

    def __init__(self, seed, lanes):
        self.seed = np.uint64(seed)
        self.lane = np.arange(lanes, dtype=np.uint64) << np.uint64(32)
        self.k = np.zeros(lanes, dtype=np.uint64)

    def take(self, which=slice(None)):
        i = self.lane[which] + self.k[which] + np.uint64(1)
        self.k[which] += np.uint64(1)
        return _splitmix(self.seed + i * np.uint64(_GAMMA))

    def until(self, make, accept):
        """Per lane: draws until accept(make(draw), lanes) holds."""
        out = np.zeros(len(self.k), dtype=np.uint64)
        left = np.arange(len(self.k))
        while len(left):
            v = make(self.take(left), left)
            ok = accept(v, left)
            out[left[ok]] = v[ok]
            left = left[~ok]
        return out


def _dev(a):
    return torch.from_numpy(np.asarray(a).astype(np.int64)).cuda()


def _combination(variant, C, seed):
    """The combination arrays (two, or sixteen): Fisher-Yates permutations
    from splitmix64, the xor variant's second one free of equal positions."""
    count = 0

    def shuffled():
        nonlocal count
        a = list(range(C))
        for i in range(C - 1, 0, -1):
            j = int(_splitmix(np.array([(seed + (count + 1) * _GAMMA) % (1 << 64)], dtype=np.uint64))[0]) % (i + 1)
            count += 1
            a[i], a[j] = a[j], a[i]
        return a

    with np.errstate(over="ignore"):
        if variant != "xor":
            return torch.tensor([shuffled() for _ in range(16)], device="cuda")
        first = shuffled()
        second = shuffled()
        while C > 1 and any(a == b for a, b in zip(first, second)):
            second = shuffled()
    return torch.tensor([first, second], device="cuda")


def _seed_xor(case, draws):
    d0, d1, d2 = draws.take(), draws.take(), draws.take()
    lo, hi = np.uint64(MASK32), np.uint64(32)
    xl = case["xl"]
    if xl == "xor128":
        w = [d0 & lo, d0 >> hi, d1 & lo, d1 >> hi]
        w[0] = np.where((w[0] | w[1] | w[2] | w[3]) == 0, np.uint64(1), w[0])
    elif xl == "xor64":
        w = [np.where(d0 == 0, np.uint64(1), d0)]
    else:
        w = [np.where(d0 & lo == 0, np.uint64(1), d0 & lo)]
    # xor64 uses all 64 bits: the int64 view keeps them
    w = [torch.from_numpy(v.view(np.int64).copy()).cuda() for v in w]

    def xor128():
        s = w[0] ^ (w[0] << 11 & MASK32)
        w[0], w[1], w[2] = w[1], w[2], w[3]
        w[3] = w[3] ^ (w[3] >> 19) ^ s ^ (s >> 8)
        return w[3]

    def xorshift32():
        z = w[0] ^ (w[0] << 13 & MASK32)
        z = z ^ (z >> 17)
        w[0] = z ^ (z << 5 & MASK32)
        return w[0]

    def xor64():
        z = w[0] ^ (w[0] << 13)
        z = z ^ ((z >> 7) & ((1 << 57) - 1))
        w[0] = z ^ (z << 17)
        return w[0] & MASK32

    return ({"xor128": xor128, "xorshift32": xorshift32, "xor64": xor64}[xl], _dev(d2 & lo), _dev(d2 >> hi), (0, 1))


def _is_prime(n, _lanes=None):
    """Miller-Rabin with bases 2, 7, 61 (exact below 2^32) for odd n < 2^31."""
    n = n.astype(np.uint64)
    d, s = n - np.uint64(1), np.zeros(len(n), dtype=np.int64)
    while True:
        even = d % np.uint64(2) == 0
        if not even.any():
            break
        d[even] >>= np.uint64(1)
        s[even] += 1
    prime = np.ones(len(n), dtype=bool)
    for a in (2, 7, 61):
        x = np.ones(len(n), dtype=np.uint64)
        b, e = np.full(len(n), a, dtype=np.uint64) % n, d.copy()
        while e.any():
            x = np.where(e & np.uint64(1) == 1, x * b % n, x)
            b = b * b % n
            e >>= np.uint64(1)
        good = (x == 1) | (x == n - np.uint64(1))
        for r in range(1, int(s.max())):
            x = x * x % n
            good |= (r < s) & (x == n - np.uint64(1))
        prime &= good
    return prime


def _blum(d, _lanes=None):
    return (np.uint64(1 << 30) + (d >> np.uint64(34))) | np.uint64(3)


def _crt_square(p, q, M, y):
    """A function that squares y modulo M = p q in place, p and q below 2^31,
    through the residues of p and q (products below 2^62)."""
    inv = _dev([pow(int(a), -1, int(b)) for a, b in zip(p.cpu().tolist(), q.cpu().tolist())])
    res = {"p": y % p, "q": y % q}

    def step():
        res["p"] = res["p"] * res["p"] % p
        res["q"] = res["q"] * res["q"] % q
        t = (res["q"] - res["p"] % q + q) % q * inv % q
        return res["p"] + p * t

    return step


def _seed_bbs(case, draws):
    p = draws.until(_blum, _is_prime)
    q = draws.until(_blum, lambda v, lanes: (v != p[lanes]) & _is_prime(v))
    M = p * q
    v = draws.until(lambda d, lanes: np.uint64(2) + d % (M[lanes] - np.uint64(2)),
                    lambda v, lanes: (v % p[lanes] != 0) & (v % q[lanes] != 0))
    d = draws.take()
    square = _crt_square(_dev(p), _dev(q), _dev(M), _dev(v))

    def word():
        t = torch.zeros(len(p), dtype=torch.int64, device="cuda")
        for _ in range(7):
            t = (t << 5 | square() & 31) & MASK32
        for _ in range(2):
            shift = square() & 3
            t = (t << shift & MASK32) | square() & ((1 << shift) - 1)
        return t

    arrays = (_dev(v & np.uint64(7)), 8 + _dev(v >> np.uint64(3) & np.uint64(7)))
    return word, _dev(d & np.uint64(MASK32)), _dev(d >> np.uint64(32)), arrays


def _seed_bbs16(case, draws):
    def factor(d, _lanes=None):
        return (np.uint64(128) + d % np.uint64(128)) | np.uint64(3)

    def prime(v, _lanes=None):
        return np.all([v % np.uint64(f) != 0 for f in (3, 5, 7, 11, 13)], axis=0)

    Ms, ys = [], []
    for _ in range(8):
        p = draws.until(factor, prime)
        q = draws.until(factor, lambda v, lanes: (v != p[lanes]) & prime(v))
        M = p * q
        ys.append(draws.until(lambda d, lanes: np.uint64(2) + d % (M[lanes] - np.uint64(2)),
                              lambda v, lanes: (v % p[lanes] != 0) & (v % q[lanes] != 0)))
        Ms.append(M)
    d = draws.take()
    M, y = torch.stack([_dev(m) for m in Ms]), torch.stack([_dev(v) for v in ys])
    weight = _dev([1 << 4 * (7 - k) for k in range(8)])[:, None]

    def one(k):
        y[k] = y[k] * y[k] % M[k]
        return y[k]

    arrays = (y[0] & 7, 8 + (y[1] & 7))

    def word():
        y.copy_(y * y % M)
        t = ((y & 15) * weight).sum(0)
        for a, b in ((2, 0), (6, 1)):
            shift = one(a) & 3
            t = (t << shift & MASK32) | one(b) & ((1 << shift) - 1)
        return t

    return word, _dev(d & np.uint64(MASK32)), _dev(d >> np.uint64(32)), arrays


_SOURCES = {"xor": _seed_xor, "bbs": _seed_bbs, "bbs16": _seed_bbs16}


def _exact_bg(case, seed):
    keys, text = _bg_inputs(case, seed)
    if case["direction"] == "decrypt":
        return [text]  # what was encrypted
    p, q, r = keys["p"], keys["q"], keys["r"]
    pool, place = np.unique(np.stack([p.cpu().numpy(), q.cpu().numpy()]), axis=1, return_inverse=True)
    inv = _dev([pow(int(a), -1, int(b)) for a, b in pool.T])[torch.from_numpy(place.reshape(-1)).cuda()]
    rp, rq = r % p * (r % p) % p, r % q * (r % q) % q
    key, out = keys["S0"].long(), torch.empty_like(text)
    for k in range(case["chunks"] + 1):
        x = rp + p * ((rq - rp % q + q) % q * inv % q)
        if k == case["chunks"]:
            return [out, x]
        key = key ^ (x & 31)
        out[:, k] = (text[:, k].long() ^ key).to(torch.uint8)
        rp, rq = rp * rp % p, rq * rq % q
