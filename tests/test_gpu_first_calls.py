"""First calls of a process, before the jump tables of the xor-like generators
exist on the device: each in a process of its own."""
import os
import subprocess
import sys

import pytest

from gpu_util import cuda_or_skip

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))

PRELUDE = """
import sys, time
sys.path[:0] = [%r, %r]
import numpy as np
import torch
import paper_1112_5239_gb300 as ci
from gpu_util import oracle_gen, u32
""" % (os.path.dirname(HERE), HERE)


def _run(code):
    cuda_or_skip()
    r = subprocess.run([sys.executable, "-c", PRELUDE + code], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("done"), r.stdout + r.stderr


@pytest.mark.parametrize("call", ["st.generate(4096, out=out)", "st.generate(20000, out=out)",
                                  "st.generate_split(4096, out=out, segments=4)"])
def test_a_captured_first_call_replays(call):
    n = 20000 if "20000" in call else 4096
    _run(f"""
S, n = 40, {n}
orc = oracle_gen("xor", "xor128", 32, 3, 0, S)
st = ci.States(S, seed=3)
out = torch.empty((S, n), dtype=torch.int32, device="cuda")
torch.cuda.synchronize()
graph = torch.cuda.CUDAGraph()
with torch.cuda.graph(graph):
    {call}
for _ in range(2):
    graph.replay()
    assert np.array_equal(u32(out), orc.streams(n))
assert np.array_equal(u32(st.generate(n)), orc.streams(n))
print("done")
""")


def test_other_streams_find_finished_tables():
    """The tables are built behind other work of the first call's stream; a call
    on another stream waits for them on the device."""
    _run("""
S = 40
orc, other = (oracle_gen("xor", "xor128", 32, seed, 0, S) for seed in (3, 4))
a, b = torch.cuda.Stream(), torch.cuda.Stream()
st, st2 = ci.States(S, seed=3), ci.States(S, seed=4)
out, out2 = (torch.empty((S, n), dtype=torch.int32, device="cuda") for n in (600, 20000))
torch.cuda.synchronize()
with torch.cuda.stream(a):
    torch.cuda._sleep(200_000_000)
st.generate(600, out=out, stream=a)
st2.generate(20000, out=out2, stream=b)
torch.cuda.synchronize()
assert np.array_equal(u32(out), orc.streams(600))
assert np.array_equal(u32(out2), other.streams(20000))
print("done")
""")


def test_a_first_call_does_not_wait():
    """Behind half a second of other work on its stream the first narrow call
    returns at once.  Kernels are loaded beforehand (the first launch of a lazily
    loaded kernel waits by itself), without torch and its many; the output lies
    in the memory of another state."""
    cuda_or_skip()
    code = """
import ctypes, importlib.util, sys, time
spec = importlib.util.spec_from_file_location("_lib", sys.argv[1])
lib = importlib.util.module_from_spec(spec)
spec.loader.exec_module(lib)

def state(S):
    h = ctypes.c_void_p()
    lib.call("ci_init_states", ctypes.byref(lib.ci_params(comb_size=32, seed=3)), S, None, ctypes.byref(h))
    d = lib.ci_states_desc()
    lib.call("ci_states_query", h, ctypes.byref(d))
    return h, d

def wait():
    lib.call("ci_export_state", small, ctypes.create_string_buffer(sd.state_bytes), sd.state_bytes, None)

big, bd = state(1 << 20)
room, rd = state(1 << 20)
small, sd = state(40)
lib.call("ci_generate_digest", big, 64, rd.state_dev, None)
wait()
for _ in range(8):
    lib.call("ci_generate_digest", big, 1 << 17, rd.state_dev, None)
t0 = time.perf_counter()
lib.call("ci_generate", small, 600, rd.state_dev, 24000, None)
t1 = time.perf_counter()
wait()
t2 = time.perf_counter()
assert t2 - t0 > 0.2, t2 - t0
assert t1 - t0 < 0.25 * (t2 - t0), (t1 - t0, t2 - t0)
print("done")
"""
    lib = os.path.join(os.path.dirname(HERE), "paper_1112_5239_gb300", "_lib.py")
    r = subprocess.run([sys.executable, "-c", code, lib], capture_output=True, text=True, timeout=300,
                       env={**os.environ, "CUDA_MODULE_LOADING": "EAGER"})
    assert r.returncode == 0 and r.stdout.strip().endswith("done"), r.stdout + r.stderr
