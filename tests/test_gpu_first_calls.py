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


def _run(code, **env):
    cuda_or_skip()
    r = subprocess.run([sys.executable, "-c", PRELUDE + code], capture_output=True, text=True, timeout=300,
                       env={**os.environ, **env})
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
