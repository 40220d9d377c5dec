"""What the workspace pool keeps, by the device's free memory, and what freeing
the last handle waits for, in a process of its own (handles of other tests keep
the pool alive)."""
import os
import subprocess
import sys

import pytest

from gpu_util import cuda_or_skip

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import sys, time
sys.path.insert(0, %r)
import torch
import paper_1112_5239_gb300 as ci
S, n = 16384, 2048          # the digests' scratch outputs: 128 MiB
def used():
    torch.cuda.synchronize()
    return -torch.cuda.mem_get_info()[0] / 2**20
def calls(memory, wait):
    st = ci.States(S, variant="bbs", seed=1, memory=memory)
    d = torch.zeros(S, dtype=torch.int64, device="cuda")
    st.generate_digest(n, digest=d)
    between = used() if wait else 0
    st.generate_digest(n, digest=d)
    if not wait:
        torch.cuda._sleep(1_000_000_000)
        st.generate_digest(n, digest=d)
    t = time.perf_counter()
    ci._lib.call("ci_free_states", st.handle)  # States.free waits for the current stream first
    t = time.perf_counter() - t
    st.handle = None
    assert memory == "library" or t < 0.1, ("ci_free_states waited", t)
    return between, used()
calls("torch", True)        # everything loaded
before = used()
for memory, wait in %r:
    between, after = calls(memory, wait)
    print(memory, wait, before, between, after)
    if wait:
        assert between > before + 100, "kept between calls"
    assert after < before + 50, "given back when the last handle is freed"
print("done")
"""


@pytest.mark.parametrize("order", [[("torch", False)], [("torch", True), ("torch", False), ("torch", True)],
                                   [("library", False), ("library", True)]])
def test_the_pool_keeps_nothing_without_handles(order):
    cuda_or_skip()
    r = subprocess.run([sys.executable, "-c", CODE % (ROOT, order)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("done"), r.stdout + r.stderr
