"""One call of kin_integrate_static on a small batch is the set-up for batches
of any size: the driver has reserved what the per-thread kernels need, and
later calls leave the device's free memory as it is.  In a process of its own,
whose first integrations these are."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(),
                                                  reason="needs a CUDA GPU")]
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = """
import sys
sys.path.insert(0, sys.argv[1])
import numpy as np, torch
from paper_1607_03884_gb300 import kin, synth
m = synth.make_mechanism("h2")
st = synth.make_states(m, 250000, 4)
def inputs(n):
    return [torch.from_numpy(np.ascontiguousarray(a[..., :n])).cuda() for a in (st.Y, st.T, st.P)]
batches = [inputs(n) for n in (8, 20000, 100000, 200000, 250000)]
free = []
for b in batches:
    kin.integrate_static(m, *b, 1e-9)
    torch.cuda.synchronize()
    free.append(torch.cuda.mem_get_info()[0])
print(free)
assert len(set(free)) == 1, [free[0] - f for f in free]
"""


def test_a_small_batch_is_the_set_up():
    r = subprocess.run([sys.executable, "-c", PROGRAM, ROOT], capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
