"""FP32 matrices of small mechanisms on four and on seven teams per block: a
state's bits do not depend on which, on both sides of the line between them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(),
                                                  reason="needs a CUDA GPU")]

from paper_1607_03884_gb300 import kin, synth  # noqa: E402
from test_gpu_team import _run, _states, _with_spectators  # noqa: E402


@pytest.mark.parametrize("ns", [13, 17, 23, 24, 25])
@pytest.mark.parametrize("form", ["mass", "mass, fd", "conc"])
def test_four_and_seven_teams(ns, form):
    h2, line = synth.make_mechanism("h2"), 14 * torch.cuda.get_device_properties(0).multi_processor_count
    m = _with_spectators(h2, ns) if ns > h2.ns else h2
    st = _states(h2, line + 5, ns, 3)
    h = kin.ConcMechanism(m) if form == "conc" else kin.Mechanism(m)
    opt = dict(layout="warp", lu_fp32=True, **({"jac_fd": True} if form == "mass, fd" else {}))
    Y, T = _run(h, st, 1e-7, **opt)
    for n in (line, line - 1, 40):
        y, t = _run(h, st.subset(np.arange(n)), 1e-7, **opt)
        np.testing.assert_array_equal(t, T[:n])
        np.testing.assert_array_equal(y, Y[:, :n])
