"""exprb43 from the smallest to the largest mechanism it takes: temperatures and
mass fractions of states that move, against the per-thread Radau kernel at a
tighter tolerance."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(),
                                                  reason="needs a CUDA GPU")]

from paper_1607_03884_gb300 import kin, synth  # noqa: E402
from test_gpu_team import _run, _states, _with_spectators  # noqa: E402


@pytest.mark.parametrize("ns", [13, 16, 17, 40, 58])
def test_species_and_temperature(ns):
    h2 = synth.make_mechanism("h2")
    m = _with_spectators(h2, ns) if ns > h2.ns else h2
    st = _states(h2, 9, ns, 12)
    Y, T = _run(kin.ExpRosenbrock(m), st, 1e-7, rtol=1e-8, atol=1e-12)
    Yq, Tq = _run(kin.Mechanism(m), st, 1e-7, layout="queue", rtol=1e-10, atol=1e-14)
    assert np.abs(Yq - st.Y).max(axis=0).min() > 1e-4
    # about a hundred steps of 1e-8 |Y| + 1e-12 each, in a norm over up to 58
    # species, with room for an igniting state's growth of errors
    assert np.all(np.abs(Y - Yq) <= 1e-8 + 1e-4 * np.abs(Yq))
    np.testing.assert_allclose(T, Tq, rtol=1e-6)


def test_the_next_size_is_refused():
    h2 = synth.make_mechanism("h2")
    with pytest.raises(kin.KinError) as e:
        kin.ExpRosenbrock(_with_spectators(h2, 59))
    assert e.value.code == kin.KIN_ERR_UNSUPPORTED
