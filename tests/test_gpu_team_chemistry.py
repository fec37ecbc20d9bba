"""kin_rhs and both kinds of kin_jacobian on teams of warps at the species
counts where their shared memory is tightest (17, 18), where the two register
slots meet (32, 33) and at the largest (63), against the oracle, for batches
that leave a team's warps idle (1), fill one team (3) and fill many (500), and
on both sides of the lines beyond which the thread kernels serve."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(),
                                                  reason="needs a CUDA GPU")]

from oracle import oracle as O  # noqa: E402
from paper_1607_03884_gb300 import kin, synth  # noqa: E402
from test_gpu_team import _dev, _states, _with_spectators  # noqa: E402

H = 3e-8  # the step that the difference increments are formed with


def _rhs(mg, y, P):
    f = torch.full(y.shape, np.nan, dtype=torch.float64, device="cuda")
    mg.rhs(_dev(y), _dev(P), f)
    return f.cpu().numpy()


def _jac(mg, y, P, scal=None):
    N, n = y.shape
    J = torch.full((N * N, n), np.nan, dtype=torch.float64, device="cuda")
    if scal is None:
        mg.jacobian(_dev(y), _dev(P), J)
    else:
        mg.jacobian(_dev(y), _dev(P), J, fd=True, h=H, scal=_dev(scal))
    return J.cpu().numpy().reshape(N, N, n)


def _against_the_oracle(ns, n):
    h2 = synth.make_mechanism("h2")
    m = _with_spectators(h2, ns)
    st = _states(h2, n, ns, 40 + ns)
    mg, om, y = kin.Mechanism(m), O.OracleMech(m), O.state_vector(st)
    scal = 1e-9 + 1e-5 * np.abs(y)
    f, J, Jfd = _rhs(mg, y, st.P), _jac(mg, y, st.P), _jac(mg, y, st.P, scal)
    eps = np.finfo(float).eps
    for i in sorted({0, n // 2, n - 1}):
        yi, P = y[:, i], st.P[i]
        fo, Jo = O.rhs(om, P, yi)[0], O.jac(om, P, yi)[0]
        assert np.all(np.abs(f[:, i] - fo) <= 1e-10 * np.abs(fo) + 1e-13 * np.abs(fo).max()), i
        colmax = np.abs(Jo).max(axis=0) + 1e-300
        assert np.max(np.abs(J[:, :, i] - Jo) / colmax) < 1e-9, i
        # difference quotients with the same increments differ by the two
        # sides' right-hand sides at the two points, over the increment; the
        # device's are taken in a batch of the same size, by the same kernel
        Jd, rc = O.jac_fd(om, P, yi, fo, H, scal[:, i])
        assert rc == 0
        fn = np.sqrt(np.mean((fo / scal[:, i]) ** 2))
        inc = np.maximum(np.sqrt(eps) * np.abs(yi), 1000.0 * H * eps * ns * fn * scal[:, i])
        yp = np.repeat(yi[:, None], ns + 1, axis=1)
        yp[np.arange(ns), 1 + np.arange(ns)] += inc
        cols = np.arange(max(n, ns + 1)) % (ns + 1)
        df = np.abs(_rhs(mg, yp[:, cols], np.full(cols.size, P))[:, :ns + 1]
                    - np.stack([O.rhs(om, P, yp[:, c])[0] for c in range(ns + 1)], axis=1))
        bound = (1e-9 * (np.abs(Jd).max(axis=0) + 1e-300)[None, :]
                 + 1.01 * (df[:, 1:] + df[:, :1]) / inc[None, :] + 1e-300)
        assert np.all(np.abs(Jfd[:, :, i] - Jd) <= bound), i
    return mg, st, y, scal, f, J, Jfd


@pytest.mark.parametrize("n", [1, 3, 500])
@pytest.mark.parametrize("ns", [17, 18, 19, 32, 33, 63])
def test_chemistry_against_the_oracle(ns, n):
    mg, st, y, scal, f, J, Jfd = _against_the_oracle(ns, n)
    # and a state's results do not depend on the batch it comes in
    for i in sorted({0, n // 3, n - 1}):
        s = slice(i, i + 1)
        np.testing.assert_array_equal(f[:, s], _rhs(mg, y[:, s], st.P[s]))
        np.testing.assert_array_equal(J[:, :, s], _jac(mg, y[:, s], st.P[s]))
        np.testing.assert_array_equal(Jfd[:, :, s], _jac(mg, y[:, s], st.P[s], scal[:, s]))


@pytest.mark.parametrize("ns", [17, 24, 63])
@pytest.mark.parametrize("kind", ["rhs and differences", "analytical"])
@pytest.mark.parametrize("over", [0, 1])
def test_both_sides_of_the_lines(ns, kind, over):
    chain = synth.make_mechanism("h2").nr * (80 + ns)
    _against_the_oracle(ns, (chain if kind != "analytical" else chain * 11 // 5) + over)
