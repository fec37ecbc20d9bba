"""Small PLAIN batches run one state per block (csrc/kin_coop.cuh) with the
per-thread kernel's arithmetic: the same bits as the QUEUE layout, which always
runs the per-thread step code, over batch sizes, options and mechanism forms."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(),
                                                  reason="needs a CUDA GPU")]

from paper_1607_03884_gb300 import kin, synth  # noqa: E402


def _without_falloff(m):
    keep = np.nonzero(m.rtype == 0)[0]
    out = synth.Mechanism(**m.__dict__)
    out.nr = len(keep)
    for f in ("reac", "prod", "arrh", "eff", "fall", "rtype"):
        setattr(out, f, np.ascontiguousarray(getattr(m, f)[keep]))
    return out


def _with_spectators(m, extra):
    """extra species that take part in no reaction, before the inert."""
    out = synth.Mechanism(**m.__dict__)
    out.ns = m.ns + extra
    at = m.ns - 1
    out.W = np.insert(m.W, [at] * extra, m.W[0])
    out.nasa = np.insert(m.nasa, [at] * extra, m.nasa[0], axis=0)
    out.eff = np.insert(m.eff, [at] * extra, 1.0, axis=1)
    return out


def _run(mg, Y, T, P, dt, **opt):
    n = T.shape[0]
    d = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (Y, T, P)]
    c = torch.zeros((8, n), dtype=torch.int32, device="cuda")
    s = torch.zeros(n, dtype=torch.int32, device="cuda")
    out = {k: torch.zeros(*shape, dtype=torch.float64, device="cuda")
           for k, shape in (("h_first", (n,)), ("z_first", (3 * mg.ns, n)))}
    mg.integrate(d[0], d[1], d[2], dt, counters=c, status=s, **out, **opt)
    torch.cuda.synchronize()
    return [a.cpu().numpy() for a in (d[0], d[1], c, s, *out.values())]


def _same(mg, st, dt, **opt):
    a = _run(mg, st.Y, st.T, st.P, dt, layout="plain", **opt)
    b = _run(mg, st.Y, st.T, st.P, dt, layout="queue", **opt)
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x, y)
    return a


@pytest.mark.parametrize("n", [1, 2, 31, 257])
@pytest.mark.parametrize("opt", [{}, {"lu_fp32": True}, {"jac_fd": True},
                                 {"jac_fd": True, "lu_fp32": True}, {"h_fixed": 1e-6 / 48},
                                 {"stop_after": 1}, {"max_steps": 9}, {"nit": 2}])
def test_small_batches_give_the_per_thread_bits(n, opt):
    m = synth.make_mechanism("h2")
    _same(kin.Mechanism(m), synth.make_states(m, n, 90 + n), 1e-6, **opt)


@pytest.mark.parametrize("form", ["no falloff", "16 species"])
@pytest.mark.parametrize("lu_fp32", [False, True])
def test_other_mechanism_forms_give_the_per_thread_bits(form, lu_fp32):
    m = synth.make_mechanism("h2")
    st = synth.make_states(m, 40, 17, mode="mixed")
    if form == "no falloff":
        m = _without_falloff(m)
    else:
        m = _with_spectators(m, 3)
        st = synth.States(np.insert(st.Y, [12] * 3, 0.0, axis=0), st.T, st.P)
    _same(kin.Mechanism(m), st, 1e-5, lu_fp32=lu_fp32)


def test_both_sides_of_the_size_rule_give_the_same_bits():
    """A batch of 5633 states (per thread) and its first 5632 (per block)."""
    m = synth.make_mechanism("h2")
    mg = kin.Mechanism(m)
    st = synth.make_states(m, 5633, 3)
    a = _run(mg, st.Y, st.T, st.P, 1e-7, layout="plain")
    sub = st.subset(np.arange(5632))
    b = _run(mg, sub.Y, sub.T, sub.P, 1e-7, layout="plain")
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x[..., :5632], y)


def test_failing_states_and_a_bad_order_are_reported_alike():
    m = synth.make_mechanism("h2")
    mg = kin.Mechanism(m)
    st = synth.make_states(m, 64, 5)
    Y, T = st.Y.copy(), st.T.copy()
    T[3], Y[2, 7], T[11] = np.nan, np.inf, 1e300
    st = synth.States(Y, T, st.P)
    s = _same(mg, st, 1e-6)[3]
    assert s[3] == 4 and s[7] == 4 and np.all(np.delete(s, [3, 7, 11]) == 0)
    order = torch.arange(63, -1, -1, dtype=torch.int32, device="cuda")
    order[5], order[9] = 64, -1
    _same(mg, st, 1e-6, order=order)
    with pytest.raises(kin.KinError):
        _run(mg, st.Y, st.T, st.P, 1e-6, layout="plain", order=order)
        mg.stats()


def test_given_first_steps_and_guesses_are_used_alike():
    m = synth.make_mechanism("h2")
    mg = kin.Mechanism(m)
    st = synth.make_states(m, 50, 8)
    h0 = torch.full((50,), 1e-9, dtype=torch.float64, device="cuda")
    z0 = torch.full((3 * m.ns, 50), 1e-9, dtype=torch.float64, device="cuda")
    _same(mg, st, 1e-6, h0=h0, z0=z0)
