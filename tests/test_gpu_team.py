"""Teams of warps (csrc/kin_team.cuh) at the edges of their sizes: panels and
register slots of the factorisations, the largest mechanisms, tables that do
not fit shared memory, small batches; the predictor's staged kernels at ragged
shapes.  The references are the per-thread kernels (QUEUE runs them at every
size), the same state in another batch, and numpy."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(),
                                                  reason="needs a CUDA GPU")]

from paper_1607_03884_gb300 import kin, synth  # noqa: E402


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _with_spectators(m, ns):
    """The mechanism with unreactive species before the inert, ns in all."""
    out, extra, at = synth.Mechanism(**m.__dict__), ns - m.ns, m.ns - 1
    out.ns = ns
    out.W = np.insert(m.W, [at] * extra, m.W[0])
    out.nasa = np.insert(m.nasa, [at] * extra, m.nasa[0], axis=0)
    out.eff = np.insert(m.eff, [at] * extra, 1.0, axis=1)
    return out


def _states(m, n, ns, seed):
    st = synth.make_states(m, n, seed, mode="mixed")
    Y = np.insert(st.Y, [m.ns - 1] * (ns - m.ns), 1e-6, axis=0)
    Y[-1] = 1.0 - Y[:-1].sum(axis=0)
    return synth.States(Y, st.T, st.P)


def _run(h, st, dt, **opt):
    Y, T, P = _dev(st.Y), _dev(st.T), _dev(st.P)
    s = torch.zeros(st.n, dtype=torch.int32, device="cuda")
    h.integrate(Y, T, P, dt, status=s, **opt)
    torch.cuda.synchronize()
    assert int(s.abs().sum()) == 0
    return Y.cpu().numpy(), T.cpu().numpy()


def _close(a, b, tol):
    for x, y in zip(a, b):
        big = np.abs(y) > 1e-9
        assert np.max(np.abs(x - y)[big] / np.abs(y)[big]) < tol


@pytest.mark.parametrize("ns", [13, 16, 31, 32, 33, 34, 63])
def test_team_sizes_against_the_thread_kernel(ns):
    """FP64 matrices: two elimination orders of rounding over about 40 steps of
    an error-controlled integration: 1e-8 (1e6 times the rounding)."""
    h2 = synth.make_mechanism("h2")
    m = _with_spectators(h2, ns) if ns > h2.ns else h2
    st = _states(h2, 37, ns, 5)
    mg = kin.Mechanism(m)
    _close(_run(mg, st, 1e-6, layout="warp"), _run(mg, st, 1e-6, layout="queue"), 1e-8)


@pytest.mark.parametrize("n", [1, 3, 153, 700])
@pytest.mark.parametrize("f32", [False, True])
def test_a_state_does_not_depend_on_its_batch(n, f32):
    ch4 = synth.make_mechanism("ch4")
    st = synth.make_states(ch4, 700, 6, T_range=(800.0, 2600.0))
    for h in (kin.Mechanism(ch4), kin.ConcMechanism(ch4)):
        Y, T = _run(h, st, 1e-7, layout="warp", lu_fp32=f32)
        y, t = _run(h, st.subset(np.arange(700 - n, 700)), 1e-7, layout="warp", lu_fp32=f32)
        np.testing.assert_array_equal(t, T[-n:])
        np.testing.assert_array_equal(y, Y[:, -n:])


@pytest.mark.parametrize("nr", [700, 1400])
def test_many_reactions_with_tables_beside_or_outside_shared_memory(nr):
    """CH4-like reactions repeated with shares of their rates: the same
    kinetics, one team per block (700) and tables in global memory (1400)."""
    ch4 = synth.make_mechanism("ch4")
    m = synth.Mechanism(**ch4.__dict__)
    idx = np.arange(nr) % ch4.nr
    share = np.bincount(idx)[idx].astype(float)
    m.nr = nr
    for f in ("reac", "prod", "arrh", "eff", "fall", "rtype"):
        setattr(m, f, np.ascontiguousarray(getattr(ch4, f)[idx]))
    m.arrh[:, 0] /= share
    m.fall[:, 0] /= share  # k0 with k_inf: the falloff factor is unchanged
    st = synth.make_states(ch4, 20, 8, T_range=(800.0, 2600.0))
    _close(_run(kin.Mechanism(m), st, 1e-7, layout="warp"),
           _run(kin.Mechanism(ch4), st, 1e-7, layout="warp"), 1e-8)
    _close(_run(kin.ConcMechanism(m), st, 1e-7), _run(kin.ConcMechanism(ch4), st, 1e-7), 1e-8)


@pytest.mark.parametrize("ns", [13, 17, 40])
def test_exprb_with_the_assembly_matrix_in_shared_and_global_memory(ns):
    """Spectator species change the error norm's count only; a tight tolerance
    keeps both step sequences within 1e-6 of the solution."""
    h2 = synth.make_mechanism("h2")
    m = _with_spectators(h2, ns) if ns > h2.ns else h2
    st = _states(h2, 9, ns, 12)
    Y, T = _run(kin.ExpRosenbrock(m), st, 1e-7, rtol=1e-8, atol=1e-12)
    Yq, Tq = _run(kin.Mechanism(m), st, 1e-7, layout="queue", rtol=1e-10, atol=1e-14)
    np.testing.assert_allclose(T, Tq, rtol=1e-6)


@pytest.mark.parametrize("n", [1, 11, 500])
def test_chemistry_on_teams_per_state(n):
    """Right-hand sides and both Jacobians of a batch equal those of its
    single states."""
    ch4 = synth.make_mechanism("ch4")
    mg, ns = kin.Mechanism(ch4), ch4.ns
    st = synth.make_states(ch4, n, 9, T_range=(800.0, 2600.0))
    y, P = _dev(np.concatenate([st.T[None], st.Y[:-1]])), _dev(st.P)
    scal = 1e-9 + 1e-5 * y.abs()

    def all_of(yy, PP, sc):
        k = PP.shape[0]
        f = torch.empty((ns, k), dtype=torch.float64, device="cuda")
        J = [torch.empty((ns * ns, k), dtype=torch.float64, device="cuda") for _ in range(2)]
        mg.rhs(yy, PP, f)
        mg.jacobian(yy, PP, J[0])
        mg.jacobian(yy, PP, J[1], fd=True, h=1e-8, scal=sc)
        return [x.cpu().numpy() for x in (f, *J)]

    whole, i = all_of(y, P, scal), n - 1
    one = all_of(y[:, i:].contiguous(), P[i:].contiguous(), scal[:, i:].contiguous())
    for a, b in zip(whole, one):
        np.testing.assert_array_equal(a[:, i:], b)


@pytest.mark.parametrize("M,d", [(1, 1), (7, 9), (1000, 160), (4099, 57)])
def test_moments_of_ragged_shapes(M, d):
    rng = np.random.default_rng(3)
    X = (rng.standard_normal((M, d)) * 10.0 ** rng.uniform(-6, 3, d) + 5.0).astype(np.float32)
    mean, std = (torch.empty(d, dtype=torch.float32, device="cuda") for _ in range(2))
    kin.moments(_dev(X), mean, std)
    x = X.astype(np.float64)
    # FP64 sums rounded once to FP32 (2^-24), the deviation's square root too
    np.testing.assert_allclose(mean.cpu().numpy(), x.mean(0), rtol=2e-7)
    np.testing.assert_allclose(std.cpu().numpy(), np.maximum(x.std(0), 1e-12), rtol=4e-7)


@pytest.mark.parametrize("n,ns", [(1, 2), (33, 13), (70, 300)])
def test_features_and_targets_of_ragged_shapes(n, ns):
    rng = np.random.default_rng(4)
    Y = 10.0 ** rng.uniform(-14, 0, (ns, n))
    Y[0, 0], Y[1, 0] = -1.0, 1.0
    T, P = rng.uniform(300, 3000, n), rng.uniform(1e4, 1e7, n)
    X = torch.empty((n, 3 + ns), dtype=torch.float32, device="cuda")
    kin.features(ns, _dev(Y), _dev(T), _dev(P), 1e-5, X)
    want = np.concatenate([np.log(T)[:, None], np.log(P)[:, None], np.full((n, 1), np.log(1e-5)),
                           np.log10(np.maximum(Y, 1e-12)).T], axis=1)
    # one rounding to FP32 of an FP64 logarithm
    np.testing.assert_allclose(X.cpu().numpy(), want, rtol=6.1e-8, atol=1e-30)
    h, z = 10.0 ** rng.uniform(-12, -6, n), rng.standard_normal((ns, n))
    tgt = torch.empty((n, 1 + ns), dtype=torch.float32, device="cuda")
    kin.targets(ns, _dev(h), _dev(z), tgt)
    np.testing.assert_allclose(tgt.cpu().numpy(), np.concatenate([np.log(h)[:, None], z.T], axis=1),
                               rtol=6.1e-8)


@pytest.mark.parametrize("width,rows", [(8, 5), (40, 129), (36, 64), (256, 300)])
def test_minibatch_gradients_of_fused_and_unfused_widths(width, rows):
    """Gathered rows (some outside the set) against the same rows given
    directly; a width of 36 takes the unfused kernels."""
    rng = np.random.default_rng(width)
    net = [kin.MLP(11, width, 21, seed=2) for _ in range(2)]
    X, T = (rng.standard_normal((400, k)).astype(np.float32) for k in (11, 21))
    idx = rng.integers(0, 400, rows).astype(np.int32)
    idx[0], idx[-1] = -1, 400
    ok = (idx >= 0) & (idx < 400)
    Xd, Td = (np.where(ok[:, None], a[np.clip(idx, 0, 399)], 0).astype(np.float32) for a in (X, T))
    loss = [torch.zeros(1, device="cuda") for _ in range(2)]
    net[0].train_step_rows(_dev(X), _dev(T), _dev(idx), 1e-3, loss_out=loss[0])
    net[1].train_step(_dev(Xd), _dev(Td), 1e-3, loss_out=loss[1])
    np.testing.assert_array_equal(net[0].get_params(), net[1].get_params())
    np.testing.assert_allclose(loss[0].item(), loss[1].item(), rtol=1e-6)
