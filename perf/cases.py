"""Performance cases: the calls a user of this library makes, over the range of
batch sizes, mechanisms, step lengths and precisions it is used with.

  listed()             the named cases
  draw(rng)            one more case of the same ranges
  prepare(case, seed)  the inputs and handles a program holds before the call
  run(state)           one pass through the public entry points, and its outputs
  work(case)           bytes and operations the pass cannot do without
  exact(case, seed)    the outputs in 64 bits by plain torch / numpy, where the
                       path computes a closed expression (not an integration)

Six kinds of work:

  radau    one global step of a batch with Radau IIA: the library's main call
           (device arrays, a captured graph with the stiffness ordering, or
           host arrays), in mass fractions or in concentrations
  exprb    the same step with exprb43
  chem     right-hand sides and analytical Jacobians of a batch (chemistry
           analysis, Jacobian spectra)
  predict  first-step prediction for a batch by the learned predictor
  train    sixteen Adam steps on gathered minibatches (the learned part's loop
           between two reads of its loss)
  dataset  a training set from recorded first steps: features, targets, moments
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1607_03884_gb300 import kin, synth

RTOL, ATOL = 1e-6, 1e-10
WIDTH = 256        # the predictor's hidden width
BATCHES = 16       # minibatches of a training pass

# temperature ranges of the synthetic workloads
T_RANGE = {"h2": (900.0, 2500.0), "ch4": (800.0, 2600.0)}


def listed():
    return [
        # a handful of cells: one warp's worth of reactors, pure latency
        dict(name="h2_few", kind="radau", mech="h2", mode="correlated", n=33, dt=1e-6,
             fp32=False, entry="device", form="mass"),
        # the paper's verification batch: 1024 PaSR states, FP64 throughout
        dict(name="h2_1024", kind="radau", mech="h2", mode="correlated", n=1024, dt=1e-6,
             fp32=False, entry="device", form="mass"),
        # the headline path at a production batch: graph replay with the
        # stiffness ordering, FP32 Newton matrices, mixed stiffness, long step
        dict(name="h2_mixed_graph", kind="radau", mech="h2", mode="mixed", n=131072, dt=1e-4,
             fp32=True, entry="graph", form="mass"),
        # a CFD code's host arrays (ragged batch), short step, FP64 matrices
        dict(name="h2_host", kind="radau", mech="h2", mode="mixed", n=50021, dt=1e-6,
             fp32=False, entry="host", form="mass"),
        # the large mechanism, long step, FP32 matrices
        dict(name="ch4_long", kind="radau", mech="ch4", mode="correlated", n=6000, dt=1e-4,
             fp32=True, entry="device", form="mass"),
        # the large mechanism, short step, FP64 matrices, ragged batch
        dict(name="ch4_fp64", kind="radau", mech="ch4", mode="correlated", n=3001, dt=1e-6,
             fp32=False, entry="device", form="mass"),
        # its concentration-based form with the sparse LU
        dict(name="ch4_conc", kind="radau", mech="ch4", mode="correlated", n=4000, dt=1e-5,
             fp32=True, entry="device", form="conc"),
        # the exponential method on the small mechanism
        dict(name="h2_exprb", kind="exprb", mech="h2", mode="mixed", n=2500, dt=1e-6),
        # chemistry of a batch of large-mechanism states
        dict(name="ch4_chem", kind="chem", mech="ch4", mode="correlated", n=2000),
        # first-step predictions for a large batch
        dict(name="predict", kind="predict", mech="ch4", mode="correlated", n=131072, dt=1e-4),
        # the training loop at its default minibatch
        dict(name="train", kind="train", mech="ch4", rows=65536, batch=4096),
        # a training set of one generation chunk
        dict(name="dataset", kind="dataset", mech="ch4", mode="correlated", n=65536, dt=1e-4),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["radau"] * 6 + ["exprb", "chem", "predict", "train", "dataset"])
    if kind == "radau":
        mech = rng.choice(["h2", "ch4"])
        form = rng.choice(["mass", "mass", "conc"]) if mech == "ch4" else "mass"
        entry = "device" if form == "conc" else rng.choice(["device", "graph", "host"])
        mode = rng.choice(["correlated", "mixed"]) if mech == "h2" else "correlated"
        dt = 10.0 ** rng.uniform(-6.0, -4.0)
        n = _log_int(rng, 1, 100000) if mech == "h2" else _log_int(rng, 1, 4000)
        return dict(kind=kind, mech=mech, mode=mode, n=n, dt=dt, fp32=rng.random() < 0.5,
                    entry=entry, form=form)
    if kind == "exprb":
        return dict(kind=kind, mech="h2", mode=rng.choice(["correlated", "mixed"]),
                    n=_log_int(rng, 8, 2000), dt=10.0 ** rng.uniform(-6.5, -5.0))
    if kind == "chem":
        mech = rng.choice(["h2", "ch4"])
        n = _log_int(rng, 16, 20000) if mech == "h2" else _log_int(rng, 16, 2000)
        return dict(kind=kind, mech=mech, mode="correlated", n=n)
    if kind == "predict":
        return dict(kind=kind, mech=rng.choice(["h2", "ch4"]), mode="correlated",
                    n=_log_int(rng, 32, 131072), dt=10.0 ** rng.uniform(-6.0, -4.0))
    if kind == "train":
        return dict(kind=kind, mech=rng.choice(["h2", "ch4"]),
                    rows=_log_int(rng, 8192, 65536), batch=_log_int(rng, 128, 8192))
    return dict(kind=kind, mech=rng.choice(["h2", "ch4"]), mode="correlated",
                n=_log_int(rng, 256, 65536), dt=10.0 ** rng.uniform(-6.0, -4.0))


# ---------------------------------------------------------------------------
# inputs (host arrays from the seed alone)
# ---------------------------------------------------------------------------

@functools.lru_cache(maxsize=None)
def _mech(kind):
    return synth.make_mechanism(kind)


def _states(case, seed):
    return synth.make_states(_mech(case["mech"]), case["n"], seed, T_range=T_RANGE[case["mech"]],
                             mode=case["mode"])


def _params(din, dout, seed):
    """Weights and biases of the four layers, unpadded and concatenated."""
    rng = np.random.default_rng(seed)
    out = []
    for a, b in ((din, WIDTH), (WIDTH, WIDTH), (WIDTH, WIDTH), (WIDTH, dout)):
        lim = math.sqrt(6.0 / a)
        out += [rng.uniform(-lim, lim, a * b), rng.uniform(-0.05, 0.05, b)]
    return np.concatenate(out).astype(np.float32)


def _layers(params, din, dout):
    out, q = [], 0
    for a, b in ((din, WIDTH), (WIDTH, WIDTH), (WIDTH, WIDTH), (WIDTH, dout)):
        out.append((params[q:q + a * b].reshape(a, b), params[q + a * b:q + a * b + b]))
        q += a * b + b
    return out


def _norm(ns):
    """Standardisation of the predictor's inputs and outputs: typical moments
    of log T, log P, log dt, log10 Y and of log h0 and the stage increments."""
    f = np.float32
    return dict(in_mean=np.concatenate([[7.3, 13.9, -10.4], np.full(ns, -7.0)]).astype(f),
                in_std=np.concatenate([[0.3, 0.7, 1.6], np.full(ns, 4.0)]).astype(f),
                out_mean=np.concatenate([[-17.0], np.zeros(3 * ns)]).astype(f),
                out_std=np.concatenate([[1.5], np.full(3 * ns, 1e-4)]).astype(f))


def _training_set(case, seed):
    """Standardised features and targets (unit variance), as a set holds them,
    and the row numbers of the minibatches."""
    ns = _mech(case["mech"]).ns
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((case["rows"], 3 + ns), dtype=np.float32)
    A = rng.standard_normal((3 + ns, 1 + 3 * ns), dtype=np.float32) / math.sqrt(3 + ns)
    T = np.tanh(X @ A) + 0.1 * rng.standard_normal((case["rows"], 1 + 3 * ns), dtype=np.float32)
    rows = np.stack([rng.permutation(case["rows"])[:case["batch"]] for _ in range(BATCHES)])
    return X, T.astype(np.float32), rows.astype(np.int32)


def _first_steps(case, seed):
    """Recorded first steps: sizes and stage increments of the accepted steps."""
    ns, n = _mech(case["mech"]).ns, case["n"]
    rng = np.random.default_rng(seed + 1)
    h = np.minimum(np.exp(rng.normal(-17.0, 1.5, n)), case["dt"])
    z = rng.standard_normal((3 * ns, n)) * 10.0 ** rng.uniform(-12.0, -3.0, (3 * ns, 1))
    return h, z


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# ---------------------------------------------------------------------------
# prepare / run
# ---------------------------------------------------------------------------

def prepare(case, seed):
    s = dict(case=case, ns=_mech(case["mech"]).ns)
    kind = case["kind"]
    if kind in ("radau", "exprb"):
        st = _states(case, seed)
        mech = _mech(case["mech"])
        if kind == "exprb":
            s["handle"] = kin.ExpRosenbrock(mech)
        elif case["form"] == "conc":
            s["handle"] = kin.ConcMechanism(mech)
        else:
            s["handle"] = kin.Mechanism(mech)
        if case.get("entry") == "host":
            pin = lambda a: torch.from_numpy(a).pin_memory()  # noqa: E731
            s["Y0"], s["T0"], s["P"] = pin(st.Y), pin(st.T), pin(st.P)
            s["status"] = torch.zeros(case["n"], dtype=torch.int32).pin_memory()
            s["Y"], s["T"] = s["Y0"].clone().pin_memory(), s["T0"].clone().pin_memory()
        else:
            s["Y0"], s["T0"], s["P"] = _dev(st.Y), _dev(st.T), _dev(st.P)
            s["status"] = torch.zeros(case["n"], dtype=torch.int32, device="cuda")
            s["Y"], s["T"] = s["Y0"].clone(), s["T0"].clone()
        if case.get("entry") == "graph":
            s["graph"] = s["handle"].capture(s["Y"], s["T"], s["P"], case["dt"], RTOL, ATOL,
                                             status=s["status"], order_by="heuristic",
                                             lu_fp32=case["fp32"])
    elif kind == "chem":
        st, ns = _states(case, seed), s["ns"]
        s["handle"] = kin.Mechanism(_mech(case["mech"]))
        s["y"], s["P"] = _dev(np.concatenate([st.T[None], st.Y[:-1]])), _dev(st.P)
        s["f"] = torch.empty((ns, case["n"]), dtype=torch.float64, device="cuda")
        s["J"] = torch.empty((ns * ns, case["n"]), dtype=torch.float64, device="cuda")
    elif kind == "predict":
        st, ns = _states(case, seed), s["ns"]
        s["net"] = kin.MLP(3 + ns, WIDTH, 1 + 3 * ns, precision="bf16")
        s["net"].set_params(_params(3 + ns, 1 + 3 * ns, seed))
        s["norm"] = {k: _dev(v) for k, v in _norm(ns).items()}
        s["Y"], s["T"], s["P"] = _dev(st.Y), _dev(st.T), _dev(st.P)
        s["h0"] = torch.empty(case["n"], dtype=torch.float64, device="cuda")
        s["z0"] = torch.empty((3 * ns, case["n"]), dtype=torch.float64, device="cuda")
    elif kind == "train":
        ns = s["ns"]
        X, T, rows = _training_set(case, seed)
        s["net"] = kin.MLP(3 + ns, WIDTH, 1 + 3 * ns, precision="bf16")
        s["params"] = _params(3 + ns, 1 + 3 * ns, seed)
        s["net"].set_params(s["params"])
        s["X"], s["T"], s["rows"] = _dev(X), _dev(T), _dev(rows)
        s["loss"] = torch.zeros(1, dtype=torch.float32, device="cuda")
    else:
        st, ns = _states(case, seed), s["ns"]
        s["Y"], s["T"], s["P"] = _dev(st.Y), _dev(st.T), _dev(st.P)
        h, z = _first_steps(case, seed)
        s["h"], s["z"] = _dev(h), _dev(z)
        e = lambda *d: torch.empty(d, dtype=torch.float32, device="cuda")  # noqa: E731
        s["X"], s["Xs"] = e(case["n"], 3 + ns), e(case["n"], 3 + ns)
        s["tgt"], s["tgts"] = e(case["n"], 1 + 3 * ns), e(case["n"], 1 + 3 * ns)
        s["mean"], s["std"] = e(3 + ns), e(3 + ns)
        s["tmean"], s["tstd"] = e(1 + 3 * ns), e(1 + 3 * ns)
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind in ("radau", "exprb"):
        s["Y"].copy_(s["Y0"])  # the integration advances its arrays in place
        s["T"].copy_(s["T0"])
        if kind == "exprb":
            s["handle"].integrate(s["Y"], s["T"], s["P"], case["dt"], RTOL, ATOL,
                                  status=s["status"])
        elif case["entry"] == "graph":
            s["graph"].replay()
        elif case["entry"] == "host":
            s["handle"].integrate_host(s["Y"], s["T"], s["P"], case["dt"], RTOL, ATOL,
                                       status=s["status"], order_by="heuristic",
                                       lu_fp32=case["fp32"])
        else:
            s["handle"].integrate(s["Y"], s["T"], s["P"], case["dt"], RTOL, ATOL,
                                  status=s["status"], lu_fp32=case["fp32"])
        return dict(T=s["T"], Y=s["Y"], status=s["status"])
    if kind == "chem":
        s["handle"].rhs(s["y"], s["P"], s["f"])
        s["handle"].jacobian(s["y"], s["P"], s["J"])
        return dict(f=s["f"], J=s["J"])
    if kind == "predict":
        s["net"].predict(s["ns"], s["Y"], s["T"], s["P"], case["dt"], s["norm"], h0=s["h0"],
                         z0=s["z0"])
        return dict(h0=s["h0"], z0=s["z0"])
    if kind == "train":
        # a late epoch's learning rate
        for b in range(BATCHES):
            s["net"].train_step_rows(s["X"], s["T"], s["rows"][b], 2e-5, loss_out=s["loss"])
        return dict(loss=s["loss"], params=s["net"].get_params())
    kin.features(s["ns"], s["Y"], s["T"], s["P"], case["dt"], s["X"])
    kin.targets(3 * s["ns"], s["h"], s["z"], s["tgt"])
    kin.moments(s["X"], s["mean"], s["std"])
    kin.moments(s["tgt"], s["tmean"], s["tstd"])
    kin.features(s["ns"], s["Y"], s["T"], s["P"], case["dt"], s["Xs"], s["mean"], s["std"])
    kin.targets(3 * s["ns"], s["h"], s["z"], s["tgts"], s["tmean"], s["tstd"])
    return dict(X=s["X"], Xs=s["Xs"], tgt=s["tgt"], tgts=s["tgts"], mean=s["mean"], std=s["std"],
                tmean=s["tmean"], tstd=s["tstd"])


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------

# Floating-point operations per event (right-hand side, Jacobian beyond its
# point's right-hand side, factorisation pair, Newton iteration, error
# estimate, accepted step) and the events per state of an integration over
# 1e-6 s and 1e-4 s; between the two they are interpolated in log dt.
_EVENT = {("h2", "mass"): (1141, 2790, 7465, 2441, 457, 650),
          ("ch4", "mass"): (9386, 36560, 498945, 31121, 6097, 2600),
          ("ch4", "conc"): (9174, 22174, 414321, 29388, 5748, 2600)}
_COUNT = {"h2": ((260, 16, 28, 72, 42, 42), (448, 32, 48, 127, 66, 66)),
          "ch4": ((285, 15, 40, 80, 46, 46), (494, 27, 58, 140, 73, 73))}


def work(case):
    ns, kind = _mech(case["mech"]).ns, case["kind"]
    params = (3 + ns) * WIDTH + 2 * WIDTH * WIDTH + WIDTH * (1 + 3 * ns)
    if kind in ("radau", "exprb"):
        ev = _EVENT[(case["mech"], case.get("form", "mass"))]
        x = min(1.0, max(0.0, (math.log10(case["dt"]) + 6.0) / 2.0))
        cnt = [a + x * (b - a) for a, b in zip(*_COUNT[case["mech"]])]
        per = sum(a * b for a, b in zip(ev, cnt))
        if kind == "exprb":  # about as many right-hand sides; a Jacobian per step
            per = cnt[0] * ev[0] + cnt[5] * ev[1]
        return dict(bytes=case["n"] * (2 * ns + 3) * 8.5, flops=case["n"] * per)
    n = case.get("n", 0)
    if kind == "chem":
        ev = _EVENT[(case["mech"], "mass")]
        return dict(bytes=8.0 * n * (2 * ns + 1 + ns * ns), flops=float(n) * (2 * ev[0] + ev[1]))
    if kind == "predict":
        return dict(bytes=8.0 * n * (ns + 2 + 3 * ns + 1) + 4.0 * params, flops=2.0 * n * params)
    if kind == "train":
        m = BATCHES * case["batch"]
        return dict(bytes=4.0 * m * (4 + 4 * ns) + 28.0 * BATCHES * params, flops=6.0 * m * params)
    return dict(bytes=8.0 * n * (ns + 2 + 3 * ns + 1) + 8.0 * n * (4 + 4 * ns),
                flops=20.0 * n * (4 + 4 * ns))


# ---------------------------------------------------------------------------
# exact
# ---------------------------------------------------------------------------

def _rhs64(m, T, Y, P):
    """dT/dt and dY/dt (all species but the last) of one state, float64 torch:
    NASA-7 thermo, reversible mass action with third bodies and Troe falloff at
    constant pressure."""
    t64 = lambda a: torch.from_numpy(np.asarray(a, np.float64))  # noqa: E731
    RU, PATM = 8314.46261815324, 101325.0
    W, nasa = t64(m.W), t64(m.nasa)
    Yf = torch.cat([Y, (1.0 - Y.sum())[None]])
    rho = P / (RU * T * (Yf / W).sum())
    C = rho * Yf / W
    a = torch.where((T < nasa[:, 1])[:, None], nasa[:, 3:10], nasa[:, 10:17])
    lnT = torch.log(T)
    cp = a[:, 0] + T * (a[:, 1] + T * (a[:, 2] + T * (a[:, 3] + T * a[:, 4])))
    h = (a[:, 0] + T * (a[:, 1] / 2 + T * (a[:, 2] / 3 + T * (a[:, 3] / 4 + T * a[:, 4] / 5)))
         + a[:, 5] / T)
    s = (a[:, 0] * lnT + T * (a[:, 1] + T * (a[:, 2] / 2 + T * (a[:, 3] / 3 + T * a[:, 4] / 4)))
         + a[:, 6])
    one = torch.ones(1, dtype=torch.float64)
    Cp, gp = torch.cat([C, one]), torch.cat([s - h, 0.0 * one])  # index -1: the empty slot
    re, pr = torch.from_numpy(m.reac.astype(np.int64)), torch.from_numpy(m.prod.astype(np.int64))
    re, pr = torch.where(re < 0, m.ns, re), torch.where(pr < 0, m.ns, pr)
    dnu = ((pr < m.ns).sum(1) - (re < m.ns).sum(1)).to(torch.float64)
    arrh, fall = t64(m.arrh), t64(m.fall)
    lnk = torch.log(arrh[:, 0]) + arrh[:, 1] * lnT - arrh[:, 2] / T
    lnKc = gp[pr].sum(1) - gp[re].sum(1) + dnu * (math.log(PATM / RU) - lnT)
    R = torch.exp(lnk) * (Cp[re].prod(1) - torch.exp(-lnKc) * Cp[pr].prod(1))
    M = (t64(m.eff) * C).sum(1)
    rt = torch.from_numpy(np.asarray(m.rtype))
    ok = rt == 2
    f = torch.where(ok[:, None], fall, torch.ones_like(fall))
    Fc = ((1 - f[:, 3]) * torch.exp(-T / f[:, 4]) + f[:, 3] * torch.exp(-T / f[:, 5])
          + torch.exp(-f[:, 6] / T))
    lnPr = torch.log(f[:, 0]) + f[:, 1] * lnT - f[:, 2] / T - lnk + torch.log(M)
    lnPr = torch.where(ok, lnPr, torch.zeros_like(lnPr))
    lF = torch.log10(torch.where(ok, Fc, 0.5 * torch.ones_like(Fc)))
    u = lnPr / math.log(10.0) - 0.4 - 0.67 * lF
    v = 0.75 - 1.27 * lF - 0.14 * u
    troe = torch.exp(lnPr) / (1 + torch.exp(lnPr)) * 10.0 ** (lF / (1 + (u / v) ** 2))
    q = R * torch.where(rt == 0, torch.ones_like(M), torch.where(rt == 1, M, troe))
    qq = q[:, None].expand(-1, 3).reshape(-1)
    wd = torch.zeros(m.ns + 1, dtype=torch.float64)
    wd = wd.index_add(0, pr.reshape(-1), qq).index_add(0, re.reshape(-1), -qq)[:m.ns]
    dT = -(h * wd).sum() * T / (C * cp).sum()
    return torch.cat([dT[None], (wd * W / rho)[:-1]])


def _features64(ns, st, dt):
    return np.concatenate([np.log(st.T)[:, None], np.log(st.P)[:, None],
                           np.full((st.n, 1), math.log(dt)),
                           np.log10(np.maximum(st.Y, 1e-12)).T], axis=1)


def exact(case, seed):
    kind, m = case["kind"], _mech(case["mech"])
    ns = m.ns
    if kind in ("radau", "exprb"):
        return None  # the result of an error-controlled step sequence
    if kind == "chem":
        st = _states(case, seed)
        y = torch.from_numpy(np.concatenate([st.T[None], st.Y[:-1]]))
        P = torch.from_numpy(st.P)
        one = lambda yy, p: _rhs64(m, yy[0], yy[1:], p)  # noqa: E731
        fs, Js = [], []
        for i in range(0, st.n, 250):
            a, p = y[:, i:i + 250].T.contiguous(), P[i:i + 250]
            fs.append(torch.func.vmap(one)(a, p))
            Js.append(torch.func.vmap(torch.func.jacfwd(one))(a, p))
        f, J = torch.cat(fs), torch.cat(Js)
        return dict(f=f.T.contiguous(), J=J.reshape(st.n, ns * ns).T.contiguous())
    if kind == "predict":
        st, nm = _states(case, seed), {k: v.astype(np.float64) for k, v in _norm(ns).items()}
        h = (_features64(ns, st, case["dt"]) - nm["in_mean"]) / nm["in_std"]
        for l, (w, b) in enumerate(_layers(_params(3 + ns, 1 + 3 * ns, seed), 3 + ns, 1 + 3 * ns)):
            h = h @ w.astype(np.float64) + b
            if l < 3:
                h = h / (1.0 + np.exp(-h))
        o = h * nm["out_std"] + nm["out_mean"]
        return dict(h0=np.clip(np.exp(o[:, 0]), 1e-14, case["dt"]),
                    z0=np.ascontiguousarray(o[:, 1:].T))
    if kind == "train":
        X, T, rows = _training_set(case, seed)
        ps = [torch.from_numpy(a.astype(np.float64)).requires_grad_(True) for l in _layers(
            _params(3 + ns, 1 + 3 * ns, seed), 3 + ns, 1 + 3 * ns) for a in l]
        opt = torch.optim.Adam(ps, lr=2e-5, betas=(0.9, 0.999), eps=1e-8)
        for b in range(BATCHES):
            h = torch.from_numpy(X[rows[b]].astype(np.float64))
            for l in range(4):
                h = h @ ps[2 * l] + ps[2 * l + 1]
                h = torch.nn.functional.silu(h) if l < 3 else h
            loss = ((h - torch.from_numpy(T[rows[b]].astype(np.float64))) ** 2).mean()
            opt.zero_grad()
            loss.backward()
            opt.step()
        return dict(loss=loss.detach().reshape(1),
                    params=np.concatenate([p.detach().numpy().ravel() for p in ps]))
    st = _states(case, seed)
    X = _features64(ns, st, case["dt"])
    h, z = _first_steps(case, seed)
    t = np.concatenate([np.log(h)[:, None], z.T], axis=1)
    stat = lambda a: (a.mean(0), np.maximum(a.std(0), 1e-12))  # noqa: E731
    (mx, sx), (mt, s_t) = stat(X), stat(t)
    # a constant column (log dt) standardises to zero
    Xs = np.where(sx > 1e-12, X - mx, 0.0) / sx
    return dict(X=X, Xs=Xs, tgt=t, tgts=(t - mt) / s_t, mean=mx, std=sx, tmean=mt, tstd=s_t)
