"""Threads that use different handles on their own streams: a kernel's shared
memory limit belongs to the process, so calls of different sizes must not lower
it under one another."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(),
                                                  reason="needs a CUDA GPU")]

from paper_1607_03884_gb300 import kin, synth  # noqa: E402
from test_gpu_team import _dev  # noqa: E402

CALLS = 4000


def _in_threads(jobs):
    """Every job called CALLS times in its own thread and stream; their errors."""
    errors, start = [], threading.Barrier(len(jobs))

    def go(job):
        s = torch.cuda.Stream()
        start.wait()
        try:
            for _ in range(CALLS):
                job(s)
        except kin.KinError as e:
            errors.append(str(e))

    threads = [threading.Thread(target=go, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    return errors


def test_chemistry_of_a_large_and_a_small_batch():
    ch4 = synth.make_mechanism("ch4")
    jobs, outs = [], []
    for n in (700, 1):
        st = synth.make_states(ch4, n, 9, T_range=(800.0, 2600.0))
        mg, y, P = kin.Mechanism(ch4), _dev(np.concatenate([st.T[None], st.Y[:-1]])), _dev(st.P)
        f = torch.empty((ch4.ns, n), dtype=torch.float64, device="cuda")
        want = torch.empty_like(f)
        mg.rhs(y, P, want)
        jobs.append(lambda s, a=(mg, y, P, f): a[0].rhs(*a[1:], stream=s))
        outs.append((f, want))
    assert not _in_threads(jobs)
    for f, want in outs:
        assert torch.equal(f, want)


def test_small_batches_of_a_large_and_a_small_mechanism():
    h2 = synth.make_mechanism("h2")
    big = synth.Mechanism(**h2.__dict__)
    big.nr = 300
    for f in ("reac", "prod", "arrh", "eff", "fall", "rtype"):
        setattr(big, f, np.ascontiguousarray(getattr(h2, f)[np.arange(300) % h2.nr]))
    st, jobs = synth.make_states(h2, 2, 3), []
    for m in (big, h2):
        a = kin.Mechanism(m), _dev(st.Y), _dev(st.T), _dev(st.P)
        jobs.append(lambda s, a=a: a[0].integrate(*a[1:], 1e-9, stream=s, layout="plain",
                                                  stop_after=1))
    assert not _in_threads(jobs)
