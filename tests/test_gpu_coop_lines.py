"""Both sides of the line between one state per block and one per thread, for
mechanisms with few reactions, give the same bits; so does QUEUE."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(),
                                                  reason="needs a CUDA GPU")]

from paper_1607_03884_gb300 import kin, synth  # noqa: E402
from test_gpu_coop import _run  # noqa: E402


def _first_reactions(m, nr):
    out = synth.Mechanism(**m.__dict__)
    out.nr = nr
    for f in ("reac", "prod", "arrh", "eff", "fall", "rtype"):
        setattr(out, f, np.ascontiguousarray(getattr(m, f)[:nr]))
    return out


@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("nr", [1, 2, 3, 5, 6, 19, 20])
def test_lines_for_few_reactions(nr, f32):
    m = _first_reactions(synth.make_mechanism("h2"), nr)
    mg = kin.Mechanism(m)
    line = 1700 if nr < 3 else (4700 if f32 else 4400) if 6 <= nr < 20 else 6912 if f32 else 5632
    st = synth.make_states(m, line + 1, 3)
    sub = st.subset(np.arange(line))
    over = _run(mg, st.Y, st.T, st.P, 1e-7, layout="plain", lu_fp32=f32)
    for layout in ("plain", "queue"):
        got = _run(mg, sub.Y, sub.T, sub.P, 1e-7, layout=layout, lu_fp32=f32)
        for x, y in zip(over, got):
            np.testing.assert_array_equal(x[..., :line], y)
