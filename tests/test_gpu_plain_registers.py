"""The thread kernel's register variants (csrc/kin_kernels.cuh, PLAIN_USE_*)
compute the same bits on both sides of every line of the rule."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(),
                                                  reason="needs a CUDA GPU")]

from paper_1607_03884_gb300 import kin, synth  # noqa: E402

LINES = (6, 17, 21)  # 64-thread blocks per SM


@pytest.mark.parametrize("f32", [False, True])
def test_register_variants_agree(f32):
    m = synth.make_mechanism("h2")
    h, tile = kin.Mechanism(m), synth.make_states(m, 997, 21)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    want = None
    for n in sorted(64 * sms * p + e for p in LINES for e in (0, 1)):
        i = np.arange(n) % tile.n
        Y, T, P = (torch.from_numpy(np.ascontiguousarray(a)).cuda()
                   for a in (tile.Y[:, i], tile.T[i], tile.P[i]))
        h.integrate(Y, T, P, 1e-8, layout="plain", lu_fp32=f32)
        got = torch.cat([T[None], Y])[:, :tile.n * (n // tile.n)].reshape(m.ns + 1, -1, tile.n)
        want = got[:, :1].clone() if want is None else want
        assert torch.equal(got, want.expand_as(got)), n
