"""The data-set kernels on both sides of the lines where their launches change:
moments by a thread per column or a cluster of eight CTAs, targets a row per
thread or in tiles."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(),
                                                  reason="needs a CUDA GPU")]

from paper_1607_03884_gb300 import kin  # noqa: E402
from test_gpu_team import _dev  # noqa: E402


@pytest.mark.parametrize("M", [2, 31, 32, 33])
@pytest.mark.parametrize("d", [1, 64, 65])
def test_moments_of_few_rows(M, d):
    rng = np.random.default_rng(M + d)
    X = (rng.standard_normal((M, d)) * 10.0 ** rng.uniform(-6, 3, d) + 5.0).astype(np.float32)
    mean, std = (torch.empty(d, dtype=torch.float32, device="cuda") for _ in range(2))
    kin.moments(_dev(X), mean, std)
    x = X.astype(np.float64)
    # FP64 sums rounded once to FP32 (2^-24), the deviation's square root too
    np.testing.assert_allclose(mean.cpu().numpy(), x.mean(0), rtol=2e-7)
    np.testing.assert_allclose(std.cpu().numpy(), np.maximum(x.std(0), 1e-12), rtol=4e-7)


@pytest.mark.parametrize("n", [99999, 100000, 100001])
@pytest.mark.parametrize("nz", [1, 27, 28])
def test_targets_by_rows_and_by_tiles(n, nz):
    rng = np.random.default_rng(nz)
    h, z = 10.0 ** rng.uniform(-12, -6, n), rng.standard_normal((nz, n))
    mu = rng.standard_normal(1 + nz).astype(np.float32)
    sd = rng.uniform(0.5, 2.0, 1 + nz).astype(np.float32)
    t = np.concatenate([np.log(h)[:, None], z.T], axis=1)
    for norm in ((), (_dev(mu), _dev(sd))):
        tgt = torch.full((n, 1 + nz), np.nan, dtype=torch.float32, device="cuda")
        kin.targets(nz, _dev(h), _dev(z), tgt, *norm)
        want = t.astype(np.float32)  # then a difference and a quotient in FP32
        if norm:
            want = (want - mu) / sd
        # log h may round to the neighbouring FP32 value: 2^-23 of |log h| < 28,
        # over the deviation
        np.testing.assert_allclose(tgt.cpu().numpy(), want, rtol=1.3e-7, atol=1e-5 if norm else 0)
