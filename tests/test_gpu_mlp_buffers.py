"""The predictor's buffers: a handle whose growth failed for lack of memory is
usable again."""
import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(),
                                                  reason="needs a CUDA GPU")]

from paper_1607_03884_gb300 import kin  # noqa: E402


@pytest.mark.parametrize("width", [64, 36])
def test_a_handle_survives_a_batch_that_does_not_fit(width):
    """2^34 rows ask for terabytes: refused at the first allocation, before any
    row is touched; then the same small batch as before gives the same bits."""
    net = kin.MLP(16, width, 40, seed=1)
    X = torch.from_numpy(np.random.default_rng(5).standard_normal((130, 16), dtype=np.float32)).cuda()
    Y = [torch.zeros((130, 40), device="cuda") for _ in range(2)]
    net.forward(X, Y[0])
    for _ in range(2):
        rc = kin.lib().kin_mlp_forward(net._h, C.c_void_p(X.data_ptr()), C.c_void_p(Y[1].data_ptr()),
                                       1 << 34, None)
        assert rc == kin.KIN_ERR_NOMEM
    net.forward(X, Y[1])
    assert torch.equal(*Y)
