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


def test_a_first_batch_allocates_what_its_path_uses():
    """Width 256, 56 inputs, 160 outputs, per row: BF16 input (64) and
    activations (3 x 256 + 160), FP32 pre-activations (3 x 256), two gradient
    pairs of 256 in both types."""
    rows = 1 << 18
    net = kin.MLP(56, 256, 160)
    X = torch.zeros((rows, 56), device="cuda")
    Y = torch.zeros((rows, 160), device="cuda")
    net.forward(X[:1], Y[:1])
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    net.forward(X, Y)
    torch.cuda.synchronize()
    per_row = 2 * (64 + 3 * 256 + 160) + 4 * 3 * 256 + 2 * (4 + 2) * 256
    # each of twelve allocations may round up to a 2 MiB page
    assert before - torch.cuda.mem_get_info()[0] <= rows * per_row + (12 << 21)
