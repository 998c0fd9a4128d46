"""A forward pass whose activations do not fit the device (refused by the allocator, nothing is launched)
leaves no activations behind: loss and backward of it are argument errors, and the handle works on."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def test_failed_forward_leaves_nothing_stale():
    from paper_2206_11009_gb300 import _lib, learn
    net = learn.WarmNet(learn.init_params(7))
    lib = net._lib
    rng = np.random.default_rng(0)
    x = torch.from_numpy(rng.standard_normal((2, 2, 20, 20)).astype(np.float32)).cuda()
    y = net.forward(x)
    g = net.backward(x, y).clone()
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())
    # 2.7e11 pixels of more than a kilobyte each
    assert lib.ot_cnn_forward(net.h, 4096, 8192, ptr(x), None) == _lib.OT_ERR_OOM
    loss = ctypes.c_float(0.0)
    dy = torch.empty_like(x)
    assert lib.ot_cnn_loss(net.h, ptr(x), ptr(dy), ctypes.byref(loss)) == _lib.OT_ERR_ARG
    assert lib.ot_cnn_backward(net.h, ptr(y), ptr(net.grad), None) == _lib.OT_ERR_ARG
    assert torch.equal(net.forward(x), y)
    assert torch.equal(net.backward(x, y), g)
