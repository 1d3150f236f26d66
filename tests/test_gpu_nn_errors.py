"""Refused calls of the network's kernels: the codes, and that the next call is not refused for them."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_refused_bias_gradient_leaves_no_error():
    """No channels are refused (by the launch, as an empty grid); the next call works."""
    import ctypes as C

    import paper_1102_2193_gb300 as P
    L = P.lib()
    d = torch.ones((64, 16), dtype=torch.float32, device="cuda")
    db = torch.zeros(16, dtype=torch.float32, device="cuda")
    a, b = C.c_void_p(d.data_ptr()), C.c_void_p(db.data_ptr())
    assert L.lc_nn_bias_grad(a, b, 64, 0, None) != 0
    half = torch.empty((64, 16), dtype=torch.bfloat16, device="cuda")
    assert L.lc_nn_cast_bf16(a, C.c_void_p(half.data_ptr()), 64 * 16, None) == 0
    assert L.lc_nn_bias_grad(a, b, 64, 16, None) == 0
    torch.cuda.synchronize()
    assert (db == 64.0).all()
