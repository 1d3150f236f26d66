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


@pytest.mark.parametrize("cin", [24, 40, 56, 64, 72, 0])
@pytest.mark.parametrize("taps", [1, 27])
def test_weight_gradient_refuses_other_channel_counts(cin, taps):
    """Input-channel counts that no layer kernel is made for are refused whichever path the tensors' alignment takes."""
    import ctypes as C

    import paper_1102_2193_gb300 as P
    L = P.lib()
    z = torch.zeros(64 * 80 + 8, dtype=torch.bfloat16, device="cuda")
    w = torch.zeros(16 * 27 * 80, dtype=torch.float32, device="cuda")
    part = torch.zeros(16 * 27 * 80, dtype=torch.float32, device="cuda")
    for off in (0, 2):
        p = C.c_void_p(z.data_ptr() + 2 * off)
        assert L.lc_nn_conv3d_wgrad(p, p, C.c_void_p(w.data_ptr()), C.c_void_p(part.data_ptr()), 4, 4, 4, cin, 16, taps,
                                    None) == -1
