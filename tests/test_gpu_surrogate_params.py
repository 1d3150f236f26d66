"""Training with entries of ``UNet.params`` replaced by tensors of the caller's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("key", ["w", "b", "gw", "mw", "w16"])
def test_replaced_parameters_are_trained(key):
    """Two training steps with one entry of two layers replaced by a copy: the same weights as with the net's own."""
    from paper_1102_2193_gb300.surrogate import LAYERS, UNet
    S = 8
    g = np.random.default_rng(1)
    st = {n: dict(w=(g.standard_normal((co, t, ci)) * 0.1).astype(np.float32), b=np.zeros(co, np.float32))
          for n, ci, co, t, _, _ in LAYERS}
    solid = torch.full((S**3,), -1.0, dtype=torch.float64, device="cuda")
    q = torch.tensor(g.standard_normal((5, S**3)) * 0.1, device="cuda")
    target = torch.tensor(g.standard_normal((5, S**3)) * 0.1, device="cuda")
    out = []
    for replace in (False, True):
        net = UNet(S=S)
        net.load(st)
        if replace:
            for n in ("c1a", "head"):
                net.params[n][key] = net.params[n][key].clone()
        for _ in range(2):
            net.set_input(solid, q, 2.0, 8.0, 0.02)
            net.set_target(target)
            net.forward()
            net.loss_and_grad()
            net.backward()
            net.adam(lr=1e-2)
        out.append(net.state())
    for n in out[0]:
        assert (out[0][n]["w"] == out[1][n]["w"]).all() and (out[0][n]["b"] == out[1][n]["b"]).all(), n
        assert (out[0][n]["w"] != st[n]["w"]).any(), n
