"""Calls that reach the step kernels by another way than ``step``, against ``step`` or the oracle."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("flow", [False, True])
def test_profile_advances_as_step(prec, flow):
    """``profile(n)`` leaves the state that ``step(n)`` leaves, with the flow frozen too: fields, forces on a mobile
    colloid and its motion (sums over faces and links run in any order: 1e-9 of the force, 1e-6 in FP32 storage)."""
    import paper_1102_2193_gb300 as P
    L, prm = (24, 20, 22), dict(synth.NEMATIC, q0=2 * np.pi / 15)
    q = synth.random_q((L[2], L[1], L[0]), 3, amp=0.05, base=(0.2, 0.05, 0.02, -0.1, 0.03))
    out = []
    for how in ("step", "profile"):
        s = P.Solver(*L, precision=P.LC_FP32 if prec == "f32" else P.LC_FP64, flow=flow, **prm)
        s.set_Q(q)
        s.add_colloid((11.3, 9.8, 10.6), 4.2, P.LC_NORMAL, 0.02, mobile=True)
        getattr(s, how)(4)
        out.append((s.get_Q(), s.colloid(0)))
    (qa, a), (qb, b) = out
    tol = 1e-6 if prec == "f32" else 1e-9
    F = np.abs(a["F_lc"]).max()
    assert F > 0
    for k in ("F_lc", "T_lc", "F_hyd", "T_hyd"):
        assert np.abs(np.asarray(a[k]) - b[k]).max() <= tol * F * (4.2 if k[0] == "T" else 1.0), k
    assert np.abs(np.asarray(a["V"]) - b["V"]).max() <= tol * np.abs(a["V"]).max()
    assert np.abs(np.asarray(a["X"]) - b["X"]).max() <= 1e-12 * 24
    assert np.abs(qa - qb).max() <= tol
