"""Step kernels at the edges of their tiles against the FP64 oracle: widths around the 64-column tiles of the
two-node path, rows of whole 16-byte pieces and others, a two-node-wide box, odd widths (one node per lane), ragged
heights, boxes one to three planes deep, walls, near-node lists that fill less than a group of 32 and several groups, and boxes without any near node.
Tolerances as the other parity tests (FP32 storage 1e-5 in Q, 1e-6 in u; FP64 1e-10, 1e-12)."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

CASES = [((64, 9, 3), False, None), ((66, 7, 5), False, (20.3, 3.1, 2.2, 1.6)), ((62, 5, 33), False, (30.2, 2.4, 15.7, 2.3)),
         ((130, 6, 10), True, (64.4, 2.9, 4.6, 2.6)), ((2, 3, 4), False, None), ((4, 1, 1), False, None),
         ((12, 10, 2), False, None), ((68, 12, 1), False, None), ((33, 17, 9), True, (15.1, 8.3, 4.4, 3.2)),
         ((1, 2, 3), False, None), ((20, 33, 18), False, (10.2, 16.4, 8.9, 7.1)),
         ((132, 7, 6), True, (66.1, 3.2, 2.7, 1.9)), ((36, 2, 5), False, None), ((128, 10, 4), False, (1.2, 9.1, 2.1, 1.7))]


@pytest.mark.parametrize("L,wall,col", CASES)
@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("pitch,flow", [(0.0, True), (12.0, True), (12.0, False)])
def test_step_edges(L, wall, col, prec, pitch, flow):
    import paper_1102_2193_gb300 as P
    prm = dict(synth.NEMATIC, q0=2 * np.pi / pitch if pitch else 0.0)
    q = synth.random_q((L[2], L[1], L[0]), 5, amp=0.02, base=(-0.1, 0.05, 0.02, -0.12, 0.03))
    s = P.Solver(*L, wall_z=wall, precision=P.LC_FP32 if prec == "f32" else P.LC_FP64, flow=flow, **prm)
    o = oracle.Oracle(*L, wall_z=wall, flow=flow, **prm)
    for k in (s, o):
        k.set_Q(q)
        if col:
            k.add_colloid(col[:3], col[3], 1, 0.02)
        k.step(5)
    fl = o.get_solid() < 0
    assert np.abs(s.get_Q() - o.get_Q())[:, fl].max() < (1e-5 if prec == "f32" else 1e-10)
    if flow:
        _, u = s.get_rho_u()
        _, ur = o.get_rho_u()
        assert np.abs(u - ur)[:, fl].max() < (1e-6 if prec == "f32" else 1e-12)
    r, ro = s.diag(), o.diag()
    assert abs(r["resid_rms"] - ro["resid_rms"]) <= (1e-4 if prec == "f32" else 1e-9) * ro["resid_rms"]
    assert abs(r["resid_max"] - ro["resid_max"]) <= (1e-3 if prec == "f32" else 1e-9) * ro["resid_max"]
    if col:
        a, b = s.colloid(0), o.colloid(0)
        F = np.abs(b["F_lc"]).max() + np.abs(b["F_hyd"]).max()
        tol = 1e-4 if prec == "f32" else 1e-9
        assert np.abs(a["F_lc"] - b["F_lc"]).max() <= tol * F and np.abs(a["F_hyd"] - b["F_hyd"]).max() <= tol * F


@pytest.mark.parametrize("anchoring,w", [(0, 0.02), (0, float("inf")), (1, 0.03)])
def test_surface_values_far_from_origin(anchoring, w):
    """FP32 surface values of colloids at positions that FP32 does not hold (the normal ones are summed in pairs of
    FP32 numbers) and across the periodic boundary: the colloid's LC force and torque after one step."""
    import paper_1102_2193_gb300 as P
    L, X, a0 = (130, 40, 34), (128.7, 39.2, 0.4), 9.3
    prm = dict(synth.NEMATIC, q0=2 * np.pi / 17)
    s, o = P.Solver(*L, precision=P.LC_FP32, **prm), oracle.Oracle(*L, **prm)
    q = synth.random_q((L[2], L[1], L[0]), 9, amp=0.05, base=(0.2, 0.05, 0.02, -0.1, 0.03))
    for k in (s, o):
        k.set_Q(q)
        k.add_colloid(X, a0, anchoring, w)
        k.step(1)
    a, b = s.colloid(0), o.colloid(0)
    assert np.abs(a["F_lc"] - b["F_lc"]).max() <= 2e-5 * np.abs(b["F_lc"]).max()
    assert np.abs(a["T_lc"] - b["T_lc"]).max() <= 1e-4 * a0 * np.abs(b["F_lc"]).max()


@pytest.mark.parametrize("scale", [0.0, 1e-12, 1e-3, 1.0, 1e6])
@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_exported_moments(scale, prec):
    """Density and velocity of populations of mixed magnitudes (the FP32 kernel adds them as integers at a common
    exponent) against FP64 sums of the exported populations.  Tolerance: 19 roundings of f, 18 of the sum and 3 of the
    quotient, 2^-53 of the sum of |f| each."""
    import paper_1102_2193_gb300 as P
    rng = np.random.default_rng(3)
    L = (33, 9, 5)
    d = rng.random((19, L[2], L[1], L[0])) * 10.0 ** rng.integers(-6, 1, (19, 1, L[1], L[0]))
    s = P.Solver(*L, precision=P.LC_FP32 if prec == "f32" else P.LC_FP64, **synth.NEMATIC)
    s.set_Q(np.zeros((5, L[2], L[1], L[0])))
    w = oracle.feq(1.0, (0, 0, 0)).reshape(19, 1, 1, 1)
    c = np.array([[0, 0, 0], [1, 0, 0], [-1, 0, 0], [0, 1, 0], [0, -1, 0], [0, 0, 1], [0, 0, -1], [1, 1, 0], [-1, -1, 0],
                  [1, -1, 0], [-1, 1, 0], [1, 0, 1], [-1, 0, -1], [1, 0, -1], [-1, 0, 1], [0, 1, 1], [0, -1, -1],
                  [0, 1, -1], [0, -1, 1]], dtype=float)
    s.set_f(w * (1.0 + scale * d))
    f, (rho, u) = s.get_f(), s.get_rho_u()
    total = np.abs(f).sum(0)
    eps = 40 * 2.0**-53
    assert (np.abs(rho - f.sum(0)) <= eps * total).all()
    m = np.einsum("qa,qzyx->azyx", c, f)
    assert (np.abs(u - m / f.sum(0)) <= 2 * eps * total / f.sum(0)).all()
