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


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("w", [0.02, float("inf")])
def test_normal_surface_values_at_low_face(axis, w):
    """FP32 surface values of a colloid across the low periodic face of a long box: its LC force and torque are those
    of the same colloid and field shifted by half the box.  Both differ by the sum of FP64 atomics and by the last bit
    of few surface values only (1e-6; an error of 4e-6 in the normal, a rounding at the size of the box, shows at 1e-5)."""
    import paper_1102_2193_gb300 as P
    L, X = [20, 22, 24], np.array([9.3, 10.6, 12.4])
    L[axis] = 256
    X[axis] = np.round(0.4 * 2.0**40) / 2.0**40
    prm = dict(synth.NEMATIC, q0=2 * np.pi / 17)
    q = synth.random_q((L[2], L[1], L[0]), 9, amp=0.05, base=(0.2, 0.05, 0.02, -0.1, 0.03))
    out = []
    for shift in (0, 128):
        s = P.Solver(*L, precision=P.LC_FP32, **prm)
        s.set_Q(np.roll(q, shift, axis=3 - axis))
        Y = X.copy()
        Y[axis] += shift
        s.add_colloid(Y, 6.3, P.LC_NORMAL, w)
        s.step(1)
        out.append(s.colloid(0))
    a, b = out
    F = np.abs(a["F_lc"]).max()
    assert F > 0 and np.abs(a["F_lc"] - b["F_lc"]).max() <= 1e-6 * F
    assert np.abs(a["T_lc"] - b["T_lc"]).max() <= 1e-6 * 6.3 * F


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("radius", [3.0, 8.5])
def test_residual_of_other_boxes_after_add_colloid(prec, radius):
    """The last step's residual of a box of a batch is the same after a colloid was added to the box before it (one
    whose near nodes fit the allocated groups, and one that takes more)."""
    import paper_1102_2193_gb300 as P
    prm = dict(synth.NEMATIC, q0=0.0)
    L = ((22, 24, 26), (26, 20, 18), (18, 18, 18))
    B = P.Batch([dict(grid=g, params=prm) for g in L], precision=P.LC_FP32 if prec == "f32" else P.LC_FP64)
    for k, s in enumerate(B.boxes):
        s.set_Q(synth.random_q(L[k][::-1], k, amp=0.05, base=(0.2, 0.05, 0.02, -0.1, 0.03)))
        s.add_colloid((9.3, 8.6, 9.1), 3.1, P.LC_NORMAL, 0.02)
    B.step(3)
    before = [s.diag() for s in B.boxes]
    B.boxes[0].add_colloid((19.6 if radius < 5 else 20.9, 20.4, 21.2), radius, P.LC_NORMAL, 0.02)
    for s, d in list(zip(B.boxes, before))[1:]:
        after = s.diag()
        assert after["resid_rms"] == d["resid_rms"] and after["resid_max"] == d["resid_max"]


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("size,gap", [(1.0, 1e-1), (1.0, 1e-2), (1.0, 3e-3), (1.0, 3e-4), (1.0, 1e-4), (1.0, 1e-5),
                                      (1.0, 1e-6), (1e-20, 0.3), (1e-22, 0.3), (1e-6, 0.1)])
def test_planar_faces_of_close_eigenvalues(prec, size, gap):
    """Planar surface values where the two largest eigenvalues of Q are ``gap`` apart (size 1: 0.16 + g/2, 0.16 - g/2,
    -0.32), and of a Q that FP32 products lose: the colloid's LC force after one step against the oracle (Jacobi).
    Tolerance: the angle of the director in FP64, 1e-17 / gap^2 (relative), ten times over, the rounding of Q as it is
    stored (FP32 and a BF16 remainder: 4e-10 / gap at most) and of the FP32 force (2e-5)."""
    import paper_1102_2193_gb300 as P
    L, X, prm = (20, 18, 16), (9.4, 8.3, 7.7), dict(synth.NEMATIC, q0=0.0)
    R = np.linalg.qr(np.random.default_rng(4).standard_normal((3, 3)))[0]
    A = size * (R * [0.16 + gap / 2, 0.16 - gap / 2, -0.32]) @ R.T
    q = np.tile(np.array([A[0, 0], A[0, 1], A[0, 2], A[1, 1], A[1, 2]]).reshape(5, 1, 1, 1), (1, L[2], L[1], L[0]))
    s, o = P.Solver(*L, precision=P.LC_FP32 if prec == "f32" else P.LC_FP64, **prm), oracle.Oracle(*L, **prm)
    for k in (s, o):
        k.set_Q(q)
        k.add_colloid(X, 4.6, 1, 0.03)
        k.step(1)
    a, b = s.colloid(0), o.colloid(0)
    F = np.abs(b["T_lc"]).max() / 4.6 + np.abs(b["F_lc"]).max()
    g = gap / 0.16
    tol = 1e-9 + 1e-16 / g**2 + (2e-5 + 4e-9 / g if prec == "f32" else 0.0)
    assert np.abs(a["F_lc"] - b["F_lc"]).max() <= tol * F
    assert np.abs(a["T_lc"] - b["T_lc"]).max() <= 4 * tol * 4.6 * F


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_export_destinations(prec):
    """Fields read into device memory, aligned to 16 bytes and to 8: the values that a host destination receives, and
    nothing beside them."""
    import ctypes as C

    import torch

    import paper_1102_2193_gb300 as P
    L, prm = (22, 9, 7), dict(synth.NEMATIC, q0=0.2)
    s = P.Solver(*L, precision=P.LC_FP32 if prec == "f32" else P.LC_FP64, **prm)
    s.set_Q(synth.random_q(L[::-1], 3, amp=0.05, base=(0.2, 0.05, 0.02, -0.1, 0.03)))
    s.add_colloid((9.3, 4.2, 3.1), 2.3, P.LC_NORMAL, 0.02)
    s.step(2)
    N = L[0] * L[1] * L[2]
    for which, nc in ((P.LC_Q, 5), (P.LC_U, 3), (P.LC_RHO, 1)):
        ref = np.empty(nc * N)
        dp = ref.ctypes.data_as(C.c_void_p)
        assert s.L.lc_lb_get_fields(s.h, which, dp, ref.nbytes, 0) == 0
        for off in (0, 1):
            out = torch.full((nc * N + 2,), 7.0, dtype=torch.float64, device="cuda")
            assert s.L.lc_lb_get_fields(s.h, which, C.c_void_p(out.data_ptr() + 8 * off), ref.nbytes, 1) == 0
            assert (out[off:off + nc * N].cpu().numpy() == ref).all()
            assert (out[:off] == 7.0).all() and (out[off + nc * N:] == 7.0).all()


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_tuned_shapes_of_frozen_and_coupled_boxes(prec, tmp_path, monkeypatch):
    """A box relaxed with the flow frozen and a coupled box of the same size are tuned apart (their steps are different
    kernels), each once; the results do not depend on the order."""
    import paper_1102_2193_gb300 as P
    L = (23, 17, 21) if prec == "f32" else (21, 17, 23)
    cache = tmp_path / "tune.txt"
    monkeypatch.setenv("LCLB_TUNE_CACHE", str(cache))
    for flow in (False, True, False, True):
        s = P.Solver(*L, precision=P.LC_FP32 if prec == "f32" else P.LC_FP64, flow=flow, **dict(synth.NEMATIC, q0=0.2))
        s.set_Q(synth.random_q(L[::-1], 3, amp=0.05, base=(0.2, 0.05, 0.02, -0.1, 0.03)))
        s.step(2)
    keys = [tuple(r.split()[:2]) for r in cache.read_text().splitlines()]
    assert len(keys) == 2 and len(set(keys)) == 2


@pytest.mark.parametrize("moving", [False, True])
@pytest.mark.parametrize("nx", [38, 37])
def test_residual_is_the_same_for_every_handle(nx, moving):
    """The FP32 residual of a box with many near nodes, summed over the list of them: the same bits from eight handles
    of the same state, also after a colloid has moved from node to node (a colloid held by its own inertia: its
    velocity is set before every step, so that sums in any order do not reach the fields)."""
    import paper_1102_2193_gb300 as P
    L, prm = (nx, 34, 36), dict(synth.NEMATIC, q0=0.3)
    q = synth.random_q(L[::-1], 3, amp=0.05, base=(0.2, 0.05, 0.02, -0.1, 0.03))
    seen = set()
    for _ in range(8):
        s = P.Solver(*L, wall_z=True, precision=P.LC_FP32, flow=False, **prm)
        s.set_Q(q)
        s.add_colloid((14.3, 16.2, 17.4), 9.6, P.LC_NORMAL, 0.02, mobile=moving)
        if moving:
            for _ in range(3):
                s.set_colloid_velocity(0, (0.4, 0.3, 0.2))
                s.step(1)
        s.step(1)
        d = s.diag()
        seen.add((d["resid_rms"], d["resid_max"]))
    assert len(seen) == 1


@pytest.mark.parametrize("w", [1e-3, 1e-12, 1e-22, 1e3])
@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_surface_energy(w, prec):
    """Free energy of weakly anchored faces alone (no bulk term, a uniform Q): (w/2)|Qs - Q0|^2 of every face against the
    oracle, over the range of w in which squares of Qs - Q leave FP32.  Tolerance: FP32 surface values (1e-6)."""
    import paper_1102_2193_gb300 as P
    L, prm = (20, 18, 16), dict(synth.NEMATIC, q0=0.0, A0=0.0)
    q = np.tile(np.array([0.2, 0.05, 0.02, -0.1, 0.03]).reshape(5, 1, 1, 1), (1, L[2], L[1], L[0]))
    s, o = P.Solver(*L, precision=P.LC_FP32 if prec == "f32" else P.LC_FP64, **prm), oracle.Oracle(*L, **prm)
    for k in (s, o):
        k.set_Q(q)
        k.add_colloid((9.4, 8.3, 7.7), 4.6, 0, w)
    a, b = s.diag()["free_energy"], o.diag()["free_energy"]
    assert b > 0 and abs(a - b) <= (1e-6 if prec == "f32" else 1e-11) * b
