"""FP32 boxes near rest against stored results.  Such a flow is driven by small differences of the stress, and a sum
of H, P or the collision rounded in another order shows in it at 2e-5 and more although it is no less exact (the
oracle cannot tell the two apart: both are that far from FP64).  The stored values are those of the first build of the
step kernels on GB300 (one node or one packed pair at a time, H and P by sums over 3x3 matrices); tolerance 1e-5, half
of what two runs of FP32 storage may differ by.  ``python tests/test_gpu_fp32_order.py FILE`` writes them."""
import os
import sys

import numpy as np
import pytest

if __name__ == "__main__":
    sys.path.insert(0, os.getcwd())
import oracle
import synth

pytestmark = pytest.mark.gpu
GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "fp32_order.npz")
C = np.array([[0, 0, 0], [1, 0, 0], [-1, 0, 0], [0, 1, 0], [0, -1, 0], [0, 0, 1], [0, 0, -1], [1, 1, 0], [-1, -1, 0],
              [1, -1, 0], [-1, 1, 0], [1, 0, 1], [-1, 0, -1], [1, 0, -1], [-1, 0, 1], [0, 1, 1], [0, -1, -1], [0, 1, -1],
              [0, -1, 1]], dtype=float)
# sides, pitch, walls, colloid (position, radius, anchoring, w), steps
CASES = {"nematic": ((32, 24, 20), 0.0, False, None, 40),
         "odd": ((31, 23, 21), 16.0, False, None, 40),
         "mobile": ((34, 30, 36), 0.0, True, ((16.3, 14.6, 16.8), 4.7, 0, float("inf")), 40),
         "mobile_planar": ((38, 28, 30), 26.0, True, ((18.1, 13.4, 14.2), 4.1, 1, 0.02), 40)}


def start(L, pitch, seed):
    """Bulk order 1/2, a helix along z or a tilted nematic, with noise of 1e-3 (whole 2^-20ths: the same everywhere)."""
    z = np.arange(L[2])[:, None, None] + np.zeros((L[2], L[1], L[0]))
    if pitch:
        n = [np.cos(2 * np.pi / pitch * z), np.sin(2 * np.pi / pitch * z), 0 * z]
    else:
        n = [np.full(z.shape, v / np.sqrt(1.13)) for v in (0.3, 0.2, 1.0)]
    q = 0.5 * np.stack([n[0] * n[0] - 1 / 3, n[0] * n[1], n[0] * n[2], n[1] * n[1] - 1 / 3, n[1] * n[2]])
    return np.round((q + 1e-3 * (2 * np.random.default_rng(seed).random(q.shape) - 1)) * 2**20) / 2**20


def run(name):
    import paper_1102_2193_gb300 as P
    L, pitch, walls, col, steps = CASES[name]
    prm = dict(synth.NEMATIC, q0=2 * np.pi / pitch if pitch else 0.0)
    s = P.Solver(*L, wall_z=walls, precision=P.LC_FP32, **prm)
    s.set_Q(start(L, pitch, 5))
    if col:
        s.add_colloid(col[0], col[1], col[2], col[3], mobile=True, F_ext=(1e-4, 4e-5, 0.0))
    s.step(steps)
    if col:
        c = s.colloid(0)
        return {"force": c["F_hyd"] + c["F_lc"]}
    return {"momentum": np.einsum("qa,qzyx->azyx", C, s.get_f()).reshape(3, -1)[:, ::3]}


@pytest.mark.parametrize("name", list(CASES))
def test_fp32_results(name):
    ref = np.load(GOLDEN)
    for k, v in run(name).items():
        r = ref[name + "_" + k].astype(float)
        assert np.linalg.norm(v - r) <= 1e-5 * np.linalg.norm(r), k


if __name__ == "__main__":
    np.savez_compressed(sys.argv[1], **{n + "_" + k: v.astype(np.float32) for n in CASES for k, v in run(n).items()})
