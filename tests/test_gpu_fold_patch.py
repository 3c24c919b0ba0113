"""Folded back-projection by patches of 2 x 2 voxels against the FP64 oracle at
the edges of its range: every coefficient group (one to 32, odd and even), several
slices per thread with a remainder, images that cut a patch, detectors narrower
and wider than the image, angles on both sides of the near-axis test, and scans
whose distinct angles lie in one quadrant only.  Tolerance 1e-5 for FP32
(relative L2 and largest element) as for the other folded operators, 1e-3 for
BF16 storage against the oracle's output rounded the same way."""
import numpy as np
import pytest

import oracle
from paper_1809_09725_gb300 import dynrecon as dr
from paper_1809_09725_gb300 import synth

from _common import assert_close, dev_tensor, host_values, to_bf16_f64

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

EPS = 4.4721e-3  # cos = 0.99999
Q = np.pi / 2
ANGLES = {
    "near_axis": np.concatenate([np.array([0.0, 1e-7, 1e-3, EPS * 0.999, EPS * 1.001, 0.05]) + a for a in (0.0, Q)] +
                                [np.array([-1e-7, -1e-3, -EPS * 0.999, -EPS * 1.001]) + a for a in (Q, 2 * Q)] +
                                [np.array([0.25, 0.75]) * np.pi]),
    "one_quadrant": np.linspace(0.02, 1.5, 11),
    "other_quadrant": np.linspace(1.6, 3.1, 13),
    "one_angle": np.array([0.6]),
    "scan": np.linspace(0.0, np.pi, 37, endpoint=False),
}

# nx, ny, nz, ns, m, angles
CASES = [(33, 31, 5, 48, 1, "scan"), (40, 24, 7, 47, 2, "near_axis"), (31, 47, 3, 20, 3, "scan"),
         (64, 64, 4, 92, 4, "near_axis"), (35, 65, 3, 75, 5, "scan"), (50, 34, 5, 30, 6, "one_quadrant"),
         (47, 33, 2, 58, 7, "near_axis"), (65, 49, 3, 200, 8, "scan"), (64, 48, 1, 80, 8, "other_quadrant"),
         (33, 34, 2, 40, 11, "near_axis"), (49, 31, 2, 60, 16, "scan"), (17, 40, 2, 24, 24, "near_axis"),
         (34, 18, 2, 36, 32, "scan"), (40, 17, 1, 44, 29, "one_angle"), (16, 16, 3, 23, 8, "one_angle")]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(map(str, c)))
@pytest.mark.parametrize("prec", [dr.F32, dr.BF16])
def test_patch_backprojection_matches_oracle(case, prec):
    nx, ny, nz, ns, m, angles = case
    a = np.sort(ANGLES[angles])
    theta = np.concatenate([a + h * np.pi for h in range(3)])
    t = np.linspace(0.0, 1.0, theta.size)
    plan = dr.Plan(nx, ny, nz, ns, theta, t, dr.LEGENDRE, m, 3, prec)
    P = oracle.Problem(nx, ny, nz, ns, theta, t, oracle.LEGENDRE, m, 3)
    plan.set_variant(dr.DIRECT, dr.FOLD)
    g = synth.random_g(synth.rng_for(4800 + m), nz, theta.size, ns)
    g = g.astype(np.float32).astype(np.float64) if prec == dr.F32 else to_bf16_f64(g)
    gd = dev_tensor(g, prec)
    outs = []
    for _ in range(2):
        u = torch.full(plan.u_shape(), float("nan"), dtype=gd.dtype, device="cuda")
        dr.dyn_radon_adj(plan, gd, u)
        plan.sync()
        outs.append(host_values(u))
    np.testing.assert_array_equal(outs[1], outs[0])
    ref = P.adj(g)
    if prec == dr.F32:
        assert_close(outs[0], ref, 1e-5)
    else:
        assert_close(outs[0], to_bf16_f64(ref), 1e-3)
