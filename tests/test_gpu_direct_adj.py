"""Direct back-projection with one and two slices per thread against the FP64
oracle: each of its three ways of staging the data (rows of whole 16-byte
vectors, other rows, bf16 rows of odd length), odd numbers of slices, images
that cut a tile, projections left over in the last stage, every coefficient
group, and u = beta u + R* g.  Tolerances are those of the other operator tests:
1e-5 in FP32, 1e-11 in FP64, 1e-3 for BF16 storage."""
import numpy as np
import pytest

import oracle
from paper_1809_09725_gb300 import dynrecon as dr
from paper_1809_09725_gb300 import synth

from _common import assert_close, dev_tensor, host_values, to_bf16_f64

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# nx, ny, nz, ns, K, m: one slice per thread first, then two
CASES = [(33, 17, 1, 40, 33, 8), (40, 50, 3, 61, 65, 5), (20, 30, 2, 30, 7, 1), (64, 33, 2, 67, 31, 16),
         (100, 90, 29, 120, 33, 8), (97, 101, 31, 131, 64, 7), (70, 100, 29, 101, 35, 2), (70, 70, 41, 64, 50, 4),
         (90, 80, 21, 97, 40, 1), (66, 80, 27, 90, 40, 12), (65, 70, 27, 75, 33, 16), (60, 65, 17, 70, 32, 24),
         (57, 64, 19, 59, 37, 32)]
TOL = {dr.F32: 1e-5, dr.F64: 1e-11, dr.BF16: 1e-3}


@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(map(str, c)))
@pytest.mark.parametrize("prec", [dr.F32, dr.F64, dr.BF16])
@pytest.mark.parametrize("beta", [0.0, 0.5])
def test_direct_backprojection_matches_oracle(case, prec, beta):
    nx, ny, nz, ns, K, m = case
    theta, t = synth.scan(K, 0.97)
    plan = dr.Plan(nx, ny, nz, ns, theta, t, dr.LEGENDRE, m, 3, prec)
    P = oracle.Problem(nx, ny, nz, ns, theta, t, oracle.LEGENDRE, m, 3)
    plan.set_variant(dr.DIRECT, dr.DIRECT)
    rng = synth.rng_for(4900 + m + nz)
    store = {dr.F64: lambda a: a, dr.F32: lambda a: a.astype(np.float32).astype(np.float64), dr.BF16: to_bf16_f64}[prec]
    g, u0 = store(synth.random_g(rng, nz, K, ns)), store(synth.random_u(rng, nz, ny, nx, m))
    gd = dev_tensor(g, prec)
    outs = []
    for _ in range(2):
        u = dev_tensor(u0, prec)
        dr.dyn_radon_adj(plan, gd, u, beta)
        plan.sync()
        outs.append(host_values(u))
    np.testing.assert_array_equal(outs[1], outs[0])
    ref = P.adj(g) + beta * u0
    assert_close(outs[0], store(ref) if prec == dr.BF16 else ref, TOL[prec])
