"""The row filter of the FBP start at the edges of its tiles, through
dr_fbp_init on small images: rows shorter than a vector, one vector past a
chunk or a tile, several chunks and tiles, rows left over in the last group, and
few rows (two per thread) as well as many (eight).  Tolerances are those of the
other FBP tests: 1e-11 in FP64, 1e-5 in FP32."""
import numpy as np
import pytest

import oracle
from paper_1809_09725_gb300 import dynrecon as dr
from paper_1809_09725_gb300 import synth

from _common import assert_close, dev_tensor, host_values

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# ns, nz, K
SIZES = [(1, 1, 16), (3, 2, 30), (5, 1, 17), (64, 3, 34), (127, 5, 66), (300, 1, 21), (301, 9, 72), (512, 4, 150),
         (513, 2, 180), (516, 1, 33), (1027, 3, 90), (2045, 1, 100), (2048, 1, 11)]


@pytest.mark.parametrize("ns,nz,K", SIZES)
@pytest.mark.parametrize("prec,tol", [(dr.F64, 1e-11), (dr.F32, 1e-5)])
def test_filter_tiles(ns, nz, K, prec, tol):
    theta, t = synth.scan(K, 2.0)
    args = (9, 8, nz, ns, theta, t, dr.FOURIER, 3, 2)
    g = synth.rng_for(720 + ns).standard_normal((nz, K, ns))
    g = g.astype(np.float32).astype(np.float64)
    P = oracle.Problem(*args)
    plan = dr.Plan(*args, prec=prec)
    u = torch.full(plan.u_shape(), 7.0, dtype=getattr(torch, plan.storage_dtype), device="cuda")
    dr.fbp_init(plan, dev_tensor(g, prec), u, 2)
    plan.sync()
    assert_close(host_values(u), P.fbp_init(g, 2), tol)
