"""An infinity or a NaN in the data reaches, in the folded back-projection, the
voxels whose two bins of that projection hold it and no other: every other voxel
is bit for bit that of the same data without it.  (A patch of 2 x 2 voxels
multiplies its neighbours' bins by zero.)"""
import numpy as np
import pytest

from paper_1809_09725_gb300 import dynrecon as dr
from paper_1809_09725_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

NX, NY, NS, K, HT = 45, 38, 52, 60, 5


@pytest.mark.parametrize("m", [1, 4, 7, 8, 12, 16, 24, 32])
@pytest.mark.parametrize("prec,beta", [(dr.F32, 0.0), (dr.F32, 0.5), (dr.BF16, 0.0)])
def test_nonfinite_data_stays_with_its_voxels(m, prec, beta):
    theta, t = synth.scan(K, HT)
    nz = 3
    plan = dr.Plan(NX, NY, nz, NS, theta, t, dr.LEGENDRE, m, 2, prec)
    plan.set_variant(dr.DIRECT, dr.FOLD)
    dt = torch.float32 if prec == dr.F32 else torch.bfloat16
    g = torch.from_numpy(synth.random_g(synth.rng_for(4950 + m), nz, K, NS)).to(dt).cuda()
    u0 = torch.from_numpy(synth.random_u(synth.rng_for(4951), nz, NY, NX, m)).to(dt).cuda()

    def back(data):
        u = u0.clone()
        dr.dyn_radon_adj(plan, data, u, beta)
        plan.sync()
        return u

    clean = back(g)
    bad = g.clone()
    spots = [(0, 0, 20, float("inf")), (1, 17, 31, float("nan")), (1, 44, 9, -float("inf"))]
    X, Y = np.meshgrid(np.arange(NX) - 0.5 * (NX - 1), np.arange(NY) - 0.5 * (NY - 1))
    hit, near = np.zeros((nz, NY, NX), bool), np.zeros((nz, NY, NX), bool)
    for z, k, b, v in spots:
        bad[z, k, b] = v
        d = np.abs(X * np.cos(theta[k]) + Y * np.sin(theta[k]) + 0.5 * (NS - 1) - b)
        hit[z] |= d < 1 - 1e-3
        near[z] |= d < 1 + 1e-3
    got = back(bad)
    finite = torch.isfinite(got).all(-1).cpu().numpy()
    assert hit.any() and not finite[hit].any()
    assert finite[~near].all()
    keep = torch.from_numpy(~near).cuda()
    assert torch.equal(got[keep], clean[keep])
