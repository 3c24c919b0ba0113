"""The row filter of the FBP start runs one row per CTA in FP64 and where there is at
most a row per SM, tiles of rows otherwise: the same sums, so the start of many
slices is bit for bit that of its slices one by one."""
import numpy as np
import pytest

from paper_1809_09725_gb300 import dynrecon as dr
from paper_1809_09725_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("ns", [1, 33, 128, 257, 512, 513])
@pytest.mark.parametrize("prec", [dr.F32, dr.BF16, dr.F64])
def test_filtered_rows_do_not_depend_on_their_number(ns, prec):
    K, nz = 60, 40  # 60 rows by themselves, 2400 together
    theta, t = synth.scan(K, 2.0)
    out = []
    for n in (nz, 1):
        plan = dr.Plan(9, 8, n, ns, theta, t, dr.FOURIER, 3, 2, prec)
        plan.set_variant(dr.DIRECT, dr.DIRECT)
        dt = getattr(torch, plan.storage_dtype)
        g = torch.from_numpy(synth.rng_for(730 + ns).standard_normal((nz, K, ns))).to(dt).cuda()
        u = torch.full((nz, 8, 9, 3), 7.0, dtype=dt, device="cuda")
        for z in range(0, nz, n):
            dr.fbp_init(plan, g[z:z + n], u[z:z + n], 2)
        plan.sync()
        out.append(u)
    assert torch.isfinite(out[0].double()).all()
    np.testing.assert_array_equal(out[0].double().cpu().numpy(), out[1].double().cpu().numpy())
