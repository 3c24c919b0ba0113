"""The back-projection kernels work on one or several slices, and on all or a share
of a voxel's coefficients, per thread, by rules on the size of the grid.  Every
form gives the same bits: a volume large enough for the many-slice and
all-coefficient forms against its slices back-projected one by one (which take the
others), at edges of tiles and with a slice left over.  The one-by-one forms are
compared with the oracle elsewhere."""
import numpy as np
import pytest

from paper_1809_09725_gb300 import dynrecon as dr
from paper_1809_09725_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _compare(nx, ny, nz, ns, K, ht, m, prec, adj):
    theta, t = synth.scan(K, ht)
    dt = torch.bfloat16 if prec == dr.BF16 else torch.float32
    gen = torch.Generator("cuda").manual_seed(nx + m)
    g = torch.randn((nz, K, ns), device="cuda", generator=gen).to(dt)
    out = []
    for n in (nz, 1):
        plan = dr.Plan(nx, ny, n, ns, theta, t, dr.LEGENDRE, m, 2, prec)
        plan.set_variant(dr.DIRECT, adj)
        u = torch.full((nz, ny, nx, m), float("nan"), device="cuda").to(dt)
        for z in range(0, nz, n):
            dr.dyn_radon_adj(plan, g[z:z + n], u[z:z + n])
        plan.sync()
        out.append(u)
    assert torch.equal(out[0], out[1])
    assert torch.isfinite(out[0]).all()


# eight tiles by 75 slices: 304 CTAs of two slices, four rounds of one-slice ones on 152 SMs
@pytest.mark.parametrize("m,nx,ny", [(1, 40, 50), (2, 64, 64), (4, 33, 49), (7, 47, 61), (8, 64, 50), (10, 30, 64),
                                     (16, 17, 49), (20, 13, 61), (32, 16, 64)])
@pytest.mark.parametrize("ns", [64, 67])
def test_direct_two_slices_are_the_one_slice_bits(m, nx, ny, ns):
    _compare(nx, ny, 75, ns, 33, 0.97, m, dr.F32, dr.DIRECT)


def test_direct_two_slices_of_bf16_rows():
    _compare(47, 61, 75, 64, 33, 0.97, 7, dr.BF16, dr.DIRECT)


# 304 CTAs of four (m <= 4) or two slices
@pytest.mark.parametrize("m,nz", [(1, 151), (2, 152), (4, 151), (5, 75), (8, 76), (7, 75)])
@pytest.mark.parametrize("prec", [dr.F32, dr.BF16])
def test_folded_slices_per_thread_are_the_one_slice_bits(m, nz, prec):
    _compare(45, 61, nz, 66, 60, 6, m, prec, dr.FOLD)


# CTAs above the line from which a thread takes all (m <= 16) or half of a voxel's coefficients
@pytest.mark.parametrize("m,nx,nz", [(10, 45, 40), (12, 64, 40), (16, 33, 100), (13, 50, 100), (24, 29, 60), (20, 32, 60),
                                     (32, 17, 80), (27, 30, 80)])
@pytest.mark.parametrize("prec", [dr.F32, dr.BF16])
def test_folded_coefficients_per_thread_are_the_same_bits(m, nx, nz, prec):
    _compare(nx, 31, nz, 66, 60, 6, m, prec, dr.FOLD)
