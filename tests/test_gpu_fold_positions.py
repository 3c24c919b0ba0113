"""The folded back-projection rounds the position of a subtile's middle one way,
fma(x, cos, y sin) + C0 in double, whatever tile it lies in: the voxels of
subtiles whose fraction the other order of that sum would round to the
neighbouring float are compared bit for bit with the same float arithmetic done
here in exact rationals.  (Image sizes 2^k + 1: the offset C0 is then free of
rounding questions itself.)"""
import math
from fractions import Fraction

import numpy as np
import pytest

from paper_1809_09725_gb300 import dynrecon as dr
from paper_1809_09725_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

NX, NY, NS = 513, 257, 577
f32 = np.float32


def _round32(x: Fraction) -> np.float32:
    """x rounded once to the nearest float (normal range)."""
    if x == 0:
        return f32(0.0)
    n, d = abs(x).numerator, abs(x).denominator
    e = n.bit_length() - d.bit_length()
    if Fraction(n, d) < Fraction(2) ** e:
        e -= 1
    m = round(abs(x) / Fraction(2) ** (e - 23))  # ties to even
    return f32(math.copysign(math.ldexp(m, e - 23), x))


def _fma(a, b, c):
    return _round32(Fraction(float(a)) * Fraction(float(b)) + Fraction(float(c)))


def _tile(th, xo, yo, row):
    """The 16 x 16 voxels round (xo, yo) of one projection at angle th."""
    c, s = math.cos(th), math.sin(th)
    inv = 1.0 / max(abs(c), abs(s))
    e0, ic2 = f32(float(Fraction(-0.5 * inv) * Fraction(inv) + Fraction(inv))), f32(inv * inv)
    C0 = (-(NX - 1) / 2 * c - (NY - 1) / 2 * s) + (NS - 1) / 2
    pos = float(Fraction(xo) * Fraction(c) + Fraction(yo * s)) + C0
    fl = math.floor(pos)
    qb = f32(pos - fl) - f32(0.5)
    out = np.zeros((16, 16), dtype=np.float32)
    for j in range(16):
        for i in range(16):
            if xo - 8 + i >= NX or yo - 8 + j >= NY:
                continue
            q = _fma(f32(j - j % 2 - 8), f32(s), _fma(f32(i - 8), f32(c), qb))
            if j % 2:
                q = q + f32(s)
            near = np.rint(q)  # ties to even, as adding 1.5 * 2^23 rounds
            b = fl + int(near)
            d = q - near
            w0, w1 = max(f32(0), _fma(-d, ic2, e0)), max(f32(0), _fma(d, ic2, e0))
            g0 = row[b] if 0 <= b < NS else f32(0)
            g1 = row[b + 1] if 0 <= b + 1 < NS else f32(0)
            out[j, i] = _fma(w1, g1, w0 * g0)
    return out


@pytest.mark.parametrize("step,xo,yo", [(8736, 360, 8), (30404, 408, 232), (33149, 440, 8), (37721, 168, 136)])
def test_position_of_a_subtile(step, xo, yo):
    th = math.pi * (step + 0.37) / 40011.0
    plan = dr.Plan(NX, NY, 1, NS, np.array([th]), np.array([0.0]), dr.LEGENDRE, 10, 2, dr.F32)
    plan.set_variant(dr.DIRECT, dr.FOLD)
    g = synth.rng_for(4900).standard_normal((1, 1, NS)).astype(np.float32)
    u = torch.zeros(plan.u_shape(), dtype=torch.float32, device="cuda")
    dr.dyn_radon_adj(plan, torch.from_numpy(g).cuda(), u)
    plan.sync()
    got = u[0, yo - 8:yo + 8, xo - 8:xo + 8, 0].cpu().numpy()  # coefficient 0: weight 1
    ref = _tile(th, xo, yo, g[0, 0])[:got.shape[0], :got.shape[1]]
    np.testing.assert_array_equal(got, ref)
