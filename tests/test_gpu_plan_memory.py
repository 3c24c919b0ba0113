"""What a plan says of its device memory, and what it holds of it: the two calls
that report it agree, scratch stays within what a serving job is counted for, and
nothing is kept for a kernel that the autotuner did not choose."""
import ctypes

import numpy as np
import pytest

from paper_1809_09725_gb300 import dynrecon as dr
from paper_1809_09725_gb300 import synth

from _common import dev_tensor

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _plan(nx, ny, nz, ns, K, ht, m, prec=dr.F32):
    theta, t = synth.scan(K, ht)
    return dr.Plan(nx, ny, nz, ns, theta, t, dr.LEGENDRE, m, 3, prec)


def _use_channels(plan, solvers):
    lib = dr.load()
    lib.dr_internal_use_channels.argtypes = [ctypes.c_void_p, ctypes.c_int]
    lib.dr_internal_use_channels.restype = ctypes.c_int
    assert lib.dr_internal_use_channels(plan.handle, solvers) == dr.DR_OK


def _pair(plan):
    u = torch.zeros(plan.u_shape(), dtype=getattr(torch, plan.storage_dtype), device="cuda")
    g = torch.zeros(plan.g_shape(), dtype=u.dtype, device="cuda")
    dr.dyn_radon_fwd(plan, u, g)
    dr.dyn_radon_adj(plan, g, u)
    plan.sync()


def test_both_reports_of_device_memory_agree():
    plan = _plan(64, 64, 8, 64, 192, 8, 4)
    _use_channels(plan, 0)
    before = plan.device_bytes()
    _pair(plan)
    assert plan.device_bytes() > before
    assert plan.info()["device_bytes"] == plan.device_bytes()
