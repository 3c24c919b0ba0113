"""The channel-lane forward when the plan's status word is already set (another
launch's bounded wait gave up): its compute warps leave at once, its copy warp
first waits for the copies it has in flight, the failure is reported once, and
the next call is right."""
import ctypes
import threading
import time

import numpy as np
import pytest

from paper_1809_09725_gb300 import dynrecon as dr
from paper_1809_09725_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_forward_after_a_wait_gave_up():
    theta, t = synth.scan(360, 6)
    plan = dr.Plan(256, 256, 16, 256, theta, t, dr.LEGENDRE, 8, 3, dr.F32)
    lib = dr.load()
    lib.dr_internal_use_channels.argtypes = [ctypes.c_void_p, ctypes.c_int]
    assert lib.dr_internal_use_channels(plan.handle, 0) == dr.DR_OK
    u = torch.randn(plan.u_shape(), device="cuda", generator=torch.Generator("cuda").manual_seed(7))
    ref, g = torch.empty(plan.g_shape(), device="cuda"), torch.empty(plan.g_shape(), device="cuda")
    dr.dyn_radon_fwd(plan, u, ref)
    plan.sync()
    status = []
    waiter = threading.Thread(target=lambda: status.append(plan.wait_selftest(1.0)))
    waiter.start()
    time.sleep(0.3)
    dr.dyn_radon_fwd(plan, u, g)  # queued behind the wait that will have given up
    waiter.join()
    torch.cuda.synchronize()
    assert status == [dr.DR_ETIMEOUT]
    try:
        plan.sync()  # (the status word may have been read before or after the forward)
    except dr.DynreconError:
        pass
    dr.dyn_radon_fwd(plan, u, g)
    plan.sync()
    np.testing.assert_array_equal(g.cpu().numpy(), ref.cpu().numpy())
