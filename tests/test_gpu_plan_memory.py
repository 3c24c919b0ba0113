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


def test_solver_on_channels_stays_within_the_partial_sums_of_a_job():
    """72 channels padded to 128: eight line chunks of them exceed what a job of this
    size is counted for, so the solve stays on the fold in two kernels (same bits)
    and holds what that holds."""
    size = (32, 32, 9, 32, 150, 3, 8)
    g = dev_tensor(synth.random_g(synth.rng_for(4971), 9, 150, 32), dr.F32)
    held, us = [], []
    for channels in (True, False):
        plan = _plan(*size)
        plan.set_fold_march(8)
        if channels:
            _use_channels(plan, 1)
        else:
            plan.set_variant(dr.FOLD2, dr.FOLD)
        u = torch.zeros(plan.u_shape(), dtype=torch.float32, device="cuda")
        dr.admm_solve(plan, g, u, dr.solve_params(dr.ADMM_CG, iters=2, n_cg=2, lambda1=0.05, lambda2=1.0, rho=0.5))
        held.append(plan.device_bytes())
        us.append(u.cpu().numpy())
    assert held[0] == held[1]
    np.testing.assert_array_equal(us[0], us[1])


@pytest.mark.parametrize("size", [(64, 64, 8, 64, 192, 8, 4), (128, 128, 6, 128, 720, 8, 8), (96, 80, 16, 101, 360, 6, 5),
                                  (256, 256, 16, 256, 1800, 10, 8)])
@pytest.mark.parametrize("prec", [dr.F32, dr.BF16])
def test_first_forward_of_a_cached_plan_recorded_into_a_graph(size, prec):
    """A plan that takes its choices from the cache has the scratch of the kernels
    that won: its first forward, recorded into a graph, gives the bits of the plan
    that timed them."""
    timed = _plan(*size, prec)
    timed.autotune()
    cached = _plan(*size, prec)
    cached.autotune()
    dt = getattr(torch, timed.storage_dtype)
    u = torch.randn(timed.u_shape(), device="cuda", generator=torch.Generator("cuda").manual_seed(3)).to(dt)
    g, recorded = (torch.empty(timed.g_shape(), dtype=dt, device="cuda") for _ in range(2))
    dr.dyn_radon_fwd(timed, u, g)
    cached.set_variant(dr.FOLD2, dr.FOLD)  # (what the thread-per-ray forms allocate by themselves)
    _pair(cached)
    cached.set_variant(-1, -1)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        dr.dyn_radon_fwd(cached, u, recorded)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(recorded, g)


@pytest.mark.parametrize("size", [(64, 64, 9, 64, 192, 8, 4), (128, 128, 7, 128, 720, 8, 8), (96, 80, 17, 101, 360, 6, 5),
                                  (256, 256, 12, 256, 1800, 10, 8)])
@pytest.mark.parametrize("prec", [dr.F32, dr.BF16])
def test_timing_keeps_nothing_of_the_kernels_that_lost(size, prec):
    """The plan that timed the kernels holds what a plan holds that takes the choices
    from the cache, once both have run the forms that allocate on first use.
    (Sizes that no other test has timed.)"""
    held = []
    for _ in range(2):
        plan = _plan(*size, prec)
        plan.autotune()
        plan.set_variant(dr.FOLD2, dr.FOLD)
        _pair(plan)
        plan.set_variant(-1, -1)
        _pair(plan)
        held.append(plan.device_bytes())
    assert held[0] == held[1]


@pytest.mark.parametrize("size,most", [((256, 256, 16, 256, 360, 4, 8), 6), ((256, 256, 16, 256, 360, 4, 16), 7)])
def test_tuned_angles_per_stage_are_what_a_stage_holds(size, most):
    """26 KB of windows: six angles of two slices with m = 8 (2 KB each), seven with
    m = 16 (3.5 KB).  A caller's own choice is kept as it is given."""
    plan = _plan(*size)
    plan.autotune()
    assert 6 <= plan.info()["fold_adj_angles"] <= most
    plan.set_fold_adj_stage(12)
    assert plan.info()["fold_adj_angles"] == 12


def test_slab_solve_leaves_partial_sums_where_they_are():
    """A slab-streamed solve that tunes its plan neither frees nor replaces the buffer
    of partial sums that an earlier forward, perhaps recorded into a graph, wrote to."""
    nz, K, n = 8, 192, 64
    plan = _plan(n, n, nz, n, K, 8, 4)
    plan.set_fold_march(3)
    plan.set_variant(dr.FOLD2, dr.FOLD)
    _pair(plan)
    held = plan.device_bytes()
    plan.set_variant(-1, -1)
    g = synth.random_g(synth.rng_for(4972), nz, K, n).astype(np.float32)
    u = np.zeros(plan.u_shape(), dtype=np.float32)
    dr.cp_solve_slabs(plan, g, u, dr.solve_params(dr.CHAMBOLLE_POCK, iters=1, lambda1=0.05, lambda2=1.0, op_norm=60.0), 3)
    assert plan.info()["tuned"] == 1
    assert plan.device_bytes() == held
