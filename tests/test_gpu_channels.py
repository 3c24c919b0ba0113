"""Channel-lane folded forward (lanes of a warp are slices x coefficients)
against the FP64 oracle, at the edges of its range: one, two and four channels
per lane, padded rows (m not a multiple of 4), partly filled blocks of slices,
detectors wider and narrower than the image, few distinct angles, lines cut
into chunks.  The kernel is forced on the plan's automatic choice, which would
otherwise depend on timing.  Tolerances are those of the other folded forwards:
1e-5 for FP32 (relative L2 and largest element), 1e-3 for BF16 storage against
the oracle's output rounded the same way."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_1809_09725_gb300 import dynrecon as dr
from paper_1809_09725_gb300 import synth

from _common import assert_close, dev_tensor, host_values, rel, to_bf16_f64

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# nx, ny, nz, ns, K, half-turns, m
CASES = [(64, 64, 8, 64, 192, 8, 4), (40, 56, 5, 70, 160, 8, 8), (33, 200, 7, 210, 240, 8, 24),
         (61, 47, 33, 64, 200, 8, 5), (128, 96, 3, 100, 720, 8, 16), (96, 96, 16, 96, 360, 6, 8),
         (24, 24, 2, 24, 240, 120, 32), (17, 23, 9, 31, 40, 8, 7)]


def _plan(case, prec, nt=3):
    nx, ny, nz, ns, K, ht, m = case
    theta, t = synth.scan(K, ht)
    plan = dr.Plan(nx, ny, nz, ns, theta, t, dr.LEGENDRE, m, nt, prec)
    return plan, oracle.Problem(nx, ny, nz, ns, theta, t, oracle.LEGENDRE, m, nt)


def _force(plan, admm=0):
    lib = dr.load()
    lib.dr_internal_use_channels.argtypes = [ctypes.c_void_p, ctypes.c_int]
    lib.dr_internal_use_channels.restype = ctypes.c_int
    assert lib.dr_internal_use_channels(plan.handle, admm) == dr.DR_OK


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("prec", [dr.F32, dr.BF16])
def test_channel_forward_matches_oracle(case, prec):
    plan, P = _plan(case, prec)
    _force(plan)
    rng = synth.rng_for(4700 + case[0])
    u = synth.random_u(rng, case[2], case[1], case[0], case[6])
    u = u.astype(np.float32).astype(np.float64) if prec == dr.F32 else to_bf16_f64(u)
    ud = dev_tensor(u, prec)
    outs = []
    for _ in range(2):
        g = torch.full(plan.g_shape(), float("nan"), dtype=ud.dtype, device="cuda")
        dr.dyn_radon_fwd(plan, ud, g)
        plan.sync()
        outs.append(host_values(g))
    np.testing.assert_array_equal(outs[1], outs[0])
    ref = P.fwd(u)
    if prec == dr.F32:
        assert_close(outs[0], ref, 1e-5)
    else:
        assert_close(outs[0], to_bf16_f64(ref), 1e-3)


def test_channel_forward_inside_solver():
    """Chambolle-Pock's data-fidelity step on the channel table, against the
    oracle's iterates (five FP32 iterations; each adds a few roundings of 6e-8)
    and replayed bit for bit."""
    case = (40, 56, 5, 70, 160, 8, 8)
    g = synth.random_g(synth.rng_for(4790), case[2], case[4], case[3])
    us = []
    for _ in range(2):
        plan, P = _plan(case, dr.F32)
        _force(plan)
        u = torch.zeros(plan.u_shape(), dtype=torch.float32, device="cuda")
        L = P.power_norm(1.0)
        dr.admm_solve(plan, dev_tensor(g, dr.F32), u,
                      dr.solve_params(dr.CHAMBOLLE_POCK, iters=5, lambda1=0.05, lambda2=1.0, op_norm=L))
        us.append(host_values(u))
    np.testing.assert_array_equal(us[0], us[1])
    uo, _ = P.chambolle_pock(g, np.zeros(us[0].shape), 5, 0.05, 1.0, L=L)
    assert rel(us[0], uo) <= 1e-5


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("nsplit", [1, 3])
def test_admm_on_channels_is_the_two_kernel_fold_bitwise(case, nsplit):
    """In the order of the thread-per-ray kernels the channel kernel gives their
    values bit for bit: residuals, CG products and the objective of a solve."""
    if case[6] > 4 and min(case[:2]) < 8 * nsplit:
        pytest.skip("fewer lines than chunks are worth")
    g = dev_tensor(synth.random_g(synth.rng_for(4795), case[2], case[4], case[3]), dr.F32)
    res = []
    for channels in (True, False):
        plan, _ = _plan(case, dr.F32)
        plan.set_fold_march(nsplit)
        if channels:
            _force(plan, admm=1)
        else:
            plan.set_variant(dr.FOLD2, dr.FOLD)
        u = torch.zeros(plan.u_shape(), dtype=torch.float32, device="cuda")
        r = dr.admm_solve(plan, g, u, dr.solve_params(dr.ADMM_CG, iters=2, n_cg=2, lambda1=0.05, lambda2=1.0, rho=0.5))
        res.append((host_values(u), r["objective"]))
    np.testing.assert_array_equal(res[0][0], res[1][0])
    np.testing.assert_array_equal(res[0][1], res[1][1])


def test_captured_call_without_scratch():
    """A call recorded into a graph before any scratch exists runs on the kernels
    that need none; a later call allocates it."""
    case = (40, 56, 5, 70, 160, 8, 8)
    plan, P = _plan(case, dr.F32)
    _force(plan)
    u = synth.random_u(synth.rng_for(4791), case[2], case[1], case[0], case[6]).astype(np.float32)
    ud = torch.from_numpy(u).cuda()
    g = torch.zeros(plan.g_shape(), dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        dr.dyn_radon_fwd(plan, ud, g)
    graph.replay()
    torch.cuda.synchronize()
    ref = P.fwd(u.astype(np.float64))
    assert_close(host_values(g), ref, 1e-5)
    dr.dyn_radon_fwd(plan, ud, g)
    plan.sync()
    assert_close(host_values(g), ref, 1e-5)


def test_recorded_forward_outlives_a_solve():
    """The partial sums of a forward recorded into a graph stay where they are when
    a solve on the same plan needs more of them (padded rows in more chunks)."""
    case = (128, 128, 5, 128, 360, 6, 8)
    plan, P = _plan(case, dr.F32)
    plan.set_fold_march(8)  # (the operator call's own chunks are four at most)
    _force(plan, admm=1)
    _force(plan)
    u = synth.random_u(synth.rng_for(4797), case[2], case[1], case[0], case[6]).astype(np.float32)
    ud = torch.from_numpy(u).cuda()
    g, gr = (torch.zeros(plan.g_shape(), dtype=torch.float32, device="cuda") for _ in range(2))
    dr.dyn_radon_fwd(plan, ud, g)
    plan.sync()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        dr.dyn_radon_fwd(plan, ud, gr)
    dr.dyn_radon_adj(plan, g, torch.empty(plan.u_shape(), dtype=torch.float32, device="cuda"))  # (its folded data)
    held = plan.device_bytes()
    x = torch.zeros(plan.u_shape(), dtype=torch.float32, device="cuda")
    dr.admm_solve(plan, g, x, dr.solve_params(dr.ADMM_CG, iters=1, n_cg=1, lambda1=0.05, lambda2=1.0, rho=0.5))
    assert plan.device_bytes() == held + plan.workspace_bytes(dr.ADMM_CG)
    gr.zero_()
    graph.replay()
    torch.cuda.synchronize()
    np.testing.assert_array_equal(host_values(gr), host_values(g))
    assert_close(host_values(g), P.fwd(u.astype(np.float64)), 1e-5)
