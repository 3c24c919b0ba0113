"""The solvers' sums do not depend on which kernel is the fastest one for a
single call: where the channel-lane forward serves the operator calls (and, in
the order of the thread-per-ray kernels, the solvers), a Chambolle-Pock solve
gives the iterates and the objective of the fold in two kernels bit for bit, in
core and in slabs."""
import ctypes

import numpy as np
import pytest

from paper_1809_09725_gb300 import dynrecon as dr
from paper_1809_09725_gb300 import synth

from _common import dev_tensor, host_values

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# nx, ny, nz, ns, K, half-turns, m: padded rows and a partly filled block; four channels per lane
CASES = [(40, 56, 5, 70, 160, 8, 7), (96, 80, 16, 101, 360, 6, 8)]


def _plan(case, prec=dr.F32):
    nx, ny, nz, ns, K, ht, m = case
    theta, t = synth.scan(K, ht)
    return dr.Plan(nx, ny, nz, ns, theta, t, dr.LEGENDRE, m, 3, prec)


def _use_channels(plan, solvers):
    lib = dr.load()
    lib.dr_internal_use_channels.argtypes = [ctypes.c_void_p, ctypes.c_int]
    lib.dr_internal_use_channels.restype = ctypes.c_int
    assert lib.dr_internal_use_channels(plan.handle, solvers) == dr.DR_OK


def _channels_everywhere(case, prec=dr.F32):
    plan = _plan(case, prec)
    plan.set_fold_march(1)
    _use_channels(plan, 1)
    _use_channels(plan, 0)
    return plan


def _params(**kw):
    return dr.solve_params(dr.CHAMBOLLE_POCK, iters=3, lambda1=0.05, lambda2=1.0, op_norm=60.0, **kw)


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("prec", [dr.F32, dr.BF16])
def test_chambolle_pock_is_the_two_kernel_fold_bitwise(case, prec):
    g = dev_tensor(synth.random_g(synth.rng_for(4801), case[2], case[4], case[3]), prec)
    res = []
    for channels in (True, False):
        if channels:
            plan = _channels_everywhere(case, prec)
        else:
            plan = _plan(case, prec)
            plan.set_fold_march(1)
            plan.set_variant(dr.FOLD2, dr.FOLD)
        u = torch.zeros(plan.u_shape(), dtype=g.dtype, device="cuda")
        r = dr.admm_solve(plan, g, u, _params())
        res.append((host_values(u), r["objective"]))
    np.testing.assert_array_equal(res[0][0], res[1][0])
    np.testing.assert_array_equal(res[0][1], res[1][1])


@pytest.mark.parametrize("case", CASES)
def test_chambolle_pock_in_slabs_is_the_in_core_one_bitwise(case):
    g = synth.random_g(synth.rng_for(4802), case[2], case[4], case[3]).astype(np.float32)
    plan = _channels_everywhere(case)
    u = torch.zeros(plan.u_shape(), dtype=torch.float32, device="cuda")
    dr.admm_solve(plan, torch.from_numpy(g).cuda(), u, _params())
    us = np.zeros(plan.u_shape(), dtype=np.float32)
    dr.cp_solve_slabs(_channels_everywhere(case), g, us, _params(), 2)
    np.testing.assert_array_equal(us, u.cpu().numpy())


# Half as many distinct angles as projections, aligned rows: the folded
# back-projection is the faster one of the two by some 12 %, but the solvers stay
# on the direct one.  A third as many: both agree on the fold.
@pytest.mark.parametrize("ht,adj", [(14, dr.DIRECT), (21, dr.FOLD)])
@pytest.mark.parametrize("algo", [dr.ADMM_CG, dr.CHAMBOLLE_POCK])
def test_solvers_back_projection_does_not_follow_the_timer(ht, adj, algo):
    case = (128, 128, 12, 128, 720, ht, 8)
    plan = _plan(case)
    plan.autotune()
    g = dev_tensor(synth.random_g(synth.rng_for(4803), case[2], case[4], case[3]), dr.F32)
    prm = dr.solve_params(algo, iters=2, n_cg=2, lambda1=0.05, lambda2=1.0, rho=0.5, op_norm=60.0)
    res = []
    for forced in (False, True):
        if forced:
            plan.set_variant(plan.info()["fwd_variant"], adj)
        u = torch.zeros(plan.u_shape(), dtype=torch.float32, device="cuda")
        r = dr.admm_solve(plan, g, u, prm)
        res.append((host_values(u), r["objective"]))
    np.testing.assert_array_equal(res[0][0], res[1][0])
    np.testing.assert_array_equal(res[0][1], res[1][1])


def test_plan_says_which_forward_runs():
    """dyn_radon_fwd on the channel kernel is a variant of its own, and does not hide
    what the solvers run."""
    case = CASES[1]
    plan = _plan(case)
    own, solvers = plan.info()["fwd_variant"], plan.solver_variants()
    assert solvers[0] == own
    _use_channels(plan, 0)
    assert plan.info()["fwd_variant_storage"] == 3
    assert plan.info()["fwd_variant"] == own and plan.solver_variants() == solvers
    _use_channels(plan, 1)
    assert plan.info()["fwd_variant"] == dr.FOLD2 and plan.solver_variants() == (3, dr.FOLD)
    plan.set_variant(dr.DIRECT, dr.DIRECT)
    assert plan.info()["fwd_variant_storage"] == dr.DIRECT and plan.solver_variants() == (dr.DIRECT, dr.DIRECT)
