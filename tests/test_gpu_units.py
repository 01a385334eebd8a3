"""Every solver in units far from one: conductivity, capacity and source times a factor, so that the
temperatures, the objective and the gradient stay and the adjoint states go with its inverse.  The
factors leave FP32 (and its subnormals) wherever a power of the operator or of its inverse is formed."""
from __future__ import annotations

import numpy as np
import pytest

import workloads as W
from oracle import Operator as OracleOp
from oracle import coarse_states_from_sequential, oneshot_pass as o_oneshot
from oracle.fem import Material
from paper_2411_19030_gb300 import PassBuffers, oneshot_pass
from tests.gpu_helpers import FP64_TOL, assert_close, dev, ensure_built, gpu_operator, host
from tests.problems import make_problem

pytestmark = pytest.mark.gpu

FORMS = {"jacobi": dict(twolevel="none"), "additive": dict(twolevel="additive"), "vcycle": dict(twolevel="vcycle"),
         "vcycle-global": dict(twolevel="vcycle", smooth_steps=1), "threelevel": {},
         "slab-local": dict(local_steps=2), "grid": dict(grid_wide=2), "streamed": dict(coarse_stream=2, fine_stream=2),
         "streamed-jacobi": dict(coarse_stream=1, fine_stream=2, local_steps=1)}


@pytest.fixture(scope="module")
def case():
    ensure_built()
    nx, ny, Nt = 40, 32, 24
    prob = make_problem(nx, ny, Nt=Nt, Ntau=4, dt=1 / 64, material="table1", sink="left_wide")
    rho = W.rho_uniform(nx, ny, 3, 0.1, 0.9)
    U, V, _ = coarse_states_from_sequential(OracleOp(prob, W.rho_warm_perturb(rho, seed=3, amp=0.05)))
    return rho, U, V, o_oneshot(OracleOp(prob, rho), U, V)


@pytest.mark.parametrize("scale", [1e-30, 1e-8, 1e8, 1e30])
@pytest.mark.parametrize("precision", ["fp64", "fp32_refine", "fp32_refine_all"])
@pytest.mark.parametrize("form", FORMS)
def test_solvers_do_not_depend_on_the_units(case, form, precision, scale):
    rho, U, V, ref = case
    nx, ny = 40, 32
    m = W.MATERIALS["table1"]
    mat = Material(**{k: v * scale if k in ("k0", "kmin", "c0", "cmin") else v for k, v in m.items()})
    prob = make_problem(nx, ny, Nt=24, Ntau=4, dt=1 / 64, material=mat, sink="left_wide",
                        q_elem=np.full(nx * ny, scale))
    op = gpu_operator(prob, precision, rtol=1e-12, **FORMS[form])
    buf = PassBuffers(op)
    for t, a in ((buf.U_T, U[0]), (buf.U_th, U[1]), (buf.V_l, V[0] / scale), (buf.V_g, V[1])):
        t.copy_(dev(a))
    op.assemble(dev(rho))
    Theta, grad = oneshot_pass(op, buf)
    assert op.stats()["status"] == 0, op.stats()
    # rtol 1e-12 in every solve, a few steps: FP64_TOL holds in every precision
    assert_close("T_hist", host(buf.T_hist), ref["T_hist"], FP64_TOL)
    assert_close("V_l", host(buf.V_l_new) * scale, ref["V"][0], FP64_TOL)
    assert_close("grad", host(grad), ref["grad"], FP64_TOL)
