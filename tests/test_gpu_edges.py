"""Sizes at which the kernels' tilings can go wrong: the strips of four elements of the sensitivity
sums, the tiles of the filter's backward, the row rings of the streamed multigrid marches, the
fields' scale in the float-pair CG."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import workloads as W
from oracle import Operator as OracleOp
from oracle import coarse_states_from_sequential, oneshot_pass as o_oneshot, sequential_pass as o_sequential
from oracle.design import Design
from oracle.fem import Material
from oracle.stepping import sensitivity_term
from paper_2411_19030_gb300 import PassBuffers, oneshot_pass, sequential_pass
from paper_2411_19030_gb300.design import DesignMap
from tests.gpu_helpers import FP64_TOL, assert_close, dev, ensure_built, gpu_operator, host
from tests.problems import make_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


@pytest.mark.parametrize("material", ["simp_k", "table1"])
@pytest.mark.parametrize("nx,ny,Nt", [(2, 2, 1), (3, 3, 2), (5, 4, 7), (31, 5, 66), (33, 127, 3)])
def test_sensitivity_strips(nx, ny, Nt, material):
    """Rows that fill no strip, one strip and many, fewer steps than time chunks."""
    prob = make_problem(nx, ny, Nt=Nt, material=material, sink="bottom")
    rho = W.rho_uniform(nx, ny, 5, 0.1, 0.9)
    rng = np.random.default_rng(7)
    T, lam = rng.uniform(-1, 1, (Nt + 1, prob.Nn)), rng.uniform(-1, 1, (Nt, prob.Nn))
    oop = OracleOp(prob, rho)
    ref = -sum(sensitivity_term(oop, lam[j - 1], T[j], T[j - 1], prob.dt) for j in range(1, Nt + 1)) / Nt
    op = gpu_operator(prob)
    op.assemble(dev(rho))
    g = torch.zeros(prob.Ne, dtype=torch.float64, device="cuda")
    op.sensitivities(dev(lam), 1, Nt, dev(T), g)
    # sums of at most 66 terms of about 50 products of order one: 1e-16 x 66 x 50 / the largest sum
    assert_close("grad", host(g), ref, 1e-12)


@pytest.mark.parametrize("nx,ny,R", [(31, 15, 1), (32, 16, 3), (33, 17, 5), (70, 40, 27), (70, 40, 28)])
def test_filter_backward_tiles(nx, ny, R):
    """Grids around the 32 x 16 tile; the widest filter of the tile kernel and the next one."""
    h = 1.0 / max(nx, ny)
    r_fil = (R - 0.25) * h
    ref = Design(nx, ny, h, r_fil, 8.0, 0.5)
    chi, y = W.rho_uniform(nx, ny, 17, 0.0, 1.0), W.rho_uniform(nx, ny, 18, -1.0, 1.0)
    _, dp_r = ref.forward(chi)
    dm = DesignMap(nx, ny, h, r_fil, 8.0, 0.5)
    rho, dp, g, gv = (torch.empty(nx * ny, dtype=torch.float64, device="cuda") for _ in range(4))
    dm.forward(dev(chi), rho, dp)
    dm.backward(dp, dev(y), g)
    dm.backward(dp, None, gv)
    assert_close("H^T", host(g), ref.backward(dp_r, y), 1e-13)
    assert_close("volume gradient", host(gv), ref.volume_gradient(dp_r), 1e-13)


@pytest.mark.parametrize("nx,ny,precision", [(72, 24, "fp64"), (80, 72, "fp32_refine"), (124, 40, "fp64"),
                                             (132, 20, "fp32_refine"), (260, 48, "fp64"), (516, 12, "fp32_refine")])
def test_streamed_marches(nx, ny, precision):
    """Rows around the shortest that go through a ring (72: none of the levels does), rows whose
    restriction ends beyond them (124), rows that a block covers several of or a third of one; the
    streamed solves against the oracle, every slice count giving other rows per block."""
    prob = make_problem(nx, ny, Nt=8, Ntau=2, dt=1 / 64, material="table1", sink="left_wide")
    rho = W.rho_uniform(nx, ny, 11, 0.2, 0.8)
    U_old, V_old, _ = coarse_states_from_sequential(OracleOp(prob, W.rho_warm_perturb(rho, seed=3, amp=0.05)))
    ref = o_oneshot(OracleOp(prob, rho), U_old, V_old)
    op = gpu_operator(prob, precision, rtol=1e-12, coarse_stream=2, fine_stream=2)
    buf = PassBuffers(op)
    for t, a in ((buf.U_T, U_old[0]), (buf.U_th, U_old[1]), (buf.V_l, V_old[0]), (buf.V_g, V_old[1])):
        t.copy_(dev(a))
    op.assemble(dev(rho))
    Theta, grad = oneshot_pass(op, buf)
    # rtol 1e-12 in every solve, a few steps: FP64_TOL holds in both precisions
    assert_close("T_hist", host(buf.T_hist), ref["T_hist"], FP64_TOL)
    assert_close("grad", host(grad), ref["grad"], FP64_TOL)
    assert op.stats()["status"] == 0


@pytest.mark.parametrize("nx,ny,Ntau,solo", [(64, 64, 2, 0), (64, 64, 2, 257), (64, 64, 160, 0), (66, 66, 2, 0),
                                             (20, 132, 4, 0), (100, 36, 2, 9), (40, 24, 160, 2)])
def test_small_levels(nx, ny, Ntau, solo):
    """The levels that one block works on: the last three, all, a coarsest level of one warp and one of
    more than 32 groups of nodes, none (solo = 2: then the coarsest level is the group's)."""
    prob = make_problem(nx, ny, Nt=Ntau, Ntau=Ntau, dt=1 / 64, material="simp_k", sink="left_wide")
    rho = W.rho_uniform(nx, ny, 12, 0.2, 0.8)
    U_old, V_old, _ = coarse_states_from_sequential(OracleOp(prob, W.rho_warm_perturb(rho, seed=3, amp=0.05)))
    ref = o_oneshot(OracleOp(prob, rho), U_old, V_old)
    op = gpu_operator(prob, "fp32_refine", rtol=1e-12, coarse_stream=2, fine_stream=2)
    if solo:
        op.set_multigrid(solo_rows=solo)
    buf = PassBuffers(op)
    for t, a in ((buf.U_T, U_old[0]), (buf.U_th, U_old[1]), (buf.V_l, V_old[0]), (buf.V_g, V_old[1])):
        t.copy_(dev(a))
    op.assemble(dev(rho))
    Theta, grad = oneshot_pass(op, buf)
    # every step's solve leaves rtol 1e-12, in the state and again in the adjoint and the gradient
    tol = max(FP64_TOL, 5 * Ntau * 1e-12)
    assert_close("T_hist", host(buf.T_hist), ref["T_hist"], tol)
    assert_close("grad", host(grad), ref["grad"], tol)
    assert op.stats()["status"] == 0


@pytest.mark.parametrize("scale", [1e-30, 1e30])
def test_float_pair_cg_is_independent_of_the_units(scale):
    """Conductivity, capacity and source times a factor far from one: the same temperatures."""
    m = W.MATERIALS["table1"]
    mat = Material(**{k: v * scale if k in ("k0", "kmin", "c0", "cmin") else v for k, v in m.items()})
    Nt = 12
    rho = W.rho_uniform(21, 13, 3, 0.1, 0.9)
    prob = make_problem(21, 13, Nt=Nt, Ntau=3, material=mat, sink="left_wide", q_elem=np.full(21 * 13, scale))
    unit = make_problem(21, 13, Nt=Nt, Ntau=3, material="table1", sink="left_wide")
    op = gpu_operator(prob, "fp64", twolevel=False)
    buf = PassBuffers(op)
    op.assemble(dev(rho))
    Theta, _ = sequential_pass(op, buf)
    ref = o_sequential(OracleOp(unit, rho))
    assert_close("T_hist", host(buf.T_hist), ref["T_hist"], FP64_TOL)
    assert abs(float(Theta.item()) - ref["Theta"]) < FP64_TOL * ref["Theta"]
    assert op.stats()["status"] == 0
