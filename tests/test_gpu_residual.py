"""The tolerance of a solve is one of its true residual b - A x: states that a pass returns satisfy it,
also after many steps and where a solve starts far from its solution, and a tolerance that rounding
does not allow is reported."""
from __future__ import annotations

import numpy as np
import pytest

import workloads as W
from oracle import Operator as OracleOp
from paper_2411_19030_gb300 import PTG_PRIMAL, PTG_SLICES_CHAINED
from paper_2411_19030_gb300._ffi import PTG_ENOCONV
from tests.gpu_helpers import dev, ensure_built, gpu_operator, host
from tests.problems import make_problem

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53
STREAMED = dict(fine_stream=2, coarse_stream=2)
PATHS = [("fp64", dict(initial_guess=1)), ("fp64", {}), ("fp32_refine", dict(initial_guess=1)), ("fp32_refine", {}),
         ("fp32_refine_all", {}), ("fp64", STREAMED), ("fp32_refine", STREAMED), ("fp32_refine_all", STREAMED)]
IDS = [f"{p}-{'-'.join(k) or 'default'}" for p, k in PATHS]


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


def _problem(Nt, Ntau):
    """Large steps under a load that changes from step to step: K outweighs C/dt, and every start is
    far from its solution."""
    q = 1.0 + 0.9 * np.cos(1.7 * np.arange(Nt + 1))
    prob = make_problem(48, 32, Nt=Nt, Ntau=Ntau, dt=0.25, material="simp_k", sink="left_wide", q_time=q)
    return prob, W.rho_uniform(48, 32, 3, 0.2, 0.8)


def _rows(oop, dt):
    """Residual of A x = C/dt xp + q f on the unknowns over ||b||, and the rounding unit of that residual."""
    A, free = oop.C / dt + oop.K, oop.free
    absA = abs(A)

    def of(x, xp, q):
        b = oop.C @ xp / dt + q * oop.f
        nb = np.linalg.norm(b[free])
        return np.linalg.norm((b - A @ x)[free]) / nb, EPS * np.linalg.norm((absA @ np.abs(x))[free]) / nb
    return of


@pytest.mark.parametrize("precision,kw", PATHS, ids=IDS)
def test_states_satisfy_the_tolerance(precision, kw):
    Nt = 512
    prob, rho = _problem(Nt, 2)
    oop = OracleOp(prob, rho)
    fine, coarse = _rows(oop, prob.dt), _rows(oop, prob.dt * Nt / 2)
    q = prob.q_time
    U_T, U_th, F_T, F_th = dev(np.zeros((3, prob.Nn))), dev(np.zeros(3)), dev(np.zeros((2, prob.Nn))), dev(np.zeros(2))
    hist, G_T = dev(np.zeros((Nt + 1, prob.Nn))), dev(np.zeros((2, prob.Nn)))

    def operator(rows, dt):
        # attainable: the rounding of x and of A x is about a unit each
        x = oop.solve(dt, q[1] * oop.f)
        rtol = 8 * rows(x, np.zeros(prob.Nn), q[1])[1]
        op = gpu_operator(prob, precision, rtol=rtol, **kw)
        op.assemble(dev(rho))
        return op, rtol

    op, rtol = operator(fine, prob.dt)
    if kw is STREAMED:                                 # (streamed fine propagators run slices in parallel)
        op.fine_propagate_slices(U_T, U_th, F_T, F_th, hist)
    else:
        op.fine_propagate_slices(U_T, U_th, F_T, F_th, hist, schedule=PTG_SLICES_CHAINED)
    assert op.stats()["status"] == 0, op.stats()
    opc, rtol_c = operator(coarse, prob.dt * Nt / 2)
    opc.coarse_sweep(PTG_PRIMAL, U_T, U_th, G_T, F_th)
    assert opc.stats()["status"] == 0, opc.stats()
    T = host(hist)
    worst = 0.0
    for j in range(1, Nt + 1):
        xp = np.zeros(prob.Nn) if j == 1 or (kw is STREAMED and j == Nt // 2 + 1) else T[j - 1]
        r, u = fine(T[j], xp, q[j])
        # the tolerance; 8 units for this evaluation of the residual and for weights that the device assembles
        worst = max(worst, (r - 8 * u) / rtol)
    G = host(G_T)
    for s in range(2):
        r, u = coarse(G[s], np.zeros(prob.Nn), q[(s + 1) * Nt // 2])
        worst = max(worst, (r - 8 * u) / rtol_c)
    print(f"worst residual / rtol {worst:.2f}")
    assert worst <= 1.0


@pytest.mark.parametrize("precision,kw", PATHS, ids=IDS)
def test_tolerance_below_rounding(precision, kw):
    """FP64 kinds on chip report it; the others end where rounding does (the rounding of x and of A x, a
    unit each), and not before."""
    Nt = 16
    prob, rho = _problem(Nt, 2)
    oop = OracleOp(prob, rho)
    q = prob.q_time
    for coarse in (False, True):
        dt = prob.dt * (Nt // 2 if coarse else 1)
        rows = _rows(oop, dt)
        unit = rows(oop.solve(dt, q[1] * oop.f), np.zeros(prob.Nn), q[1])[1]
        op = gpu_operator(prob, precision, rtol=unit / 16, **kw)
        op.assemble(dev(rho))
        U_T, U_th, F_T, F_th = op.zeros(3, prob.Nn), op.zeros(3), op.zeros(2, prob.Nn), op.zeros(2)
        hist = op.zeros(Nt + 1, prob.Nn)
        if coarse:
            op.coarse_sweep(PTG_PRIMAL, U_T, U_th, F_T, F_th)
            pairs = [(host(F_T)[s], np.zeros(prob.Nn), q[(s + 1) * Nt // 2]) for s in range(2)]
        else:
            op.fine_propagate_slices(U_T, U_th, F_T, F_th, hist)
            T = host(hist)
            pairs = [(T[j], np.zeros(prob.Nn) if j % (Nt // 2) == 1 else T[j - 1], q[j]) for j in range(1, Nt + 1)]
        fp64 = precision == "fp64" or (coarse and precision == "fp32_refine")
        st = op.stats()
        assert st["status"] == (PTG_ENOCONV if fp64 and kw is not STREAMED else 0), st
        for x, xp, qj in pairs:
            r, u = rows(x, xp, qj)
            assert r <= (2 + 8) * u, f"residual of {r / u:.1f} units"
