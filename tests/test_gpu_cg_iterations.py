"""The CG on chip, one reduction per iteration, takes as many iterations as the textbook arrangement with a
dot product of its own for (p, A p), also where K outweighs C/dt by far: near-binary designs, long steps
and starts that leave one slow and one fast mode."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import Operator as OracleOp
from oracle.fem import Material
from paper_2411_19030_gb300 import PTG_SLICES_CHAINED
from tests.gpu_helpers import dev, ensure_built, gpu_operator, host
from tests.problems import make_problem

pytestmark = pytest.mark.gpu

N = 16


def _iterations(A, b, x, real, inner_rtol, rtol):
    """Jacobi CG inside an FP64 residual loop as the library has it: A, r, p, q and d in `real`, z in
    FP32, each CG down to inner_rtol or to half of what is left to the tolerance."""
    Ar, minv = A.astype(real), (1.0 / A.diagonal()).astype(np.float32)
    total = 0
    for sweep in range(9):
        r64 = b - A @ x
        nr, goal = np.linalg.norm(r64), rtol * np.linalg.norm(b)
        if nr <= goal or sweep == 8:
            break
        r = (r64 / nr).astype(real)
        target = max(inner_rtol, 0.5 * goal / nr) ** 2 * float(r @ r)
        d = np.zeros_like(r)
        p, q = d.copy(), d.copy()
        rz_old = None
        while float(r @ r) > target and total < 20000:
            z = (minv * r.astype(np.float32)).astype(real)
            rz = r @ z
            beta = real(0) if rz_old is None else rz / rz_old
            p, q, rz_old = z + beta * p, Ar @ z + beta * q, rz
            alpha = rz / (p @ q)
            d, r = d + alpha * p, r - alpha * q
            total += 1
        x = x + nr * d.astype(np.float64)
    return total, nr <= goal


def _checkers(n):
    iy, ix = np.divmod(np.arange((n + 1) ** 2), n + 1)
    return 1e-3 * (-1.0) ** (iy + ix)


@pytest.mark.parametrize("precision,dt,design,sink,start", [
    ("fp64", 1e2, "binary", "left", "zero"), ("fp64", 1e2, "solid", "none", "checkers"),
    ("fp64", 1e4, "binary", "left", "zero"), ("fp32_refine", 1e2, "solid", "none", "checkers"),
    ("fp32_refine", 1e4, "solid", "none", "checkers"), ("fp32_refine", 1e4, "binary", "left", "zero")])
def test_iterations_of_ill_conditioned_steps(precision, dt, design, sink, start):
    ensure_built()
    rho = np.ones(N * N) if design == "solid" else (np.random.default_rng(1).random(N * N) < 0.4) * 1.0
    mat = Material(k0=1.0, kmin=1e-6 if design == "binary" else 1e-3, pk=3.0, c0=1.0, cmin=1.0, pc=1.0)
    prob = make_problem(N, Nt=1, Ntau=1, dt=dt, material=mat, sink=sink)
    oop = OracleOp(prob, rho)
    x0 = _checkers(N) * (start == "checkers") * oop.free
    A = (oop.C / dt + oop.K).tocsr()[oop.fidx][:, oop.fidx]
    b = (oop.C @ x0 / dt + oop.f)[oop.fidx]
    # the residuals of these steps can be brought to the rounding of x and A x (K / (C / dt) units of 1e-16)
    rtol = 1e-10 if dt < 1e3 else 1e-8
    real, inner = (np.float64, 0.0) if precision == "fp64" else (np.float32, 1e-4)
    ref, converged = _iterations(A, b, x0[oop.fidx], real, inner, rtol)
    op = gpu_operator(prob, precision, rtol=rtol, cg_iters_max=20000)
    op.assemble(dev(rho))
    U, U_th = dev(np.stack([x0, 0 * x0])), dev(np.zeros(2))
    F, F_th = dev(np.zeros((1, prob.Nn))), dev(np.zeros(1))
    op.fine_propagate_slices(U, U_th, F, F_th, schedule=PTG_SLICES_CHAINED)
    st = op.stats()
    print(f"iterations {st['cg_iters']}, reference {ref}")
    if converged:                     # FP32 is at its end where K outweighs C/dt by 1e7
        assert st["status"] == 0, st
    assert np.isfinite(host(F)).all()
    # rounding moves a count by some per cent; one refinement more or less is the CG's own share of it
    assert st["cg_iters"] <= 1.3 * ref + 5
