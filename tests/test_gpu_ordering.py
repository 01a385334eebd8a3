"""Node rows that the CTAs of a cluster read from one another's global memory: the ring of states that
a fine step's start is extrapolated through.  Short steps at a loose tolerance take few CG iterations,
so a ring row is read soon after it was written; the FP32 kinds keep the halo rows that they
extrapolated for the rest of the slice, so a stale row would stay in the result."""
from __future__ import annotations

import numpy as np
import pytest

import workloads as W
from paper_2411_19030_gb300 import PassBuffers, sequential_pass
from tests.gpu_helpers import dev, ensure_built, gpu_operator, host
from tests.problems import make_problem

pytestmark = pytest.mark.gpu

FINE_PRI, FINE_ADJ = 0, 3


@pytest.mark.parametrize("precision", ["fp64", "fp32_refine"])
def test_ring_rows_of_neighbouring_slabs(precision):
    ensure_built()
    Nt, rtol = 256, 1e-7
    prob = make_problem(48, 62, Nt=Nt, Ntau=2, dt=1 / 4096, material="simp_k", sink="left_wide")
    rho = W.rho_uniform(48, 62, 3, 0.2, 0.8)
    runs = {}
    for cs in (16, 1):
        op = gpu_operator(prob, precision, rtol=rtol)
        op.set_plan(FINE_PRI, cs, 1 if cs > 1 else 3)
        op.set_plan(FINE_ADJ, cs, 1 if cs > 1 else 3)
        buf = PassBuffers(op)
        op.assemble(dev(rho))
        Theta, grad = sequential_pass(op, buf)
        runs[cs] = (host(buf.T_hist), host(buf.V_l), host(grad))
        assert op.stats()["status"] == 0
    # every solve leaves a residual of at most rtol ||b||, so an error of rtol cond(C) ||x|| (cond(C)
    # at most 36 for the consistent mass matrix with its boundary); the steps' errors add up, in both runs
    # and again in the adjoint, which T drives as T^7
    tol = 2 * Nt * 36 * rtol
    for name, a, b, f in zip(("T_hist", "V_l", "grad"), runs[16], runs[1], (1, 8, 9)):
        err = np.linalg.norm(a - b) / np.linalg.norm(b)
        assert err <= f * tol, f"{name}: {err:.2e}"
