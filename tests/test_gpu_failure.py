"""Failure detection on the device without faulting it: the bounded wait of a grid barrier is
made to run out (ptg_op_set_wait_limit with a limit of one poll), so the cooperative launch
records PTG_ETIMEOUT in the op's status word and every CTA stops waiting and returns.  The
error is read on the host through ptg_get_stats; after ptg_reset_stats and the default limit
the same op gives the oracle's result again.  Nothing here traps or hangs the GPU: every wait is
bounded and every loop of the stepper has an iteration limit."""
from __future__ import annotations

import pytest
import torch

import workloads as W
from oracle import Operator as OracleOp, sequential_pass as o_sequential
from oracle import coarse_states_from_sequential, oneshot_pass as o_oneshot
from paper_2411_19030_gb300 import PassBuffers, oneshot_pass, sequential_pass
from paper_2411_19030_gb300._ffi import PTG_ETIMEOUT
from paper_2411_19030_gb300.batch import Batch
from tests.gpu_helpers import FP64_TOL, assert_close, dev, ensure_built, gpu_operator, host
from tests.problems import make_problem

pytestmark = pytest.mark.gpu


def test_grid_barrier_wait_limit_reports_timeout_and_op_recovers():
    ensure_built()
    prob = make_problem(13, 9, Nt=24, Ntau=4, dt=1 / 24, material="table1", sink="left_wide",
                        q_time=W.q_time_paper(24, 1 / 24))
    rho = W.rho_uniform(13, 9, 3, 0.05, 0.95)
    seq = o_sequential(OracleOp(prob, rho))
    # small iteration limits: once the barrier is broken the reductions are meaningless and the
    # solves run to their limits, which keeps the broken launch short
    op = gpu_operator(prob, "fp64", grid_wide=2, cg_iters_max=40, refine_max=2)
    assert op.plan(0, 1)["cs"] > 1          # a cooperative grid of several CTAs per system
    buf = PassBuffers(op)
    op.assemble(dev(rho))
    op.set_wait_limit(1)
    sequential_pass(op, buf)
    torch.cuda.synchronize()
    st = op.stats()
    assert st["status"] == PTG_ETIMEOUT, st
    assert st["fail_kind"] in (10, 13), st   # recorded by a fine primal or fine adjoint launch
    # the context is intact and the op recovers with the default limit
    op.set_wait_limit(0)
    op.reset_stats()
    op2 = gpu_operator(prob, "fp64", grid_wide=2)
    for o in (op, op2):
        o.set_wait_limit(0)
    op.close()
    b2 = PassBuffers(op2)
    op2.assemble(dev(rho))
    Theta, grad = sequential_pass(op2, b2)
    torch.cuda.synchronize()
    assert_close("T_hist after recovery", host(b2.T_hist), seq["T_hist"], FP64_TOL)
    assert_close("grad after recovery", host(grad), seq["grad"], FP64_TOL)
    assert op2.stats()["status"] == 0


def test_wait_limit_rejects_negative_values():
    ensure_built()
    prob = make_problem(6, Nt=4, Ntau=2, dt=0.25)
    op = gpu_operator(prob, "fp64")
    with pytest.raises(Exception):
        op.set_wait_limit(-1)


def _problem():
    prob = make_problem(24, 18, Nt=24, Ntau=4, dt=1 / 24, material="table1", sink="left_wide",
                        q_time=W.q_time_paper(24, 1 / 24))
    return prob, W.rho_uniform(24, 18, 3, 0.05, 0.95)


@pytest.mark.parametrize("precision,twolevel", [("fp64", "threelevel"), ("fp64", "vcycle"), ("fp32_refine", "additive"),
                                                ("fp32_refine_all", "threelevel")])
def test_cluster_wait_limit_reports_timeout_and_op_recovers(precision, twolevel):
    """The exchanges of a cluster run out of their one poll: every launch of the pass ends with the error,
    and the same op gives the oracle's result with the default limit."""
    ensure_built()
    prob, rho = _problem()
    U_old, V_old, _ = coarse_states_from_sequential(OracleOp(prob, W.rho_warm_perturb(rho, seed=3, amp=0.05)))
    ref = o_oneshot(OracleOp(prob, rho), U_old, V_old)
    op = gpu_operator(prob, precision, rtol=1e-12, twolevel=twolevel)
    assert op.plan(0, 4)["cs"] > 1 and op.plan(2, 1)["cs"] > 1
    buf = PassBuffers(op)
    op.assemble(dev(rho))
    for limit in (1, 0):
        for t, a in ((buf.U_T, U_old[0]), (buf.U_th, U_old[1]), (buf.V_l, V_old[0]), (buf.V_g, V_old[1])):
            t.copy_(dev(a))
        op.set_wait_limit(limit)
        op.reset_stats()
        Theta, grad = oneshot_pass(op, buf)
        torch.cuda.synchronize()
        assert op.stats()["status"] == (PTG_ETIMEOUT if limit else 0), op.stats()
    # rtol 1e-12 in every solve, a few steps
    assert_close("T_hist after recovery", host(buf.T_hist), ref["T_hist"], FP64_TOL)
    assert_close("grad after recovery", host(grad), ref["grad"], FP64_TOL)


def test_row_ring_wait_limit_reports_timeout_and_op_recovers():
    """One CTA per slice, which waits for no other CTA: what runs out is the wait for the rows that it
    copies to shared memory."""
    ensure_built()
    prob = make_problem(80, 24, Nt=160, Ntau=160, dt=1 / 64, material="simp_k", sink="left_wide")
    rho = W.rho_uniform(80, 24, 12, 0.2, 0.8)
    op = gpu_operator(prob, "fp32_refine", rtol=1e-10, coarse_stream=2, fine_stream=2)
    assert op.plan(0, 160)["cs"] == 1
    U_T, F_T = op.zeros(161, prob.Nn), [op.zeros(160, prob.Nn) for _ in range(3)]
    U_th, F_th = op.zeros(161), op.zeros(160)
    op.assemble(dev(rho))
    for F, limit in zip(F_T, (0, 1, 0)):
        op.set_wait_limit(limit)
        op.reset_stats()
        op.fine_propagate_slices(U_T, U_th, F, F_th)
        torch.cuda.synchronize()
        st = op.stats()
        assert st["status"] == (PTG_ETIMEOUT if limit else 0), st
    assert torch.equal(F_T[0], F_T[2]) and float(F_T[0].abs().max()) > 0


def test_batch_does_not_pass_on_a_broken_cluster():
    """One design's waits run out: the designs whose tasks its clusters take afterwards report it too, the
    others have the oracle's result."""
    ensure_built()
    prob, rho = _problem()
    small = make_problem(16, Nt=24, Ntau=4, dt=1 / 24, material="simp_k", sink="left_wide")
    rho_s = W.rho_uniform(16, 16, 5, 0.05, 0.95)
    refs = [o_sequential(OracleOp(p, r)) for p, r in ((prob, rho), (small, rho_s), (small, rho_s))]
    ops = [gpu_operator(prob, "fp64")] + [gpu_operator(small, "fp64") for _ in range(2)]
    ops[0].set_wait_limit(1)
    batch = Batch(ops)
    for d, r in enumerate((rho, rho_s, rho_s)):
        batch.buffers(d)["rho"].copy_(dev(r))
    batch.assemble()
    batch.sequential_pass()
    torch.cuda.synchronize()
    status = [op.stats()["status"] for op in ops]
    assert status[0] == PTG_ETIMEOUT
    for d in (1, 2):
        assert status[d] in (0, PTG_ETIMEOUT)
        if status[d] == 0:
            b = batch.buffers(d)
            assert_close(f"T_hist[{d}]", host(b["T_hist"]), refs[d]["T_hist"], FP64_TOL)
            assert_close(f"grad[{d}]", host(b["V_g"][0]), refs[d]["grad"], FP64_TOL)
