"""The measured schedule choice (fc_autotune: FFT stage orders per continued length and
warps per CTA per length class) changes rounding only: after tuning, the operator still
matches the oracle within the RHS tolerance, and the batched, per-patch and graph
schedules stay bit-identical to each other (they share the tuned plans)."""
import numpy as np
import pytest
import torch

from oracle import solver as S
from paper_2506_16076_gb300 import workloads as W
from tests.gpu_helpers import from_dev, rel_err, smooth_mu, to_dev, to_dev_scalar_field

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tuned(gpu_lib):
    w = W.small_multipatch(W.ADIABATIC)
    ctx = gpu_lib.Context(w)
    rep = ctx.autotune()
    return w, ctx, S.Solver(w), rep


def test_report(tuned):
    w, ctx, sv, rep = tuned
    assert rep["lengths"] >= 1 and rep["classes"] >= 1
    assert 0 <= rep["lengths_changed"] <= rep["lengths"] and 0 <= rep["classes_changed"] <= rep["classes"]
    assert 0.0 < rep["ms_after"] <= rep["ms_before"]


def test_rhs_parity_after_tuning(tuned):
    w, ctx, sv, rep = tuned
    st = W.random_smooth_state(w, seed=11, amp=0.2)
    mu = smooth_mu(w, seed=3, scale=0.01)
    ref = sv.rhs(st, mu)
    e = to_dev(st)
    out = torch.empty_like(e)
    ctx.rhs(e, out, to_dev_scalar_field(mu))
    torch.cuda.synchronize()
    errs = rel_err(from_dev(out, w), ref)
    assert max(errs) < 1e-11, errs


def test_schedules_agree_after_tuning(tuned, gpu_lib):
    w, ctx, sv, rep = tuned
    st = W.random_smooth_state(w, seed=31, amp=0.05)
    outs = []
    for flags in (0, gpu_lib.STEP_PER_PATCH, gpu_lib.STEP_GRAPH):
        e = to_dev(st)
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            dt = torch.zeros(1, dtype=torch.float64, device="cuda")
            mu = torch.zeros(e.shape[1], dtype=torch.float64, device="cuda")
            for n in range(2):
                ctx.rk_step(e, dt, mu, flags | (1 if n else 0))
        s.synchronize()
        outs.append(e.cpu())
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])


def test_graph_steps_across_tuning(gpu_lib):
    # a step graph captured before tuning is captured again after it: from one common
    # post-tuning state, a graph step and a plain step (both with the tuned plans) agree
    # bit for bit, whatever the tuner chose
    w = W.small_multipatch()
    ctx = gpu_lib.Context(w)
    st = W.random_smooth_state(w, seed=5, amp=0.05)
    s = torch.cuda.Stream()
    n = None
    with torch.cuda.stream(s):
        e = to_dev(st)
        n = e.shape[1]
        dt = torch.zeros(1, dtype=torch.float64, device="cuda")
        mu = torch.zeros(n, dtype=torch.float64, device="cuda")
        ctx.rk_step(e, dt, mu, gpu_lib.STEP_GRAPH | 1)
        ctx.autotune()
        outs = []
        for flags in (gpu_lib.STEP_GRAPH | 1, 1):
            ei = e.clone()
            dti = torch.zeros(1, dtype=torch.float64, device="cuda")
            mui = torch.zeros(n, dtype=torch.float64, device="cuda")
            ctx.rk_step(ei, dti, mui, flags)
            outs.append((ei, dti, mui))
    s.synchronize()
    (eg, dtg, mug), (ep, dtp, mup) = outs
    assert torch.equal(dtg.cpu(), dtp.cpu()) and torch.equal(mug.cpu(), mup.cpu())
    assert torch.equal(eg.cpu(), ep.cpu())
    assert not torch.equal(eg.cpu(), e.cpu())


def test_tuning_on_a_side_stream(gpu_lib):
    # fc_autotune called on a non-default stream orders its own copies on that stream
    w = W.small_multipatch_grid()
    ctx = gpu_lib.Context(w)
    sv = S.Solver(w)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        rep = ctx.autotune()
    s.synchronize()
    assert rep["lengths"] >= 1
    st = W.random_smooth_state(w, seed=13, amp=0.2)
    mu = smooth_mu(w, seed=3, scale=0.01)
    ref = sv.rhs(st, mu)
    e = to_dev(st)
    out = torch.empty_like(e)
    ctx.rhs(e, out, to_dev_scalar_field(mu))
    torch.cuda.synchronize()
    errs = rel_err(from_dev(out, w), ref)
    assert max(errs) < 1e-11, errs


def _box(n1, n2):
    fs = (1.4, 1.0, 0.3, 1.0)
    p = W.PatchDesc(W.AFFINE, n1, n2, (0.0, 1.0, 0.0, 0.7), (W.DIRICHLET,) * 4, bc=(fs,) * 4)
    return W.Workload(f"box_{n1}x{n2}", [p], W.Params(c_policy=0), fs, "freestream", 1)


def test_report_covers_the_launches_of_a_step(gpu_lib):
    # one continued length, contracted in both directions: one launch each, nothing to choose
    rep = gpu_lib.Context(_box(101, 101)).autotune()
    assert (rep["lengths"], rep["lengths_changed"], rep["classes"], rep["classes_changed"]) == (1, 0, 2, 0)
    assert 0.0 < rep["ms_after"] == rep["ms_before"]
    # q1 lines of 2025 + 27 = 2052 points stay on the FFT kernels, q2 lines are contracted
    rep = gpu_lib.Context(_box(2025, 101)).autotune()
    assert (rep["lengths"], rep["classes"]) == (2, 2)
