"""An affine strip with fewer than 2d points along one direction, inside an O-grid's annulus: all
its points are receivers and it has lines along the other direction only. The operator, a filtered
step and the adjoint of one against the oracle (tolerance of the other parity tests: 1e-11)."""
import numpy as np
import pytest
import torch

from oracle import adjoint as A, solver as S
from paper_2506_16076_gb300 import workloads as W
from tests.gpu_helpers import from_dev, rel_err, to_dev, to_dev_scalar_field

pytestmark = pytest.mark.gpu

FS = (1.4, 0.6, 0.2, 1.0)


def _layout(n1, n2):
    og = W.PatchDesc(W.OGRID, 96, 40, (0.0, 0.0, 0.5, 1.5), (W.PERIODIC, W.PERIODIC, W.SLIPWALL, W.DIRICHLET), bc=(FS,) * 4)
    a, b = 0.0175 * (n1 - 1) / 2, 0.0175 * (n2 - 1) / 2
    strip = W.PatchDesc(W.AFFINE, n1, n2, (1.0 - a, 1.0 + a, -b, b), (W.INTERNAL,) * 4, bc=(FS,) * 4)
    return W.Workload(f"strip{n1}x{n2}", [og, strip], W.Params(c_policy=2), FS, "freestream", 1)


@pytest.mark.parametrize("n1,n2", [(24, 8), (8, 24), (8, 8)])
def test_strip_with_lines_along_one_direction(gpu_lib, n1, n2):
    w = _layout(n1, n2)
    sv = S.Solver(w)
    st = sv.project(W.random_smooth_state(w, seed=3, amp=0.1))
    mu = [0.003 * (1 + np.cos(2 * g.x) * np.sin(g.y)) ** 2 for g in sv.geos]
    assert min(m.min() for m in mu) > 0.0
    ctx = gpu_lib.Context(w)
    e, mud = to_dev(st), to_dev_scalar_field(mu)
    out = torch.empty_like(e)
    for m, md in ((mu, mud), ([0.0 * a for a in mu], 0.0 * mud)):
        ctx.rhs(e, out, md)
        errs = rel_err(from_dev(out, w), sv.rhs(st, m))
        assert max(errs) < 1e-11, errs
    dt = 1e-4
    dtt = torch.tensor([dt], dtype=torch.float64, device="cuda")
    lam = [np.random.default_rng(5).normal(size=a.shape) for a in st]
    lam_n, gbc = torch.empty_like(e), torch.zeros_like(e)
    ctx.adjoint_step(e, mud, dtt, to_dev(lam), lam_n, gbc, gpu_lib.STEP_FILTER)
    errs = rel_err(from_dev(lam_n, w), A.step_adjoint(sv, st, mu, dt, lam, filt=True)[0])
    assert max(errs) < 1e-11, errs
    for flags in (0, gpu_lib.STEP_PER_PATCH):
        now = e.clone()
        ctx.rk_step(now, dtt, mud.clone(), flags | gpu_lib.STEP_FROZEN_MU | gpu_lib.STEP_FIXED_DT | gpu_lib.STEP_FILTER)
        errs = rel_err(from_dev(now, w), A.step_forward(sv, st, mu, dt, filt=True)[0][5])
        assert max(errs) < 1e-11, errs
