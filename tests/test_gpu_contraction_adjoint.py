"""The transposed contractions (adjoint of a filtered step) at the sizes where their layout changes:
inner lengths 128 / 129, 256 / 258 and 512 (results at end and continuation points lie behind the
digits in shared memory), odd lengths next to them, tiles with absent lines; affine and curvilinear
patches, viscous and inviscid tiles.

Tolerance as for the operator: 1e-11, or twice the error of an FP64 FFT evaluation of the same adjoint
where that is larger."""
import numpy as np
import pytest
import torch

from oracle import adjoint as A, solver as S
from paper_2506_16076_gb300 import workloads as W
from tests.gpu_helpers import fp64_floor, from_dev, rel_err, to_dev, to_dev_scalar_field

pytestmark = pytest.mark.gpu

# n + 27: even 256 / 258, 512 / 516, 1024; odd 255, 259, 511 (and 37 to 41 across)
CASES = [(229, 14, False), (231, 11, False), (485, 13, False), (489, 11, False), (997, 12, False), (228, 10, False),
         (232, 13, False), (484, 12, False), (485, 13, True), (231, 10, True), (228, 14, True)]


@pytest.mark.parametrize("n1,n2,grid", CASES)
def test_adjoint_at_the_length_edges(gpu_lib, n1, n2, grid):
    fs = (1.4, 1.0, 0.3, 1.0)
    p = W.PatchDesc(W.AFFINE, n1, n2, (0.0, 1.0, 0.0, 0.7), (W.DIRICHLET,) * 4, bc=(fs,) * 4)
    w = W.Workload(f"box_{n1}x{n2}", [W.as_grid(p, bump=0.04) if grid else p], W.Params(c_policy=0), fs, "freestream", 1)
    sv = S.Solver(w)
    st = sv.project(W.random_smooth_state(w, seed=n1 + n2, amp=0.1))
    mu = [0.003 * (1 + np.cos(2 * g.x) * np.sin(g.y)) ** 2 for g in sv.geos]
    mu[0][:, : n1 // 2] = 0.0  # column tiles with and without viscosity
    mu[0][: n2 // 2] = 0.0  # row tiles
    dt = 0.5 * sv.dt(st, mu)
    lam = [np.random.default_rng(5).normal(size=a.shape) for a in st]

    def adjoint():
        return A.step_adjoint(sv, st, mu, dt, lam, filt=True)[0]
    ref = adjoint()
    tol = max(1e-11, 2 * max(rel_err(fp64_floor(sv, adjoint), ref)))
    ctx = gpu_lib.Context(w)
    lam_n = torch.empty_like(to_dev(st))
    dtt = torch.tensor([dt], dtype=torch.float64, device="cuda")
    ctx.adjoint_step(to_dev(st), to_dev_scalar_field(mu), dtt, to_dev(lam), lam_n, torch.zeros_like(lam_n), gpu_lib.STEP_FILTER)
    errs = rel_err(from_dev(lam_n, w), ref)
    assert max(errs) < tol, (errs, tol)
