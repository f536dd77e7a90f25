"""The tensor-core contraction of FC lines on the GPU at the sizes where it can go wrong:
inner lengths around the padding to 16 and around the CTA sizes (128 / 129, 256 / 258), the
longest contracted lengths and the first ones left to the transforms, odd lengths, tiles
with absent lines; lines of zeros and non-finite values.

Tolerance of the operator as in the other edge cases: 1e-11, or twice the error of an FP64
FFT evaluation where that is larger."""
import dataclasses

import numpy as np
import pytest
import torch

from oracle import solver as S
from paper_2506_16076_gb300 import workloads as W
from tests.gpu_helpers import fp64_floor, from_dev, rel_err, smooth_mu, to_dev, to_dev_scalar_field, ulp_floor

pytestmark = pytest.mark.gpu


def _box(n1, n2):
    fs = (1.4, 1.0, 0.3, 1.0)
    p = W.PatchDesc(W.AFFINE, n1, n2, (0.0, 1.0, 0.0, 0.7), (W.DIRICHLET,) * 4, bc=(fs,) * 4)
    return W.Workload(f"box_{n1}x{n2}", [p], W.Params(c_policy=0), fs, "freestream", 1)


# n + 27: 64, 66, 128, 256 / 258 (inner 128 / 129), 512 / 516 (256 / 258), odd 255, 259 and 513, 1024 and
# 1026 (transforms)
CASES = [(37, 39), (101, 10), (229, 231), (485, 13), (489, 11), (228, 14), (232, 17), (486, 10), (997, 12), (999, 10)]


@pytest.mark.parametrize("n1,n2", CASES)
def test_rhs_and_filter_at_the_length_edges(gpu_lib, n1, n2):
    w = _box(n1, n2)
    ctx = gpu_lib.Context(w)
    sv = S.Solver(w)
    st = W.random_smooth_state(w, seed=n1 + n2, amp=0.2)
    mu = smooth_mu(w, seed=2, scale=0.01)
    mu[0][:, : n1 // 2] = 0.0  # inviscid and viscous column tiles
    e = to_dev(st)
    out = torch.empty_like(e)
    ctx.rhs(e, out, to_dev_scalar_field(mu))
    ref = sv.rhs(st, mu)
    tol = max(1e-11, 2 * max(rel_err(fp64_floor(sv, lambda: sv.rhs(st, mu)), ref)))
    errs = rel_err(from_dev(out, w), ref)
    assert max(errs) < tol, (errs, tol)
    ctx.filter(e)
    ref = sv.filter(st)
    tol = max(1e-11, 2 * max(rel_err(fp64_floor(sv, lambda: sv.filter(st)), ref)))
    errs = rel_err(from_dev(e, w), ref)
    assert max(errs) < tol, (errs, tol)


@pytest.mark.parametrize("alpha,p", [(2000.0, 2), (-5.0, 2), (10.0, 0)])
def test_filters_of_any_width(gpu_lib, alpha, p):
    """Continued lengths 512 and 255; sigma from 1 over few modes to e^5, and e^-10 throughout. A
    filter of few modes takes up the rounding of the end values that the continuation weighs by
    thousands, so the bound includes twice the effect of one rounding of the input (ulp_floor)."""
    w = _box(485, 228)
    w = dataclasses.replace(w, params=dataclasses.replace(w.params, alpha_f=alpha, p_f=p))
    ctx = gpu_lib.Context(w)
    sv = S.Solver(w)
    st = W.random_smooth_state(w, seed=9, amp=0.2)
    e = to_dev(st)
    ctx.filter(e)
    ref = sv.filter(st)
    tol = max([1e-11] + [2 * x for x in rel_err(fp64_floor(sv, lambda: sv.filter(st)), ref) + ulp_floor(sv.filter, st)])
    errs = rel_err(from_dev(e, w), ref)
    assert max(errs) < tol, (errs, tol)


def test_odd_filter_power_runs_as_transforms(gpu_lib):
    """With an odd p, sigma(2k/L) differs for k and -k: such a filter is a multiplier of the packed
    transforms of (rho, rho u) and (rho v, theta), as on the lines that are too long for contractions."""
    from oracle import euler, fc
    w = _box(101, 37)
    prm = w.params = dataclasses.replace(w.params, alpha_f=0.5, p_f=1)
    st = W.random_smooth_state(w, seed=9, amp=0.2)[0]

    def lines(f):
        n = f.shape[-1]
        c = fc.extend_ld(f, prm.d, fc.choose_C(n, prm.C0, prm.c_policy, prm.d))
        L = c.shape[-1]
        s = np.exp(-prm.alpha_f * (2.0 * np.fft.fftfreq(L, 1.0 / L).round() / L) ** prm.p_f)
        if L % 2 == 0:
            s[L // 2] = np.exp(-prm.alpha_f)
        z = np.fft.ifft(s * np.fft.fft(c[0::2] + 1j * c[1::2], axis=-1), axis=-1)[..., :n]
        return np.stack([z[0].real, z[0].imag, z[1].real, z[1].imag])

    q = lines(np.stack([st[0], st[1], st[2], euler.temperature(st, prm.gamma)]))
    q = np.swapaxes(lines(np.ascontiguousarray(np.swapaxes(q, 1, 2))), 1, 2)
    ref = np.stack([q[0], q[1], q[2], euler.energy_from_theta(*q, prm.gamma)])
    e = to_dev([st])
    gpu_lib.Context(w).filter(e)
    errs = rel_err(from_dev(e, w), [ref])
    assert max(errs) < 1e-11, errs


def test_uniform_gas_at_rest_stays_exactly_at_rest(gpu_lib):
    # u = v = 0: the momentum lines are zero, their derivatives exactly zero
    w = _box(101, 37)
    st = [W.prim_to_cons(np.full((37, 101), 1.4), np.zeros((37, 101)), np.zeros((37, 101)), np.full((37, 101), 1.0))]
    e = to_dev(st)
    ctx = gpu_lib.Context(w)
    ctx.filter(e)
    assert torch.equal(e[1:3], torch.zeros_like(e[1:3]))
    out = torch.empty_like(e)
    ctx.rhs(e, out, torch.zeros(e.shape[1], dtype=torch.float64, device="cuda"))
    assert torch.equal(out[0], torch.zeros_like(out[0])) and torch.equal(out[3], torch.zeros_like(out[3]))


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_non_finite_point_spoils_its_lines_only(gpu_lib, bad):
    w = _box(101, 39)
    n1, n2 = 101, 39
    st = W.random_smooth_state(w, seed=4, amp=0.2)
    mu = torch.zeros(n1 * n2, dtype=torch.float64, device="cuda")
    ctx = gpu_lib.Context(w)
    e = to_dev(st)
    good, out = torch.empty_like(e), torch.empty_like(e)
    ctx.rhs(e, good, mu)
    j, i = 20, 33
    e[3, j * n1 + i] = bad
    ctx.rhs(e, out, mu)
    fin = torch.isfinite(out).reshape(4, n2, n1)
    # packed pairs (0, 1) and (2, 3): the x flux has p in both, the y flux in the second only
    assert not fin[:, j, :].any() and not fin[2:, :, i].any()
    keep = torch.ones(n2, n1, dtype=torch.bool, device="cuda")
    keep[j, :] = False
    keep[:, i] = False
    assert torch.equal(out.reshape(4, n2, n1)[:, keep], good.reshape(4, n2, n1)[:, keep])


@pytest.mark.parametrize("wall_form", [0, 1])
def test_curvilinear_patch_after_affine_ones(gpu_lib, wall_form):
    # the scratch of a curvilinear patch starts at another index than its points; 126 radial
    # lines leave a tile with absent lines
    w = W.small_multipatch(W.ADIABATIC)
    og = dataclasses.replace(w.patches[0], n1=126)
    w = dataclasses.replace(w, patches=w.patches[1:] + [og], params=dataclasses.replace(w.params, wall_form=wall_form))
    ctx = gpu_lib.Context(w)
    sv = S.Solver(w)
    st = W.random_smooth_state(w, seed=6, amp=0.2)
    mu = smooth_mu(w, seed=2, scale=0.01)
    e = to_dev(st)
    out = torch.empty_like(e)
    ctx.rhs(e, out, to_dev_scalar_field(mu))
    errs = rel_err(from_dev(out, w), sv.rhs(st, mu))
    assert max(errs) < 1e-11, errs


@pytest.mark.parametrize("k", [-400, 400])
def test_viscosity_of_a_scaled_state_has_the_same_bits(gpu_lib, k):
    """Quotients from a shared reciprocal (exponents in the middle of the range) against
    divisions (the state times 2^400 or 2^-400): velocity, Mach number and sound speed do not
    depend on the scale, so neither do the classes and the viscosity, to the last bit."""
    w = _box(301, 203)
    ctx = gpu_lib.Context(w)
    g = np.random.default_rng(7)
    st = W.random_smooth_state(w, seed=5, amp=0.2)
    st[0] = np.array(st[0])
    st[0][:, :, 100:] *= 1.0 + 1e-3 * g.standard_normal(st[0][:, :, 100:].shape)  # all significands
    st[0][2][:, :200] = 0.0  # no velocity across
    e = to_dev(st)
    mu, mu_s = torch.empty_like(e[0]), torch.empty_like(e[0])
    tau, tau_s = (torch.empty(e.shape[1], dtype=torch.int32, device="cuda") for _ in range(2))
    ctx.viscosity(e, mu, tau)
    ctx.viscosity(e * 2.0**k, mu_s, tau_s)
    assert int(tau.min()) < int(tau.max()) and float(mu.max()) > 0.0
    assert torch.equal(tau, tau_s) and torch.equal(mu, mu_s)


def test_pass_products_count_the_contracted_lines(gpu_lib):
    # L = 128 = 2 x 64 along both directions: 21 digit pairs, 2 parts of 64 x 64 and 16 columns of 27
    # continuation points, 4 components
    per_line = 2 * 21 * 4 * (2 * 64 * 64 + 16 * 27)
    ctx = gpu_lib.Context(_box(101, 101))
    assert ctx.pass_products("cart_q2") == (2 * 101 * per_line, 0)
    assert ctx.pass_products("filter_q1") == (101 * per_line, 0)
    # 2025 + 27 points: transforms
    ctx = gpu_lib.Context(_box(2025, 101))
    assert ctx.pass_products("cart_q1") == (0.0, 101) and ctx.pass_products("cart_q2") == (2 * 2025 * per_line, 0)
