"""The time step against the plain maximum of |u| + |v| + a over the points, to the last bit: a
patch whose points all have the state that attains the maximum has the same time step."""
import numpy as np
import pytest
import torch

from paper_2506_16076_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _boxes(sizes, gamma):
    fs = (1.4, 1.0, 0.3, 1.0)
    ps = [W.PatchDesc(W.AFFINE, n1, n2, (2.0 * k, 2.0 * k + 1.0, 0.0, 1.0), (W.DIRICHLET,) * 4, bc=(fs,) * 4)
          for k, (n1, n2) in enumerate(sizes)]
    return W.Workload("boxes", ps, W.Params(c_policy=0, gamma=gamma), fs, "freestream", 1)


def _speed(e, gamma):
    """|u| + |v| + a, every operation rounded on its own."""
    u, v = e[1] / e[0], e[2] / e[0]
    ke = (0.5 * e[0]) * (u * u + v * v)
    return (u.abs() + v.abs()) + torch.sqrt((gamma * ((gamma - 1.0) * (e[3] - ke))) / e[0])


def _attaining(e, gamma, off):
    """Every point replaced by the state of its patch's largest speed."""
    out = e.clone()
    for a, b in zip(off, off[1:]):
        k = int(torch.argmax(_speed(e[:, a:b], gamma)))
        out[:, a:b] = e[:, a + k:a + k + 1]
    return out


def _state(rng, P, gamma, spread, speed):
    """Densities over two octaves, temperatures within `spread` of each other, velocities up to `speed`."""
    rho = np.exp2(rng.uniform(-1.0, 1.0, P))
    p = rho * (1.0 + spread * rng.uniform(-1.0, 1.0, P))
    u, v = speed * rng.uniform(-1.0, 1.0, (2, P))
    e = np.stack([rho, rho * u, rho * v, p / (gamma - 1.0) + 0.5 * rho * (u * u + v * v)])
    return torch.from_numpy(e).cuda()


def _check(gpu_lib, sizes, gamma, states):
    w = _boxes(sizes, gamma)
    ctx = gpu_lib.Context(w)
    P = w.total_points
    mu = torch.zeros(P, dtype=torch.float64, device="cuda")
    got, ref = (torch.zeros(len(states), dtype=torch.float64, device="cuda") for _ in range(2))
    for k, e in enumerate(states):
        ctx.timestep(e, mu, got[k:k + 1])
        ctx.timestep(_attaining(e, gamma, w.offsets), mu, ref[k:k + 1])
    assert torch.equal(got, ref), (got / ref - 1.0).abs().max()
    return ctx, mu


@pytest.mark.parametrize("gamma", [1.001, 1.002, 1.0200359, 1.033, 1.4, 5.0 / 3.0])
def test_time_step_is_that_of_the_largest_speed(gpu_lib, gamma):
    rng = np.random.default_rng(11)
    # one patch of whole blocks of 1024 points, then three whose boundaries lie inside blocks
    for sizes in ([(64, 48)], [(37, 29), (64, 64), (45, 23)]):
        P = sum(a * b for a, b in sizes)
        states = [_state(rng, P, gamma, s, v) for s in (1e-6, 1e-5, 1e-2) for v in (0.0, 0.3, 4.0) for _ in range(10)]
        ctx, mu = _check(gpu_lib, sizes, gamma, states)
    e = states[0].clone()
    e[3, 37 * 29 + 5] = float("nan")
    dt = torch.zeros(1, dtype=torch.float64, device="cuda")
    ctx.timestep(e, mu, dt)
    assert bool(torch.isnan(dt).all())


@pytest.mark.parametrize("k", [60, 80, 100, -60, -100])
def test_time_step_of_scaled_states(gpu_lib, k):
    """Densities times 2^k and pressures times 2^-k (speeds times 2^-k): values that FP32 holds,
    with squares of the sound speed that it does not."""
    rng = np.random.default_rng(12)
    scale = torch.tensor([2.0**k, 1.0, 1.0, 2.0**-k], dtype=torch.float64, device="cuda")[:, None]
    _check(gpu_lib, [(64, 48)], 1.4, [_state(rng, 64 * 48, 1.4, 0.5, 0.3) * scale for _ in range(20)])
