"""Long lines whose contraction would leave half of a wave empty run on the FFT kernels. The choice
looks at the whole workload, so every schedule and every rank of a sharded run makes the same one."""
import numpy as np
import pytest
import torch

from paper_2506_16076_gb300 import shard, workloads as W
from tests.gpu_helpers import to_dev

pytestmark = pytest.mark.gpu

N1, N2 = 997, 313  # continued lengths 1024 and 340


def _boxes(k):
    fs = (1.4, 1.0, 0.3, 1.0)
    ps = [W.PatchDesc(W.AFFINE, N1, N2, (2.0 * i, 2.0 * i + 1.0, 0.0, 0.7), (W.DIRICHLET,) * 4, bc=(fs,) * 4) for i in range(k)]
    return W.Workload(f"boxes{k}", ps, W.Params(c_policy=0), fs, "freestream", 1)


def _step(gpu_lib, ctx, e0, flags):
    e = e0.clone()
    dt = torch.full((1,), 1e-5, dtype=torch.float64, device="cuda")
    mu = torch.full((e.shape[1],), 1e-4, dtype=torch.float64, device="cuda")
    ctx.rk_step(e, dt, mu, flags | gpu_lib.STEP_FILTER | gpu_lib.STEP_FROZEN_MU | gpu_lib.STEP_FIXED_DT)
    torch.cuda.synchronize()
    return e


def test_schedules_and_ranks_agree_on_long_lines(gpu_lib):
    w = _boxes(2)  # 626 lines of L = 1024: 158 tiles
    e0 = to_dev(W.random_smooth_state(w, seed=9, amp=0.1))
    P = N1 * N2
    both = _step(gpu_lib, gpu_lib.Context(w), e0, 0)
    assert torch.equal(_step(gpu_lib, gpu_lib.Context(w), e0, gpu_lib.STEP_PER_PATCH), both)
    # rank 0 of two, with one box (nothing to exchange between the two)
    ctx = gpu_lib.Context(w)
    hub = shard.LocalHub(1)
    ctx.shard(2, 0, [0, 1], shard.LocalComm(hub, 0))
    assert torch.equal(_step(gpu_lib, ctx, e0, 0)[:, :P], both[:, :P])
    # one box alone: 313 lines, contracted. Equal up to the rounding of FP64 transforms of such lines
    # (5e-11 of an operator's largest value, which counts dt = 1e-5, and 3e-15 of the filter's)
    one = _step(gpu_lib, gpu_lib.Context(_boxes(1)), e0[:, :P].contiguous(), 0)
    assert not torch.equal(one, both[:, :P])
    assert float((one - both[:, :P]).abs().max()) < 1e-11 * float(both.abs().max())
