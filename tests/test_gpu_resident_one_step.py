"""Resident launches of one time step while another stream keeps the GPU busy, so that
the tiles of a launch start at different times: a tile must not write its state back
before its neighbours have read their first halo from it.  Traces bit for bit against the
per-step kernels, the misfit to rounding of its sum, gradients to the bound of the tests
that reorder the imaging sum (relative L2 1e-6)."""
import contextlib

import numpy as np
import pytest

from paper_2110_03345_gb300 import inputs
from _helpers import gpu_forward, gpu_gradient, rel_l2

pytestmark = pytest.mark.gpu


@contextlib.contextmanager
def busy_gpu(n=400):
    """Elementwise kernels over 64 MB on another stream, some 10 ms of them in flight."""
    import torch
    x = torch.ones(1 << 24, device="cuda")
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        for _ in range(n):
            x.mul_(1.0)
    yield
    s.synchronize()


def problem(shape, nt, shots):
    return inputs.breast_problem(shape, 0.3e-3, nt, nelem=24, shots=shots, order=8, nb=10,
                                 radius=0.3 * min(shape) * 0.3e-3)


# one tile row and several, one phase and two; 513 steps end on a launch of one step (a
# launch runs 512 at most), and so do 17 steps with checkpoints every 8 or 16
@pytest.mark.parametrize("shape,shots", [((70, 140), 2), ((256, 256), 1), ((300, 400), 3), ((700, 748), 2),
                                         ((905, 1024), 1)])
@pytest.mark.parametrize("nt", [18, 514])
def test_one_step_launches_on_a_busy_gpu(shape, shots, nt):
    p = problem(shape, nt, shots=[8 * i for i in range(shots)])
    ref, per_step = gpu_forward(p, tile=6)
    for _ in range(4):
        with busy_gpu():
            got, plan = gpu_forward(p)
        # (the exchange buffer of the resident kernels is part of the workspace)
        assert plan.stats()["workspace_bytes"] > per_step.stats()["workspace_bytes"] + (1 << 20)
        assert np.array_equal(got, ref)
    # residuals: half the data, or a constant before the waves arrive (over hundreds of
    # steps the adjoint of a constant keeps few correct digits in FP32)
    obs = 0.5 * ref if nt > 18 else ref + 1e-3
    J0, g0, _, _ = gpu_gradient(p, obs, tile=6, shots_per_cta=1)
    for k in (-1, 8, 16) if nt <= 18 else (-1,):
        with busy_gpu():
            J1, g1, d1, plan = gpu_gradient(p, obs, ckpt_every=k)
        assert plan.stats()["launches"] < 2 * (nt - 1)   # (one per step and direction otherwise)
        assert np.array_equal(d1, ref)
        assert abs(J1 - J0) <= 1e-12 * J0 and rel_l2(g1, g0) < 1e-6
