"""The 3D PML on the plane ring: several column tiles and z chunks against the
FP64 oracle (the tolerances of test_gpu_pml.py), and planes crowded with
injection entries (found by bisection) against the same receivers a few at a
time: the gradient is linear in the residual, so the sums agree to the rounding
of a dozen FP32 sums (relative L2 2e-6)."""
import numpy as np
import pytest

import oracle
from oracle import pml as opml
from paper_2110_03345_gb300 import binding, inputs
from _helpers import TOL_GRAD, TOL_TRACES, rel_l2, to_dev

pytestmark = pytest.mark.gpu


def setup(shape, order, nb, nt, vd):
    dx = 0.5e-3
    vp, rho = inputs.random_smooth_model(shape, dx, 3)
    if vd:   # constant over the layer and the stencil's reach
        m = nb + order // 2 + 1
        core = tuple(slice(m, n - m) for n in shape)
        full = np.full(shape, 1000.0)
        full[core] = rho[core]
        rho = full
    dt = 0.4 * dx / vp.max()
    w = inputs.ricker(0.25 * 1500.0 / dx / 4.0, dt, nt)[None, None, :]
    ctr = np.array([[(n / 2 + 0.3) * dx for n in shape]])[None]
    return dx, dt, vp, (rho if vd else None), w, ctr


def run(shape, dx, dt, nt, order, nb, vp, rho, src, rec, w, obs):
    plan = binding.Plan(shape, dx, nt, dt, order=order, sponge=nb, c_ref=1500.0)
    plan.set_options(boundary=binding.BOUNDARY_PML)
    J, g, d = plan.gradient(to_dev(vp), to_dev(rho) if rho is not None else None, binding.Geometry(src, rec),
                            to_dev(w), to_dev(obs), traces=True)
    out = J, g.cpu().numpy().astype(np.float64), d.cpu().numpy().astype(np.float64)
    plan.close()
    return out


@pytest.mark.parametrize("shape,order,vd", [((33, 26, 131), 10, True), ((70, 33, 65), 8, False),
                                            ((27, 41, 64), 8, True)])
def test_several_tiles_against_the_oracle(shape, order, vd):
    nb, nt = 5, 80
    dx, dt, vp, rho, w, src = setup(shape, order, nb, nt, vd)
    rec = np.concatenate([inputs.random_points(6, shape, dx, 4, margin=nb + 2),
                          inputs.random_points(6, shape, dx, 5, margin=1)])
    g = oracle.Grid(shape, dx, dt=dt, nt=nt, order=order, nb=nb, c_ref=1500.0)
    obs = opml.forward(g, vp * 1.03, src[0], w[0], rec, rho=rho)[None]
    J_ref, g_ref, d_ref = opml.gradient(g, vp, src[0], w[0], rec, obs[0], rho=rho)
    J, gg, d = run(shape, dx, dt, nt, order, nb, vp, rho, src, rec, w, obs)
    assert rel_l2(d[0], d_ref) <= TOL_TRACES and abs(J - J_ref) <= 1e-3 * abs(J_ref)
    assert rel_l2(gg, g_ref) <= TOL_GRAD


def test_crowded_planes():
    shape, order, nb, nt = (40, 44, 70), 10, 6, 90
    dx, dt, vp, rho, w, src = setup(shape, order, nb, nt, True)
    # twelve receivers in one plane of one tile (48 entries in each of two planes)
    rec = np.array([[20.4, 16.0 + 0.5 * i, 8.0 + 3.3 * i] for i in range(12)]) * dx
    obs = np.random.default_rng(0).standard_normal((1, 12, nt)) * 1e-4
    args = (shape, dx, dt, nt, order, nb, vp, rho, src)
    J, g, _ = run(*args, rec, w, obs)
    Js, gs = 0.0, np.zeros(shape)
    for i in range(0, 12, 2):
        Ji, gi, _ = run(*args, rec[i:i + 2], w, obs[:, i:i + 2])
        Js, gs = Js + Ji, gs + gi
    assert abs(J - Js) <= 1e-12 * Js and rel_l2(g, gs) < 2e-6
