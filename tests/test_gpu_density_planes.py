"""3D plane rings leave out the density terms on planes of a column that no density
gradient reaches.  The terms left out are zeros, so the leapfrog's forward gives the bits
of the one-point kernels, which add them, and its gradient agrees with theirs to the
rounding of 40 adjoint steps in another order (a few 6e-8 per step, adding up as their
root: 3e-6 relative L2; one plane of the smallest inclusion left out is 1e-4): densities that vary everywhere, nowhere, and only at
inclusions on, next to and across the edges of columns and z chunks, at the faces, and
along one axis only (a gradient that the adjoint's stencil alone reaches).  The PML runs
against the FP64 oracle (the tolerances of test_gpu_pml.py)."""
import numpy as np
import pytest

import oracle
from oracle import pml as opml
from paper_2110_03345_gb300 import binding, inputs
from _helpers import TOL_GRAD, TOL_TRACES, rel_l2, to_dev

pytestmark = pytest.mark.gpu

BOXES = [(slice(30, 34), slice(15, 17), slice(60, 68)), (slice(0, 3), slice(0, 2), slice(0, 5)),
         (slice(41, 45), slice(26, 30), slice(125, 131)), (slice(12, 13), slice(8, 9), slice(64, 65)),
         (slice(20, 21), slice(22, 24), slice(96, 97)), (slice(20, 22), slice(14, 16), slice(96, 99))]


def density(kind, shape):
    rho = np.full(shape, 1000.0)
    if kind == "everywhere":
        rho += 50.0 * np.random.default_rng(0).random(shape)
    elif kind in ("x", "y", "z"):
        rho[tuple(slice(25, None) if a == kind else slice(None) for a in "zyx")] = 1100.0
    elif kind.startswith("box"):
        rho[BOXES[int(kind[3:])]] = 1300.0
    return rho


@pytest.mark.parametrize("order,tile", [(8, 0), (10, 0), (10, 9), (8, 10), (10, 11)])
def test_kernels_that_add_every_term(order, tile):
    shape, nt = (45, 30, 131), 40
    p = inputs.skull_problem(shape, 0.5e-3, nt, nrec=24, every=24, order=order, nb=5, f0=250e3)
    geo = binding.Geometry(p.src_xyz, p.rec_xyz)
    vp, w = to_dev(p.vp), to_dev(p.wavelet)
    obs = to_dev(1e-3 * np.random.default_rng(1).standard_normal((p.src_xyz.shape[0], p.rec_xyz.shape[0], nt)))
    plans = []
    for t in (tile, 5):
        plan = binding.Plan(p.shape, p.spacing, nt, p.dt, order=order, sponge=p.nb, c_ref=p.c_ref)
        plan.set_options(tile=t)
        plans.append(plan)
    # (one plan for all densities: each call's flags are its own)
    for kind in ["everywhere", "constant", "x", "y", "z"] + ["box%d" % i for i in range(len(BOXES))]:
        rho = to_dev(density(kind, shape))
        out = [plan.gradient(vp, rho, geo, w, obs, traces=True) for plan in plans]
        (J0, g0, d0), (J1, g1, d1) = [(J, g.cpu().numpy(), d.cpu().numpy()) for J, g, d in out]
        assert np.array_equal(d0, d1) and J0 == J1 and rel_l2(g0, g1) < 3e-6, kind
        assert np.abs(g0).max() > 0
    for plan in plans:
        plan.close()


@pytest.mark.parametrize("kind,order", [("box0", 10), ("box3", 8), ("box5", 10)])
def test_pml_against_the_oracle(kind, order):
    shape, nb, nt, dx = (45, 30, 131), 3, 60, 0.5e-3
    vp, _ = inputs.random_smooth_model(shape, dx, 3)
    rho = density(kind, shape)
    dt = 0.4 * dx / vp.max()
    w = inputs.ricker(0.25 * 1500.0 / dx / 4.0, dt, nt)[None, None, :]
    src = np.array([[[(n / 2 + 0.3) * dx for n in shape]]])
    rec = inputs.random_points(8, shape, dx, 4, margin=nb + 2)
    g = oracle.Grid(shape, dx, dt=dt, nt=nt, order=order, nb=nb, c_ref=1500.0)
    obs = opml.forward(g, vp * 1.03, src[0], w[0], rec, rho=rho)[None]
    J_ref, g_ref, d_ref = opml.gradient(g, vp, src[0], w[0], rec, obs[0], rho=rho)
    plan = binding.Plan(shape, dx, nt, dt, order=order, sponge=nb, c_ref=1500.0)
    plan.set_options(boundary=binding.BOUNDARY_PML)
    J, gg, d = plan.gradient(to_dev(vp), to_dev(rho), binding.Geometry(src, rec), to_dev(w), to_dev(obs),
                             traces=True)
    plan.close()
    assert rel_l2(d.cpu().numpy()[0], d_ref) <= TOL_TRACES and abs(J - J_ref) <= 1e-3 * abs(J_ref)
    assert rel_l2(gg.cpu().numpy(), g_ref) <= TOL_GRAD
