"""Calls whose grid points over all slots are enough for the density flags (three million, the
PML a million) against the same shots one at a time, whose launches add every density
term: what the flags leave out are zeros, so traces and misfits are equal, and gradients
to the order in which the shots are summed (32 terms of 6e-8 each add up as their root:
1e-6 relative L2).  The densities of test_gpu_density_planes.py."""
import numpy as np
import pytest

from paper_2110_03345_gb300 import binding, inputs
from _helpers import rel_l2, to_dev
from test_gpu_density_planes import density

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scheme,order,shots", [("leapfrog", 8, 32), ("leapfrog", 10, 32), ("att2", 10, 32),
                                                ("pml", 10, 8), ("pml", 8, 8)])
def test_flags_against_every_term(scheme, order, shots):
    shape, nt, dx = (45, 30, 131), 44, 0.5e-3
    p = inputs.skull_problem(shape, dx, nt, nrec=64, every=1, order=order, nb=5, f0=250e3)
    src = p.src_xyz[:shots]
    assert len(src) == shots and np.prod(shape) * shots >= (1e6 if scheme == "pml" else 3e6)
    geo = binding.Geometry(src, p.rec_xyz)
    vp = to_dev(p.vp)
    w = to_dev(np.broadcast_to(np.asarray(p.wavelet)[:1, :1], (shots, 1, nt)))
    obs = to_dev(1e-3 * np.random.default_rng(1).standard_normal((shots, p.rec_xyz.shape[0], nt)))
    plans = []
    for batch in (shots, 1):
        plan = binding.Plan(shape, dx, nt, p.dt, order=order, sponge=p.nb, c_ref=p.c_ref)
        opts = dict(boundary=binding.BOUNDARY_PML) if scheme == "pml" else {}
        plan.set_options(batch=batch, **opts)
        if scheme == "att2":
            plan.set_attenuation(to_dev(np.full(shape, 5.756 / (2 * np.pi * 1e6) ** 2)), 2)
        plans.append(plan)
    for kind in ("constant", "x", "y", "z", "box0", "box1", "box2", "box3", "box5"):
        rho = to_dev(density(kind, shape))
        (J0, g0, d0), (J1, g1, d1) = [plan.gradient(vp, rho, geo, w, obs, traces=True) for plan in plans]
        assert plans[0].stats()["batch"] == shots and plans[1].stats()["batch"] == 1
        assert np.array_equal(d0.cpu().numpy(), d1.cpu().numpy()), kind
        assert abs(J0 - J1) <= 1e-12 * J1
        assert np.abs(g0.cpu().numpy()).max() > 0 and rel_l2(g0.cpu().numpy(), g1.cpu().numpy()) < 1e-6, kind
    for plan in plans:
        plan.close()
