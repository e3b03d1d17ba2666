"""A plan whose budget is the estimate of its request gives the bits of a plan with all the
memory: the serving loop runs requests so.  Shot counts around the line between resident
and per-step kernels, which lies elsewhere with and without density (a gradient differs in
its last bits between the two)."""
import numpy as np
import pytest

from paper_2110_03345_gb300 import binding, inputs
from _helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nshots", [1, 6, 8, 9, 10, 11, 12, 13, 16])
@pytest.mark.parametrize("vd", [True, False])
def test_the_estimate_leaves_room_for_the_same_kernels(nshots, vd):
    nt = 60
    p = inputs.breast_problem((456, 485), 0.3e-3, nt, nelem=64, shots=[4 * i for i in range(nshots)], order=8, nb=10,
                              radius=0.3 * 456 * 0.3e-3)
    geo = binding.Geometry(p.src_xyz, p.rec_xyz)
    vp, rho, w = to_dev(p.vp), to_dev(p.rho) if vd else None, to_dev(p.wavelet)
    obs = to_dev(1e-3 * np.random.default_rng(0).standard_normal((nshots, 64, nt)))
    out = []
    budget = 0
    for _ in range(2):
        plan = binding.Plan(p.shape, p.spacing, nt, p.dt, order=8, sponge=p.nb, c_ref=p.c_ref, budget=budget)
        budget = plan.estimate(geo, gradient=True)
        J, g, _ = plan.gradient(vp, rho, geo, w, obs)
        out.append((J, g.cpu().numpy(), plan.stats()["launches"], plan.stats()["ckpt_every"]))
        plan.close()
    (J0, g0, n0, k0), (J1, g1, n1, k1) = out
    assert J0 == J1 and np.array_equal(g0, g1) and (n0, k0) == (n1, k1)
