"""The 3D y = 2 attenuation on the plane ring: where a tight budget has no room
for its two fields the gradient (forward and adjoint) runs on the one-point
kernels.  The families' traces agree to 1e-6 (relative L2), so the residual of
half the data to 2e-6, the misfit to 4e-6 and the gradient, linear in the
residual and in the history, to 3e-6."""
import numpy as np
import pytest

from paper_2110_03345_gb300 import binding, inputs
from _helpers import rel_l2, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,order,vd", [((33, 41, 130), 10, True), ((40, 24, 67), 8, False)])
def test_ring_and_one_point_kernels_agree(shape, order, vd):
    nt = 60
    p = inputs.skull_problem(shape, 0.5e-3, nt, nrec=32, every=32, order=order, nb=6, f0=250e3)
    a0 = to_dev(1e-13 * (1 + np.indices(shape).sum(0) % 3))
    geo = binding.Geometry(p.src_xyz, p.rec_xyz)
    vp, rho, w = to_dev(p.vp), to_dev(p.rho) if vd else None, to_dev(p.wavelet)

    def gradient(budget, obs):
        plan = binding.Plan(p.shape, p.spacing, nt, p.dt, order=order, sponge=p.nb, c_ref=p.c_ref,
                            budget=budget)
        plan.set_options(ckpt_every=-1)
        plan.set_attenuation(a0, 2)
        tr = plan.forward(vp, rho, geo, w)
        J, g, _ = plan.gradient(vp, rho, geo, w, 0.5 * tr if obs is None else obs)
        out = (J, g.cpu().numpy().astype(np.float64), tr, plan.stats())
        plan.close()
        return out

    J0, g0, tr, st = gradient(0, None)
    R = order // 2
    field = 4 * (-(-shape[2] // 128) * 128 + 16) * (-(-shape[1] // 64) * 64 + 2 * R) * (shape[0] + 2 * R)
    seen = {st["launches"]}
    for less in range(6):
        try:
            J1, g1, tr1, st1 = gradient(st["workspace_bytes"] - less * field // 2, 0.5 * tr)
        except binding.FwiError:
            break
        seen.add(st1["launches"])
        assert np.array_equal(tr1.cpu().numpy(), tr.cpu().numpy())
        assert abs(J1 - J0) <= 4e-6 * J0 and rel_l2(g1, g0) < 3e-6
    assert len(seen) == 2   # with and without the ring's extra pass
