"""The 2D PML on the shot-loop tiles and the frame of its layer, against the FP64
oracle (the tolerances of test_gpu_pml.py): several tiles each way with ragged
edges, shot groups that do not divide the shots, a layer as wide as the tile rows,
grids with no point away from the layer, no layer at all, receivers and sources on
both sides of the line between the two forms, one and two steps."""
import numpy as np
import pytest

import oracle
from oracle import pml as opml
from paper_2110_03345_gb300 import binding, inputs
from _helpers import TOL_GRAD, TOL_TRACES, rel_l2, to_dev
from test_gpu_pml import density_with_constant_rim

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,order,nb,vd,shots,spc,ckpt,nt",
                         [((77, 270), 8, 7, True, 3, 2, -1, 150),
                          ((263, 83), 10, 19, False, 2, 2, 17, 150),
                          ((45, 259), 10, 9, True, 3, 3, 31, 120),
                          ((21, 134), 8, 8, False, 2, 1, -1, 120),
                          ((140, 33), 10, 16, False, 1, 1, -1, 120),
                          ((40, 141), 8, 0, False, 2, 2, -1, 100),
                          ((50, 60), 8, 6, False, 2, 2, -1, 2),
                          ((50, 60), 8, 6, False, 2, 2, -1, 3)])
def test_against_the_oracle(shape, order, nb, vd, shots, spc, ckpt, nt):
    dx = 0.5e-3
    vp, _ = inputs.random_smooth_model(shape, dx, 7)
    rho = density_with_constant_rim(shape, dx, nb + order // 2 + 1) if vd else None
    dt = 0.4 * dx / vp.max()
    w = np.ones(nt) if nt < 60 else inputs.ricker(0.25 * 1500.0 / dx / 4.0, dt, nt)
    w = np.broadcast_to(w, (shots, 1, nt)).copy()
    src = inputs.random_points(shots, shape, dx, 8, margin=min(nb + 3, min(shape) // 2 - 3))[:, None, :]
    rec = inputs.random_points(14, shape, dx, 9, margin=1)   # in the layer, next to it, away from it
    rec = np.concatenate([rec, src[:1, 0] + 0.3 * dx])       # reached within a step
    g = oracle.Grid(shape, dx, dt=dt, nt=nt, order=order, nb=nb, c_ref=1500.0)
    obs = np.random.default_rng(1).standard_normal((shots, len(rec), nt)) * 1e-3
    J_ref, g_ref, d_ref = 0.0, np.zeros(shape), []
    for s in range(shots):
        J_s, g_s, d_s = opml.gradient(g, vp, src[s], w[s], rec, obs[s], rho=rho)
        J_ref, g_ref = J_ref + J_s, g_ref + g_s
        d_ref.append(d_s)
    plan = binding.Plan(shape, dx, nt, dt, order=order, sponge=nb, c_ref=1500.0)
    plan.set_options(boundary=binding.BOUNDARY_PML, ckpt_every=ckpt, shots_per_cta=spc)
    J, gg, d = plan.gradient(to_dev(vp), to_dev(rho) if vd else None, binding.Geometry(src, rec),
                             to_dev(w), to_dev(obs), traces=True)
    plan.close()
    assert rel_l2(d.cpu().numpy(), np.stack(d_ref)) <= TOL_TRACES
    assert abs(J - J_ref) <= 1e-3 * abs(J_ref)
    assert rel_l2(gg.cpu().numpy(), g_ref) <= TOL_GRAD
