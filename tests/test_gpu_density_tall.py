"""A 3D grid of more planes than a launch has blocks along z (65535), with density
gradients at both ends: the planes' density flags are made for all of them.  Bits of the
forward and 3e-6 of the gradient against the kernels that add every term, as in
test_gpu_density_planes.py."""
import numpy as np
import pytest

from paper_2110_03345_gb300 import binding, inputs
from _helpers import rel_l2, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nz", [65536, 70001])
def test_more_planes_than_blocks(nz):
    shape, nt, dx, nb = (nz, 9, 12), 14, 0.5e-3, 3
    vp = np.full(shape, 1500.0, np.float32)
    rho = np.full(shape, 1000.0, np.float32)
    for z in (40, nz - 30):
        rho[z:z + 3, 3:6, 4:9] = 1300.0
    dt = 0.4 * dx / 1500.0
    ends = np.array([38.3, nz - 31.4])
    src = np.stack([[[z * dx, 4.2 * dx, 5.7 * dx]] for z in ends])
    rec = np.array([[(z + d) * dx, 4.6 * dx, 6.1 * dx] for z in ends for d in (-2.0, 1.5, 4.5)])
    w = np.broadcast_to(inputs.ricker(0.25 * 1500.0 / dx / 4.0, dt, nt), (2, 1, nt))
    geo = binding.Geometry(src, rec)
    out = []
    for tile in (0, 5):
        plan = binding.Plan(shape, dx, nt, dt, order=8, sponge=nb, c_ref=1500.0)
        plan.set_options(tile=tile, batch=1)
        J, g, d = plan.gradient(to_dev(vp), to_dev(rho), geo, to_dev(w), to_dev(np.zeros((2, len(rec), nt))),
                                traces=True)
        out.append((J, g.cpu().numpy(), d.cpu().numpy()))
        plan.close()
    (J0, g0, d0), (J1, g1, d1) = out
    assert np.abs(d0[0, :3]).max() > 0 and np.abs(d0[1, 3:]).max() > 0
    assert np.array_equal(d0, d1) and J0 == J1 and rel_l2(g0, g1) < 3e-6
