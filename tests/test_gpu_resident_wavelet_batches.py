"""Wavelet gradient of the resident 2D kernels over batches of shots whose last one is
not full (and with several sources per shot): dJ/dq of every shot against the per-step
kernels, relative L2 1e-6 (the same sums; the residuals agree bit for bit)."""
import numpy as np
import pytest

from paper_2110_03345_gb300 import binding, inputs
from _helpers import gpu_plan, rel_l2, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nshots,batch,nsrc", [(3, 2, 1), (5, 4, 1), (5, 3, 3), (7, 6, 2), (4, 2, 1)])
@pytest.mark.parametrize("interp", [binding.INTERP_LINEAR, binding.INTERP_SINC])
def test_partial_last_batch(nshots, batch, nsrc, interp):
    nt = 150
    shape = (140, 300)
    p = inputs.breast_problem(shape, 0.3e-3, nt, nelem=48, shots=list(range(nshots)), order=8, nb=10,
                              radius=0.3 * min(shape) * 0.3e-3)
    ring = np.asarray(p.rec_xyz)
    src = np.stack([[ring[(5 * i + 16 * k) % len(ring)] for k in range(nsrc)] for i in range(nshots)])
    w = np.asarray(p.wavelet, dtype=np.float64)[:, :1, :] * np.linspace(1.0, 0.5, nsrc)[None, :, None]
    geo = binding.Geometry(src, ring)
    out = []
    for opts in (dict(tile=6, shots_per_cta=1), dict()):
        plan = gpu_plan(p, batch=batch, interp=interp, **opts)
        tr = plan.forward(to_dev(p.vp), to_dev(p.rho), geo, to_dev(w))
        plan.misfit_forward(to_dev(p.vp), to_dev(p.rho), geo, to_dev(w), 0.5 * tr)
        g, q = plan.misfit_backward_ex()
        out.append([a.cpu().numpy().astype(np.float64) for a in (tr, g, q)])
        plan.close()
    (tr0, g0, q0), (tr1, g1, q1) = out
    assert np.array_equal(tr1, tr0) and rel_l2(g1, g0) < 1e-6
    assert q1.shape == (nshots, nsrc, nt)
    for s in range(nshots):
        assert np.abs(q0[s]).max() > 0 and rel_l2(q1[s], q0[s]) < 1e-6
