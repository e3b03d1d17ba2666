"""Resident 2D calls that span several launches: the hand-over of state, exchange tags and
samples between launches of 512 steps, and launches cut shorter by the buffer of raw samples
(eight million floats).  Each run is shown to be resident: one launch per step and direction
would make stats()['launches'] at least the number counted here.  Traces bit for bit against
the per-step kernels, gradients to 1e-6 (relative L2), as in test_gpu_resident.py."""
import numpy as np
import pytest

from paper_2110_03345_gb300 import binding, inputs
from _helpers import gpu_plan, rel_l2, to_dev

pytestmark = pytest.mark.gpu


def run(shape, nt, nshots, nelem, vd=True, **opts):
    """Traces, misfit, gradient and launches (forward, gradient) for tile 6 and the default."""
    p = inputs.breast_problem(shape, 0.3e-3, nt, nelem=nelem, shots=[i * (nelem // nshots) for i in range(nshots)],
                              order=8, nb=10, radius=0.3 * min(shape) * 0.3e-3)
    geo = binding.Geometry(p.src_xyz, p.rec_xyz)
    vp, rho, w = to_dev(p.vp), to_dev(p.rho) if vd else None, to_dev(p.wavelet)
    out, obs = [], None
    for o in (dict(tile=6, shots_per_cta=1), dict()):
        plan = gpu_plan(p, **{k: v for k, v in opts.items() if k == "interp" or not o}, **o)
        tr = plan.forward(vp, rho, geo, w)
        n = [plan.stats()["launches"]]
        obs = 0.5 * tr if obs is None else obs
        J, g, d = plan.gradient(vp, rho, geo, w, obs, traces=True)
        n.append(plan.stats()["launches"])
        assert np.array_equal(d.cpu().numpy(), tr.cpu().numpy())
        out.append((tr.cpu().numpy(), J, g.cpu().numpy().astype(np.float64), n))
        plan.close()
    return out


def check(ref, got, nt):
    assert np.abs(ref[0]).max() > 0 and np.array_equal(got[0], ref[0])
    assert abs(got[1] - ref[1]) <= 1e-12 * ref[1] and rel_l2(got[2], ref[2]) < 1e-6
    assert ref[3][0] >= nt - 1 and ref[3][1] >= 2 * (nt - 1)
    assert got[3][0] < nt - 1 and got[3][1] < 2 * (nt - 1)


@pytest.mark.parametrize("nt", [513, 514, 1025, 1026])
@pytest.mark.parametrize("vd", [True, False])
def test_several_launches(nt, vd):
    ref, got = run((150, 171), nt, 2, 24, vd=vd)
    check(ref, got, nt)
    assert got[3][0] <= 3 * -(-(nt - 1) // 512) + 2   # a launch and a combination of samples per 512 steps


@pytest.mark.parametrize("nshots,nelem", [(1, 512), (2, 512), (1, 2048)])
def test_launches_cut_by_the_sample_buffer(nshots, nelem):
    nt = 600                                            # 64 nodes per receiver: 256, 128 and 64 steps
    ref, got = run((300, 300), nt, nshots, nelem, interp=binding.INTERP_SINC)
    check(ref, got, nt)
    assert got[3][0] > 2 * (nt // 512 + 1)


@pytest.mark.parametrize("nshots", [2, 5, 16])
@pytest.mark.parametrize("opts", [dict(), dict(batch=2), dict(ckpt_every=40)])
def test_several_shots_run_resident(nshots, opts):
    nt = 120
    ref, got = run((150, 171), nt, nshots, 32, **opts)
    batches = -(-nshots // opts["batch"]) if "batch" in opts else 1
    assert got[3][0] < batches * (nt - 1) and got[3][1] < batches * 2 * (nt - 1)
    assert np.array_equal(got[0], ref[0]) and rel_l2(got[2], ref[2]) < 1e-6
