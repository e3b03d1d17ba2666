"""Resident 2D launches (a shot's wavefields stay on chip for many steps)
against the per-step kernels: the forward bit for bit, the gradient up to the
rounding of the density terms and of the imaging sum (relative L2 1e-6, the
bound of the other tests that reorder those sums).  Grids at the edges of the
tiles (128 points wide, one or two phases high), several shots side by side
and in turn, both orders and density modes, sinc points, one-step launches."""
import threading

import numpy as np
import pytest

from paper_2110_03345_gb300 import binding, inputs
from _helpers import gpu_forward, gpu_gradient, gpu_plan, rel_l2, to_dev

pytestmark = pytest.mark.gpu


def problem(shape, nt, shots, order=8, nelem=24):
    return inputs.breast_problem(shape, 0.3e-3, nt, nelem=nelem, shots=shots, order=order, nb=10,
                                 radius=0.3 * min(shape) * 0.3e-3)


def resident(plan, nt):
    return plan.stats()["launches"] < nt   # far fewer launches than time steps


@pytest.mark.parametrize("shape", [(40, 37), (64, 128), (129, 257), (97, 640), (640, 130), (700, 260),
                                   (905, 1024)])
@pytest.mark.parametrize("order,vd", [(8, False), (8, True), (10, False), (10, True)])
def test_matches_the_per_step_kernels(shape, order, vd):
    nt = 130
    p = problem(shape, nt, shots=[0], order=order)
    ref, _ = gpu_forward(p, variable_density=vd, tile=6)
    got, plan = gpu_forward(p, variable_density=vd)
    assert resident(plan, nt)
    assert np.abs(ref).max() > 0 and np.array_equal(got, ref)
    obs = 0.5 * ref
    J0, g0, d0, _ = gpu_gradient(p, obs, variable_density=vd, tile=6)
    J1, g1, d1, plan = gpu_gradient(p, obs, variable_density=vd)
    assert resident(plan, 2 * nt)
    assert J1 == J0 and np.array_equal(d1, d0)
    assert rel_l2(g1, g0) < 1e-6


@pytest.mark.parametrize("nshots", [2, 5, 16])
def test_shots_side_by_side_and_in_turn(nshots):
    nt = 120
    p = problem((150, 171), nt, shots=list(range(nshots)))
    ref, _ = gpu_forward(p, tile=6)
    got, plan = gpu_forward(p)
    assert resident(plan, nt * nshots) and np.array_equal(got, ref)
    obs = 0.5 * ref
    J0, g0, _, _ = gpu_gradient(p, obs, tile=6, shots_per_cta=1)
    for opts in (dict(), dict(batch=max(1, nshots // 2)), dict(ckpt_every=9)):
        J1, g1, d1, _ = gpu_gradient(p, obs, **opts)
        assert np.array_equal(d1, ref) and abs(J1 - J0) <= 1e-12 * J0
        assert rel_l2(g1, g0) < 1e-6


@pytest.mark.parametrize("nt", [2, 3, 17])
def test_short_runs(nt):
    p = problem((70, 140), nt, shots=[0, 7])
    ref, _ = gpu_forward(p, tile=6)
    got, _ = gpu_forward(p)
    assert np.array_equal(got, ref)
    J0, g0, _, _ = gpu_gradient(p, ref + 1e-3, tile=6, shots_per_cta=1)
    for k in (-1, 1, 2):   # K = 1: launches of one step
        J1, g1, _, _ = gpu_gradient(p, ref + 1e-3, ckpt_every=k)
        assert abs(J1 - J0) <= 1e-12 * J0 and rel_l2(g1, g0) < 1e-6


def test_sinc_points_and_the_wavelet_gradient():
    nt = 150
    p = problem((140, 300), nt, shots=[0, 9])
    geo = binding.Geometry(p.src_xyz, p.rec_xyz)
    out = []
    for tile in (6, 0):
        plan = gpu_plan(p, tile=tile, interp=binding.INTERP_SINC, shots_per_cta=1 if tile else 0)
        tr = plan.forward(to_dev(p.vp), to_dev(p.rho), geo, to_dev(p.wavelet))
        plan.misfit_forward(to_dev(p.vp), to_dev(p.rho), geo, to_dev(p.wavelet), 0.5 * tr)
        g, q = plan.misfit_backward_ex()
        out.append([a.cpu().numpy().astype(np.float64) for a in (tr, g, q)])
        plan.close()
    assert np.array_equal(out[0][0], out[1][0])
    assert rel_l2(out[1][1], out[0][1]) < 1e-6 and rel_l2(out[1][2], out[0][2]) < 1e-6


def test_concurrent_streams_give_the_same_bits():
    """Resident launches of several threads share the GPU: each result is the
    one the plan gives alone."""
    import torch
    ps = [problem(s, 200, shots=[0]) for s in ((300, 400), (512, 512), (150, 171), (700, 260))]
    obs = [0.5 * gpu_forward(p)[0] for p in ps]
    ref = [gpu_gradient(p, o)[:2] for p, o in zip(ps, obs)]
    got = [[] for _ in ps]

    def work(i):
        p = ps[i]
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(3):
                plan = gpu_plan(p)
                got[i].append(gpu_gradient(p, obs[i], plan=plan)[:2])
                plan.close()

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(ps))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for (J, g), runs in zip(ref, got):
        assert len(runs) == 3
        assert all(Jr == J and np.array_equal(gr, g) for Jr, gr in runs)
