"""Resident launches of several threads: plans of different sizes run at once on streams of
their own, and each gives the bits it gives alone (a launch must not change the
shared-memory limit under another thread's launch)."""
import threading

import numpy as np
import pytest
import torch

from paper_2110_03345_gb300 import binding, inputs
from _helpers import to_dev

pytestmark = pytest.mark.gpu


def test_plans_of_different_sizes_at_once():
    dx, nt = 0.5e-3, 60
    jobs = []
    for n in ((96, 130), (700, 748), (256, 256), (1000, 900)):
        vp, rho = inputs.random_smooth_model(n, dx, 1)
        dt = 0.4 * dx / vp.max()
        src = inputs.random_points(1, n, dx, 2, margin=12)[:, None, :]
        rec = src[0] + dx * np.array([[3.0, 2.0], [-4.0, 1.0], [5.5, -6.0], [-7.0, -3.5]])   # reached early
        w = inputs.ricker(0.25 * 1500.0 / dx / 4.0, dt, nt)[None, None, :]
        jobs.append((n, dt, to_dev(vp), to_dev(rho), binding.Geometry(src, rec), to_dev(w)))

    def plan_of(job, stream):
        return binding.Plan(job[0], dx, nt, job[1], order=8, sponge=10, c_ref=1500.0, budget=2 << 30,
                            stream=stream)

    def run(plan, job):
        return plan.forward(job[2], job[3], job[4], job[5])

    alone = []
    for job in jobs:
        plan = plan_of(job, torch.cuda.current_stream())
        alone.append(run(plan, job).cpu().numpy())
        plan.close()
    assert all(np.abs(a).max() > 0 for a in alone)
    errors = []

    def work(i):
        try:
            st = torch.cuda.Stream()
            with torch.cuda.stream(st):
                plan = plan_of(jobs[i], st)
                for _ in range(40):
                    got = run(plan, jobs[i])
                    st.synchronize()
                    if not np.array_equal(got.cpu().numpy(), alone[i]):
                        errors.append((i, "bits"))
                plan.close()
        except Exception as e:   # noqa: BLE001 - reported by the main thread
            errors.append((i, repr(e)))

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
