"""A captured batch whose plans get other inputs: every replay is of the inputs stored last."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2201_08500_gb300 import bpm
from test_gpu_parity import deformed_small

pytestmark = pytest.mark.gpu


def load(p, w, u):
    p.set_geometry(getattr(w, "tan_psi", 0.0))
    p.set_crystal_shape(getattr(w, "mask", None))
    p.set_crystal(w.chi0, w.chih, w.chihb, w.theta_B, w.lambda_B, w.x_surface, w.thickness, u=u)
    pulse(p, w)


def pulse(p, w):
    p.set_pulse(w.omega, w.S, w.theta_i, w.x0, w.w0, w.zx, w.zR)


def results(p):
    return p.e0(), p.eh(), p.eh_time(), p.reflectivity()[0]


def alone(w, u, shard=None):
    p = bpm.plan_from_workload(w, u=u)
    if shard:
        p.set_channel_shard(*shard)
    p.run()
    p.sync()
    got = results(p)
    p.close()
    return got


@pytest.mark.parametrize("change", ["beam", "spacing", "tilted beam", "shard", "shard spacing",
                                    "displacement", "no displacement", "cut", "shape", "crystal",
                                    "cap", "nothing"])
def test_a_replay_uses_the_inputs_stored_last(change):
    ws = [deformed_small(512, nz=70, n_ch=5, seed=1), deformed_small(2048, nz=40, n_ch=3, seed=2)]
    us = [torch.from_numpy(w.u).cuda() for w in ws]
    other = torch.from_numpy(deformed_small(512, nz=70, n_ch=5, seed=3).u).cuda()
    b = bpm.Batch()
    plans = [bpm.plan_from_workload(w, u=u) for w, u in zip(ws, us)]
    shard = None
    if change.startswith("shard"):
        shard = (2, 9, 1.5e11)
        plans[0].set_channel_shard(*shard)
    for p in plans:
        b.submit(p)

    def check(w, u, shard):
        for _ in range(2):
            b.run_graph()
            b.sync()
        for p, want in zip(plans, (alone(w, u, shard), alone(ws[1], us[1]))):
            for x, y in zip(results(p), want):
                assert np.array_equal(x, y)

    check(ws[0], us[0], shard)
    w, u, p = dataclasses.replace(ws[0]), us[0], plans[0]
    if change == "beam":
        w.x0, w.w0 = w.x0 + 9 * w.dx, 1.5 * w.w0
        pulse(p, w)
    elif change == "spacing":  # scales the time response
        w.omega = w.omega[0] + 1.25 * (w.omega - w.omega[0])
        pulse(p, w)
    elif change == "tilted beam":
        w.theta_i, w.zx, w.zR = w.theta_i + 1e-6, 2e-4, 1e-3
        pulse(p, w)
    elif change.startswith("shard"):
        shard = (2, 9, 2e11) if change == "shard spacing" else (3, 8, 1.5e11)
        pulse(p, w)
        p.set_channel_shard(*shard)
    elif change == "displacement":  # (the buffer before lives on)
        w.u, u = None, other
        load(p, w, u)
    elif change == "no displacement":
        w.u, u = None, None
        load(p, w, u)
    elif change == "cut":
        w.tan_psi = 0.1
        load(p, w, u)
    elif change == "shape":
        w.mask = np.random.default_rng(4).random((w.nz, w.nx)) < 0.3
        load(p, w, u)
    elif change == "crystal":
        w.chih, w.thickness = 2 * w.chih, w.thickness / 2
        load(p, w, u)
    elif change == "cap":
        b.set_max_blocks(2)
    else:
        load(p, w, u)
    check(w, u, shard)
    b.close()
    for p in plans:
        p.close()


def test_a_crystal_that_the_stored_pulse_does_not_go_with_is_refused():
    w = deformed_small(512, nz=30, n_ch=4, seed=5)
    p = bpm.plan_from_workload(w)
    b = bpm.Batch()
    b.submit(p)
    b.run_graph()
    b.sync()
    want = p.e0(), p.eh()
    crystal = (w.chi0, w.chih, w.chihb, w.theta_B, w.lambda_B, w.x_surface, w.thickness)
    p.set_crystal(*crystal[:4], 0.5 * w.lambda_B, *crystal[5:], u=w.u)  # k <= h/2
    with pytest.raises(bpm.BpmError):
        b.run_graph()
    p.set_crystal(*crystal, u=w.u)
    b.run_graph()
    b.sync()
    for x, y in zip((p.e0(), p.eh()), want):
        assert np.array_equal(x, y)
    b.close()
    p.close()
