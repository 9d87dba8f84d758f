"""Marches of more channels than fit at a time, in equal shares of the SMs' blocks,
against plans of few channels, which march whole."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2201_08500_gb300 import bpm
from test_gpu_parity import deformed_small

pytestmark = pytest.mark.gpu


# extra: channels beyond the slots, one or a tenth of the SMs' worth (each slot's
# cuts then lie within a step of one another, or spread over the march)
@pytest.mark.parametrize("extra", [1, 0.1])
@pytest.mark.parametrize("nx,order,form,group,per_sm",
                         [(256, 4, 0, 1, 2), (512, 1, 0, 1, 1), (1024, 1, 3, 2, 1),
                          (1024, 1, 2, 1, 5), (1024, 4, 2, 1, 8), (2048, 2, 3, 1, 2),
                          (4096, 1, 3, 1, 2), (4096, 4, 2, 1, 1), (8192, 1, 3, 1, 1)])
def test_shares_give_the_bits_of_whole_channels(nx, order, form, group, per_sm, extra):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    slots = sms * per_sm * group
    n_ch = slots + (1 if extra == 1 else int(extra * sms * group))
    nz = 40
    w = deformed_small(nx, nz=nz, n_ch=n_ch, seed=nx + order)
    w.split_order = order
    p = bpm.plan_from_workload(w)
    p.set_launch(form=form, channels_per_block=group)
    got = []
    for steps in ((nz,), (nz,), (3, 17, 20)):  # the marks are clean again after each
        p.set_pulse(w.omega, w.S, w.theta_i, w.x0, w.w0, w.zx, w.zR)
        for n in steps:
            p.run(n)
        p.sync()
        got.append((p.e0(), p.eh(), *p.reflectivity()[:2]))
        if len(steps) == 1:
            assert p.stats()["blocks"] == per_sm * sms
    p.close()
    for g in got[1:]:
        for a, b in zip(got[0], g):
            assert np.array_equal(a, b)
    part = max(1, sms // 2)
    for lo in range(0, n_ch, part):  # whole channels: no more than an SM each
        v = dataclasses.replace(w, omega=w.omega[lo:lo + part], S=w.S[lo:lo + part])
        v.split_order = order
        q = bpm.plan_from_workload(v)
        q.run()
        q.sync()
        for a, b in zip(got[0], (q.e0(), q.eh(), *q.reflectivity()[:2])):
            assert np.array_equal(a[lo:lo + part], b)
        q.close()
