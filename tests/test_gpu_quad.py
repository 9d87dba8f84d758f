"""The march with 8 Nx/16 threads a channel (few channels) against the grouped resident form."""
import numpy as np
import pytest

from paper_2201_08500_gb300 import bpm
from test_gpu_parity import deformed_small

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [1, 2, 4])
@pytest.mark.parametrize("nx,n_ch,maxg", [(256, 1, 16), (256, 35, 16), (512, 1, 8), (512, 160, 8),
                                          (1024, 1, 4), (1024, 155, 4)])
def test_few_channels_give_the_resident_forms_bits(nx, n_ch, maxg, order):
    """Fields and reflectivities bitwise equal; a split run ends where a whole one does."""
    w = deformed_small(nx, nz=61, n_ch=n_ch, seed=nx + order)
    w.split_order = order
    out = []
    for group, steps in ((maxg, (61,)), (1, (61,)), (1, (1, 40, 20))):
        p = bpm.plan_from_workload(w)
        p.set_launch(form=0, channels_per_block=group)
        for n in steps:
            p.run(n)
        p.sync()
        out.append((p.e0(), p.eh(), *p.reflectivity()[:2]))
        p.close()
    for got in out[1:]:
        for a, b in zip(out[0], got):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("sms", [0, 4])
def test_work_queue_singles_and_full_items_give_the_plans_bits(sms):
    """Plans of small grids in one batch, on either side of the line between
    single channels and resident items (on four SMs the larger counts fill
    these), each as marched alone."""
    ws = []
    for nx, order, counts in ((256, 1, (1, 64)), (256, 2, (31,)), (256, 4, (61, 3)),
                              (512, 1, (1, 15, 40)), (512, 2, (9,)), (512, 4, (6, 32)),
                              (1024, 2, (2, 7))):
        for n_ch in counts:
            w = deformed_small(nx, nz=20 + n_ch, n_ch=n_ch, seed=n_ch)
            w.split_order = order
            ws.append(w)
    want = []
    for w in ws:
        p = bpm.plan_from_workload(w)
        p.run()
        p.sync()
        want.append((p.e0(), p.eh(), p.reflectivity()[0]))
        p.close()
    b = bpm.Batch()
    b.set_max_blocks(sms)
    plans = [bpm.plan_from_workload(w) for w in ws]
    for p in plans:
        b.submit(p)
    b.step(13)
    b.run()
    b.sync()
    for p, (e0, eh, R) in zip(plans, want):
        assert np.array_equal(p.e0(), e0) and np.array_equal(p.eh(), eh)
        assert np.array_equal(p.reflectivity()[0], R)
    b.close()
    for p in plans:
        p.close()


@pytest.mark.parametrize("nx,order,n_ch", [(256, 1, 1700), (512, 2, 3), (1024, 1, 160),
                                           (1024, 2, 310), (1024, 4, 307), (2048, 1, 5),
                                           (2048, 4, 305), (4096, 1, 153), (4096, 4, 155),
                                           (8192, 2, 3)])
def test_default_forms_give_the_resident_forms_bits(nx, order, n_ch):
    """A plan that names no form, on either side of the lines between forms."""
    w = deformed_small(nx, nz=9, n_ch=n_ch, seed=nx + n_ch)
    w.split_order = order
    group = {256: 16, 512: 8, 1024: 4, 2048: 2}.get(nx, 1)
    out = []
    for forced in (False, True):
        p = bpm.plan_from_workload(w)
        if forced:
            p.set_launch(form=0, channels_per_block=group)
        p.run(4)
        p.run(5)
        p.sync()
        out.append((p.e0(), p.eh(), *p.reflectivity()[:2]))
        p.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
