"""Which kernel a launch takes: the few-channel march and the two kinds of work-queue items."""
import pytest

from paper_2201_08500_gb300 import bpm
from test_gpu_parity import deformed_small

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [1, 2, 4])
@pytest.mark.parametrize("nx,n_ch", [(256, 1), (256, 35), (512, 1), (512, 160), (1024, 1),
                                     (1024, 155)])
def test_few_channels_take_eight_times_the_threads(nx, n_ch, order):
    w = deformed_small(nx, nz=4, n_ch=n_ch, seed=1)
    w.split_order = order
    p = bpm.plan_from_workload(w)
    p.set_launch(form=0, channels_per_block=1)
    p.run()
    assert p.stats()["threads_per_channel"] == nx // 2
    maxg = 4096 // nx
    p.set_launch(form=0, channels_per_block=maxg)
    assert p.stats()["threads_per_channel"] == nx // 16
    p.close()


# full resident items on four SMs (four items of 16 or 8 channels), single channels on all
@pytest.mark.parametrize("nx,order,n_ch", [(256, 1, 64), (256, 4, 64), (512, 1, 32), (512, 4, 32)])
def test_queue_items_are_full_or_single_channels(nx, order, n_ch):
    items = {}
    for cap in (0, 4):
        w = deformed_small(nx, nz=6, n_ch=n_ch, seed=2)
        w.split_order = order
        p = bpm.plan_from_workload(w)
        b = bpm.Batch()
        b.set_max_blocks(cap)
        b.submit(p)
        b.run()
        b.sync()
        items[cap] = tuple(b.info()["last_items"])
        b.close()
        p.close()
    assert items == {0: (n_ch, 0), 4: (4, 0)}
