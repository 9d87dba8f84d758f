"""The march with an envelope a half block (few channels of 2048 points) against the
parked and resident forms."""
import numpy as np
import pytest

from paper_2201_08500_gb300 import bpm
from test_gpu_parity import deformed_small

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_ch", [1, 152, 200])  # one block, one an SM, shares
@pytest.mark.parametrize("order,other", [(1, 3), (2, 3), (4, 2)])
@pytest.mark.parametrize("crystal", [True, False])
def test_envelopes_side_by_side_give_the_parked_forms_bits(order, other, n_ch, crystal):
    w = deformed_small(2048, nz=61, n_ch=n_ch, seed=order)
    w.split_order = order
    if not crystal:
        w.thickness = 0.0
    out = []
    for form, steps in ((other, (61,)), (0, (61,)), (0, (1, 40, 20))):
        p = bpm.plan_from_workload(w)
        p.set_launch(form=form, channels_per_block=1)
        for n in steps:
            p.run(n)
        p.sync()
        assert form or p.stats()["threads_per_channel"] == 256
        out.append((p.e0(), p.eh(), *p.reflectivity()[:2]))
        p.close()
    for got in out[1:]:
        for a, b in zip(out[0], got):
            assert np.array_equal(a, b)
