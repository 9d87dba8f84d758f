"""The share of a batch's budget that a plan took is what its end gives back."""
import pytest

from paper_2201_08500_gb300 import bpm
from test_gpu_parity import deformed_small

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("end", ["done", "cancelled"])
@pytest.mark.parametrize("before,after", [(None, (0, 611)), ((0, 611), (0, 8)), ((2, 13), (2, 11))])
def test_a_shard_declared_in_the_batch_leaves_the_budget_balanced(before, after, end):
    """Its time response and that transform's tables grow or shrink the plan meanwhile."""
    ws = [deformed_small(256, nz=20, n_ch=4, seed=k) for k in (1, 2)]
    plans = [bpm.plan_from_workload(w) for w in ws]
    if before:
        plans[0].set_channel_shard(*before, 1.0e11)
    b = bpm.Batch(hbm_budget_bytes=1 << 30)
    b.submit(plans[1])
    own = b.info()["used_bytes"]
    t = b.submit(plans[0])
    plans[0].set_channel_shard(*after, 1.0e11)
    if end == "done":
        b.run()
        b.sync()
        assert b.poll(t)
    else:
        b.cancel(t)
    assert b.info()["used_bytes"] == own
    b.close()
    for p in plans:
        p.close()
