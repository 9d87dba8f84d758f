"""The form that a plan takes by itself is one that the tuner tries, a caller can force
and a tune file can name."""
import numpy as np
import pytest

from paper_2201_08500_gb300 import bpm
from test_gpu_parity import deformed_small

pytestmark = pytest.mark.gpu

FORM = ("form", "channels_per_block", "row_threads")


@pytest.fixture(autouse=True)
def untuned():
    bpm.tune_clear()
    yield
    bpm.tune_clear()


# on either side of the default forms' lines (152 SMs)
@pytest.mark.parametrize("order", [1, 2, 4])
@pytest.mark.parametrize("nx,counts", [(256, (1, 2000)), (512, (1, 700)),
                                       (1024, (1, 290, 611)), (2048, (1, 240, 310)),
                                       (4096, (1, 160)), (8192, (1, 160))])
def test_the_default_form_is_a_candidate_of_the_tuner(nx, counts, order):
    for n_ch in counts:
        w = deformed_small(nx, nz=16 * 8, n_ch=n_ch, seed=nx)
        w.split_order, w.u = order, None
        p = bpm.plan_from_workload(w)

        def ran():
            p.run(16)
            s = p.stats()
            return {k: s[k] for k in ("threads_per_channel", "channels_per_block", "blocks",
                                      "smem_bytes")}

        default, forms = ran(), []
        for f in bpm.tune(2, nx, 1, w.dx, 0.0, w.dz, n_ch, split_order=order)[1]:
            p.set_launch(**{k: f[k] for k in FORM})
            forms.append(ran())
        assert default in forms, (n_ch, default, forms)
        p.close()


def test_strang_takes_the_two_channel_form_from_a_caller_and_a_file(tmp_path):
    w = deformed_small(1024, nz=40, n_ch=311, seed=6)
    w.split_order = 2
    want = dict(form=3, channels_per_block=2, row_threads=256)
    bpm.tune(2, 1024, 1, w.dx, 0.0, w.dz, w.n_ch, split_order=2)
    path = tmp_path / "tune.txt"
    bpm.tune_save(str(path))
    lines = path.read_text().splitlines()
    lines[-1] = " ".join(lines[-1].split()[:6] + ["3", "2", "256", "0.1"])
    path.write_text("\n".join(lines) + "\n")
    bpm.tune_clear()
    out = []
    for how in ("resident", "forced", "file"):
        if how == "file":
            assert bpm.tune_load(str(path)) == 1
        p = bpm.plan_from_workload(w)
        if how == "resident":
            p.set_launch(form=0, channels_per_block=4)
        elif how == "forced":
            p.set_launch(**want)
        assert how == "resident" or p.launch() == want
        p.run()
        p.sync()
        out.append((p.e0(), p.eh(), *p.reflectivity()[:2]))
        p.close()
    for got in out[1:]:
        for a, b in zip(out[0], got):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("n_ch", [400, 512, 700])
def test_a_few_tuning_steps_name_the_form_of_a_long_march(n_ch):
    """Where a form's one-time costs decided in 16 steps: what the tuner names then is what
    it names in 300 (the forms are 4 % apart or more in the lengthened run)."""
    named = [bpm.tune(2, 2048, 1, 5e-7, 0.0, 5e-7, n_ch, steps=s)[0] for s in (16, 300)]
    assert {k: named[0][k] for k in FORM} == {k: named[1][k] for k in FORM}
