"""GPU tests of the order of fp32 additions: which form of a sweep runs, with how
many threads and where its state lies, must not show in the results."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2511_17245_gb300 import Model, _lib
from paper_2511_17245_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
RULES = ["metropolis", "heat_bath", "opt_metropolis"]


@pytest.mark.parametrize("lo", [(1 << 24) - 20, 1 << 25, -(1 << 25) - 3, (1 << 22) + 1])
@pytest.mark.parametrize("width", [12, 40, 90, 150, 230])
def test_heat_bath_beyond_2_24_is_the_level_orders(lo, width):
    """Values whose steps of 1 round in fp32: blocked and level order form them alike."""
    inst = wl.batch_instance({"index": 0, "n": 70, "width": width, "dense": True, "deg": 0, "seed": width})
    inst = dict(inst, lower=inst["lower"] + lo, upper=inst["upper"] + lo)
    model = Model(inst)
    for tpr in (32, 128, 512):
        kw = dict(threads_per_replica=tpr, seed=5, t_max=1e9, t_min=1e7)
        ref = model.run("heat_bath", 8, 24, flags=_lib.SA_FLAG_NO_SPECULATION, **kw)
        got = model.run("heat_bath", 8, 24, **kw)
        for key in ("states", "accepts", "energies"):
            assert torch.equal(ref[key], got[key]), (tpr, key)
