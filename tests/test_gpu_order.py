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


def test_tracked_energies_of_narrow_levels():
    """Per-sweep energies of an fp32 model with levels of about 13 variables.
    Couplings and values are whole numbers, so fields and energy changes are exact
    and both orders make the same moves; what is left is the rounding of the sums
    of changes.  It falls with the root of the number of partial sums (32 lanes of
    a block against the threads of a level), so blocks may be no worse than half as
    much again as levels."""
    n, S, R = 1000, 4, 64
    inst = wl.quio_sparse_int(4, n, 20 * n, 0, 200)
    inst = dict(inst, coeffs=inst["coeffs"].astype(np.float32), coef_type="f32")
    model = Model(inst)
    assert 8 <= n / model.info["n_levels"] <= 16

    def run(rule, flags):
        tr = torch.zeros((S, R, n), dtype=torch.int32, device="cuda")
        et = torch.zeros((S, R), dtype=torch.float64, device="cuda")
        model.run(rule, S, R, seed=3, trace=tr, trace_replicas=R, energy_trace=et, flags=flags,
                  t_max=1e7, t_min=1e6)
        return tr, et

    for rule in ("metropolis", "opt_metropolis"):
        (ta, ea), (tb, eb) = run(rule, 0), run(rule, _lib.SA_FLAG_NO_SPECULATION)
        assert torch.equal(ta, tb)
        true = torch.stack([model.energy(ta[s]) for s in range(S)])
        rms = [float(((e - true)[:-1] ** 2).mean().sqrt()) for e in (ea, eb)]
        assert rms[1] > 0 and rms[0] <= 1.5 * rms[1], (rule, rms)
        assert torch.equal(ea[-1], true[-1])     # recomputed in FP64 at the end, whole numbers
