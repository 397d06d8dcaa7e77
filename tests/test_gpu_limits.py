"""GPU tests of calls whose shared memory lies at the limits of a kernel's
static plus dynamic share.  Integer or exactly summed results; each call is
compared with sa_run or numpy."""
import os
import subprocess
import sys

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2511_17245_gb300 import (Model, make_params, sa_batch_create, sa_batch_destroy, sa_batch_get_info,
                                    sa_batch_result, sa_batch_run)
from paper_2511_17245_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _banded(n, step, coef_type="f32"):
    """Variables k and k + step coupled: levels of `step` variables.  Whole-number
    couplings, so that fp32 fields and FP64 energies are exact."""
    rng = np.random.default_rng(n)
    i = np.arange(n - step)
    pairs = np.stack([i, i + step], axis=1)
    lin = rng.integers(-9, 10, n)
    cpl = rng.choice([-3, -2, -1, 1, 2, 3], len(pairs))
    offs = np.concatenate([np.arange(n + 1), n + 2 * np.arange(1, len(pairs) + 1)]).astype(np.int64)
    flat = np.concatenate([np.arange(n), pairs.ravel()]).astype(np.int32)
    dt = np.float32 if coef_type == "f32" else np.int32
    return {"n_vars": n, "lower": np.zeros(n, np.int64), "upper": np.full(n, 7, np.int64), "term_offsets": offs,
            "term_vars": flat, "coeffs": np.concatenate([lin, cpl]).astype(dt), "coef_type": coef_type}


@pytest.mark.parametrize("n", [2600, 2613, 2617, 2620, 2640, 2829, 2832])
def test_batch_shapes_that_fill_shared_memory(n):
    """Fifteen (fourteen) replicas of 32 threads whose regions and argument copies
    end within a few hundred bytes of a block's shared memory."""
    model = Model(_banded(n, 64))
    p = make_params(rule="metropolis", n_sweeps=6, n_replicas=40, seed=9)
    b = sa_batch_create([model.handle], [p])
    try:
        info = sa_batch_get_info(b)
        assert info["threads_per_replica"] == 32 and info["replicas_per_block"] >= 13
        sa_batch_run(b)
        torch.cuda.synchronize()
        st, en, ac = np.zeros((40, n), np.int32), np.zeros(40), np.zeros(40, np.uint64)
        sa_batch_result(b, 0, st, en, ac)
    finally:
        sa_batch_destroy(b)
    ref = model.run("metropolis", 6, 40, seed=9)
    assert np.array_equal(st, ref["states"].cpu().numpy())
    assert np.array_equal(en, ref["energies"].cpu().numpy())
