"""GPU tests of calls whose shared memory lies at the limits of a kernel's
static plus dynamic share.  Integer or exactly summed results; each call is
compared with sa_run or numpy."""
import os
import subprocess
import sys

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2511_17245_gb300 import (Model, _lib, make_params, sa_batch_create, sa_batch_destroy, sa_batch_get_info,
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


@pytest.mark.parametrize("n,hi,n_states", [(12288, 255, 1216), (12273, 255, 1216), (6144, 300, 1216), (6137, 300, 1216),
                                           (49152, 255, 3), (49089, 255, 3), (24576, 300, 3), (12288, 255, 3)])
def test_energies_at_48_kb_of_staged_states(n, hi, n_states):
    """Staged states of 48 KB and the first size whose static scratch reaches past
    it, in a process that has made no larger call: whole numbers, exact."""
    code = f"""
import sys; sys.path.insert(0, {ROOT!r})
import numpy as np, torch
from paper_2511_17245_gb300 import Model
rng = np.random.default_rng(1)
n, hi = {n}, {hi}
i = np.arange(n - 1)
inst = dict(n_vars=n, lower=np.zeros(n, np.int64), upper=np.full(n, hi, np.int64), coef_type="i32",
            term_offsets=np.concatenate([np.arange(n + 1), n + 2 * np.arange(1, n)]).astype(np.int64),
            term_vars=np.concatenate([np.arange(n), np.stack([i, i + 1], 1).ravel()]).astype(np.int32),
            coeffs=rng.integers(-9, 10, 2 * n - 1).astype(np.int32))
z = rng.integers(0, hi + 1, ({n_states}, n))
c = inst["coeffs"].astype(np.int64)
want = z @ c[:n] + (z[:, :-1] * z[:, 1:]) @ c[n:]
got = Model(inst).energy(torch.from_numpy(z.astype(np.int32)).cuda()).cpu().numpy()
assert np.array_equal(got, want), (got, want)
"""
    res = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert res.returncode == 0, res.stderr[-2000:]


@pytest.mark.parametrize("n,first", [(20_000, 0), (20_000, 19_000), (188, 0), (188, 9), (189, 3)])
def test_unused_variables_take_no_coefficient_slots(n, first):
    """A multilinear HUIO model, 60 of whose variables occur in terms: 100 replicas
    of 20,000 variables take 2.7 MB of the fixed scratch of sa_run_noalloc, not 18.
    With 128 unused variables the slots are padded, with 129 they are not."""
    from oracle import oracle as orc
    from paper_2511_17245_gb300 import sa_run_noalloc
    small = wl.random_small(3, 60, 4, np.full(60, -3), np.full(60, 4), 300, repeat=False)
    used = first + 3 * np.arange(60)
    inst = dict(small, n_vars=n, lower=np.full(n, -3, np.int64), upper=np.full(n, 4, np.int64),
                term_vars=used[small["term_vars"]].astype(np.int32))
    model, om = Model(inst), orc.Model(inst)
    R, S = 100, 12
    tmax, tmin = om.auto_temperatures()
    st = torch.empty((R, n), dtype=torch.int32, device="cuda")
    en = torch.empty(R, dtype=torch.int64, device="cuda")
    tr = torch.zeros((S, 3, n), dtype=torch.int32, device="cuda")
    sa_run_noalloc(model.handle, make_params(rule="metropolis", n_sweeps=S, n_replicas=R, seed=4, t_max=tmax,
                                             t_min=tmin, flags=_lib.SA_FLAG_STATE_IN_GLOBAL, trace=tr,
                                             trace_replicas=3), st, en)
    torch.cuda.synchronize()
    res = om.run("metropolis", S, 4, tmax, tmin, r_begin=0, r_end=3, trace=tr.cpu().numpy(), trace_replicas=3)
    assert res["follow"]["mismatch"] == 0, res["follow"]
    assert np.array_equal(res["states"], st[:3].cpu().numpy())
    assert torch.equal(en, model.energy(st))


@pytest.mark.parametrize("lows", [(-2,), (-2, -1)])
def test_levels_with_more_changes_than_list_places(lows):
    """Levels of more than 256 variables that nearly all change: the lists that find
    no place are walked by their lanes, from compact records (one lower bound) and
    full ones (two), to the oracle's states."""
    from oracle import oracle as orc
    n, S, R = 1800, 4, 3
    rng = np.random.default_rng(8)
    lo = np.resize(np.asarray(lows), n)
    terms = [[k] for k in range(n)] + [sorted(rng.choice(n, 1 + int(rng.integers(1, 4)), replace=False))
                                       for _ in range(n // 2)]
    offs = np.concatenate([[0], np.cumsum([len(t) for t in terms])]).astype(np.int64)
    inst = {"n_vars": n, "lower": lo.astype(np.int64), "upper": (lo + 9).astype(np.int64), "term_offsets": offs,
            "term_vars": np.concatenate(terms).astype(np.int32),
            "coeffs": rng.integers(1, 6, len(terms)).astype(np.int32), "coef_type": "i32"}
    model, om = Model(inst), orc.Model(inst)
    later = {int(v) for t in terms for v in t[1:]}   # (members after a term's first have an earlier neighbour)
    assert n - len(later) > 512                      # variables of the first level
    for rule in ("metropolis", "opt_metropolis"):
        tr = torch.zeros((S, R, n), dtype=torch.int32, device="cuda")
        out = model.run(rule, S, R, seed=3, t_max=1e6, t_min=1e5, trace=tr, trace_replicas=R)
        res = om.run(rule, S, 3, 1e6, 1e5, r_begin=0, r_end=R, trace=tr.cpu().numpy(), trace_replicas=R)
        assert res["follow"]["mismatch"] == 0, res["follow"]
        assert np.array_equal(res["states"], out["states"].cpu().numpy())
        assert np.array_equal(res["energy"], out["energies"].cpu().numpy())


def test_a_model_holds_one_record_per_incidence():
    """Compact records: 16 bytes an incidence beside the term lists' 16 and 8 per
    term (at least two incidences); with full records it was 100 and more."""
    inst = wl.huio_zipf(1, n=2000, n_quad=8000, n_cubic=20_000, n_quartic=5000)
    lens = np.diff(inst["term_offsets"])
    incidences = int(lens[lens > 1].sum())
    assert Model(inst).info["device_bytes"] <= 36 * incidences + 200 * 2000 + (1 << 16)


def test_calls_of_two_threads_with_different_state_sizes():
    """Two host threads on streams of their own call the same kernels with 56 and
    200 KB of shared memory: neither call's limit may reach the other's launch."""
    import threading
    errors = []

    def work(n, n_states):
        try:
            model = Model(_banded(n, 4000))
            big = Model(_banded(n_states, 4000))
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                z = torch.ones((1300, n_states), dtype=torch.int32, device="cuda")
                want = model.run("metropolis", 1, 1, seed=1, threads_per_replica=32)["states"].clone()
                for _ in range(300):
                    got = model.run("metropolis", 1, 1, seed=1, threads_per_replica=32)["states"]
                    big.energy(z)
                stream.synchronize()
                assert torch.equal(got, want)
        except Exception as ex:   # (reported by the main thread)
            errors.append(ex)

    threads = [threading.Thread(target=work, args=a) for a in ((11_000, 14_000), (40_000, 50_000))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
