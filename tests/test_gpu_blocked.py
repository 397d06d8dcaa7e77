"""GPU tests of the sweep's blocked form, of HUIO incidence records and of the
energy kernel, at the sizes where they can go wrong.

Blocked sweeps (32 consecutive variables per warp) must give the states, change
counts, per-attempt traces and, at the same thread count, energies of the
level-by-level order, bit for bit; that order is checked against the oracle in
test_gpu_parity.py.  Energies are compared with numpy: exactly for integers, and
for floats within n_terms * 2^-53 of the sum of the terms' magnitudes, the
largest error that adding them in FP64 in any order can make.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as orc
from paper_2511_17245_gb300 import Model, _lib
from paper_2511_17245_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
RULES = ["metropolis", "heat_bath", "opt_metropolis"]


def _complete_float(n, width, seed=3):
    return wl.batch_instance({"index": 0, "n": n, "width": width, "dense": True, "deg": 0, "seed": seed})


def _wide(inst):
    """The same integer model with couplings beyond int32 (the blocks' int64 table)."""
    inst = dict(inst)
    inst["coeffs"] = inst["coeffs"].astype(np.int64) * ((1 << 33) + 12345)
    inst["coef_type"] = "i64"
    return inst


CASES = {
    # one block, its edges, two and three blocks, complete integer graphs
    **{f"complete_int_{n}": (lambda n=n: wl.quio_complete(n, n=n, lo=-8, hi=7)) for n in (2, 31, 32, 33, 64, 65, 97)},
    # enough threads for two deciding warps, ragged last block
    "complete_int_301": lambda: wl.quio_complete(1, n=301, lo=-30, hi=31),
    # fp32: one warp, two warps, narrow and wide heat-bath ranges
    "complete_float_33_w40": lambda: _complete_float(33, 40),
    "complete_float_130_w2": lambda: _complete_float(130, 2),
    "complete_float_257_w300": lambda: _complete_float(257, 300),
    # zero couplings: rows by columns; couplings beyond int32
    "dense_zeros_70": lambda: wl.quio_dense_small(9, n=70, lo=-3, hi=4),
    "dense_wide_coefficients_40": lambda: _wide(wl.quio_dense_small(4, n=40, lo=-8, hi=7)),
    # narrow levels that are not single variables, short and long rows
    "sparse_narrow_181": lambda: wl.quio_sparse_int(2, 181, 181 * 53 // 2, -20, 20),
    "chain_100": lambda: wl.quio_chain(5, n=100, lo=-30, hi=30, n_long=5),
}


@pytest.mark.parametrize("case", sorted(CASES))
@pytest.mark.parametrize("rule", RULES)
def test_blocks_equal_level_order(case, rule):
    model = Model(CASES[case]())
    S, R, n = 12, 9, model.n

    def run(**kw):
        tr = torch.zeros((S, R, n), dtype=torch.int32, device="cuda")
        out = model.run(rule, S, R, seed=7, trace=tr, trace_replicas=R, **kw)
        return {**out, "trace": tr}

    for tpr in (0, 32, 64, 128, 512):
        ref = run(flags=_lib.SA_FLAG_NO_SPECULATION, threads_per_replica=tpr)
        got = run(threads_per_replica=tpr)
        for key in ("states", "accepts", "trace", "energies"):
            assert torch.equal(ref[key], got[key]), (case, rule, tpr, key)
    # without traces the last block's changes of a sweep wait for the next one
    plain = model.run(rule, S, R, seed=7)
    assert torch.equal(plain["states"], run()["states"])
    glob = model.run(rule, S, R, seed=7, flags=_lib.SA_FLAG_STATE_IN_GLOBAL)
    assert torch.equal(plain["states"], glob["states"])


@pytest.mark.parametrize("lo,order,n", [(-3, 3, 40), ([-3, -2] * 20, 3, 40), (-1, 6, 24)])
def test_huio_incidence_records_follow_the_oracle(lo, order, n):
    """Multilinear terms of up to 4 members with one lower bound (compact
    records) and with two (full records), and terms of more than 4 members."""
    lo = np.broadcast_to(np.asarray(lo), (n,))
    inst = wl.random_small(5, n, order, lo, lo + 5, 6 * n, repeat=False, cmax=1 << 20)
    model, om = Model(inst), orc.Model(inst)
    tmax, tmin = om.auto_temperatures()
    for rule in RULES:
        S, R = 40, 6
        tr = torch.zeros((S, R, n), dtype=torch.int32, device="cuda")
        out = model.run(rule, S, R, seed=3, t_max=tmax, t_min=tmin, trace=tr, trace_replicas=R)
        res = om.run(rule, S, 3, tmax, tmin, r_begin=0, r_end=R, trace=tr.cpu().numpy(), trace_replicas=R)
        assert res["follow"]["mismatch"] == 0, res["follow"]
        assert np.array_equal(res["states"], out["states"].cpu().numpy())
        assert np.array_equal(res["energy"], out["energies"].cpu().numpy())


@pytest.mark.parametrize("scale", [1, (1 << 27) - 1, (1 << 33) + 7])
def test_carries_between_the_words_of_a_field(scale):
    """64-bit fields are updated word by word: couplings that fill the low word
    and reach into the high one, with both signs, end in the exact energies."""
    inst = wl.quio_sparse_int(11, 700, 5000, -40, 40)
    inst["coeffs"], inst["coef_type"] = inst["coeffs"].astype(np.int64) * scale, "i64"
    model = Model(inst)
    for flags in (0, _lib.SA_FLAG_STATE_IN_GLOBAL):
        out = model.run("metropolis", 30, 20, seed=1, flags=flags)
        assert torch.equal(out["energies"], model.energy(out["states"]))


@pytest.mark.parametrize("n,edges", [(2, 1), (40, 255), (40, 257), (300, 1025), (70, 2240), (70, 2241), (65536, 70000),
                                     (65537, 70000)])
@pytest.mark.parametrize("lo,hi", [(-1, 1), (0, 255), (-4095, 4095), (-4096, 4095)])
def test_energies_from_the_pair_list(n, edges, lo, hi):
    """Around the limits of the pair list (variables, values, row lengths), of a
    thread's four pairs and of the states per block."""
    inst = wl.quio_sparse_wide(5, n=n, n_edges=edges, lo=lo, hi=hi)
    model = Model(inst)
    c = inst["coeffs"].astype(np.float64)
    pairs = inst["term_vars"][3 * n:].reshape(-1, 2)
    for n_states in ((3,) if n > 1000 else (3, 1217)):
        states = wl.initial_states(4, inst, n_states)
        got = model.energy(torch.from_numpy(states).cuda()).cpu().numpy()
        z = states.astype(np.float64)
        terms = np.concatenate([z * c[:n], z * z * c[n:2 * n], z[:, pairs[:, 0]] * z[:, pairs[:, 1]] * c[2 * n:]], axis=1)
        bound = (terms.shape[1] + 4) * 2.0 ** -52 * np.abs(terms).sum(axis=1)
        assert np.all(np.abs(got - terms.sum(axis=1)) <= bound)


@pytest.mark.parametrize("n_states", [1, 5, 1215, 1216, 1219])
@pytest.mark.parametrize("lo,hi,coef", [(0, 255, "f32"), (-300, 300, "i32"), (-40, 90000, "f64"),
                                        (-(1 << 25), 1 << 25, "f64")])
def test_energies_by_state_width_and_count(n_states, lo, hi, coef):
    n, edges = 67, 300
    if coef == "i32":
        inst = wl.quio_sparse_int(3, n, edges, lo, hi)
    else:
        inst = wl.quio_sparse_wide(3, n=n, n_edges=edges, lo=lo, hi=hi, coef_type=coef)
    states = wl.initial_states(4, inst, n_states)
    got = Model(inst).energy(torch.from_numpy(states).cuda()).cpu().numpy()
    z = states.astype(np.int64 if coef == "i32" else np.float64)
    c = inst["coeffs"].astype(z.dtype)
    pairs = inst["term_vars"][3 * n:].reshape(-1, 2)
    terms = np.concatenate([z * c[:n], z * z * c[n:2 * n], z[:, pairs[:, 0]] * z[:, pairs[:, 1]] * c[2 * n:]], axis=1)
    if coef == "i32":
        assert np.array_equal(got, terms.sum(axis=1))
    else:
        bound = (terms.shape[1] + 4) * 2.0 ** -52 * np.abs(terms).sum(axis=1)
        assert np.all(np.abs(got - terms.sum(axis=1)) <= bound)
