"""The workloads that the library's speed is judged on, through its public entry points.

Every kind of call that a user makes is here: single runs of the three rules
on sparse, dense and complete QUIO and on HUIO with and without powers, with
integer and fp32 coefficients; an uneven batch; a mixed set of served
requests; and the energies of many states.  Shapes are those of the
generators in `paper_2511_17245_gb300.workloads` (the benchmark's sparse wide
model, the dense 32-variable model, the Zipf HUIO model, the paper's
random-interaction and multilinear models, the uneven batch and the request
stream), with fewer sweeps where a full anneal would take seconds: the
schedule still runs from the model's T_max to its T_min, so hot, accepting
sweeps and cold, rejecting ones are both present.

fp32 couplings of sparse models are rounded to multiples of 1/64, as instances
prepared for fixed-precision solvers are: sums of them are exact in fp32, so a
run of such a model gives the same states every time, whatever order the
concurrent updates of a field are added in.  Complete fp32 models, whose
fields have one writer at a time, keep Gaussian couplings.
"""
from __future__ import annotations

import numpy as np
import torch

import paper_2511_17245_gb300 as sa
from paper_2511_17245_gb300 import workloads as wl

RULES = ("metropolis", "heat_bath", "opt_metropolis")


def listed():
    return [
        # the smallest call: a short run of the dense 32-variable model, where
        # the host path and the launch are most of the time
        {"name": "dense32_short", "kind": "dense_int", "n": 32, "lo": -8, "hi": 7, "replicas": 64, "sweeps": 10,
         "rule": "metropolis"},
        # the same model's full 1000-sweep heat-bath anneal
        {"name": "dense32_heat_bath", "kind": "dense_int", "n": 32, "lo": -8, "hi": 7, "replicas": 64,
         "sweeps": 1000, "rule": "heat_bath"},
        # the benchmark model: 10,000 variables in [0, 255], mean degree 16,
        # 1024 replicas, more than the GPU holds at once
        {"name": "sparse_wide_metropolis", "kind": "sparse", "n": 10000, "degree": 16, "lo": 0, "hi": 255,
         "coef": "f32", "replicas": 1024, "sweeps": 60, "rule": "metropolis"},
        {"name": "sparse_wide_heat_bath", "kind": "sparse", "n": 10000, "degree": 16, "lo": 0, "hi": 255,
         "coef": "f32", "replicas": 1024, "sweeps": 40, "rule": "heat_bath"},
        # an ordinary sparse model of odd size, optimal-transition proposals
        {"name": "sparse_otm", "kind": "sparse", "n": 1501, "degree": 16, "lo": 0, "hi": 63, "coef": "f32",
         "replicas": 512, "sweeps": 100, "rule": "opt_metropolis"},
        # exact integer arithmetic over ranges of 601 values, ragged replicas
        {"name": "sparse_int_heat_bath", "kind": "sparse", "n": 3333, "degree": 9, "lo": -300, "hi": 300,
         "coef": "i32", "replicas": 333, "sweeps": 20, "rule": "heat_bath"},
        # HUIO with hub variables of thousands of terms
        {"name": "zipf_metropolis", "kind": "zipf", "n": 2000, "lo": -50, "hi": 50, "coef": "i32",
         "replicas": 256, "sweeps": 100, "rule": "metropolis"},
        # the paper's random-interaction model with powers up to 4: 1000 terms
        # on 100 variables over [-100, 100], 100 samples
        {"name": "powers_otm", "kind": "powers", "n": 100, "order": 4, "u": 100, "terms": 1000, "replicas": 100,
         "sweeps": 200, "rule": "opt_metropolis"},
        # a complete graph with Gaussian fp32 couplings: every change touches
        # every field
        {"name": "complete_metropolis", "kind": "complete", "n": 1000, "width": 300, "replicas": 152,
         "sweeps": 50, "rule": "metropolis"},
        # the uneven batch: dense and sparse instances of 50 to 2000 variables
        # in one launch
        {"name": "batch_uneven", "kind": "batch", "instances": 48, "n_min": 50, "n_max": 2000, "w_min": 2,
         "w_max": 1024, "replicas": 32, "sweeps": 40, "rule": "metropolis", "sizes": 3},
        # a closed loop of served requests of all rules and both model kinds
        {"name": "served_mix", "kind": "serve", "requests": 20, "n_min": 100, "n_max": 3000, "w_min": 2,
         "w_max": 1024, "s_min": 50, "s_max": 200, "replicas": 32, "sizes": 4},
        # energies of many states of the benchmark model
        {"name": "energies", "kind": "energy", "n": 10000, "degree": 16, "lo": 0, "hi": 255, "coef": "f32",
         "states": 4096},
    ]


def _log_int(rng, a, b):
    return int(round(float(a) * (float(b) / float(a)) ** rng.random()))


def draw(rng):
    """One more case: a kind, a rule and sizes spread over the ranges above; the
    sweep count is lowered where the call would cost more than the listed ones."""
    kind = rng.choice(["dense_int", "sparse", "sparse", "zipf", "powers", "complete", "batch", "serve", "energy"])
    rule = rng.choice(RULES)
    if kind == "dense_int":
        half = rng.choice([1, 3, 8, 40])
        c = {"kind": kind, "n": _log_int(rng, 16, 300), "lo": -half, "hi": half - rng.randrange(2),
             "replicas": _log_int(rng, 8, 400), "sweeps": _log_int(rng, 10, 1000), "rule": rule}
    elif kind == "sparse":
        coef = rng.choice(["f32", "i32"])
        hi = rng.choice([1, 15, 63, 255] if coef == "f32" else [1, 31, 255, 700])
        lo = 0 if coef == "f32" else -rng.randrange(0, hi + 1)
        c = {"kind": kind, "n": _log_int(rng, 300, 10000), "degree": rng.randrange(4, 25), "lo": lo, "hi": hi + lo,
             "coef": coef, "replicas": _log_int(rng, 32, 1024), "sweeps": _log_int(rng, 10, 200), "rule": rule}
    elif kind == "zipf":
        coef = rng.choice(["i32", "i32", "f32"])
        u = rng.choice([1, 4]) if coef == "f32" else rng.choice([1, 9, 50])
        c = {"kind": kind, "n": _log_int(rng, 200, 2000), "lo": -u, "hi": u, "coef": coef,
             "replicas": _log_int(rng, 16, 256), "sweeps": _log_int(rng, 10, 100), "rule": rule}
    elif kind == "powers":
        n = _log_int(rng, 40, 400)
        c = {"kind": kind, "n": n, "order": rng.randrange(2, 5), "u": rng.choice([1, 7, 30, 100]),
             "terms": 10 * n, "replicas": _log_int(rng, 16, 200), "sweeps": _log_int(rng, 10, 200), "rule": rule}
    elif kind == "complete":
        c = {"kind": kind, "n": _log_int(rng, 60, 1100), "width": _log_int(rng, 2, 1024),
             "replicas": _log_int(rng, 32, 304), "sweeps": _log_int(rng, 10, 50), "rule": rule}
    elif kind == "batch":
        c = {"kind": kind, "instances": _log_int(rng, 8, 48), "n_min": 50, "n_max": _log_int(rng, 300, 2000),
             "w_min": 2, "w_max": _log_int(rng, 16, 1024), "replicas": rng.choice([7, 16, 32]),
             "sweeps": _log_int(rng, 10, 40), "rule": rule, "sizes": rng.randrange(1 << 20)}
    elif kind == "serve":
        c = {"kind": kind, "requests": _log_int(rng, 2, 20), "n_min": 100, "n_max": _log_int(rng, 300, 3000),
             "w_min": 2, "w_max": _log_int(rng, 16, 1024), "s_min": 20, "s_max": 200, "replicas": rng.choice([8, 32]),
             "sizes": rng.randrange(1 << 20)}
    else:
        hi = rng.choice([1, 63, 255])
        c = {"kind": kind, "n": _log_int(rng, 300, 10000), "degree": rng.randrange(4, 25), "lo": 0, "hi": hi,
             "coef": rng.choice(["f32", "i32"]), "states": _log_int(rng, 16, 4096)}
    if "sweeps" in c:
        # full sweeps of a heat bath over wide ranges, dense couplings and hub
        # variables cost more per attempt than the work that they must do
        per = {"sparse": 6.1e8, "dense_int": 2.1e6, "zipf": 5.1e7, "powers": 2.0e6, "complete": 7.6e6,
               "batch": 3.0e7}[c["kind"]]
        if rule == "heat_bath":
            per /= 4.0
        cap = int(per / (_sites(c) * c["replicas"]))
        c["sweeps"] = max(1, min(c["sweeps"], cap))
    return c


def _sites(c):
    """Variables of a run, summed over a batch's instances (their mean size)."""
    if c["kind"] == "batch":
        return c["instances"] * (c["n_max"] - c["n_min"]) / np.log(c["n_max"] / c["n_min"])
    return c["n"]


# ------------------------------------------------------------------ inputs
def _quantised(inst):
    if inst["coef_type"] == "f32":
        for key in ("coeffs", "h", "J"):
            if key in inst:
                inst[key] = (np.round(inst[key].astype(np.float64) * 64.0) / 64.0).astype(np.float32)
    return inst


def _instance(c, seed):
    kind = c["kind"]
    if kind == "dense_int":
        return wl.quio_dense_small(seed, n=c["n"], lo=c["lo"], hi=c["hi"])
    if kind in ("sparse", "energy"):
        edges = c["n"] * c["degree"] // 2
        if c["coef"] == "i32":
            return wl.quio_sparse_int(seed, c["n"], edges, c["lo"], c["hi"])
        return _quantised(wl.quio_sparse_wide(seed, n=c["n"], n_edges=edges, lo=c["lo"], hi=c["hi"]))
    if kind == "zipf":
        n = c["n"]
        inst = wl.huio_zipf(seed, n=n, n_quad=4 * n, n_cubic=10 * n, n_quartic=5 * n // 2, lo=c["lo"], hi=c["hi"])
        if c["coef"] == "f32":     # whole-number couplings given in fp32
            inst["coeffs"], inst["coef_type"] = inst["coeffs"].astype(np.float32), "f32"
        return inst
    if kind == "powers":
        return wl.random_interaction(c["n"], c["order"], c["u"], n_terms=c["terms"], seed=seed, integer=True,
                                     int_scale=50)
    if kind == "complete":
        return wl.batch_instance({"index": 0, "n": c["n"], "width": c["width"], "dense": True, "deg": 0,
                                  "seed": seed})
    raise ValueError(kind)


def _specs(c, seed):
    """The instances' or requests' sizes (the case's own) with couplings of `seed`."""
    if c["kind"] == "batch":
        specs = wl.batch_specs(c["sizes"], c["instances"], c["n_min"], c["n_max"], c["w_min"], c["w_max"])
    else:
        specs = wl.serving_specs(c["sizes"], c["requests"], c["n_min"], c["n_max"], c["w_min"], c["w_max"],
                                 c["s_min"], c["s_max"], c["replicas"])
        for s in specs:
            s["int"] = True   # exact models: results do not depend on what else is running
            if s["huio"]:     # products of four values stay far inside int64
                s["width"] = min(s["width"], 256)
    for s in specs:
        s["seed"] = (s["seed"] + 7919 * seed) % (1 << 31)
    return specs


class _Batch:
    """Models, batch handle and output tensors, as a program that repeats a batch keeps them."""

    def __init__(self, c, seed):
        specs = _specs(c, seed)
        self.models = []
        for s in specs:
            inst = wl.batch_instance(s)
            self.models.append(sa.Model(inst if s["dense"] else _quantised(inst)))
        R = c["replicas"]
        params = [sa.make_params(rule=c["rule"], n_sweeps=c["sweeps"], n_replicas=R, seed=seed, instance_id=i)
                  for i in range(len(specs))]
        self.handle = sa.sa_batch_create([m.handle for m in self.models], params)
        self.at = np.concatenate([[0], np.cumsum([R * m.n for m in self.models])])
        self.R = R

    def run(self):
        st = torch.cuda.current_stream().cuda_stream
        k = len(self.models)
        states = torch.empty(int(self.at[-1]), dtype=torch.int32, device="cuda")
        energies = torch.empty((k, self.R), dtype=torch.float64, device="cuda")
        accepts = torch.empty((k, self.R), dtype=torch.int64, device="cuda")
        sa.sa_batch_run(self.handle, st)
        for i in range(k):
            sa.sa_batch_result(self.handle, i, states[int(self.at[i]):], energies[i], accepts[i], st)
        return {"states": states, "energies": energies, "accepts": accepts}

    def __del__(self):
        if getattr(self, "handle", None):
            sa.sa_batch_destroy(self.handle)


class _Served:
    """A server and the models of its requests, as a serving program keeps them."""

    def __init__(self, c, seed):
        specs = _specs(c, seed)
        self.models, self.params, self.bufs = [], [], []
        for i, s in enumerate(specs):
            m = sa.Model(wl.serving_instance(s))
            self.models.append(m)
            self.params.append(sa.make_params(rule=s["rule"], n_sweeps=s["sweeps"], n_replicas=s["replicas"],
                                              seed=seed, instance_id=i))
            self.bufs.append([np.empty((s["replicas"], m.n), np.int32), np.empty(s["replicas"], np.int64),
                              np.empty(s["replicas"], np.uint64)])
        self.handle = sa.sa_server_create(budget_bytes=1 << 32, max_running=256)

    def run(self):
        tickets = [sa.sa_server_submit(self.handle, m.handle, p) for m, p in zip(self.models, self.params)]
        for t, (s, e, a) in zip(tickets, self.bufs):
            sa.sa_server_wait(self.handle, t, 60_000_000)
            sa.sa_server_result(self.handle, t, s, e, a)
        return {"states": [b[0] for b in self.bufs], "energies": np.stack([b[1] for b in self.bufs]),
                "accepts": np.stack([b[2] for b in self.bufs]).astype(np.int64)}

    def __del__(self):
        if getattr(self, "handle", None):
            sa.sa_server_destroy(self.handle)


def _random_states(inst, count, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    lo, hi = int(inst["lower"][0]), int(inst["upper"][0])
    return torch.randint(lo, hi + 1, (count, inst["n_vars"]), generator=g, device="cuda", dtype=torch.int32)


def prepare(case, seed):
    c = case
    if c["kind"] == "batch":
        return {"case": c, "job": _Batch(c, seed)}
    if c["kind"] == "serve":
        return {"case": c, "job": _Served(c, seed)}
    inst = _instance(c, seed)
    state = {"case": c, "seed": seed, "model": sa.Model(inst)}
    if c["kind"] == "energy":
        state["states"] = _random_states(inst, c["states"], seed)
    return state


def run(state):
    c = state["case"]
    if "job" in state:
        return state["job"].run()
    if c["kind"] == "energy":
        return {"energies": state["model"].energy(state["states"])}
    return state["model"].run(rule=c["rule"], n_sweeps=c["sweeps"], n_replicas=c["replicas"], seed=state["seed"])


# ------------------------------------------------------------------ floors
def _values(c):
    """Values of a variable's range."""
    if c["kind"] == "powers":
        return 2 * c["u"] + 1
    if "width" in c:
        return c["width"]
    return c["hi"] - c["lo"] + 1


def work(case):
    """Bytes: the model read once, the outputs (states, energies, counts) written
    once.  Operations: per attempt the energy change of a proposal and its
    acceptance (about 8), or the weight of every value of the range (5 each) for
    the heat bath; the updates after accepted changes, whose number depends on
    the run, are left out."""
    c = case
    if c["kind"] == "energy":
        links = c["n"] * c["degree"] // 2
        return {"bytes": 4.0 * c["states"] * c["n"] + 8.0 * c["states"] + 12.0 * links + 8.0 * c["n"],
                "flops": c["states"] * (3.0 * links + 4.0 * c["n"])}
    if c["kind"] == "serve":
        specs = _specs(c, 0)
        att = float(sum(s["n"] * s["sweeps"] * s["replicas"] for s in specs))
        out = float(sum(s["n"] * s["replicas"] for s in specs))
        return {"bytes": 4.0 * out + 16.0 * sum(s["n"] * s["deg"] for s in specs), "flops": 8.0 * att}
    sites = float(_sites(c))
    per = 8.0
    if c["rule"] == "heat_bath" and c["kind"] != "zipf":     # (multilinear models use the closed form)
        per = 5.0 * (c["w_max"] / np.log(c["w_max"] / c["w_min"]) if c["kind"] == "batch" else _values(c))
    links = {"dense_int": 12.0 * sites * sites, "complete": 4.0 * sites * sites,
             "sparse": 8.0 * sites * c.get("degree", 0), "zipf": 16.5 * 12.0 * sites,
             "powers": 12.0 * c.get("terms", 0) * c.get("order", 0),
             "batch": 2.0 * sites * c.get("n_max", 0)}[c["kind"]]
    return {"bytes": links + 4.0 * sites * c["replicas"] + 16.0 * c["replicas"],
            "flops": per * sites * c["replicas"] * c["sweeps"]}


def exact(case, seed):
    """Energies in 64 bits from the definition.  A run's outputs are the end of a
    random trajectory: no formula gives them."""
    c = case
    if c["kind"] != "energy":
        return None
    inst = _instance(c, seed)
    if c["coef"] == "i32":
        return None     # whole numbers: compared bit for bit
    z = _random_states(inst, c["states"], seed).double()
    n, edges = c["n"], c["n"] * c["degree"] // 2
    co = torch.from_numpy(inst["coeffs"].astype(np.float64)).cuda()
    pairs = torch.from_numpy(inst["term_vars"][3 * n:].astype(np.int64)).cuda().view(edges, 2)
    e = z @ co[:n] + (z * z) @ co[n:2 * n]
    for a in range(0, edges, 4000):
        p, w = pairs[a:a + 4000], co[2 * n + a:2 * n + a + 4000]
        e += (z[:, p[:, 0]] * z[:, p[:, 1]]) @ w
    return {"energies": e}
