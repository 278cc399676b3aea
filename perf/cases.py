"""The work a user of this library has it do, as cases to time.

Every case calls the public entry points of paper_1804_02867_gb300.efmgraph
on seeded networks.  A case fixes the network's shape and the limits; the
seed of prepare() permutes the order in which the network lists its
reactions (as two files of one model would), so every seed gives other
arrays and other supports for the same amount of work: the traversal's
choices depend on metabolites only, never on the order of the reactions.

Kinds of case
  paths     traversals of a loaded network: the supports and counters of
            every target (or of one seed set), fetched to the host
  query     one whole query from a model's arrays: load the network, find
            the pathways of one target, fetch them, take their flux vectors
  batch     many uneven networks in one launch, every result fetched
  walks     Monte-Carlo walks
  gradient  loss and gradient of the proposal model over its training rows
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1804_02867_gb300 import efmgraph, synth

# genome targets whose 1000 smallest pathways lie within a 2^20 frontier
# budget: a first-K answer is exact there, whatever the order of the search
FIRSTK_TARGETS = (924, 572, 319, 823, 907, 301, 976, 154, 128, 673, 35, 232, 653, 992, 248, 967)

# reaction pairs of the core network that pathways run through
SEED_RXN = ("74 27", "70 61", "65 62", "11 92", "90 77", "40 78")


def listed():
    return [
        # the smallest call: a 12 x 16 network, one target, default budget -- a
        # notebook or a unit test; latency and launches
        dict(name="tiny", kind="paths", net="tiny", n_targets=1, max_len=12, max_sec=2, budget=0),
        # an interactive question about a core model, from its arrays to flux vectors
        dict(name="core-query", kind="query", net="core", target=1, max_len=15, max_sec=4, budget=1 << 20),
        # all targets of a core model under a modest budget: a parameter scan's step
        dict(name="core-scan", kind="paths", net="core", n_targets=8, max_len=30, max_sec=4, budget=1 << 17),
        # the same under the benchmark's budget: the exhaustive run
        dict(name="core-full", kind="paths", net="core", n_targets=8, max_len=30, max_sec=4, budget=1 << 26),
        # pathways through two given reactions (Prop. 1 seed set), an odd budget
        dict(name="core-seedset", kind="paths", net="core", seed_rxn="74 27", max_len=29, max_sec=3, budget=1_500_007),
        # Eq. 5 steps on a core model: rows that carry the flux vector
        dict(name="core-subtractive", kind="paths", net="core", n_targets=4, max_len=24, max_sec=2, budget=1 << 17,
             variant=1),
        # a mid-size network (400 internal metabolites), every target
        dict(name="mid-400", kind="paths", net="mid400", n_targets=6, max_len=40, max_sec=4, budget=1 << 17),
        # genome-scale enumeration at the benchmark's budget
        dict(name="genome", kind="paths", net="genome", n_targets=4, max_len=40, max_sec=4, budget=1 << 22),
        # the thousand smallest pathways of genome targets, arena order
        dict(name="genome-firstk", kind="paths", net="genome", targets="572 319 301", max_len=40, max_sec=4,
             budget=1 << 22, first_k=1000),
        # 512 uneven networks in one launch (a screening run)
        dict(name="batch-512", kind="batch", jobs=512, first=0, max_len=30, max_sec=4, budget=1 << 12),
        # random walks, the paper's own method
        dict(name="walks", kind="walks", net="core", target=3, max_len=30, max_sec=4, walks=1 << 20),
        # one full-batch gradient of the proposal model
        dict(name="model-gradient", kind="gradient", rows=100_003, pos_weight=4.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tiny", "core", "core", "core", "seedset", "subtractive", "mid", "genome", "genome", "firstk",
                       "firstk", "query", "batch", "batch", "walks", "gradient"])
    sec = rng.randint(1, 4)
    if kind == "tiny":
        return dict(kind="paths", net="tiny", n_targets=rng.randint(1, 4), max_len=rng.randint(6, 16), max_sec=sec,
                    budget=_log(rng, 1 << 10, 1 << 22))
    if kind == "core":
        return dict(kind="paths", net="core", n_targets=rng.randint(1, 8), max_len=rng.randint(12, 34), max_sec=sec,
                    budget=_log(rng, 1 << 13, 1 << 24))
    if kind == "seedset":
        return dict(kind="paths", net="core", seed_rxn=rng.choice(SEED_RXN), max_len=rng.randint(16, 34), max_sec=sec,
                    budget=_log(rng, 1 << 13, 1 << 23))
    if kind == "subtractive":
        return dict(kind="paths", net="core", n_targets=rng.randint(1, 6), max_len=rng.randint(12, 30), max_sec=sec,
                    budget=_log(rng, 1 << 12, 1 << 18), variant=1)
    if kind == "mid":
        return dict(kind="paths", net=rng.choice(["mid200", "mid400"]), n_targets=rng.randint(1, 6),
                    max_len=rng.randint(20, 40), max_sec=sec, budget=_log(rng, 1 << 12, 1 << 19))
    if kind == "genome":
        return dict(kind="paths", net="genome", n_targets=rng.randint(1, 4), max_len=rng.randint(20, 40), max_sec=sec,
                    budget=_log(rng, 1 << 14, 1 << 22))
    if kind == "firstk":
        return dict(kind="paths", net="genome", targets=str(rng.choice(FIRSTK_TARGETS)), max_len=40, max_sec=4,
                    budget=1 << 22, first_k=_log(rng, 20, 1000), learned=rng.random() < 0.5)
    if kind == "query":
        return dict(kind="query", net=rng.choice(["core", "mid200"]), target=rng.randint(0, 5),
                    max_len=rng.randint(10, 18), max_sec=sec, budget=_log(rng, 1 << 13, 1 << 18))
    if kind == "batch":
        return dict(kind="batch", jobs=_log(rng, 16, 512), first=rng.randint(0, 64), max_len=rng.randint(16, 34),
                    max_sec=sec, budget=_log(rng, 1 << 8, 1 << 12))
    if kind == "walks":
        return dict(kind="walks", net=rng.choice(["core", "mid200", "genome"]), target=rng.randint(0, 5),
                    max_len=rng.randint(12, 40), max_sec=sec, walks=_log(rng, 1 << 10, 1 << 18))
    return dict(kind="gradient", rows=_log(rng, 1000, 150_000), pos_weight=float(rng.randint(1, 20)))


# --- networks -----------------------------------------------------------------

@functools.lru_cache(maxsize=None)
def _network(name):
    if name == "tiny":
        return synth.tiny(3)
    if name == "core":
        return synth.core()
    if name == "genome":
        return synth.genome()
    n_int = int(name[3:])
    shape = {200: dict(n_targets=6, n_hubs=6, n_substrates=2, n_rxn=500, n_rev=100, hub_degree=(40, 100)),
             400: dict(n_targets=6, n_hubs=10, n_substrates=3, n_rxn=1000, n_rev=250, hub_degree=(80, 200))}[n_int]
    return synth.generate(n_int=n_int, size_range=(2, 6), coef_probs=synth.CORE_COEFS, gamma=2.2,
                          seed=5_000_000 + n_int, name=name, **shape)


@functools.lru_cache(maxsize=None)
def _member(i):
    return synth.batched_member(i)


def _permuted(net, rng):
    """The same network with its reactions listed in another order, and the map from old to new reaction index."""
    perm = rng.permutation(net.n_rxn).astype(np.int32)
    col = perm[net.col_idx]
    row = np.repeat(np.arange(net.n_met), np.diff(net.row_ptr))
    order = np.lexsort((col, row))
    rev = np.empty_like(net.reversible)
    rev[perm] = net.reversible
    return synth.Network(net.n_met, net.n_rxn, net.row_ptr, np.ascontiguousarray(col[order]),
                         np.ascontiguousarray(net.coef[order]), rev, net.external, list(net.targets), net.name), perm


class _Handles:
    """The library handles a program keeps, released with the state."""

    def __init__(self):
        self.nets, self.models = [], []

    def __del__(self):
        for n in self.nets:
            n.close()
        for m in self.models:
            efmgraph.efm_model_free(m)


# --- the contract ---------------------------------------------------------------

def prepare(case, seed):
    rng = np.random.default_rng(seed)
    keep = _Handles()
    kind = case["kind"]
    if kind == "gradient":
        x, y, params = _training_set(case, seed)
        m = efmgraph.efm_model_create(seed)
        keep.models.append(m)
        efmgraph.efm_model_params(m, params)
        efmgraph.efm_model_add_rows(m, x, y)
        return case, keep, m, None
    if kind == "batch":
        nets = [_permuted(_member(case["first"] + i), rng)[0] for i in range(case["jobs"])]
        keep.nets = [efmgraph.Network(n) for n in nets]
        return case, keep, [n.handle for n in keep.nets], [n.targets[0] for n in nets]
    net, perm = _permuted(_network(case["net"]), rng)
    if kind == "query":
        return case, keep, net, net.targets[case["target"]]
    nw = efmgraph.Network(net)
    keep.nets.append(nw)
    if kind == "walks":
        return case, keep, nw, (net.targets[case["target"]], seed)
    if "seed_rxn" in case:
        # the seed set: forward columns of reactions, named as the unpermuted model names them
        rxn, direction = efmgraph.efm_column_map(nw.handle)
        cols = [int(np.nonzero((rxn == perm[int(r)]) & (direction == 1))[0][0]) for r in case["seed_rxn"].split()]
        return case, keep, nw, cols
    model = None
    if case.get("learned"):
        model = efmgraph.efm_model_create(seed)
        keep.models.append(model)
    targets = [int(t) for t in case["targets"].split()] if "targets" in case else net.targets[:case["n_targets"]]
    return case, keep, nw, (targets, model)


def _ints(sup):
    return sup.view(np.int64)


def _row(ctr):
    return np.array([ctr[f] for f in efmgraph.COUNTER_FIELDS], dtype=np.int64)


def run(state):
    case, keep, a, b = state
    kind = case["kind"]
    if kind == "gradient":
        grad, loss = efmgraph.efm_model_gradient(a, case["pos_weight"])
        return {"grad": grad, "loss": np.float32(loss)}
    if kind == "batch":
        job, _ = efmgraph.efm_find_pathways_batch(a, b, case["max_len"], case["max_sec"], 0, case["budget"])
        try:
            got = [efmgraph.efm_fetch_results(job, i) for i in range(len(a))]
        finally:
            efmgraph.efm_free_job(job)
        return {"supports": np.concatenate([_ints(s).ravel() for s, _, _ in got]),
                "counts": np.array([len(s) for s, _, _ in got], dtype=np.int64),
                "counters": np.stack([_row(c) for _, c, _ in got])}
    if kind == "walks":
        target, seed = b
        sup, ctr = efmgraph.sample_target(a, target, case["max_len"], case["max_sec"], seed, case["walks"])
        return {"supports": _ints(sup), "counters": _row(ctr)}
    if kind == "query":
        with efmgraph.Network(a) as nw:
            (sup, ctr), = efmgraph.enumerate_targets(nw, [b], case["max_len"], case["max_sec"], 0, case["budget"])
            flux, status = efmgraph.efm_flux_vectors(nw.handle, sup)
            rxn, _ = efmgraph.efm_column_map(nw.handle)
        return {"supports": _ints(sup), "counters": _row(ctr), "flux": flux, "flux_status": status, "reactions": rxn}
    # the column map is what a program reads supports with
    rxn, _ = efmgraph.efm_column_map(a.handle)
    if isinstance(b, list):
        sup, ctr = efmgraph.enumerate_from(a, b, case["max_len"], case["max_sec"], 0, case["budget"])
        return {"supports": _ints(sup), "counters": _row(ctr), "reactions": rxn}
    targets, model = b
    k = case.get("first_k", 0)
    got = efmgraph.enumerate_targets(a, targets, case["max_len"], case["max_sec"], 0, case["budget"], first_k=k,
                                     proposal=efmgraph.EFM_LEARNED if model else efmgraph.EFM_PLAIN, model=model,
                                     variant=case.get("variant", 0))
    # a first-K search's work counters depend on the order in which results
    # arrive; its answer and status do not
    return {"pathways": [{"supports": _ints(s), "counters": np.int64(c["status"]) if k else _row(c)} for s, c in got],
            "reactions": rxn}


# Columns, internal rows, and what a state holds at the least: its support, one
# bit a column, and the few unbalanced rows (a row index and a value each).
_SHAPE = {"tiny": (20, 8, 3), "core": (114, 58, 10), "mid200": (600, 200, 9), "mid400": (1250, 400, 9),
          "genome": (3125, 850, 12), "member": (130, 52, 9)}


def work(case):
    """Bytes: every state of the search written once and read once (in the
    smallest exact form: support bits and the unbalanced rows).  Operations:
    one multiply-add per unbalanced row of every child."""
    kind = case["kind"]
    if kind == "gradient":
        n = case["rows"]
        return {"bytes": n * (2 * 128 + 4) + 2 * 4 * (256 * 128 + 257), "flops": 2 * 2 * n * 128 * 256}
    if kind == "walks":
        N, M, nz = _SHAPE[case["net"]]
        steps = min(20, case["max_len"])
        return {"bytes": 24 * N, "flops": 2.0 * case["walks"] * steps * M}
    if kind == "batch":
        N, M, nz = _SHAPE["member"]
        children = case["jobs"] * 3.0 * case["budget"]
    else:
        N, M, nz = _SHAPE[case["net"]]
        n_t = len(case["targets"].split()) if "targets" in case else max(1, case.get("n_targets", 1))
        budget = case["budget"] or 4096
        # a search ends a few levels after its frontier nears the budget, or runs out of length before
        grow = min(4.0 * budget, 2.0 ** case["max_len"] * 2) if case["net"] in ("tiny", "core") else 3.0 * budget
        children = n_t * (min(grow, 2000.0) if case["net"] == "tiny" else grow)
    state = N / 8 + 6 * nz
    return {"bytes": 2 * children * state, "flops": 2.0 * children * nz}


def _training_set(case, seed):
    """Rows of the model's feature kind: small fractions, a constant 1, a hashed embedding of a support; parameters as
    a partly trained model has them.  All values are exact in BF16, so that the product inputs are the same for
    everyone."""
    g = torch.Generator().manual_seed(int(seed) & 0x7FFFFFFF)
    n = case["rows"]
    x = torch.rand((n, 128), generator=g)
    x[:, 15:64] = 0.0
    size = torch.randint(4, 30, (n, 1), generator=g).float()
    bits = torch.randint(-2, 3, (n, 64), generator=g).float()
    x[:, 64:] = bits * (torch.rand((n, 64), generator=g) < 0.4) / size.sqrt()
    x[:, 10] = 1.0
    x = x.to(torch.bfloat16).float()
    w1 = (torch.rand((256, 128), generator=g) * 2 - 1) * math.sqrt(6 / 128)
    w2 = (torch.rand(256, generator=g) * 2 - 1) * math.sqrt(3 / 256)
    params = torch.cat([w1.to(torch.bfloat16).float().ravel(), w2, torch.full((1,), -0.25)])
    y = (torch.rand(n, generator=g) < 0.2).float()
    return x.numpy(), y.numpy(), params.numpy()


def exact(case, seed):
    """Every output but the gradient's is whole numbers."""
    if case["kind"] != "gradient":
        return None
    x, y, params = (torch.from_numpy(a).double() for a in _training_set(case, seed))
    w1, w2, b2 = params[:256 * 128].view(256, 128), params[256 * 128:-1], params[-1]
    h = x @ w1.T
    a = h.clamp(min=0)
    s = a @ w2 + b2
    wt = torch.where(y > 0.5, case["pos_weight"], 1.0)
    n = len(y)
    loss = (wt * (torch.nn.functional.softplus(s) - y * s)).sum() / n
    ds = wt * (torch.sigmoid(s) - y) / n
    dh = ds[:, None] * w2 * (h > 0)
    grad = torch.cat([(dh.T @ x).ravel(), a.T @ ds, ds.sum()[None]])
    return {"grad": grad.numpy(), "loss": np.float64(loss)}
