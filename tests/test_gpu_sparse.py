"""Sparse states of the level pass: sizes where the layout's edges lie.

* dense reactions (20-60 metabolites each): a state's entries exceed what the
  payload pool holds per row, so levels are run again with a larger pool;
* coefficients whose rows share divisors (the entries are divided);
* column lists that end at and around a 16-byte unit (4, 12, 20 columns),
  reached by budgets that stop at different depths.

Supports and every counter must equal the oracle's.
"""
import numpy as np
import pytest

from paper_1804_02867_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def efm():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_02867_gb300 import build, efmgraph

    build.build()
    efmgraph.load_library()
    return efmgraph


def check(oracle_lib, efm, net, targets, max_len, max_sec, budget, **kw):
    with efm.Network(net) as nw:
        got = efm.enumerate_targets(nw, targets, max_len, max_sec, 0, budget, **kw)
    out = []
    for t, (sup, ctr) in zip(targets, got):
        osup, octr = oracle_lib.enumerate_pathways(net, t, oracle_lib.Limits(max_len, max_sec, 0, budget))
        assert np.array_equal(sup, osup), (net.name, t, budget)
        assert ctr == octr, (net.name, t, budget, ctr, octr)
        out.append(ctr)
    return out


@pytest.mark.parametrize("size_range,budget", [((20, 60), 1 << 10), ((20, 60), 1 << 13), ((6, 14), 1 << 12)])
def test_dense_reactions(oracle_lib, efm, size_range, budget):
    net = synth.generate(n_int=100, n_targets=3, n_hubs=3, n_substrates=2, n_rxn=160, n_rev=40, size_range=size_range,
                         coef_probs={1: 0.5, 2: 0.3, 3: 0.2}, gamma=None, hub_degree=(5, 20), seed=77,
                         name=f"dense-{size_range[1]}")
    out = check(oracle_lib, efm, net, net.targets, 24, 2, budget)
    assert any(c["frontier_max"] > 100 for c in out)


@pytest.mark.parametrize("max_len", [3, 4, 5, 12, 13, 20, 21])
def test_list_unit_edges(oracle_lib, efm, max_len):
    """A chain-like network (few branches) whose supports grow to max_len."""
    net = synth.generate(n_int=70, n_targets=2, n_hubs=2, n_substrates=2, n_rxn=90, n_rev=20, size_range=(2, 3),
                         coef_probs={1: 0.4, 2: 0.4, 4: 0.2}, gamma=None, hub_degree=(5, 20), seed=91, name="chainlike")
    check(oracle_lib, efm, net, net.targets + [-1], max_len, 3, 1 << 12)


@pytest.mark.parametrize("max_results", [1, 50])
def test_capped(oracle_lib, efm, max_results):
    net = synth.generate(n_int=120, n_targets=2, n_hubs=3, n_substrates=2, n_rxn=300, n_rev=60, size_range=(2, 5),
                         coef_probs=synth.CORE_COEFS, gamma=2.2, hub_degree=(20, 60), seed=5, name="mid-120")
    with efm.Network(net) as nw:
        got = efm.enumerate_targets(nw, net.targets, 20, 2, max_results, 1 << 14)
    for t, (sup, ctr) in zip(net.targets, got):
        osup, octr = oracle_lib.enumerate_pathways(net, t, oracle_lib.Limits(20, 2, max_results, 1 << 14))
        assert np.array_equal(sup, osup) and ctr == octr, (t, ctr, octr)


EDGES = {
    # narrow form: long columns (past the eight a lane keeps), divisors, int32 left
    "narrow": dict(n_int=40, n_rxn=70, n_rev=15, size_range=(2, 14), coef_probs={1: 0.3, 6: 0.3, 10: 0.3, 524287: 0.1}),
    # 64 rows, 128 columns: the last narrow network
    "narrow-last": dict(n_int=64, n_rxn=104, n_rev=24, size_range=(2, 5), coef_probs={1: 0.6, 2: 0.2, 4: 0.2}),
    # one row, one column more: the next two forms
    "bits": dict(n_int=65, n_rxn=104, n_rev=24, size_range=(2, 5), coef_probs={1: 0.6, 2: 0.2, 4: 0.2}),
    "list": dict(n_int=64, n_rxn=105, n_rev=24, size_range=(2, 5), coef_probs={1: 0.6, 2: 0.2, 4: 0.2}),
    # one support word
    "one-word": dict(n_int=30, n_rxn=50, n_rev=10, size_range=(2, 5), coef_probs={1: 0.5, 3: 0.5}),
}


def edge_network(name):
    return synth.generate(n_targets=3, n_hubs=2, n_substrates=2, gamma=None, hub_degree=(3, 10), seed=11, name=name,
                          **EDGES[name])


@pytest.mark.parametrize("name", sorted(EDGES))
def test_forms(oracle_lib, efm, name):
    net = edge_network(name)
    out = check(oracle_lib, efm, net, net.targets + [-1], 16, 3, 1 << 13)
    if name == "narrow":
        assert any(c["overflow"] for c in out)
    with efm.Network(net) as nw:
        for t in net.targets:
            (got, _), = efm.enumerate_targets(nw, [t], 9, 2, 0, 1 << 16, first_k=5)
            want, _ = oracle_lib.first_k(net, t, 5, 9, 2)
            assert np.array_equal(got, want), (name, t)


@pytest.mark.parametrize("name", ["narrow", "narrow-last", "one-word"])
def test_lane_walks(oracle_lib, efm, name):
    """A walk per lane: divisions, int32 left, both support words."""
    net = edge_network(name)
    with efm.Network(net) as nw:
        for t in net.targets + [-1]:
            for n in (1, 33, 4000):
                sup, ctr = efm.sample_target(nw, t, 20, 3, 5, n)
                osup, octr = oracle_lib.sample_pathways(net, t, oracle_lib.Limits(20, 3), 5, n)
                assert np.array_equal(sup, osup) and ctr == octr, (name, t, n, ctr, octr)


@pytest.mark.parametrize("name,n", [("one-word", 10000), ("one-word", 12000), ("narrow-last", 5000),
                                    ("narrow-last", 6000), ("narrow", 16000), ("narrow", 18000)])
def test_walk_kernels(oracle_lib, efm, name, n):
    """A warp per walk below the line and a lane per walk above it (152 SMs):
    one and two rows a lane, short and long columns."""
    net = edge_network(name)
    with efm.Network(net) as nw:
        for t in net.targets[:2] + [-1]:
            sup, ctr = efm.sample_target(nw, t, 20, 3, 5, n)
            osup, octr = oracle_lib.sample_pathways(net, t, oracle_lib.Limits(20, 3), 5, n)
            assert np.array_equal(sup, osup) and ctr == octr, (t, ctr, octr)


@pytest.mark.parametrize("budget", [2**6, 2**10, 2**14])
def test_batch_slices(efm, budget):
    # levels that outgrow a job's slice are run alone; the rows come back in
    # one copy: counters and rows equal single calls' at every budget
    nets = [synth.batched_member(20 + i) for i in range(64)] + [synth.core()]
    loaded = [efm.Network(n) for n in nets]
    try:
        targets = [n.targets[0] for n in nets]
        job, _ = efm.efm_find_pathways_batch([w.handle for w in loaded], targets, 24, 3, 0, budget)
        try:
            got = [efm.efm_fetch_results(job, i) for i in range(len(nets))]
        finally:
            efm.efm_free_job(job)
        for net, w, target, (sup, ctr, _) in zip(nets, loaded, targets, got):
            (ssup, sctr), = efm.enumerate_targets(w, [target], 24, 3, 0, budget)
            assert np.array_equal(sup, ssup) and ctr == sctr, net.name
    finally:
        for w in loaded:
            w.close()


def ladder(steps, sides):
    """steps rungs from one external metabolite to another, each carrying
    1 + sides internal metabolites on; two reactions have twins with two and
    three times their coefficients, so there are four pathways."""
    n_int = steps * (1 + sides)
    rxn = [[(n_int, -1)] + [(s, 1) for s in range(1 + sides)]]
    for i in range(1, steps):
        a, b = (i - 1) * (1 + sides), i * (1 + sides)
        rxn.append([(a + s, -1 - s % 2) for s in range(1 + sides)] + [(b + s, 1 + s % 2) for s in range(1 + sides)])
    a = (steps - 1) * (1 + sides)
    rxn.append([(a + s, -1) for s in range(1 + sides)] + [(n_int + 1, 1)])
    rxn[0] = [(m, v * (1 if m == n_int else 1 + m % (1 + sides) % 2)) for m, v in rxn[0]]
    rxn[-1] = [(m, v * (1 if m == n_int + 1 else 1 + (m - a) % 2)) for m, v in rxn[-1]]
    rxn.append([(m, 3 * v) for m, v in rxn[steps // 2]])
    rxn.append([(m, 2 * v) for m, v in rxn[steps // 3]])
    S = np.zeros((n_int + 2, len(rxn)), dtype=np.int64)
    for j, ents in enumerate(rxn):
        for m, v in ents:
            S[m, j] = v
    external = [0] * n_int + [1, 1]
    return synth.Network.from_dense(S, [0] * len(rxn), external, [n_int + 1], f"ladder-{steps}-{sides}")


@pytest.mark.parametrize("steps,sides", [(31, 0), (32, 0), (33, 0), (32, 1), (13, 4), (63, 0), (61, 1), (2, 40)])
def test_rank_rows(oracle_lib, efm, steps, sides):
    # the minimality test at 31 to 33, 64, 65 and 122 rows, and at 64 columns
    net = ladder(steps, sides)
    out = check(oracle_lib, efm, net, net.targets, min(64, steps + 2), 2, 1 << 12)
    assert out[0]["results"] >= 4


@pytest.mark.parametrize("budget", [1, 30, 500, 1024, 1025, 3000])
def test_small_levels(oracle_lib, efm, budget):
    # searches that end, are cut or are capped at levels of one CTA and just
    # past them, from few seeds and from many
    for net in (synth.core(), edge_network("list"), synth.batched_member(3)):
        check(oracle_lib, efm, net, [net.targets[0], -1], min(12, net.split_columns()), 2, budget)
    net = edge_network("bits")
    with efm.Network(net) as nw:
        for cap in (1, 3):
            (sup, ctr), = efm.enumerate_targets(nw, [net.targets[0]], 12, 2, cap, budget)
            osup, octr = oracle_lib.enumerate_pathways(net, net.targets[0], oracle_lib.Limits(12, 2, cap, budget))
            assert np.array_equal(sup, osup) and ctr == octr, (cap, ctr, octr)


LONG = {
    # columns past the 8 entries of a narrow lane; with common divisors; leaving int32
    "narrow": dict(n_int=60, n_rxn=90, n_rev=20, size_range=(7, 20), coef_probs={1: 0.5, 2: 0.3, 3: 0.2}),
    "narrow-even": dict(n_int=30, n_rxn=50, n_rev=10, size_range=(8, 12), coef_probs={2: 0.4, 4: 0.4, 6: 0.2}),
    "narrow-large": dict(n_int=40, n_rxn=60, n_rev=10, size_range=(8, 12), coef_probs={1: 0.3, 999: 0.4, 524287: 0.3}),
    # columns past 32 entries, states past 64; bitsets and lists
    "bits": dict(n_int=100, n_rxn=100, n_rev=20, size_range=(28, 60), coef_probs={1: 0.5, 2: 0.3, 3: 0.2}),
    "bits-even": dict(n_int=100, n_rxn=100, n_rev=20, size_range=(30, 40), coef_probs={2: 0.4, 4: 0.4, 6: 0.2}),
    "list": dict(n_int=300, n_rxn=500, n_rev=100, size_range=(30, 80), coef_probs={1: 0.5, 2: 0.3, 3: 0.2}),
    "list-large": dict(n_int=90, n_rxn=130, n_rev=10, size_range=(31, 36), coef_probs={1: 0.3, 999: 0.4, 524287: 0.3}),
}


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("name", sorted(LONG))
def test_long_columns(oracle_lib, efm, name, variant):
    # reactions of dozens of metabolites: at budgets that one CTA's levels reach and past them
    net = synth.generate(n_targets=3, n_hubs=3, n_substrates=2, gamma=None, hub_degree=(5, 20), seed=77, name=name,
                         **LONG[name])
    max_len, targets = (12, net.targets[:2]) if variant == 0 else (6, net.targets[:1])
    for budget in (300, 3000):
        with efm.Network(net) as nw:
            got = efm.enumerate_targets(nw, targets, max_len, 2, 0, budget, variant=variant)
        seen = 0
        for t, (sup, ctr) in zip(targets, got):
            osup, octr = oracle_lib.enumerate_pathways(net, t, oracle_lib.Limits(max_len, 2, 0, budget, subtractive=bool(variant)))
            assert np.array_equal(sup, osup) and ctr == octr, (t, budget, ctr, octr)
            seen = max(seen, octr["frontier_max"])
        assert seen > 20
