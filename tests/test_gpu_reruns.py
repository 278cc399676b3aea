"""Levels that are run again, and what must not happen twice when they are.

The network is a set of ladders to one target: a ladder of `steps` rungs
carries 1 + sides metabolites from rung to rung, and each rung but the first
and the last can be taken by `alts` parallel reactions (multiples of one
column), so level l of a search has alts^l states of 1 + sides entries.
With many sides a state takes more payload than a work area starts with and
a level is run again with a larger one; with many short pathways the superset
rule's index has to grow.  Supports and counters must equal the oracle's, and
the library's trace of the level state must show that it happened.
"""
import re

import numpy as np
import pytest

from paper_1804_02867_gb300 import synth

STOP_RERUN, STOP_INDEX = 4, 6


def ladders(*spec):
    """spec: (alts, steps, sides) per ladder."""
    n_int = sum((steps + 1) * (1 + sides) for _, steps, sides in spec)
    source, target = n_int, n_int + 1
    rxn, at = [], 0
    for alts, steps, sides in spec:
        w = 1 + sides
        rxn.append([(source, -1)] + [(at + s, 1) for s in range(w)])
        for i in range(steps):
            a, b = at + i * w, at + (i + 1) * w
            for q in range(alts):
                rxn.append([(a + s, -1 - q) for s in range(w)] + [(b + s, 1 + q) for s in range(w)])
        last = at + steps * w
        rxn.append([(last + s, -1) for s in range(w)] + [(target, 1)])
        at += (steps + 1) * w
    S = np.zeros((n_int + 2, len(rxn)), dtype=np.int64)
    for j, ents in enumerate(rxn):
        for m, v in ents:
            S[m, j] = v
    name = "ladders" + "".join(f"-{a}x{n}x{s}" for a, n, s in spec)
    return synth.Network.from_dense(S, [0] * len(rxn), [0] * n_int + [1, 1], [target], name)


def stops(err):
    """The stop codes of the library's level trace."""
    return {int(x) for x in re.findall(r"stop (\d+)", err)}


def test_ladders_by_the_oracle(oracle_lib):
    net = ladders((3, 4, 2), (5, 2, 0))
    sup, ctr = oracle_lib.enumerate_pathways(net, net.targets[0], oracle_lib.Limits(10, 0, 0, 1 << 12))
    assert len(sup) == 3 ** 4 + 5 ** 2 and ctr["frontier_max"] == 81 + 0


@pytest.fixture(scope="module")
def efm():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_02867_gb300 import build, efmgraph

    build.build()
    efmgraph.load_library()
    return efmgraph


# (bitset form; list form), both with more payload a state than 16 units a row
RERUN = {"bits": ((6, 5, 80),), "list": ((15, 3, 80), (45, 2, 0))}


@pytest.mark.gpu
@pytest.mark.parametrize("form", sorted(RERUN))
def test_level_run_again_on_the_grid(oracle_lib, efm, form, capfd, monkeypatch):
    net = ladders(*RERUN[form])
    budget = 8000 if form == "bits" else 6000
    monkeypatch.setenv("EFM_DEBUG", "1")
    with efm.Network(net) as nw:
        assert (nw.n_columns > 128) == (form == "list")
        capfd.readouterr()
        (sup, ctr), = efm.enumerate_targets(nw, net.targets, 10, 1, 0, budget)
    assert STOP_RERUN in stops(capfd.readouterr().err)
    osup, octr = oracle_lib.enumerate_pathways(net, net.targets[0], oracle_lib.Limits(10, 1, 0, budget))
    assert np.array_equal(sup, osup) and ctr == octr, (ctr, octr)
    assert ctr["status"] == 0


@pytest.mark.gpu
@pytest.mark.parametrize("max_results", [0, 10])
@pytest.mark.parametrize("spec", [((8, 2, 0),), ((9, 2, 0), (2, 5, 0)), ((17, 2, 0), (3, 4, 0)), ((30, 2, 1),)])
def test_small_levels_with_many_results(oracle_lib, efm, spec, max_results):
    """64, 81, 289 and 900 balanced children at a level that one CTA runs (its
    warps judge up to 64 of them), as the last level and with more to come."""
    net = ladders(*spec)
    with efm.Network(net) as nw:
        got = efm.enumerate_targets(nw, net.targets * 2, 10, 1, max_results, 1 << 12)
    osup, octr = oracle_lib.enumerate_pathways(net, net.targets[0], oracle_lib.Limits(10, 1, max_results, 1 << 12))
    assert octr["balanced"] >= 64
    for sup, ctr in got:
        assert np.array_equal(sup, osup) and ctr == octr, (ctr, octr)


@pytest.mark.gpu
@pytest.mark.parametrize("spec", [((46, 2, 0), (3, 4, 0)), ((55, 2, 0), (4, 5, 0))])
def test_index_grows(oracle_lib, efm, spec, capfd, monkeypatch):
    """More results at one level than the superset rule's index has room for,
    and levels after it: bitset form and list form."""
    net = ladders(*spec)
    monkeypatch.setenv("EFM_DEBUG", "1")
    with efm.Network(net) as nw:
        assert (nw.n_columns > 128) == (spec[0][0] == 55)
        capfd.readouterr()
        (sup, ctr), = efm.enumerate_targets(nw, net.targets, 10, 1, 0, 1 << 13)
    assert STOP_INDEX in stops(capfd.readouterr().err)
    osup, octr = oracle_lib.enumerate_pathways(net, net.targets[0], oracle_lib.Limits(10, 1, 0, 1 << 13))
    assert np.array_equal(sup, osup) and ctr == octr, (ctr, octr)


@pytest.mark.gpu
def test_trace_takes_a_level_once(efm, capfd, monkeypatch):
    """A first-K search with every pathway among its K: the traced levels hold
    6^0 + ... + 6^5 states (the seed's level among them), whether or not
    levels were run again on the way."""
    net = ladders(*RERUN["bits"])
    want = sum(6 ** i for i in range(6))
    monkeypatch.setenv("EFM_DEBUG", "1")
    for budget in (8000, 1 << 17):
        m = efm.efm_model_create(4)
        try:
            with efm.Network(net) as nw:
                capfd.readouterr()
                efm.efm_model_trace(m, nw.handle, net.targets, 7, 1, 6 ** 5, budget, rows_per_level=1 << 16)
            assert (STOP_RERUN in stops(capfd.readouterr().err)) == (budget == 8000)
            n, pos = efm.efm_model_rows(m)
        finally:
            efm.efm_model_free(m)
        assert (n, pos) == (want, want), budget  # every state lies inside a pathway


@pytest.mark.gpu
def test_timing_counts_what_ran(efm, capfd, monkeypatch):
    """expand_launches and expand_bytes of a search whose states are known: 6^l
    states of 81 entries at level l (43 units and a header each), the children
    of the last level balanced; with a small budget, levels run again count
    again; a first-K search counts its chunks."""
    net = ladders(*RERUN["bits"])
    state = 16 * (1 + 2 + 41)
    want = sum(state * (6 ** l + (6 ** (l + 1) if l < 5 else 0)) + 16 * 6 ** min(l + 1, 5) for l in range(6))
    monkeypatch.setenv("EFM_DEBUG", "1")
    with efm.Network(net) as nw:
        (_, _, t), = efm.enumerate_targets(nw, net.targets, 10, 1, 0, 1 << 17, timing=True)
        assert (t["expand_launches"], t["expand_bytes"]) == (6, want)
        capfd.readouterr()
        (_, _, t), = efm.enumerate_targets(nw, net.targets, 10, 1, 0, 8000, timing=True)
        again = len(re.findall(r"stop 4", capfd.readouterr().err))
        assert again > 0 and t["expand_launches"] == 6 + again and t["expand_bytes"] > want
    net = ladders((21, 3, 0))  # 9261 states before the last level: two chunks
    with efm.Network(net) as nw:
        capfd.readouterr()
        (sup, _, t), = efm.enumerate_targets(nw, net.targets, 5, 1, 0, 1 << 15, first_k=21 ** 3, timing=True)
        err = capfd.readouterr().err
    assert len(sup) == 21 ** 3
    lines = len(re.findall(r"efm: level", err))
    runs = len(re.findall(r"efm: level 0 .* children so far 0 ", err))
    assert runs == 5 and t["expand_launches"] == lines - runs
    core = synth.core()
    with efm.Network(core) as nw:  # walks, minimality test, a sort of two results
        sup, _, t = efm.sample_target(nw, core.targets[4], 20, 2, 7, 1 << 12, timing=True)
    assert len(sup) == 2 and t["kernel_launches"] == 1 + 1 + 3
