"""Batched runs whose Full is kept as a hash set (from 2^18 rows after the
first semi-naive round): rounds that outgrow the room for their new
tuples and the table, retirement before the switch, copy rules beside the
joins, a stop at max_iters, with the rounds driven by the host and captured
in a graph -- each against the form with sorted rows."""
import numpy as np
import pytest

from paper_2501_13051_gb300 import workloads as W

pytestmark = pytest.mark.gpu
R = W.Rule


@pytest.fixture(scope="module")
def cdl():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a GPU"
    from paper_2501_13051_gb300 import build as B
    B.build()
    from paper_2501_13051_gb300 import cdl as C
    return C


def run(cdl, prog, **opts):
    with cdl.Engine(**opts) as e:
        e.load_program(prog)
        st = e.run()
        return {nm: e.export(nm, device=True) for nm in prog.idb()}, st


def same(cdl, prog, count, **opts):
    import torch
    rows, st0 = run(cdl, prog, n_instances=count, dense_bits=-1)
    got, st = run(cdl, prog, n_instances=count, **opts)
    for nm in rows:
        assert all(torch.equal(a, b) for a, b in zip(got[nm], rows[nm])), nm
    assert st.delta_per_round == st0.delta_per_round
    assert st.iters_per_instance == st0.iters_per_instance
    assert st.iterations == st0.iterations and st.rounds == st0.rounds
    assert st0.derived_tuples > 1 << 22
    return st


def inst(i, edges):
    return np.concatenate([np.full((len(edges), 1), i, np.uint32), edges.astype(np.uint32)], axis=1)


def chain(at, n):
    return np.stack([np.arange(at, at + n), np.arange(at + 1, at + n + 1)], axis=1), at + n


def fan(at, n):
    return np.stack([np.full(n, at), np.arange(at + 1, at + 1 + n)], axis=1), at + n


def bursts(f1, f2):
    """A chain into a fan of f1, and from its last leaf a longer chain (by
    whose end every other path has ended) into a fan of f2."""
    a, at = chain(0, 6)
    b, at = fan(at, f1)
    c, at = chain(at, 12)
    d, at = fan(at, f2)
    return np.concatenate([a, b, c, d])


@pytest.mark.parametrize("graph", [False, True, 64])
def test_bursts(cdl, graph):
    rng = np.random.default_rng(1)
    tc = np.concatenate([inst(0, bursts(2_200_000, 1_500_001)), inst(2, W.er_graph(3000, 3600, 2)),
                         inst(4, bursts(3, 70_000))])
    sg = np.concatenate([inst(1, W.random_forest(4000, 3)), inst(3, W.random_forest(700, 4))])
    prog = W.batched_program([], [])
    prog.edb["tc_edge"], prog.edb["sg_edge"] = rng.permutation(tc), rng.permutation(sg)
    st = same(cdl, prog, 5, graph=graph)
    assert st.graph_retirements == 0


@pytest.mark.parametrize("graph,retire", [(False, True), (True, True), (True, False)])
def test_instances(cdl, graph, retire):
    graphs, kinds = W.batched_instances(64, 91, 2e4, 3e5)
    same(cdl, W.batched_program(graphs, kinds), 64, graph=graph, retire=retire)


def test_copy_rules_and_filters(cdl):
    e = np.concatenate([inst(0, bursts(2_200_000, 5)), inst(1, W.er_graph(3000, 4500, 7))])
    rules = [R(("p", ("i", "x", "y")), (("e", ("i", "x", "y")),)),
             R(("q", ("i", "y", "x")), (("p", ("i", "x", "y")),)),
             R(("p", ("i", "x", "z")), (("p", ("i", "x", "y")), ("e", ("i", "y", "z"))), (("x", "z"),)),
             R(("q", ("i", "z", "x")), (("q", ("i", "y", "x")), ("e", ("i", "y", "z"))))]
    same(cdl, W.Program({"e": 3, "p": 3, "q": 3}, rules, {"e": e}), 2)


@pytest.mark.parametrize("graph", [False, True])
def test_stop_at_max_iters(cdl, graph):
    prog = W.batched_program([], [])
    prog.edb["tc_edge"] = inst(0, bursts(2_200_000, 90_000))
    prog.edb["sg_edge"] = inst(1, W.random_forest(300, 4))
    with pytest.raises(cdl.CdlError) as ex:
        run(cdl, prog, n_instances=2, graph=graph, max_iters=9)
    assert ex.value.name == "CDL_E_MAXITER"
