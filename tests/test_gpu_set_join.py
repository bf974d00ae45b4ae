"""One-pass joins into Full's bitmap: rounds whose outputs outgrow the room
their last round suggested (the round's joins run again), rows with long
ranges (taken in chunks), star joins and filters, several rules into one
relation, with the rounds driven by the host and captured in a graph; each
against the form with sorted rows, and small ones against the oracle."""
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


def same(cdl, prog, **opts):
    rows, st0 = cdl.run_program(prog, dense_bits=-1)
    got, st = cdl.run_program(prog, **opts)
    for nm in prog.arity:
        assert np.array_equal(got[nm], rows[nm]), nm
    assert st.delta_per_round == st0.delta_per_round
    assert (st.iterations, st.rounds) == (st0.iterations, st0.rounds)
    return got, st


def bursts(fans, chain=4):
    """Chains that end in fans of the given sizes, one behind the other."""
    edges, at = [], 0
    for f in fans:
        for _ in range(chain):
            edges.append((at, at + 1))
            at += 1
        edges += [(at, at + 1 + i) for i in range(f)]
        edges.append((at + 1, at + 1 + f))
        at += 1 + f
    return np.array(edges, dtype=np.uint32)


@pytest.mark.parametrize("graph", [False, True, 64])
@pytest.mark.parametrize("fans", [(5, 6000, 3), (2048, 2049, 1), (1, 9000, 1, 4500), (15000,)])
def test_bursts(cdl, oracle_lib, fans, graph):
    prog = W.tc_program(bursts(fans))
    got, _ = same(cdl, prog, graph=graph)
    assert np.array_equal(got["path"], oracle_lib.run_program(prog).relations["path"])


@pytest.mark.parametrize("graph", [False, True, 64])
@pytest.mark.parametrize("n", [255, 257, 2047, 2049, 9001])
@pytest.mark.parametrize("make", [lambda n: W.tc_program(W.er_graph(n, n + n // 3, n)),
                                  lambda n: W.sg_program(W.random_forest(n, n)),
                                  lambda n: W.sg_paper_program(W.random_forest(n, n))])
def test_sizes(cdl, make, n, graph):
    same(cdl, make(n), graph=graph)


@pytest.mark.parametrize("graph", [False, True])
def test_star_bursts(cdl, graph):
    """Same generation where a pair of parents has 70 x 70 children."""
    edges, nxt, level = [], 1, [0]
    for width in (3, 1, 70, 1, 2):
        new = []
        for p in level[:40]:
            for _ in range(width):
                edges.append((p, nxt))
                new.append(nxt)
                nxt += 1
        level = new
    e = np.array(edges, dtype=np.uint32)
    same(cdl, W.sg_program(e), graph=graph)
    same(cdl, W.sg_paper_program(e), graph=graph)


@pytest.mark.parametrize("graph", [False, True, 64])
def test_rules_into_one_relation(cdl, graph):
    a, b = W.er_graph(1500, 1700, 1), bursts((4, 7000, 2))
    rules = [R(("t", ("x", "y")), (("e", ("x", "y")),)),
             R(("t", ("x", "z")), (("t", ("x", "y")), ("e", ("y", "z")))),
             R(("t", ("x", "z")), (("t", ("x", "y")), ("f", ("y", "z"))), (("x", "z"),)),
             R(("u", ("y", 3, "x")), (("t", ("x", "y")), ("e", ("y", "y2"))))]
    prog = W.Program({"e": 2, "f": 2, "t": 2, "u": 3}, rules, {"e": a, "f": b})
    same(cdl, prog, graph=graph)
