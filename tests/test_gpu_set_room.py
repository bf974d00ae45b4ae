"""Room for the new tuples of relations kept as sets: counted joins behind a
one-pass join that found too little of it; each against the form with sorted
rows, and against the oracle."""
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


def phases(fans, n=4096):
    """t walks n rows through len(fans) phases, one a round; in phase r rule
    k into h has fans[r][k] outputs a row (all of them new tuples)."""
    nph, nk = len(fans), len(fans[0])
    edb = {"s": np.stack([np.arange(n), np.zeros(n)], axis=1),
           "next": np.stack([np.arange(nph - 1), np.arange(1, nph)], axis=1)}
    rules = [R(("t", ("x", "y")), (("s", ("x", "y")),)),
             R(("t", ("x", "z")), (("t", ("x", "y")), ("next", ("y", "z"))))]
    at = nph
    for k in range(nk):
        rows = [(nph, at)]  # (a node of no phase: the relation is not empty)
        for r in range(nph):
            rows += [(r, at + 1 + i) for i in range(fans[r][k])]
            at += 1 + fans[r][k]
        edb["e%d" % k] = np.array(rows)
        rules.append(R(("h", ("x", "z")), (("t", ("x", "y")), ("e%d" % k, ("y", "z")))))
    edb = {nm: v.astype(np.uint32) for nm, v in edb.items()}
    return W.Program(dict({nm: 2 for nm in edb}, t=2, h=2), rules, edb)


# The counted first rule leaves the buffer with room for half as much again;
# the second, expected to be small, overruns it; the third's outputs would
# have fitted beside the second's expected ones.
@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("third", [(5, 2), (5, 1), (0, 60)])
def test_counted_after_overrun(cdl, oracle_lib, third, graph):
    a, b = third
    prog = phases([(10, 0, a), (10, 0, a), (10, 8, b), (10, 0, a)])
    rows, st0 = cdl.run_program(prog, dense_bits=-1)
    got, st = cdl.run_program(prog, graph=graph)
    want = oracle_lib.run_program(prog)
    for nm in ("t", "h"):
        assert np.array_equal(got[nm], rows[nm]) and np.array_equal(got[nm], want.relations[nm]), nm
    assert st.delta_per_round == st0.delta_per_round
