"""A round's merges of several relations as one set of launches: relations of
one to three columns and of very different sizes side by side, some that
change and some that stop changing, at and across the tiles of 4,096 rows,
each against the oracle."""
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


@pytest.mark.parametrize("sizes", [(1, 2, 3), (40, 4096, 4097, 8192), (9000, 30, 700, 5000, 2, 12000, 1, 4095)])
@pytest.mark.parametrize("dense_bits", [0, -1])
def test_relations_side_by_side(cdl, oracle_lib, sizes, dense_bits):
    rng = np.random.default_rng(len(sizes))
    arity, edb, rules = {"next": 2}, {}, []
    edb["next"] = np.stack([np.arange(40), np.arange(1, 41)], axis=1).astype(np.uint32)
    for i, n in enumerate(sizes):
        a, p, u, t = "a%d" % i, "p%d" % i, "u%d" % i, "t%d" % i
        arity.update({a: 2, p: 2, u: 1, t: 3})
        edb[a] = np.unique(np.stack([rng.integers(0, 30 + i, n), rng.integers(0, 3 * n + 50, n)], axis=1)
                           .astype(np.uint32), axis=0)
        rules += [R((p, ("x", "y")), ((a, ("x", "y")),)),
                  R((p, ("z", "y")), ((p, ("x", "y")), ("next", ("x", "z")))),
                  R((u, ("y",)), ((p, ("x", "y")), (p, ("x", "x2")))) if n < 50 else
                  R((u, ("y",)), ((p, ("x", "y")),)),
                  R((t, ("y", "x", i)), ((p, ("x", "y")), ("next", ("x", "z"))))]
    prog = W.Program(arity, rules, edb)
    got, st = cdl.run_program(prog, dense_bits=dense_bits)
    want = oracle_lib.run_program(prog)
    for nm in arity:
        assert np.array_equal(got[nm], want.relations[nm]), nm
    assert st.iterations == want.iterations and st.rounds == want.rounds
    per_round = [sum(want.deltas[nm][k] for nm in prog.idb()) for k in range(want.rounds)]
    assert st.delta_per_round == per_round
