"""Full kept as a bitmap of the tuple space (new tuples appended to delta as
their bits are set, no sort and no merge), from the start in small tuple
spaces and after a switch from sorted rows in larger ones; and hub joins,
which OR a hub key's bitmap row into its probe rows' head rows.  Each against
the oracle, or against the sorted-rows form where the oracle's sets would
take minutes."""
import numpy as np
import pytest

from paper_2501_13051_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cdl():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a GPU"
    from paper_2501_13051_gb300 import build as B
    B.build()
    from paper_2501_13051_gb300 import cdl as C
    return C


@pytest.mark.parametrize("stop", [0, 9])
@pytest.mark.parametrize("spread", [1, 16, 17, 60, 130])
def test_closure_with_spread_ids(cdl, oracle_lib, tmp_path, spread, stop):
    """338,124 pairs in 37 rounds over tuple spaces of 2^20 to 2^34: a bitmap
    from the first round up to 2^28, sorted rows that go over to one above;
    a checkpoint taken on the way holds sorted versions either way."""
    prog = W.tc_program(W.er_graph(1000, 1500, 1) * np.uint32(spread))
    want = oracle_lib.run_program(prog)
    if stop:
        path = str(tmp_path / "ckpt.bin")
        with cdl.Engine(max_iters=stop) as e:
            e.load_program(prog)
            with pytest.raises(cdl.CdlError) as ex:
                e.run()
            assert ex.value.name == "CDL_E_MAXITER"
            e.checkpoint_save(path)
        with cdl.Engine() as e:
            for nm, ar in prog.arity.items():
                e.relation(nm, ar)
            for r in prog.rules:
                e.rule(r.head, r.body, r.neq)
            e.checkpoint_load(path)
            st = e.run()
            got = {nm: e.export(nm) for nm in prog.arity}
    else:
        got, st = cdl.run_program(prog)
    for nm in prog.arity:
        assert np.array_equal(got[nm], want.relations[nm]), nm
    assert st.iterations == want.iterations and st.rounds == want.rounds
    assert st.delta_per_round == want.deltas["path"][:want.rounds]


def hub_edges(sizes, n, cols=1):
    """(z, x) pairs: hub z has sizes[z] distinct x below n (and, with cols 2,
    a second key column)."""
    rng = np.random.default_rng(5)
    parts = []
    for z, d in enumerate(sizes):
        x = rng.permutation(n)[:d].astype(np.uint32)
        key = [np.full(d, z * 3 + c, np.uint32) for c in range(cols)]
        parts.append(np.stack(key + [x], axis=1))
    return np.concatenate(parts)


R = W.Rule
SIZES = [2100, 40, 33, 32, 31, 5, 1, 300]  # around the smallest hub (32 rows)


@pytest.mark.parametrize("name", ["pairs", "const", "two-keys", "read", "key-last", "filter", "one-sided"])
@pytest.mark.parametrize("n", [2100, 4096, 5000])
def test_hub_joins_equal_sorted_rows(cdl, n, name):
    e = {"e": hub_edges(SIZES, n)}
    ar = {"e": 2, "h": 2}
    if name == "pairs":
        rules = [R(("h", ("x", "y")), (("e", ("z", "x")), ("e", ("z", "y"))))]
    elif name == "const":
        ar = {"e": 2, "h": 3}
        rules = [R(("h", ("x", 3, "y")), (("e", ("z", "x")), ("e", ("z", "y"))))]
    elif name == "two-keys":
        ar, e = {"e": 3, "h": 3}, {"e": hub_edges(SIZES, n, 2)}
        rules = [R(("h", ("z", "y", "x")), (("e", ("z", "w", "x")), ("e", ("z", "w", "y"))))]
    elif name == "read":  # Full of h is read by a rule: the bitmap holds a round's new tuples
        ar = {"e": 2, "h": 2, "g": 1}
        rules = [R(("h", ("x", "y")), (("e", ("z", "x")), ("e", ("z", "y")))),
                 R(("g", ("x",)), (("h", ("x", "y")), ("h", ("y", "x"))))]
    elif name == "key-last":  # the last head column is the key: no hub row
        rules = [R(("h", ("x", "z")), (("e", ("z", "x")), ("e", ("z", "y"))))]
    elif name == "filter":
        rules = [R(("h", ("x", "y")), (("e", ("z", "x")), ("e", ("z", "y"))), (("x", "y"),))]
    else:  # the hubs of one side meet few rows of the other
        ar, e = {"e": 2, "f": 2, "h": 2}, dict(e, f=hub_edges([2099] + [3] * 7, n))
        rules = [R(("h", ("y", "x")), (("e", ("z", "x")), ("f", ("z", "y"))))]
    prog = W.Program(ar, rules, e)
    rows, st0 = cdl.run_program(prog, dense_bits=-1)
    got, st = cdl.run_program(prog, dense_bits=34)
    assert len(rows["h"]) > 2000
    for nm in ar:
        assert np.array_equal(got[nm], rows[nm]), nm
    assert st.delta_per_round == st0.delta_per_round and st.iterations == st0.iterations


def test_hub_join_equals_oracle(cdl, oracle_lib):
    prog = W.Program({"e": 2, "h": 2}, [R(("h", ("x", "y")), (("e", ("z", "x")), ("e", ("z", "y"))))],
                     {"e": hub_edges(SIZES, 2111)})
    got, _ = cdl.run_program(prog)
    assert np.array_equal(got["h"], oracle_lib.run_program(prog).relations["h"])
