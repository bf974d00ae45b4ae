"""Memory the set forms of Full need: programs whose joins have far more
outputs than new tuples, and batched runs, in as much memory as sorted rows
took (under a memory limit, and from an allocator that hands out no more)."""
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


def arena(cdl, budget):
    class Arena(cdl._TorchArena):
        def __init__(self, device):
            super().__init__(device)
            self.sizes = {}

        def _alloc(self, nbytes, ctx):
            if sum(self.sizes.values()) + nbytes > budget:
                return None
            p = super()._alloc(nbytes, ctx)
            if p:
                self.sizes[p] = nbytes
            return p

        def _free(self, ptr, nbytes, ctx):
            self.sizes.pop(ptr, None)
            super()._free(ptr, nbytes, ctx)
    return Arena


def run(cdl, prog, **opts):
    with cdl.Engine(**opts) as e:
        e.load_program(prog)
        st = e.run()
        return {nm: e.export(nm) for nm in prog.idb()}, st


def same(a, b):
    for nm in a[0]:
        assert np.array_equal(a[0][nm], b[0][nm]), nm
    assert a[1].delta_per_round == b[1].delta_per_round
    assert a[1].iters_per_instance == b[1].iters_per_instance


def repeats(n=300000, fan=60, nph=5):
    """n rows walk through the phases; two rules give 36M outputs a round,
    `fan` new tuples each."""
    edb = {"s": np.stack([np.arange(n), np.zeros(n)], axis=1),
           "next": np.stack([np.arange(nph - 1), np.arange(1, nph)], axis=1)}
    rules = [R(("t", ("x", "y")), (("s", ("x", "y")),)),
             R(("t", ("x", "z")), (("t", ("x", "y")), ("next", ("y", "z"))))]
    for k in range(2):
        edb["e%d" % k] = np.array([(r, 60000 + 100 * r + i + 7 * k) for r in range(nph) for i in range(fan)])
        rules.append(R(("h", (4095 - k, "z")), (("t", ("x", "y")), ("e%d" % k, ("y", "z")))))
    edb = {nm: v.astype(np.uint32) for nm, v in edb.items()}
    return W.Program(dict({nm: 2 for nm in edb}, t=2, h=2), rules, edb)


# sorted rows beside a round's bitmap ran from 360 MB
@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("how", ["limit", "allocator"])
def test_repeats(cdl, monkeypatch, how, graph):
    prog = repeats()
    want = run(cdl, prog, dense_bits=-1)
    if how == "allocator":
        monkeypatch.setattr(cdl, "_TorchArena", arena(cdl, 365_000_000))
        same(run(cdl, prog, graph=graph), want)
    else:
        same(run(cdl, prog, graph=graph, mem_limit=365_000_000), want)


# sorted rows ran from 242 MB; with less than the sets' tables need the run
# begins with sets or without, and changes over on the way
@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("budget", [245_000_000, 270_000_000, 300_000_000, 400_000_000])
def test_batched(cdl, monkeypatch, budget, graph):
    graphs, kinds = W.batched_instances(40, 91, 2e3, 6e4)
    prog = W.batched_program(graphs, kinds)
    want = run(cdl, prog, n_instances=40, dense_bits=-1)
    monkeypatch.setattr(cdl, "_TorchArena", arena(cdl, budget))
    same(run(cdl, prog, n_instances=40, graph=graph), want)


# Captured rounds that are outgrown by a burst: the round the host then runs
# may be the one that finds no memory for its sets, and the graph is captured
# again with sorted rows.
@pytest.mark.parametrize("graph", [True, 64])
def test_back_to_rows_behind_captured_rounds(cdl, monkeypatch, graph):
    from tests.test_gpu_hash_set import bursts, inst
    prog = W.batched_program([], [])
    prog.edb["tc_edge"] = np.concatenate([inst(0, bursts(60_000, 400_001)), inst(2, W.er_graph(3000, 3600, 2)),
                                          inst(4, bursts(3, 70_000))])
    prog.edb["sg_edge"] = np.concatenate([inst(1, W.random_forest(2500, 3)), inst(3, W.random_forest(700, 4))])
    want = run(cdl, prog, n_instances=5, dense_bits=-1)
    assert want[1].derived_tuples > 1 << 18

    def at(budget, **opts):
        with monkeypatch.context() as m:
            m.setattr(cdl, "_TorchArena", arena(cdl, budget))
            try:
                return run(cdl, prog, n_instances=5, **opts)
            except cdl.CdlError as ex:
                assert ex.name == "CDL_E_NOMEM"

    budget, ran = 200_000_000, 0
    while budget < 2_000_000_000:
        got = at(budget, graph=graph)
        if got:
            same(got, want)
            ran += 1
        else:  # no more than sorted rows take
            assert not at(int(budget * 0.95), dense_bits=-1, graph=graph), budget
        budget = int(budget * 1.1)
    assert ran > 8
