"""Steps that take more memory to be faster, where there is no more: merges of
several relations at once, and the index a join's hub keys want on its probe
side.  The run goes on without them."""
import numpy as np
import pytest

from paper_2501_13051_gb300 import workloads as W
from tests.test_gpu_set_memory import arena, run, same

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


def walks(k=8, n=200000, nph=6):
    """k relations of n rows a round, ids too large for a bitmap."""
    x, ids = np.arange(n) * 5000, 4000000000 + np.arange(nph)
    edb, arity, rules = {"next": np.stack([ids[:-1], ids[1:]], axis=1)}, {"next": 2}, []
    for i in range(k):
        s, t = "s%d" % i, "t%d" % i
        edb[s], arity[s], arity[t] = np.stack([x + i, np.full(n, ids[0])], axis=1), 2, 2
        rules += [R((t, ("x", "y")), ((s, ("x", "y")),)),
                  R((t, ("x", "z")), ((t, ("x", "y")), ("next", ("y", "z"))))]
    return W.Program(arity, rules, {nm: v.astype(np.uint32) for nm, v in edb.items()})


# one merge after the other ran from 173 MB
def test_merges_one_by_one(cdl, monkeypatch):
    prog = walks()
    want = run(cdl, prog, dense_bits=-1)
    monkeypatch.setattr(cdl, "_TorchArena", arena(cdl, 176_000_000))
    same(run(cdl, prog), want)


def hubs(n=1000000, fan=40, nph=4):
    """40M outputs a round from n rows of one hub key, `fan` new tuples."""
    edb = {"s": np.stack([np.arange(n), np.zeros(n)], axis=1),
           "next": np.stack([np.arange(nph - 1), np.arange(1, nph)], axis=1),
           "e": np.array([(r, 1000 + 100 * r + i) for r in range(nph) for i in range(fan)])}
    rules = [R(("t", ("x", "y")), (("s", ("x", "y")),)),
             R(("t", ("x", "z")), (("t", ("x", "y")), ("next", ("y", "z")))),
             R(("h", (1, "z")), (("t", ("x", "y")), ("e", ("y", "z"))))]
    edb = {nm: v.astype(np.uint32) for nm, v in edb.items()}
    return W.Program(dict({nm: 2 for nm in edb}, t=2, h=2), rules, edb)


# (the index alone takes 16 MB while it is built)
@pytest.mark.parametrize("limit", [54_000_000, 58_000_000, 100_000_000])
def test_hubs_without_index(cdl, limit):
    prog = hubs()
    want = run(cdl, prog, dense_bits=-1)
    same(run(cdl, prog, mem_limit=limit), want)
