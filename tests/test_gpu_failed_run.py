"""What a run that stopped for want of memory leaves behind: the tuples of
its completed rounds, whichever form Full had, and none of the round it
stopped in."""
import numpy as np
import pytest

from paper_2501_13051_gb300 import workloads as W
from tests.test_gpu_set_room import phases

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


def stopped(cdl, prog, **opts):
    with cdl.Engine(**opts) as e:
        e.load_program(prog)
        with pytest.raises(cdl.CdlError) as ex:
            e.run()
        assert ex.value.name == "CDL_E_NOMEM"
        return {nm: e.export(nm) for nm in prog.idb()}


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("at", [1, 3, 4])
def test_completed_rounds_alone(cdl, oracle_lib, at, graph):
    """Phase `at` needs an intermediate table of 20M rows (1,024 x 20,000)
    after the same round's first rules have derived their tuples."""
    n = 1024
    prog = phases([(3, 2)] * 6, n)
    wide = np.stack([np.full(20000, at), np.arange(20000)], axis=1)
    narrow = np.stack([np.arange(20000), np.zeros(20000)], axis=1)
    more = {"w1": wide.astype(np.uint32), "w2": narrow.astype(np.uint32)}
    full = W.Program(dict(prog.arity, w1=2, w2=2, g=2),
                     prog.rules + [R(("g", ("x", "w")), (("t", ("x", "y")), ("w1", ("y", "z")), ("w2", ("z", "w"))))],
                     dict(prog.edb, **more))
    got = stopped(cdl, full, mem_limit=64 << 20, graph=graph)
    # phase r is reached in round r + 1; its rules fire in round r + 2
    t = np.concatenate([np.stack([np.arange(n), np.full(n, r)], axis=1) for r in range(at + 1)])
    t = t[np.lexsort((t[:, 1], t[:, 0]))]
    assert np.array_equal(got["t"], t)
    cut = dict(prog.edb, next=prog.edb["next"][:at - 1])
    want = oracle_lib.run_program(W.Program(prog.arity, prog.rules, cut))
    assert np.array_equal(got["h"], want.relations["h"])
    assert len(got["g"]) == 0
    rows = stopped(cdl, full, mem_limit=64 << 20, graph=graph, dense_bits=-1)
    for nm in got:
        assert np.array_equal(got[nm], rows[nm]), nm
