"""Batched runs of 2^18 to 2^22 tuples, the smallest whose Full becomes a hash
set, and smaller ones that keep sorted rows, against sorted rows throughout."""
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


def run(cdl, prog, count, **opts):
    with cdl.Engine(n_instances=count, timing=True, **opts) as e:
        e.load_program(prog)
        st = e.run()
        out = {nm: e.export(nm, device=True) for nm in prog.idb()}
        return out, st, {d["kernel"]: d["launches"] for d in e.kernel_profile()}


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("count,hi,sets", [(24, 2.2e4, True), (7, 1.6e5, True), (1, 3e5, None), (6, 6e3, False)])
def test_small_sets(cdl, count, hi, sets, graph):
    import torch
    graphs, kinds = W.batched_instances(count, 31, 2e3 if count > 1 else 2.9e5, hi)
    prog = W.batched_program(graphs, kinds)
    rows, st0, _ = run(cdl, prog, count, dense_bits=-1)
    got, st, prof = run(cdl, prog, count, graph=graph)
    for nm in rows:
        assert all(torch.equal(a, b) for a, b in zip(got[nm], rows[nm])), nm
    assert st.delta_per_round == st0.delta_per_round
    assert st.iters_per_instance == st0.iters_per_instance
    assert st0.derived_tuples < 1 << 22
    if sets is not None:
        assert (st0.derived_tuples > 1 << 18) == sets
        assert (prof.get("dense", 0) > 0) == sets, sorted(prof)
