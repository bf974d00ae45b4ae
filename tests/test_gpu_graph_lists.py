"""Captured rounds whose rows with long ranges need more chunks than the list
of them holds: the round leaves the graph once, and the next graph has room."""
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


def hub_into_chains(chains, length, fan):
    """Every round of the closure reaches one more node of each chain from the
    hub, which `fan` nodes lead to: chains x ceil(fan / 2048) chunks a round."""
    leaf = 1 + np.arange(fan)
    edges = [np.stack([np.zeros(fan, np.int64), leaf], axis=1)]
    at = 1 + fan
    for _ in range(chains):
        c = at + np.arange(length)
        edges.append(np.stack([c, np.append(c[1:], 0)], axis=1))
        at += length
    return np.concatenate(edges).astype(np.uint32)[:, ::-1]


# option graph = 64: lists of 64 chunks to begin with, against 40 x 3 a round
def test_list_outgrown_once(cdl):
    prog = W.tc_program(hub_into_chains(40, 12, 5000))
    rows, st0 = cdl.run_program(prog, dense_bits=-1)
    got, st = cdl.run_program(prog, graph=64)
    assert np.array_equal(got["path"], rows["path"])
    assert st.delta_per_round == st0.delta_per_round
    assert st.graph_rounds >= st.rounds - 4 and st.graph_builds <= 3, (st.graph_rounds, st.graph_builds)


# 65,536 chunks, where the list starts by default: 12,000 x 6 a round
def test_default_list_outgrown_once(cdl):
    prog = W.tc_program(hub_into_chains(12000, 8, 11000))
    opts = {"dense_bits": 34}
    with cdl.Engine(graph=True, **opts) as e:
        e.load_program(prog)
        st = e.run()
        n = e.size("path")
    assert n == sum(st.delta_per_round)
    assert st.graph_rounds >= st.rounds - 4 and st.graph_builds <= 3, (st.graph_rounds, st.graph_builds)
