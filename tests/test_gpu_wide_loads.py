"""Loads of more than four columns, one relation at a time: every column's
bound counts (it says how many bits of the column are sorted and joined)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cdl():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a GPU"
    from paper_2501_13051_gb300 import build as B
    B.build()
    from paper_2501_13051_gb300 import cdl as C
    return C


@pytest.mark.parametrize("arity", [5, 6, 7, 8])
@pytest.mark.parametrize("n", [100, 5000, 300_000])
def test_columns_past_the_fourth(cdl, arity, n):
    rng = np.random.default_rng(arity)
    rows = rng.integers(0, 3, (n, arity)).astype(np.uint32)
    rows[:, arity - 1] = rng.integers(0, 1 << 20, n)
    with cdl.Engine() as e:
        e.relation("r", arity)
        e.load("r", rows)
        got = e.export("r")
    assert np.array_equal(got, np.unique(rows, axis=0))
