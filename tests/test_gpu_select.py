"""Copy rules (selection and projection) at the edges of a block's 2,048 rows:
constants, repeated variables, inequalities, constant and repeated head
columns, none and all rows kept, against the oracle."""
import numpy as np
import pytest

from paper_2501_13051_gb300 import workloads as W

pytestmark = pytest.mark.gpu
R = W.Rule

RULES = {
    "copy": R(("h", ("y", "x")), (("e", ("x", "y", "z")),)),
    "const": R(("h", ("x", "z")), (("e", ("x", 3, "z")),)),
    "same": R(("h", ("x", "y")), (("e", ("x", "y", "x")),)),
    "neq": R(("h", ("x", "z")), (("e", ("x", "y", "z")),), (("x", "z"), ("y", "z"))),
    "head": R(("h", (7, "z")), (("e", (1, "z", "z")),)),
    "none": R(("h", ("x", "y")), (("e", ("x", "y", 99)),)),
}


@pytest.fixture(scope="module")
def cdl():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a GPU"
    from paper_2501_13051_gb300 import build as B
    B.build()
    from paper_2501_13051_gb300 import cdl as C
    return C


@pytest.mark.parametrize("name", RULES)
@pytest.mark.parametrize("n", [1, 31, 256, 2047, 2048, 2049, 30_001])
@pytest.mark.parametrize("dense_bits", [0, -1])
def test_copy_rules(cdl, oracle_lib, name, n, dense_bits):
    e = np.unique(np.random.default_rng(n).integers(0, max(6, int(n ** 0.4)), (n, 3)).astype(np.uint32), axis=0)
    prog = W.Program({"e": 3, "h": 2}, [RULES[name]], {"e": e})
    got, _ = cdl.run_program(prog, dense_bits=dense_bits)
    assert np.array_equal(got["h"], oracle_lib.run_program(prog).relations["h"])
