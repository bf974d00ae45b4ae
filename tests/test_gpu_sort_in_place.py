"""cdl_sort_unique with its output over its input (in place, columns crossed,
shifted), in every form of the sort: one block, a bitmap, buckets, buckets of
wide tuples' leading columns, radix passes."""
import ctypes

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


FORMS = {"one-block": (4096, 2, 18), "bitmap": (300000, 2, 11), "buckets": (300001, 2, 20),
         "buckets-32": (100003, 2, 32), "wide": (200003, 4, 32), "wide-8": (50021, 8, 31),
         "uneven": (300000, 2, 24)}


@pytest.mark.parametrize("over", ["in place", "crossed", "shifted"])
@pytest.mark.parametrize("form", FORMS)
def test_output_over_input(cdl, form, over):
    import torch
    n, k, bits = FORMS[form]
    rng = np.random.default_rng(n)
    rows = rng.integers(0, (1 << bits) - 1, size=(n, k), dtype=np.uint64).astype(np.uint32)
    rows[n // 2:] = rows[rng.integers(0, n // 2, n - n // 2)]
    if form == "uneven":
        rows[: n // 3, 0] = 77  # (far past what one bucket holds)
    want = np.unique(rows, axis=0)
    step = (n + 63) // 64 * 64 + 64
    buf = torch.zeros(step * (k + 1), dtype=torch.int32, device="cuda")
    cols = [buf[c * step: c * step + n] for c in range(k)]
    for c in range(k):
        cols[c].copy_(torch.from_numpy(rows[:, c].view(np.int32)))
    if over == "in place":
        outs = cols
    elif over == "crossed":
        outs = cols[::-1]
    else:
        outs = [buf[c * step + 32: c * step + 32 + n] for c in range(k)]
    L, P = cdl.lib(), cdl._ptrs
    need, got_n = ctypes.c_size_t(0), ctypes.c_uint64(0)
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    pi, po = P(cols), P(outs)
    assert L.cdl_sort_unique(pi, k, n, po, ctypes.byref(got_n), None, ctypes.byref(need), s) == 0
    ws = torch.empty(need.value, dtype=torch.uint8, device="cuda")
    assert L.cdl_sort_unique(pi, k, n, po, ctypes.byref(got_n), ws.data_ptr(), ctypes.byref(need), s) == 0
    assert got_n.value == len(want)
    got = np.stack([o[:len(want)].cpu().numpy().view(np.uint32) for o in outs], axis=1)
    assert np.array_equal(got, want)
