"""cdl_join_write, the write half of a sized join: only behind the cdl_join it
belongs to (anything else is CDL_E_INVALID and writes nothing), as often as
wanted, with and without room for the rows' first matches."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
OK, INVALID, CAPACITY = 0, -1, -3


@pytest.fixture(scope="module")
def cdl():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a GPU"
    from paper_2501_13051_gb300 import build as B
    B.build()
    from paper_2501_13051_gb300 import cdl as C
    return C


class Call:
    """One join's arguments; key = column 0 on both sides."""

    def __init__(self, cdl, n_probe, n_build, neq=False, seed=0, keys=None):
        import torch
        self.L, self.cdl, self.neq = cdl.lib(), cdl, neq
        rng = np.random.default_rng(seed)
        keys = keys or max(1, n_build // 2)
        self.probe = np.stack([rng.integers(0, keys, n_probe), rng.integers(0, 3, n_probe)])
        self.build = np.stack([np.sort(rng.integers(0, keys, n_build)), rng.integers(0, 3, n_build)])
        dev = lambda a: [torch.from_numpy(np.ascontiguousarray(c.astype(np.int32))).cuda() for c in a]
        self.p, self.b = dev(self.probe), dev(self.build)
        self.spec = (cdl.ColRef * 3)(cdl.ColRef(0, 0), cdl.ColRef(0, 1), cdl.ColRef(1, 1))
        self.nq = (cdl.ColRef * 2)(cdl.ColRef(0, 1), cdl.ColRef(1, 1))
        self.need = ctypes.c_size_t(0)
        self.n = ctypes.c_uint64(0)
        assert self.join(None, None, 0) == OK
        self.ws = torch.empty(self.need.value, dtype=torch.uint8, device="cuda")

    def args(self):
        P = self.cdl._ptrs
        self.hold = P(self.p), P(self.b)
        return (self.hold[0], 2, self.p[0].numel(), 0, self.hold[1], 2, self.b[0].numel(), 0, self.spec, 3,
                self.nq, 1 if self.neq else 0)

    def call(self, f, ws, outs, cap, size=None):
        import torch
        need = ctypes.c_size_t(size if size is not None else self.need.value)
        o = self.cdl._ptrs(outs) if outs else None
        st = f(*self.args(), o, cap, ctypes.byref(self.n), ws, ctypes.byref(need),
               ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        if not ws:
            self.need = need
        return st

    def join(self, ws, outs, cap, size=None):
        return self.call(self.L.cdl_join, ws, outs, cap, size)

    def write(self, outs, cap, size=None):
        return self.call(self.L.cdl_join_write, self.ws.data_ptr(), outs, cap, size)

    def outs(self, n):
        import torch
        return [torch.full((n,), -1, dtype=torch.int32, device="cuda") for _ in range(3)]

    def want(self):
        a = np.searchsorted(self.build[0], self.probe[0], "left")
        e = np.searchsorted(self.build[0], self.probe[0], "right")
        rows = [(self.probe[0][i], self.probe[1][i], self.build[1][j])
                for i in range(len(a)) for j in range(a[i], e[i])
                if not self.neq or self.probe[1][i] != self.build[1][j]]
        return np.array(sorted(rows)).reshape(-1, 3)

    def got(self, outs, n):
        r = np.stack([o[:n].cpu().numpy() for o in outs], axis=1)
        return r[np.lexsort((r[:, 2], r[:, 1], r[:, 0]))]


def old_size(c):
    """The workspace without the rows' first matches."""
    up = lambda b: (b + 255) & ~255
    return c.need.value - up(4 * max(1, c.p[0].numel()))


@pytest.mark.parametrize("neq", [False, True])
@pytest.mark.parametrize("starts", [True, False])
@pytest.mark.parametrize("n", [(1, 1), (2047, 300), (5000, 4097)])
def test_write_after_query(cdl, n, starts, neq):
    c = Call(cdl, *n, neq=neq, seed=n[0])
    size = None if starts else old_size(c)
    assert c.join(c.ws.data_ptr(), None, 0, size) == CAPACITY
    total, want = c.n.value, c.want()
    for _ in range(2):  # the second write gives the same rows
        outs = c.outs(total)
        c.n.value = total
        assert c.write(outs, total, size) == OK
        assert c.n.value == len(want)
        assert np.array_equal(c.got(outs, len(want)), want)
    outs = c.outs(total)  # and the whole call in one
    assert c.join(c.ws.data_ptr(), outs, total, size) == OK
    assert np.array_equal(c.got(outs, c.n.value), want)


def refused(c, total, size=None):
    outs = c.outs(total)
    c.n.value = total
    assert c.write(outs, total, size) == INVALID
    assert all(int((o != -1).sum()) == 0 for o in outs)


# (the workspace is a well-formed one of another call, or zeros: a library
# without the check reads and writes within its buffers all the same.  Of five
# rows the workspace has no room for the write's splits.)
@pytest.mark.parametrize("n", [(3000, 2000, None), (5, 400000, 2)])
def test_write_without_its_query(cdl, n):
    c = Call(cdl, n[0], n[1], keys=n[2])
    assert c.join(c.ws.data_ptr(), None, 0) == CAPACITY
    total = c.n.value
    assert total > 4
    head = c.ws[:256].clone()
    c.ws[:256].zero_()
    refused(c, total)                     # the query's words are gone
    c.ws[:256].copy_(head)
    refused(c, total, old_size(c))        # its workspace had another layout
    assert c.join(c.ws.data_ptr(), None, 0, old_size(c)) == CAPACITY
    refused(c, total)
    assert c.join(c.ws.data_ptr(), None, 0) == CAPACITY
    outs = c.outs(total)
    c.n.value = total
    assert c.write(outs, total) == OK and c.n.value == total
    assert int((outs[0] == -1).sum()) == 0


def test_write_of_another_size(cdl):
    c = Call(cdl, 3000, 2000)
    assert c.join(c.ws.data_ptr(), None, 0) == CAPACITY
    total = c.n.value
    refused(c, total - 1)                 # fewer rows than counted
    for side in ("p", "b"):               # a row less on one side
        keep = getattr(c, side)
        setattr(c, side, [x[:-1] for x in keep])
        refused(c, total)
        setattr(c, side, keep)
    outs = c.outs(total)
    c.n.value = total
    assert c.write(outs, total) == OK
    assert np.array_equal(c.got(outs, total), c.want())
