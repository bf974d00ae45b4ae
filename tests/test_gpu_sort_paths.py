"""sort_unique and the engine's sorts at the edges of their forms -- one
block up to 4,096 tuples, a bitmap of a small tuple space, buckets from 2^18
tuples of at most 64 bits, the radix sort for the rest and for uneven
buckets -- against NumPy."""
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


def dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.uint32).view(np.int32)).cuda()


def unique_rows(cols):
    order = np.lexsort(cols[::-1])
    s = [c[order] for c in cols]
    new = np.ones(len(order), bool)
    if len(order):
        new[1:] = np.logical_or.reduce([c[1:] != c[:-1] for c in s])
    return [c[new] for c in s]


def check(cdl, cols):
    cols = [np.asarray(c, dtype=np.uint32) for c in cols]
    d = [dev(c) for c in cols]
    got = cdl.sort_unique(d)
    for g, w in zip(got, unique_rows(cols)):
        assert np.array_equal(g.cpu().numpy().view(np.uint32), w)
    for c, h in zip(d, cols):  # the input is left as it was
        assert np.array_equal(c.cpu().numpy().view(np.uint32), h)


def draw(rng, n, arity, bits):
    return [rng.integers(0, 1 << bits, n, dtype=np.uint64).astype(np.uint32) for _ in range(arity)]


@pytest.mark.parametrize("n", [1, 2, 31, 33, 1000, 1023, 1024, 1025, 2049, 4095, 4096, 4097])
@pytest.mark.parametrize("arity,bits", [(1, 1), (1, 32), (2, 5), (2, 18), (3, 31), (5, 7), (8, 32)])
def test_small(cdl, n, arity, bits):
    check(cdl, draw(np.random.default_rng(n), n, arity, bits))


@pytest.mark.parametrize("n,arity,bits", [(5000, 2, 9), (5000, 1, 18), (4097, 1, 19), (100_003, 3, 7),
                                          (300_000, 2, 12), (70_000, 5, 4), (270_000, 1, 25)])
def test_small_tuple_space(cdl, n, arity, bits):
    check(cdl, draw(np.random.default_rng(n), n, arity, bits))


@pytest.mark.parametrize("n", [(1 << 18) - 1, 1 << 18, 300_007, 393_216, 393_217, 1_000_003])
@pytest.mark.parametrize("arity,bits", [(1, 32), (2, 18), (2, 32), (3, 21), (4, 16), (8, 8), (3, 22)])
def test_large(cdl, n, arity, bits):
    cols = draw(np.random.default_rng(n), n, arity, bits)
    for c in cols:  # repeats
        c[: n // 5] = c[n // 5: 2 * (n // 5)]
    check(cdl, cols)


@pytest.mark.parametrize("kind", ["one-value", "half-one-value", "dense-range", "zeros-but-one",
                                  "gaps", "constant-columns"])
def test_uneven(cdl, kind):
    n, rng = 300_001, np.random.default_rng(3)
    a, b = draw(rng, n, 2, 31)
    if kind == "one-value":
        a[:], b[:] = 2 ** 31 - 1, 77
    elif kind == "half-one-value":
        a[: n // 2], b[: n // 2] = 12345, 99
    elif kind == "dense-range":
        a[1:] = rng.integers(1 << 20, (1 << 20) + 5000, n - 1)
    elif kind == "zeros-but-one":
        a[:], b[:] = 0, 0
        a[7] = 2 ** 32 - 2
    elif kind == "gaps":
        a &= 0x70000FFF
    else:
        check(cdl, [np.full(n, 2 ** 32 - 2), a, np.zeros(n)])
        check(cdl, [np.zeros(n), a, b])
        return
    check(cdl, [a, b])


@pytest.mark.parametrize("uneven", [False, True])
@pytest.mark.parametrize("n", [1, 4096, 4097, 262_143, 262_144, 700_001])
def test_engine_sorts_loaded_rows(cdl, n, uneven):
    rng = np.random.default_rng(n)
    rows = np.stack(draw(rng, n, 2, 30), axis=1)
    if uneven:
        rows[: n // 2 + 1, 0] = 5
    want = np.stack(unique_rows([rows[:, 0], rows[:, 1]]), axis=1)
    with cdl.Engine() as e:
        for nm in ("a", "b"):
            e.relation(nm, 2)
        e.load("a", rows)
        e.rule(("b", ["y", "x"]), [("a", ["x", "y"])])
        e.run()
        assert np.array_equal(e.export("a"), want)
        b = e.export("b")
    assert np.array_equal(b, np.stack(unique_rows([want[:, 1], want[:, 0]]), axis=1))
