"""Joins over both forms of the build side's index -- entries by key where the
largest key is near the number of rows, hash slots elsewhere -- at the line
between the two, with absent keys below and above the largest one, and with
runs of one key, against NumPy."""
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


def slots(n):
    return 1 << max(4, (2 * n).bit_length())


def reference(probe, build):
    lo, hi = np.searchsorted(build[0], probe[0], "left"), np.searchsorted(build[0], probe[0], "right")
    n = hi - lo
    row = np.repeat(np.arange(len(n)), n)
    at = np.arange(n.sum()) - np.repeat(np.cumsum(n) - n, n) + np.repeat(lo, n)
    return [probe[1][row], build[1][at]]


@pytest.mark.parametrize("n_build,n_probe", [(1, 5), (255, 256), (256, 257), (1000, 2049), (70000, 100003)])
@pytest.mark.parametrize("last", ["rows", "below", "at", "above", "far"])
@pytest.mark.parametrize("run", [1, 3, 200])
def test_join_over_either_index(cdl, n_build, n_probe, last, run):
    rng = np.random.default_rng(n_build + run)
    line = 2 * slots(n_build)  # the direct form holds keys below it
    top = {"rows": n_build, "below": line - 1, "at": line, "above": line + 1, "far": 0xFFFFFFFE}[last]
    key = np.sort(rng.integers(0, top + 1, (n_build + run - 1) // run).repeat(run)[:n_build])
    key[-1] = top
    build = [key.astype(np.uint32), rng.integers(0, 1 << 30, n_build).astype(np.uint32)]
    pk = np.where(rng.random(n_probe) < 0.5, key[rng.integers(0, n_build, n_probe)],
                  rng.integers(0, 2 * top + 2, n_probe)).clip(0, 0xFFFFFFFE)
    pk[:5] = [0, top, max(top - 1, 0), min(top + 1, 0xFFFFFFFE), 0xFFFFFFFE]
    probe = [pk.astype(np.uint32), rng.integers(0, 1 << 30, n_probe).astype(np.uint32)]
    want = reference(probe, build)
    got = cdl.join([dev(c) for c in probe], 0, [dev(c) for c in build], 0, [(0, 1), (1, 1)])
    for g, w in zip(got, want):
        assert np.array_equal(g.cpu().numpy().view(np.uint32), w)
    # an inequality leaves the same tuples in some order
    got = cdl.join([dev(c) for c in probe], 0, [dev(c) for c in build], 0, [(0, 1), (1, 1)],
                   neq=[((0, 1), (1, 1))])
    keep = want[0] != want[1]
    a = np.sort(got[0].cpu().numpy().view(np.uint32).astype(np.uint64) << 32
                | got[1].cpu().numpy().view(np.uint32))
    assert np.array_equal(a, np.sort(want[0][keep].astype(np.uint64) << 32 | want[1][keep]))


def test_join_refuses_a_small_output(cdl):
    a = [dev(np.arange(10)), dev(np.arange(10))]
    with pytest.raises(cdl.CdlError) as ex:
        cdl.join(a, 0, a, 0, [(0, 1), (1, 1)], out_cap=9)
    assert ex.value.name == "CDL_E_CAPACITY"
    assert len(cdl.join(a, 0, a, 0, [(0, 1), (1, 1)], out_cap=12)[0]) == 10
    empty = [dev(np.zeros(0)), dev(np.zeros(0))]
    assert len(cdl.join(a, 0, empty, 0, [(0, 1)])[0]) == 0
    assert len(cdl.join(empty, 0, a, 0, [(0, 1)])[0]) == 0


@pytest.mark.parametrize("kind", ["unique", "runs", "one-key", "gap", "sparse", "dense-then-far"])
def test_join_over_offsets(cdl, kind):
    """From 2^22 build rows the entries by key become offsets: gaps and runs
    longer than a tile of the fill, and keys that leave them to the hash form."""
    n = (1 << 22) + 5
    rng = np.random.default_rng(7)
    if kind == "unique":
        key = np.unique(rng.integers(0, 3 * n, 2 * n))[:n]
    elif kind == "runs":
        key = np.sort(rng.integers(0, 900, n))
    elif kind == "one-key":
        key = np.full(n, 123_457)
    elif kind == "gap":
        key = np.concatenate([np.arange(n // 2), np.arange(n - n // 2) + 3 * n])
    elif kind == "sparse":
        key = np.sort(rng.integers(0, 1 << 32, n) & 0xFFFFFFFE)
    else:
        key = np.arange(n)
        key[-1] = 0xFFFFFFFE
    m = 100_003
    build = [key.astype(np.uint32), rng.integers(0, 1 << 30, len(key)).astype(np.uint32)]
    probe = [np.where(rng.random(m) < 0.5, key[rng.integers(0, len(key), m)],
                      rng.integers(0, int(key[-1]) + 1000, m)).clip(0, 0xFFFFFFFE).astype(np.uint32),
             rng.integers(0, 1 << 30, m).astype(np.uint32)]
    if kind in ("runs", "one-key"):  # few probe rows meet long runs
        probe = [c[:4 if kind == "one-key" else 50] for c in probe]
    got = cdl.join([dev(c) for c in probe], 0, [dev(c) for c in build], 0, [(0, 1), (1, 1)])
    for g, w in zip(got, reference(probe, build)):
        assert np.array_equal(g.cpu().numpy().view(np.uint32), w)
