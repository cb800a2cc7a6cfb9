"""Count and range over wide windows (needs a GPU): one warp per query, windows in shared memory, in pieces when they
hold more than 512 elements; keys stored many times in a level and over the levels.  Exact against the ordered map."""

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TOP = (1 << 31) - 1


@pytest.fixture(scope="module")
def g(lsm_lib):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return lsm_lib


@pytest.mark.parametrize("r", [1, 2, 3, 7, 21, 31])
@pytest.mark.parametrize("space", [1, 40, 3000, 200000, TOP])
def test_wide_windows(g, r, space):
    b, rng = 700, np.random.default_rng(r * 7 + space % 101)
    lsm, o1 = g.LSM(b, 64 * b), oracle.MapOracle(b)
    for t in range(r):
        n = b if t % 4 else b - 300           # short batches: many copies of one element
        k = rng.integers(0, space, n).astype(np.uint32)
        v = rng.integers(0, 1 << 32, n, dtype=np.uint64).astype(np.uint32)
        d = (rng.random(n) < 0.3).astype(np.uint8)
        lsm.call("update", k, v, d)
        o1.call("update", k, v, d)
    # windows of about 0 .. all elements, empty and reversed intervals, the ends of the key range
    w = space / max(1, r * b)
    k1 = rng.integers(0, space, 400)
    k2 = k1 + (rng.choice([0, 30, 45, 100, 500, 515, 2000, 30000], 400) * w).astype(np.int64) - 1
    k1 = np.concatenate([k1, [0, 0, 5, space]])
    k2 = np.concatenate([np.clip(k2, 0, TOP - 1), [TOP - 1, 0xFFFFFFFF, 4, TOP - 1]])
    k1, k2 = k1.astype(np.uint32), k2.astype(np.uint32)
    for _ in range(2):
        np.testing.assert_array_equal(g.to_numpy_u32(lsm.count(k1, k2)), o1.count(k1, k2))
        off, rk, rv = lsm.range(k1, k2)
        eo, ek, ev = o1.range(k1, k2)
        np.testing.assert_array_equal(off.cpu().numpy().astype(np.uint64), eo)
        np.testing.assert_array_equal(g.to_numpy_u32(rk), ek)
        np.testing.assert_array_equal(g.to_numpy_u32(rv), ev)
        lsm.cleanup()                          # the second time over what a cleanup leaves
    assert lsm.device_errors() == 0
    lsm.close()


@pytest.mark.parametrize("nq", [1, 8191, 8192, 8193, 70000, (1 << 20) + 77])
@pytest.mark.parametrize("qdist", ["mixed", "one", "narrow"])
def test_bulk_lookups_agree(g, nq, qdist):
    """Lookups grouped by key range against the same ones in input order: ragged tiles, all queries in one part of
    the range, keys outside the levels' range and above the user keys."""
    rng = np.random.default_rng(nq)
    lsm = g.LSM(5000, 32 * 5000)
    keys = (1 << 27) + rng.integers(0, 1 << 26, 11 * 5000)
    for t in range(11):
        k = keys[t * 5000:(t + 1) * 5000].astype(np.uint32)
        lsm.update(k, rng.integers(0, 1 << 32, 5000, dtype=np.uint64).astype(np.uint32), (rng.random(5000) < 0.2).astype(np.uint8))
    q = np.where(rng.random(nq) < 0.5, rng.choice(keys, nq), rng.integers(0, 1 << 32, nq))
    if qdist == "one":
        q = np.full(nq, keys[77])
    elif qdist == "narrow":
        q = keys[5] + rng.integers(0, 9, nq)
    q = g.as_device_u32(q.astype(np.uint32), 0)
    out = []
    for mode in (g.LOOKUP_DIRECT, g.LOOKUP_SORTED, g.LOOKUP_AUTO):
        lsm.set_lookup_mode(mode)
        out.append(lsm.lookup(q))
    for val, found in out[1:]:
        assert torch.equal(val, out[0][0]) and torch.equal(found, out[0][1])
    assert int(out[0][1].sum()) > 0 or nq == 1 or qdist != "mixed"
    lsm.close()
