"""The batch sort over key ranges and repetitions (needs a GPU).

The bucket sort splits the sampled key range of the batch; these inputs put its edges to work: ranges of a few keys,
ranges away from zero and at the top, outliers that the sample misses, clusters that overflow one bucket, hot keys
(alone, several in one bucket, with the padding of a short batch among them).  Every comparison is exact.
"""

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


def draw(dist, n, rng):
    """n keys below 2^31 - 1."""
    if dist == "one":
        return np.full(n, 12345, np.uint32)
    if dist == "two":
        return rng.integers(TOP - 2, TOP, n).astype(np.uint32)
    if dist == "ids":
        return rng.permutation(n).astype(np.uint32)
    if dist == "offset":
        return (1500000000 + rng.integers(0, 3 * n, n)).astype(np.uint32)
    if dist == "outliers":   # a few keys far from the rest: the range they span leaves most buckets empty
        k = 700000000 + rng.integers(0, 1 << 18, n)
        at = rng.integers(0, n, max(1, n // 5000))
        k[at] = rng.integers(0, TOP, len(at))
        return k.astype(np.uint32)
    if dist == "cluster":    # half of the keys in 2^12 values, the rest spread
        return np.where(rng.random(n) < 0.5, 5000 + rng.integers(0, 1 << 12, n), rng.integers(0, TOP, n)).astype(np.uint32)
    if dist == "hot":        # one key three tenths, two neighbours a tenth each
        u = rng.random(n)
        k = rng.integers(0, TOP, n)
        return np.where(u < 0.3, 1 << 30, np.where(u < 0.4, (1 << 30) + 1, np.where(u < 0.5, (1 << 30) - 7, k))).astype(np.uint32)
    if dist == "zipf":
        return ((rng.zipf(1.1, n) % (1 << 30)).astype(np.uint64) * 0x9E3779B1 % (1 << 30)).astype(np.uint32)
    raise ValueError(dist)


DISTS = ["one", "two", "ids", "offset", "outliers", "cluster", "hot", "zipf"]


@pytest.mark.parametrize("n", [1, 511, 4097, 70001, 1 << 18, 1 << 20])
@pytest.mark.parametrize("dist", DISTS)
def test_sort_over_ranges(g, dist, n):
    rng = np.random.default_rng(n * 31 + DISTS.index(dist))
    # keys of sort_pairs are whole 32-bit words; values are positions, so stability shows
    keys = (draw(dist, n, rng) << np.uint32(1)) | rng.integers(0, 2, n).astype(np.uint32)
    vals = np.arange(n, dtype=np.uint32)
    lsm = g.LSM(n, n)
    kd, vd = g.as_device_u32(keys, 0), g.as_device_u32(vals, 0)
    ko, vo = torch.zeros_like(kd), torch.zeros_like(vd)
    g.lsm_sort_pairs(lsm.h, kd.data_ptr(), vd.data_ptr(), ko.data_ptr(), vo.data_ptr(), n,
                     torch.cuda.current_stream().cuda_stream)
    order = np.argsort(keys, kind="stable")
    np.testing.assert_array_equal(g.to_numpy_u32(ko), keys[order])
    np.testing.assert_array_equal(g.to_numpy_u32(vo), vals[order])
    assert lsm.device_errors() == 0
    lsm.close()


@pytest.mark.parametrize("short", [0, 1, 20000])
@pytest.mark.parametrize("dist", DISTS)
def test_levels_over_ranges(g, dist, short):
    """Five batches, the last one short (padded), against the structural oracle and the ordered map."""
    b, rng = 30000, np.random.default_rng(short + DISTS.index(dist))
    lsm, s, o1 = g.LSM(b, 8 * b), oracle.StructuralOracle(b), oracle.MapOracle(b)
    seen = []
    for t in range(5):
        n = b if t < 4 else b - short
        k = draw(dist, n, rng)
        v = rng.integers(0, 1 << 32, n, dtype=np.uint64).astype(np.uint32)
        d = (rng.random(n) < 0.2).astype(np.uint8)
        for x in (lsm, s, o1):
            x.call("update", k, v, d)
        seen.append(k)
    lv = lsm.levels()
    assert lsm.r == s.r
    for i, (kv, vv) in lv.items():
        ekv, ev = s.level(i)
        np.testing.assert_array_equal(kv, ekv)
        np.testing.assert_array_equal(vv, ev)
    keys = np.concatenate(seen)
    q = np.concatenate([rng.choice(keys, 4000), rng.choice(keys, 500) + 1, [0, TOP - 1, TOP, 0xFFFFFFFF],
                        rng.integers(0, TOP, 2000)]).astype(np.uint32)
    val, found = lsm.lookup(q)
    ev, ef = o1.lookup(q)
    np.testing.assert_array_equal(found.cpu().numpy(), ef)
    np.testing.assert_array_equal(g.to_numpy_u32(val), ev)
    k1 = np.minimum(q[:3000], TOP - 1)
    k2 = np.minimum(k1.astype(np.int64) + rng.integers(0, 300, len(k1)), TOP - 1).astype(np.uint32)
    np.testing.assert_array_equal(g.to_numpy_u32(lsm.count(k1, k2)), o1.count(k1, k2))
    assert lsm.device_errors() == 0
    lsm.close()


@pytest.mark.parametrize("n", [(1 << 20) + 1, 129 * 8192 - 1, 129 * 8192, 2500001])
@pytest.mark.parametrize("dist", ["one", "ids", "hot", "zipf"])
def test_long_sort_over_ranges(g, dist, n):
    """Above 2^20 elements: the four 8-bit passes, at the edges of their 8192-element tiles."""
    test_sort_over_ranges(g, dist, n)


@pytest.mark.parametrize("b", [64, 5000, (1 << 20) + 5])
def test_refused_batches_between_folds(g, b):
    """A batch with a key out of range is refused at every counter value: its fold may have been enqueued, and must
    leave the levels, the batch kept as level 0 and the later batches alone."""
    rng = np.random.default_rng(b)
    lsm, s = g.LSM(b, 16 * b), oracle.StructuralOracle(b)
    for t in range(9):
        for _ in range(1 + t % 3):
            bad = rng.integers(0, TOP, b).astype(np.uint32)
            bad[rng.integers(0, b)] = TOP + int(rng.integers(0, 3))
            with pytest.raises(g.LSMError) as e:
                lsm.insert(bad, np.zeros(b, np.uint32))
            assert e.value.status == g.LSM_ERR_KEY_RANGE
            assert lsm.r == s.r == t
        k, v = rng.integers(0, TOP, b).astype(np.uint32), rng.integers(0, 1 << 31, b).astype(np.uint32)
        lsm.insert(k, v)
        s.call("insert", k, v)
    for i, (kv, vv) in lsm.levels().items():
        ekv, ev = s.level(i)
        np.testing.assert_array_equal(kv, ekv)
        np.testing.assert_array_equal(vv, ev)
    lsm.close()


@pytest.mark.parametrize("b", [1, 33, 5119, 5120, 5121])
@pytest.mark.parametrize("dist", ["one", "ids", "hot", "zipf"])
def test_small_batches(g, dist, b):
    """Batches at the edge of the one-kernel sort, full and short, with the key check waited for and deferred (a bad
    batch then becomes placebos that no query sees)."""
    rng = np.random.default_rng(b)
    lsm, s, o1 = g.LSM(b, 32 * b), oracle.StructuralOracle(b), oracle.MapOracle(b)
    seen = []
    for t in range(9):
        n = b if t % 3 else max(1, b - b // 3)
        k, v = draw(dist, n, rng), rng.integers(0, 1 << 31, n).astype(np.uint32)
        d = (rng.random(n) < 0.3).astype(np.uint8)
        for x in (lsm, s, o1):
            x.call("update", k, v, d)
        seen.append(k)
    for i, (kv, vv) in lsm.levels().items():
        ekv, ev = s.level(i)
        np.testing.assert_array_equal(kv, ekv)
        np.testing.assert_array_equal(vv, ev)
    bad = draw(dist, b, rng)
    bad[-1] = TOP
    with pytest.raises(g.LSMError):
        lsm.insert(bad, np.zeros(b, np.uint32))
    g.lsm_set_option(lsm.h, g.LSM_OPT_KEY_CHECK, 1)
    lsm.insert(bad, np.zeros(b, np.uint32))
    assert lsm.r == 10 and lsm.device_errors() & 1
    q = np.concatenate(seen + [np.arange(50)]).astype(np.uint32)
    val, found = lsm.lookup(q)
    ev, ef = o1.lookup(q)
    np.testing.assert_array_equal(found.cpu().numpy(), ef)
    np.testing.assert_array_equal(g.to_numpy_u32(val), ev)
    lsm.close()


@pytest.mark.parametrize("n", [1, 4095, 4096, 4097, 13 * 4096 + 5, (1 << 20) + 3])
@pytest.mark.parametrize("dist", ["one", "ids", "zipf"])
def test_one_run_rebuilds(g, dist, n):
    """Bulk builds (twice, the second with the kept scratch) and cleanups of a single full level: the run is counted
    and written tile by tile.  Levels against the structural oracle."""
    b, rng = max(1, n // 5), np.random.default_rng(n)
    lsm = g.LSM(b, 8 * b + n)
    for _ in range(2):
        g.lsm_reset(lsm.h)
        k, v = draw(dist, n, rng), rng.integers(0, 1 << 31, n).astype(np.uint32)
        lsm.bulk_build(k, v)
        s = oracle.StructuralOracle(b)
        s.call("insert", k, v)
        s.cleanup()
        assert lsm.r == s.r
        for i, (kv, vv) in lsm.levels().items():
            ekv, ev = s.level(i)
            np.testing.assert_array_equal(kv, ekv)
            np.testing.assert_array_equal(vv, ev)
    g.lsm_reset(lsm.h)
    s = oracle.StructuralOracle(b)
    for t in range(2):   # two batches: one full level with deletes and old versions
        k, v = draw(dist, b, rng), rng.integers(0, 1 << 31, b).astype(np.uint32)
        d = (rng.random(b) < 0.4).astype(np.uint8)
        lsm.update(k, v, d)
        s.call("update", k, v, d)
    lsm.cleanup()
    s.cleanup()
    assert lsm.r == s.r
    for i, (kv, vv) in lsm.levels().items():
        ekv, ev = s.level(i)
        np.testing.assert_array_equal(kv, ekv)
        np.testing.assert_array_equal(vv, ev)
    assert lsm.device_errors() == 0
    lsm.close()
@pytest.mark.parametrize("n", [4095, 4096, 30000, 1 << 18, 1 << 20])
@pytest.mark.parametrize("words", ["many", "ends", "runs", "pair"])
def test_hot_words(g, words, n):
    """Words that a sort puts in buckets of their own: more of them than it has room for, the smallest and largest
    32-bit words, neighbours, and hot words with nothing else in the batch."""
    rng = np.random.default_rng(n + len(words))
    hot = {"many": 1 + rng.permutation(1 << 20)[:60] * 4093, "ends": [0, 1, 2, (1 << 32) - 3, (1 << 32) - 2, (1 << 32) - 1],
           "runs": list(range(1 << 31, (1 << 31) + 20)), "pair": [77, 3 << 30]}[words]
    keys = rng.choice(np.asarray(hot, np.int64), n)
    if words != "pair":
        keys = np.where(rng.random(n) < 0.3, rng.integers(0, 1 << 32, n), keys)
    keys = keys.astype(np.uint32)
    lsm = g.LSM(n, n)
    kd, vd = g.as_device_u32(keys, 0), g.as_device_u32(np.arange(n, dtype=np.uint32), 0)
    ko, vo = torch.zeros_like(kd), torch.zeros_like(vd)
    g.lsm_sort_pairs(lsm.h, kd.data_ptr(), vd.data_ptr(), ko.data_ptr(), vo.data_ptr(), n,
                     torch.cuda.current_stream().cuda_stream)
    order = np.argsort(keys, kind="stable")
    np.testing.assert_array_equal(g.to_numpy_u32(ko), keys[order])
    np.testing.assert_array_equal(g.to_numpy_u32(vo), order.astype(np.uint32))
    assert lsm.device_errors() == 0
    lsm.close()


@pytest.mark.parametrize("b", [1, 33, 1051, 5119, 5120, 5121])
@pytest.mark.parametrize("dist", ["two", "ids", "outliers", "hot"])
def test_small_batches_over_ranges(g, dist, b):
    """Batches around the largest that one CTA sorts, whose prefix-index entries several CTAs write: levels, and
    lookups and counts across the whole key range."""
    rng = np.random.default_rng(b + DISTS.index(dist))
    lsm, s, o1 = g.LSM(b, 8 * b), oracle.StructuralOracle(b), oracle.MapOracle(b)
    for t in range(5):
        n = b if t != 2 else max(1, b // 3)
        k, v = draw(dist, n, rng), rng.integers(0, 1 << 31, n).astype(np.uint32)
        d = (rng.random(n) < 0.2).astype(np.uint8)
        for x in (lsm, s, o1):
            x.call("update", k, v, d)
        for i, (kv, vv) in lsm.levels().items():
            ekv, ev = s.level(i)
            np.testing.assert_array_equal(kv, ekv)
            np.testing.assert_array_equal(vv, ev)
        q = np.concatenate([k, np.minimum(k + 1, TOP), np.linspace(0, TOP - 1, 3000).astype(np.uint32)]).astype(np.uint32)
        val, found = lsm.lookup(q)
        ev, ef = o1.lookup(q)
        np.testing.assert_array_equal(found.cpu().numpy(), ef)
        np.testing.assert_array_equal(g.to_numpy_u32(val), ev)
        k1 = np.sort(q)[:-1]
        k2 = np.sort(q)[1:]
        np.testing.assert_array_equal(g.to_numpy_u32(lsm.count(k1, k2)), o1.count(k1, k2))
    assert lsm.device_errors() == 0
    lsm.close()


@pytest.mark.parametrize("deletes", [0.0, 0.7, 1.0])
@pytest.mark.parametrize("batches", [1, 2, 4])
@pytest.mark.parametrize("b", [1, 5, 1000, 5200])
def test_cleanup_of_one_level(g, b, batches, deletes):
    """A single full level cleaned up into itself, into smaller levels or into nothing, and its prefix index."""
    rng = np.random.default_rng(b + batches)
    lsm, s, o1 = g.LSM(b, 8 * b), oracle.StructuralOracle(b), oracle.MapOracle(b)
    keys = draw("outliers" if b > 100 else "ids", b, rng)
    for t in range(batches):
        k = np.where(rng.random(b) < 0.5, keys, rng.integers(0, TOP, b)).astype(np.uint32)
        v, d = rng.integers(0, 1 << 31, b).astype(np.uint32), (rng.random(b) < deletes).astype(np.uint8)
        for x in (lsm, s, o1):
            x.call("update", k, v, d)
    lsm.cleanup()
    s.cleanup()
    assert lsm.r == s.r
    for i, (kv, vv) in lsm.levels().items():
        ekv, ev = s.level(i)
        np.testing.assert_array_equal(kv, ekv)
        np.testing.assert_array_equal(vv, ev)
    q = np.concatenate([keys, k, np.linspace(0, TOP - 1, 2000).astype(np.uint32)]).astype(np.uint32)
    val, found = lsm.lookup(q)
    ev, ef = o1.lookup(q)
    np.testing.assert_array_equal(found.cpu().numpy(), ef)
    np.testing.assert_array_equal(g.to_numpy_u32(val), ev)
    assert lsm.device_errors() == 0
    lsm.close()
