"""Keys that are not spread over their range (needs a GPU): results, and times that stay in proportion.

The batch sort's buckets are equal parts of the range that samples of the batch span, so clusters, long tails and a few
outliers put most of a batch in one bucket.  Comparisons of results are exact; comparisons of times have room for more
than twice the ratio that was measured.
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
    if dist == "spread":
        return rng.integers(0, TOP, n).astype(np.uint32)
    if dist == "log":        # as many keys in every octave: three quarters of them in the lowest 256th of the range
        return np.exp(rng.random(n) * np.log(TOP - 1)).astype(np.uint32)
    if dist == "tail":       # ids below 2^24, one key in fifty anywhere
        return np.where(rng.random(n) < 0.02, rng.integers(0, TOP, n), rng.integers(0, 1 << 24, n)).astype(np.uint32)
    if dist == "clusters":   # ten clusters of 2^14 keys
        return (rng.integers(0, TOP - (1 << 16), 10)[rng.integers(0, 10, n)] + rng.integers(0, 1 << 14, n)).astype(np.uint32)
    if dist == "pile":       # a cluster of 2^8 keys and a long tail on both sides
        return np.clip((1 << 30) + rng.standard_cauchy(n) * 100, 0, TOP - 1).astype(np.uint32)
    raise ValueError(dist)


def seconds(f, reps):
    """Shortest of some timings of `reps` calls."""
    f()
    a, z = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = 1e9
    for _ in range(5):
        torch.cuda.synchronize()
        a.record()
        for _ in range(reps):
            f()
        z.record()
        z.synchronize()
        best = min(best, a.elapsed_time(z) * 1e-3 / reps)
    return best


def sorter(g, dist, n, seed=5):
    rng = np.random.default_rng(n + seed)
    keys = (draw(dist, n, rng) << np.uint32(1)) | rng.integers(0, 2, n).astype(np.uint32)
    lsm = g.LSM(n, n)
    kd, vd = g.as_device_u32(keys, 0), g.as_device_u32(np.arange(n, dtype=np.uint32), 0)
    ko, vo = torch.zeros_like(kd), torch.zeros_like(vd)
    st = torch.cuda.current_stream().cuda_stream

    def run():
        g.lsm_sort_pairs(lsm.h, kd.data_ptr(), vd.data_ptr(), ko.data_ptr(), vo.data_ptr(), n, st)
    return lsm, keys, ko, vo, run


@pytest.mark.parametrize("n", [15400, 70001, 1 << 18, 1 << 20])
@pytest.mark.parametrize("dist", ["log", "tail", "clusters", "pile"])
def test_sort(g, dist, n):
    lsm, keys, ko, vo, run = sorter(g, dist, n)
    for _ in range(2):
        run()
        order = np.argsort(keys, kind="stable")
        np.testing.assert_array_equal(g.to_numpy_u32(ko), keys[order])
        np.testing.assert_array_equal(g.to_numpy_u32(vo), order.astype(np.uint32))
    assert lsm.device_errors() == 0
    lsm.close()


@pytest.mark.parametrize("dist", ["log", "tail"])
def test_sort_time_grows_with_the_batch(g, dist):
    """Four times the keys take about four times as long, not sixteen.  (Keys whose samples span the whole range at
    any size, so that the crowded bucket is as wide and holds the same share of the keys.)"""
    t = []
    for n in (1 << 18, 1 << 20):
        lsm, _, _, _, run = sorter(g, dist, n)
        t.append(seconds(run, 3))
        lsm.close()
    assert t[1] < 8.0 * t[0], t


@pytest.mark.parametrize("short", [0, 1, 30000])
@pytest.mark.parametrize("dist", ["log", "tail", "clusters", "pile"])
def test_levels(g, dist, short):
    """Batches with deletes, the last one padded, in both forms of the dictionary against the structural oracle."""
    b, rng = 100000, np.random.default_rng(short + len(dist))
    lsm, s, multi = g.LSM(b, 8 * b), oracle.StructuralOracle(b), g.MultiLSM([b, 33], 8)
    for t in range(3):
        n = b if t < 2 else b - short
        k, v = draw(dist, n, rng), rng.integers(0, 1 << 32, n, dtype=np.uint64).astype(np.uint32)
        d = (rng.random(n) < 0.2).astype(np.uint8)
        lsm.update(k, v, d)
        s.call("update", k, v, d)
        pad = [np.concatenate([x, np.zeros(b - n + 33, x.dtype)]) for x in (k, v, d)]
        multi.update(*pad, counts=np.asarray([n, 33], np.uint32))
    assert multi.sync()[0] == g.LSM_OK
    for lv in (lsm.levels(), multi.levels(0)):
        for i, (kv, vv) in lv.items():
            ekv, ev = s.level(i)
            np.testing.assert_array_equal(kv, ekv)
            np.testing.assert_array_equal(vv, ev)
    lsm.close()
    multi.close()


@pytest.mark.parametrize("sizes", [[1, 7, 8, 9], [63, 64, 65], [66, 200, 5000], [3, 64, 65, 1000]])
@pytest.mark.parametrize("shape", ["low", "high", "spread", "both"])
def test_searches_in_crowded_bins(g, sizes, shape):
    """Bins of the prefix index (2^15 keys wide here) of chosen sizes, with the keys at either end of the bin or spread
    over it: lookups and counts at every key, beside it and between the bins."""
    rng = np.random.default_rng(sum(sizes) + len(shape))
    keys = []
    for i, m in enumerate(sizes * 6):
        x = {"low": np.arange(m), "high": (1 << 15) - 1 - np.arange(m), "spread": rng.choice(1 << 15, m, replace=False),
             "both": np.concatenate([np.arange(m // 2), (1 << 15) - 1 - np.arange(m - m // 2)])}[shape]
        keys.append(((3 * i + 1) << 15) + x)
    keys = np.sort(np.concatenate(keys + [[TOP - 1]])).astype(np.uint32)
    vals = rng.integers(0, 1 << 31, len(keys)).astype(np.uint32)
    lsm = g.LSM(len(keys), len(keys))
    lsm.bulk_build(keys, vals)
    q = np.unique(np.concatenate([keys, keys - 1, keys + 1, np.arange(0, TOP, 1 << 22), [0, TOP - 1, TOP]])).astype(np.uint32)
    at = np.minimum(np.searchsorted(keys, q), len(keys) - 1)
    hit = keys[at] == q
    val, found = lsm.lookup(q)
    np.testing.assert_array_equal(found.cpu().numpy(), hit.astype(np.uint8))
    np.testing.assert_array_equal(g.to_numpy_u32(val), np.where(hit, vals[at], 0))
    k1 = q[q < TOP]
    k2 = np.minimum(k1.astype(np.int64) + rng.integers(0, 70000, len(k1)), TOP - 1).astype(np.uint32)
    want = np.searchsorted(keys, k2, side="right") - np.searchsorted(keys, k1)
    np.testing.assert_array_equal(g.to_numpy_u32(lsm.count(k1, k2)), want)
    lsm.close()


def repeated(dist, n, space, rng):
    """Keys below `space` of which most are stored many times: evenly, as Zipf's, or a few runs among single keys."""
    if dist == "even":
        return rng.integers(0, space, n)
    if dist == "zipf":
        return (rng.zipf(1.3, n) * 7919) % space
    return np.where(rng.random(n) < 0.9, rng.integers(0, 9, n) * (space // 9), rng.integers(0, space, n))


@pytest.mark.parametrize("batches", [1, 3, 8, 16, 31])
@pytest.mark.parametrize("dist,space", [("even", 100), ("even", 3000), ("even", 1 << 16), ("zipf", 1 << 20), ("runs", 1 << 16)])
def test_windows_of_repeated_keys(g, batches, dist, space):
    """Counts and ranges over windows of one to all keys, each stored many times in a level and over the levels, with
    deletes and short batches, against the ordered map."""
    b, rng = 20000, np.random.default_rng(batches + space)
    lsm, o1 = g.LSM(b, 32 * b), oracle.MapOracle(b)
    for t in range(batches):
        n = b if t % 5 != 4 else b // 3
        k = repeated(dist, n, space, rng).astype(np.uint32)
        v = rng.integers(0, 1 << 32, n, dtype=np.uint64).astype(np.uint32)
        d = (rng.random(n) < (0.0 if t % 3 else 0.3)).astype(np.uint8)
        lsm.update(k, v, d)
        o1.call("update", k, v, d)
    k1 = np.concatenate([rng.integers(0, space, 200), rng.choice(k, 50), [0, 0, space]])
    w = rng.choice([0, 1, 2, 7, 40, 300, 2500, 1 << 14, 1 << 16, 1 << 20], len(k1))
    k2 = np.minimum(k1 + w, TOP - 1)
    k1, k2 = k1.astype(np.uint32), k2.astype(np.uint32)
    np.testing.assert_array_equal(g.to_numpy_u32(lsm.count(k1, k2)), o1.count(k1, k2))
    off, rk, rv = lsm.range(k1, k2)
    eo, ek, ev = o1.range(k1, k2)
    np.testing.assert_array_equal(off.cpu().numpy().astype(np.uint64), eo)
    np.testing.assert_array_equal(g.to_numpy_u32(rk), ek)
    np.testing.assert_array_equal(g.to_numpy_u32(rv), ev)
    assert lsm.device_errors() == 0
    lsm.close()


def test_repeated_keys_are_skipped(g):
    """Counts over all of 31 batches: windows of as many elements are counted in less than half of the time when each
    key is stored a hundred times (a seventh was measured), since old versions are not read."""
    b, t = 1 << 17, []
    for space in (1 << 15, TOP):
        rng = np.random.default_rng(space % 101)
        lsm = g.LSM(b, 32 * b)
        for _ in range(31):
            lsm.insert(rng.integers(0, space, b).astype(np.uint32), np.zeros(b, np.uint32))
        k1 = g.as_device_u32(np.arange(256), 0)
        k2 = g.as_device_u32(np.full(256, TOP - 1), 0)
        t.append(seconds(lambda: lsm.count(k1, k2), 2))
        lsm.close()
    assert t[0] < 0.5 * t[1], t
