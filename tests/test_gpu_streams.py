"""What a call leaves running on its stream, and calls on several streams (needs a GPU)."""

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


@pytest.mark.parametrize("n", [3000, 1 << 19, 6000001])
def test_bulk_build_has_ended_when_it_returns(g, n):
    """A bulk build and a refused one leave nothing on their stream: their input may be overwritten and the levels
    used from another stream at once."""
    b, rng = max(64, n // 40), np.random.default_rng(n)
    lsm, s = g.LSM(b, 2 * n), oracle.StructuralOracle(b)
    k, v = rng.integers(0, TOP, n).astype(np.uint32), rng.integers(0, 1 << 31, n).astype(np.uint32)
    bad = k.copy()
    bad[n // 2] = TOP
    kd, vd, bd = (g.as_device_u32(x, 0) for x in (k, v, bad))
    side, other = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(3):
        with torch.cuda.stream(side):
            with pytest.raises(g.LSMError) as e:
                lsm.bulk_build(bd, vd)
            assert side.query() and e.value.status == g.LSM_ERR_KEY_RANGE and lsm.r == 0
            lsm.bulk_build(kd, vd)
            assert side.query()
        with torch.cuda.stream(other):
            val, found = lsm.lookup(kd)
            other.synchronize()
        assert bool(found.all())
        g.lsm_reset(lsm.h)
    lsm.bulk_build(kd, vd)
    s.call("insert", k, v)
    s.cleanup()
    for i, (kv, vv) in lsm.levels().items():
        ekv, ev = s.level(i)
        np.testing.assert_array_equal(kv, ekv)
        np.testing.assert_array_equal(vv, ev)
    lsm.close()


def built(g, n, rng):
    """A dictionary of n pairs in one go (its queries wait for no fold, so that they can be captured)."""
    lsm = g.LSM(4096, 2 * n)
    k = rng.choice(TOP, n, replace=False).astype(np.uint32) if n < 1 << 20 else np.arange(n, dtype=np.uint32) * 31
    lsm.bulk_build(k, rng.integers(0, 1 << 31, n).astype(np.uint32))
    return lsm, k


def test_grouped_lookups_on_two_streams(g):
    """Grouped lookups issued on two streams without an order between them, of growing and shrinking sizes."""
    rng = np.random.default_rng(3)
    lsm, k = built(g, 300000, rng)
    lsm.set_lookup_mode(g.LOOKUP_DIRECT)
    sizes = [70001, 1 << 20, 8193, 600000, (1 << 20) + 5, 300000]
    qs = [g.as_device_u32(np.where(rng.random(m) < 0.5, rng.choice(k, m), rng.integers(0, TOP, m)).astype(np.uint32), 0)
          for m in sizes]
    want = [lsm.lookup(q) for q in qs]
    lsm.set_lookup_mode(g.LOOKUP_SORTED)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    out = [tuple(torch.empty_like(x) for x in w) for w in want]
    torch.cuda.synchronize()
    for _ in range(5):
        for j, q in enumerate(qs):
            g.lsm_lookup(lsm.h, q.data_ptr(), q.numel(), out[j][0].data_ptr(), out[j][1].data_ptr(),
                         streams[j & 1].cuda_stream)
        torch.cuda.synchronize()
        for (val, found), (ev, ef) in zip(out, want):
            assert torch.equal(val, ev) and torch.equal(found, ef)
            val.zero_(), found.fill_(7)
        torch.cuda.synchronize()
    lsm.close()


def test_lookup_beside_captured_calls(g):
    """A captured count stays good when a later lookup needs more scratch, and a grouped lookup may be issued (and
    its scratch grow) while another stream is being captured."""
    rng = np.random.default_rng(4)
    lsm, k = built(g, 300000, rng)
    k1 = rng.integers(0, TOP - (1 << 20), 5000)
    a, z = g.as_device_u32(k1, 0), g.as_device_u32(k1 + rng.integers(0, 1 << 20, 5000), 0)
    want = lsm.count(a, z)
    got = torch.zeros_like(want)
    q = g.as_device_u32(rng.choice(k, 3 << 20), 0)
    val, found = torch.empty_like(q), torch.empty(q.numel(), dtype=torch.uint8, device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    lsm.set_lookup_mode(g.LOOKUP_SORTED)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        g.lsm_count(lsm.h, a.data_ptr(), z.data_ptr(), a.numel(), got.data_ptr(), torch.cuda.current_stream().cuda_stream)
        g.lsm_lookup(lsm.h, q.data_ptr(), 1 << 20, val.data_ptr(), found.data_ptr(), side.cuda_stream)
    torch.cuda.synchronize()
    assert bool(found[:1 << 20].all())
    for m in (2 << 20, 3 << 20):
        found.zero_()
        g.lsm_lookup(lsm.h, q.data_ptr(), m, val.data_ptr(), found.data_ptr(), torch.cuda.current_stream().cuda_stream)
        got.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(got, want) and int(found.sum()) == m
    lsm.close()
