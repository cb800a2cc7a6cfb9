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
