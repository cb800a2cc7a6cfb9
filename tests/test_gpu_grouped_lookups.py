"""Lookups grouped by key range where the groups are uneven (needs a GPU): exact against the same in input order."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TOP = (1 << 31) - 1


@pytest.fixture(scope="module")
def g(lsm_lib):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return lsm_lib


def dictionary(g, b, batches, rng):
    lsm, keys = g.LSM(b, 128 * b), []
    for _ in range(batches):
        k = rng.integers(0, TOP, b).astype(np.uint32)
        lsm.update(k, rng.integers(0, 1 << 31, b).astype(np.uint32), (rng.random(b) < 0.2).astype(np.uint8))
        keys.append(k)
    return lsm, np.concatenate(keys)


def agree(g, lsm, q, mode):
    lsm.set_lookup_mode(g.LOOKUP_DIRECT)
    want = lsm.lookup(q)
    lsm.set_lookup_mode(mode)
    for _ in range(2):
        got = lsm.lookup(q)
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


@pytest.mark.parametrize("tiles", [512, 513, 600, 1100])
def test_parts_with_runs_in_few_tiles(g, tiles):
    """A part of the range with queries in the first and the last of many tiles of 8192 only, so that a chunk reaches
    over more than 512 of them: over a window of tiles without any, and into the last one."""
    rng = np.random.default_rng(tiles)
    lsm, keys = dictionary(g, 3000, 21, rng)
    low, high = keys[keys < 1 << 29], keys[keys > 3 << 29]
    q = np.full(tiles * 8192 - 5, low[7])
    for at in (0, len(q) - 40):
        q[at:at + 40] = np.concatenate([rng.choice(high, 20), rng.integers(3 << 29, TOP, 20)])
    q[4096:4096 + 3000] = rng.choice(keys, 3000)   # more than a chunk of some other parts, in one tile
    agree(g, lsm, g.as_device_u32(q.astype(np.uint32), 0), g.LOOKUP_SORTED)
    lsm.close()


def test_grouping_chosen_by_itself(g):
    """Seven levels and enough queries: the automatic mode groups them (several kernels instead of one)."""
    rng = np.random.default_rng(9)
    lsm, keys = dictionary(g, 1000, 127, rng)
    q = np.where(rng.random(1500000) < 0.5, rng.choice(keys, 1500000), rng.integers(0, 1 << 32, 1500000))
    q = g.as_device_u32(q.astype(np.uint32), 0)
    lsm.lookup(q)
    before = g.kernel_launches()
    lsm.lookup(q)
    assert g.kernel_launches() - before > 1
    agree(g, lsm, q, g.LOOKUP_AUTO)
    lsm.close()
