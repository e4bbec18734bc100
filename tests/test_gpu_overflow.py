"""Grouped levels whose slabs or fine buckets overflow: the build goes to the
path that needs no bounds and ends as it does there, with the oracle's function
or with MPHF_EDUPLICATE, whatever the arenas held before."""
import numpy as np
import pytest

import oracle
from paper_1702_03154_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1702_03154_gb300 import mphf
    return mphf


def duplicate(M, build):
    with pytest.raises(M.MPHFError) as e:
        build()
    assert e.value.code == M.EDUPLICATE


# gamma 200: 4400 fine buckets of 655 keys (capacity 928), 35 slabs of 84e3
# (86.3e3): 300 equal keys overflow a bucket, 10000 a slab as well
@pytest.mark.parametrize("copies", [300, 1000, 10000, 500000])
@pytest.mark.parametrize("together", [True, False])
def test_equal_keys(M, copies, together):
    keys = inputs.splitmix64_keys(2200 * 262144 // 200, 61)
    at = slice(7, 7 + copies) if together else slice(7, None, (keys.size - 7) // copies)
    keys[at] = keys[0]
    buf = torch.from_numpy(keys.view(np.int64)).cuda()
    duplicate(M, lambda: M.MPHF.build(buf, gamma=200.0))
    good = inputs.splitmix64_keys(keys.size, 62)  # the same arenas again
    g = M.MPHF.build(torch.from_numpy(good.view(np.int64)).cuda(), gamma=200.0, seed=4)
    o = oracle.build(good, gamma=200.0, levels=25, seed=4)
    assert g.build_path == 1 and g.levels() == o.levels() and np.array_equal(g.bits(), o.bits())


@pytest.mark.parametrize("scale", [0.5, 0.8, 0.975])
def test_small_capacities(M, scale):
    keys = inputs.splitmix64_keys(2200 * 262144 // 200, 63)
    o = oracle.build(keys, gamma=200.0, levels=25, seed=4)
    M.debug_config(0, scale)
    try:
        g = M.MPHF.build(torch.from_numpy(keys.view(np.int64)).cuda(), gamma=200.0, seed=4)
    finally:
        M.debug_config(0, 1.0)
    assert g.build_path == 2
    assert g.levels() == o.levels()
    assert np.array_equal(g.bits(), o.bits())
    assert np.array_equal(g.rank(), o.rank())
    assert np.array_equal(g.fallback(), o.fallback())


# gamma 2: a fine bucket has 2112 slots to spare
@pytest.mark.parametrize("copies", [3000, 5000, 1_000_000])
def test_equal_keys_of_a_large_set(M, copies):
    keys = M.keygen(300_000_000, 64)
    keys[11::keys.numel() // copies] = keys[0].clone()
    duplicate(M, lambda: M.MPHF.build(keys))


def test_equal_keys_of_a_large_part(M):
    keys = M.keygen(650_000_000, 65)
    keys[11::130_000] = keys[0].clone()
    duplicate(M, lambda: M.PartitionedMPHF.build(keys, 2, 77))
