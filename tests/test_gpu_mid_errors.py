"""What can go wrong with the cooperative launch of the mid-sized levels."""
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


def same(M, keys, f):
    o = oracle.build(keys, gamma=2.0, levels=25, seed=4)
    assert f.levels() == o.levels() and np.array_equal(f.bits(), o.bits())


# entered at level 0 and from buckets
@pytest.mark.parametrize("n", [100_003, 5_000_011])
def test_a_wait_that_gives_up(M, n):
    keys = inputs.splitmix64_keys(n, 71)
    buf = torch.from_numpy(keys.view(np.int64)).cuda()
    M.debug_mid(polls=0)
    try:
        with pytest.raises(M.MPHFError) as e:
            M.MPHF.build(buf, seed=4)
    finally:
        M.debug_mid()
    assert e.value.code == M.ETIMEOUT
    same(M, keys, M.MPHF.build(buf, seed=4))  # the context is usable


# a grid larger than the device holds, which the launch call refuses: the
# levels run in buckets, also behind grouped levels (3e8 keys)
@pytest.mark.parametrize("n", [16_385, 100_003, 5_000_011])
def test_a_refused_launch(M, n):
    keys = inputs.splitmix64_keys(n, 72)
    buf = torch.from_numpy(keys.view(np.int64)).cuda()
    M.debug_mid(ctas=1 << 20)
    try:
        f = M.MPHF.build(buf, seed=4)
        g = M.MPHF.build_host(keys, seed=4)
    finally:
        M.debug_mid()
    assert f.build_path == 1
    same(M, keys, f)
    same(M, keys, g)


def test_a_refused_launch_behind_grouped_levels(M):
    keys = M.keygen(300_000_000, 73)
    want = M.MPHF.build(keys, seed=4)
    M.debug_mid(ctas=1 << 20)
    try:
        f = M.MPHF.build(keys, seed=4)
    finally:
        M.debug_mid()
    q = keys[::1000].contiguous()
    assert f.build_path == 1 and f.levels() == want.levels()
    assert torch.equal(f.lookup(q), want.lookup(q))
