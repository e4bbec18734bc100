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
