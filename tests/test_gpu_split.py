"""The write-combining split of the bucketed build at its edges, against the oracle.

Every value must reach its bucket whatever the ring size (chosen by the number
of buckets), the alignment and order of the keys, and the rest of a round."""
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


def check(M, keys, gamma, shift=0, path=1):
    buf = torch.empty(keys.size + shift, dtype=torch.int64, device="cuda")
    buf[shift:] = torch.from_numpy(keys.view(np.int64)).cuda()
    g = M.MPHF.build(buf[shift:], gamma=gamma, levels=25, seed=4)
    o = oracle.build(keys, gamma=gamma, levels=25, seed=4)
    assert g.build_path == path
    assert g.levels() == o.levels()
    assert np.array_equal(g.bits(), o.bits())
    assert np.array_equal(g.rank(), o.rank())
    assert np.array_equal(g.fallback(), o.fallback())


# buckets at level 0 (262144 positions each) around the ring sizes: quanta of
# 32, 16, 8 and 4 values; one owned bucket per thread and two; past 2048, the
# two-step grouping (its last slab and last batch partly filled)
@pytest.mark.parametrize("buckets", [388, 395, 775, 790, 1024, 1025, 1545, 1570, 2048, 2049, 4500])
def test_ring_sizes(M, buckets):
    keys = inputs.splitmix64_keys(buckets * 262144 // 200, 5)
    check(M, keys, 200.0)


@pytest.mark.parametrize("n", [16385, 16384 + 1024, 152 * 1024 - 1, 152 * 1024 + 1,
                               152 * 8192 - 1, 152 * 8192 + 1, 2 * 152 * 8192 + 513])
@pytest.mark.parametrize("shift", [0, 1])
def test_rounds_and_alignment(M, n, shift):
    check(M, inputs.splitmix64_keys(n, 6), 2.0, shift)


@pytest.mark.parametrize("n", [50000, 3_000_017])
def test_keys_in_position_order(M, n):
    # a table laid out by the function itself and built again: every round's
    # values share a bucket, so the rings overflow all the time
    keys = inputs.splitmix64_keys(n, 7)
    o = oracle.build(keys, gamma=2.0, levels=25, seed=4)
    table = np.empty_like(keys)
    table[o.lookup(keys).astype(np.int64)] = keys
    check(M, table, 2.0)
