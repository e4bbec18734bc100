"""The single-CTA level loop at its edges, against the oracle: one warp and the
block, one and several keys a thread, gammas whose level sizes take the integer
and the double form, fallbacks left by either, in a build and in a batch."""
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


def same(g, o):
    assert g.levels() == o.levels()
    assert np.array_equal(g.bits(), o.bits())
    assert np.array_equal(g.rank(), o.rank())
    assert np.array_equal(g.fallback(), o.fallback())


@pytest.mark.parametrize("n", [1, 2, 31, 33, 127, 128, 129, 1023, 1025, 2048, 2049, 4097, 8192,
                               8193, 16383, 16384])
@pytest.mark.parametrize("gamma,levels", [(2.0, 25), (1.0, 3), (1.3, 25), (5.0, 1), (1.1, 6),
                                          (3000.0, 25)])
def test_tail_sizes(M, n, gamma, levels):
    if gamma > 100 and n > 1025:
        pytest.skip("the sizes of a level, not its keys, are the point at this gamma")
    keys = inputs.splitmix64_keys(n, 71)
    o = oracle.build(keys, gamma=gamma, levels=levels, seed=6)
    same(M.MPHF.build(torch.from_numpy(keys.view(np.int64)).cuda(), gamma=gamma, levels=levels,
                      seed=6), o)


@pytest.mark.parametrize("gamma,levels", [(2.0, 25), (1.3, 25), (1.0, 2), (9.0, 25)])
def test_batched_tails(M, gamma, levels):
    sizes = [0, 1, 5, 127, 128, 129, 511, 513, 1024, 1025, 4095, 4097, 8192, 8193, 20000]
    keys = inputs.splitmix64_keys(sum(sizes), 72)
    off = np.concatenate(([0], np.cumsum(sizes)))
    fs = M.build_batched(torch.from_numpy(keys.view(np.int64)).cuda(), off, gamma=gamma,
                         levels=levels, seed=7)
    for s, f in enumerate(fs):
        same(f, oracle.build(keys[off[s]:off[s + 1]], gamma=gamma, levels=levels, seed=7))
