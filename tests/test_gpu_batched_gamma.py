"""Batched sets around the largest one that a tail takes whole, at gammas whose
tails need more than half a multiprocessor's shared memory, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1702_03154_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gamma", [7.9, 8.1, 12.0, 15.9, 16.1, 40.0])
def test_sets_of_a_whole_tail(gamma):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1702_03154_gb300 import mphf as M
    sizes = [2048, 2049, 4096, 4097, 8191, 8192, 8193, 1, 20000]
    keys = [inputs.splitmix64_keys(n, 50 + i) for i, n in enumerate(sizes)]
    flat = torch.from_numpy(np.concatenate(keys).view(np.int64)).cuda()
    fs = M.build_batched(flat, np.concatenate(([0], np.cumsum(sizes))), gamma=gamma, seed=3)
    for f, k in zip(fs, keys):
        o = oracle.build(k, gamma=gamma, levels=25, seed=3)
        assert f.build_path == 3
        assert f.levels() == o.levels()
        assert np.array_equal(f.bits(), o.bits())
        assert np.array_equal(f.fallback(), o.fallback())
