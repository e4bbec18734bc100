"""Lookup descriptors of several functions share one allocation: releasing or
re-storing some of the functions leaves the others' answers as they are."""
import numpy as np
import pytest

import oracle
from paper_1702_03154_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batched", [False, True])
def test_shared_descriptors_outlive_their_neighbours(batched):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1702_03154_gb300 import mphf as M
    sizes = [1, 777, 20011, 64, 9000]
    keys = [inputs.splitmix64_keys(n, 30 + i) for i, n in enumerate(sizes)]
    want = [oracle.build(k, gamma=2.0, levels=25, seed=2).lookup(k) for k in keys]
    dk = [torch.from_numpy(k.view(np.int64)).cuda() for k in keys]
    if batched:
        fs = M.build_batched(torch.cat(dk), np.concatenate(([0], np.cumsum(sizes))), seed=2)
    else:
        fs = [M.MPHF.build(k, seed=2) for k in dk]

    def check(which):
        outs = M.lookup_multi([fs[i] for i in which], [dk[i] for i in which])
        for i, o in zip(which, outs):
            assert np.array_equal(M.to_u64(o), want[i])

    check([2, 2])            # one function twice, its descriptor made once
    check([0, 1, 2, 3, 4])   # the others' made together
    fs[1].free()
    fs[3].free()
    check([4, 0, 2])
    fs[0].set_layout(8)
    fs[2].set_layout(64)
    check([0, 2, 4])
    fs[2].free()
    check([0, 4])
