"""The one-launch level loop between the buckets and the tail, against the
oracle: its smallest and largest sets, entered at level 0 and from buckets,
left to the tail, to a large fallback, and with nothing left."""
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


@pytest.mark.parametrize("n,gamma,levels", [
    (16385, 2.0, 25), (17000, 1.3, 25), (152 * 1024 + 1, 1.0, 25), (300001, 5.0, 25),
    (1_500_000, 11.0, 25),               # near the most bits of a level
    (1_600_000, 11.0, 25),               # past them: buckets first
    (3_500_000, 1.0, 25), (3_500_001, 1.0, 25), (3_500_001, 2.0, 25),
    (200_003, 1.0, 1), (1_000_003, 1.0, 3),   # a fallback past the tail's reach
    (1_000_003, 2.0, 6), (5_000_011, 1.0, 4),
    (20_000, 2000.0, 25),                # nothing left early
])
@pytest.mark.parametrize("shift", [0, 1])
def test_mid_levels(M, n, gamma, levels, shift):
    keys = inputs.splitmix64_keys(n, 91)
    buf = torch.empty(n + shift, dtype=torch.int64, device="cuda")
    buf[shift:] = torch.from_numpy(keys.view(np.int64)).cuda()
    g = M.MPHF.build(buf[shift:], gamma=gamma, levels=levels, seed=9)
    o = oracle.build(keys, gamma=gamma, levels=levels, seed=9)
    assert g.build_path == 1
    assert g.levels() == o.levels()
    assert np.array_equal(g.bits(), o.bits())
    assert np.array_equal(g.rank(), o.rank())
    assert np.array_equal(g.fallback(), o.fallback())


@pytest.mark.parametrize("copies", [2, 30000])
def test_equal_keys(M, copies):
    keys = inputs.splitmix64_keys(500000, 92)
    keys[:copies] = keys[copies]
    with pytest.raises(M.MPHFError) as e:
        M.MPHF.build(torch.from_numpy(keys.view(np.int64)).cuda())
    assert e.value.code == M.EDUPLICATE
