"""The write-combining split in sets past the reach of the one-launch level loop
(3.5e6 keys, 2^24 bits): rests of a round, alignment, and keys in position order,
whose rings overflow all the time; in one split, in grouped levels and by part."""
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


def launched(M, build):
    """(result, names of the kernels of a build)"""
    M.profile_report()
    M.profile_enable(True)
    try:
        g = build()
        torch.cuda.synchronize()
    finally:
        M.profile_enable(False)
    return g, set(M.profile_report())


def check(M, keys, gamma, kernels, shift=0):
    buf = torch.empty(keys.size + shift, dtype=torch.int64, device="cuda")
    buf[shift:] = torch.from_numpy(keys.view(np.int64)).cuda()
    g, names = launched(M, lambda: M.MPHF.build(buf[shift:], gamma=gamma, levels=25, seed=4))
    o = oracle.build(keys, gamma=gamma, levels=25, seed=4)
    assert g.build_path == 1 and kernels <= names
    assert g.levels() == o.levels()
    assert np.array_equal(g.bits(), o.bits())
    assert np.array_equal(g.rank(), o.rank())
    assert np.array_equal(g.fallback(), o.fallback())


# one value, most or all of a round of 152 CTAs more or less; a gamma of few keys
@pytest.mark.parametrize("n,gamma", [(3_500_001, 2.0), (3 * 152 * 8192 - 1, 2.0),
                                     (3 * 152 * 8192 + 1, 2.0), (4 * 152 * 8192 + 513, 2.0),
                                     (100_003, 200.0), (16_385, 2000.0)])
@pytest.mark.parametrize("shift", [0, 1])
def test_rounds_and_alignment(M, n, gamma, shift):
    check(M, inputs.splitmix64_keys(n, 6), gamma, {"split"}, shift)


def in_position_order(keys, gamma):
    o = oracle.build(keys, gamma=gamma, levels=25, seed=4)
    table = np.empty_like(keys)
    table[o.lookup(keys).astype(np.int64)] = keys
    return table


@pytest.mark.parametrize("n,gamma,kernels", [
    (4_000_037, 2.0, {"split"}), (20_000_003, 2.0, {"split"}), (400_009, 100.0, {"split"}),
    (2200 * 262144 // 200, 200.0, {"split_coarse", "split_fine"}),
    (4500 * 262144 // 500, 500.0, {"split_coarse", "split_fine"})])
def test_keys_in_position_order(M, n, gamma, kernels):
    check(M, in_position_order(inputs.splitmix64_keys(n, 7), gamma), gamma, kernels)


def test_large_set_in_position_order(M):
    keys = M.keygen(300_000_000, 66)
    f = M.MPHF.build(keys, seed=4)
    idx = f.lookup(keys)
    table = torch.empty_like(keys)
    table[idx] = keys
    del idx
    g, names = launched(M, lambda: M.MPHF.build(table, seed=4))
    assert g.build_path == 1 and {"split_coarse", "split_fine", "split"} <= names
    assert g.levels() == f.levels()
    q = keys[::100].contiguous()
    assert torch.equal(g.lookup(q), f.lookup(q))


@pytest.mark.parametrize("K", [2, 5])
def test_parts_in_order(M, K):
    # the keys of a part one after another: all go to the part's few rings
    n = 18_000_000 * K + 77
    keys = M.keygen(n, 67)
    p, names = launched(M, lambda: M.PartitionedMPHF.build(keys, K, 77, seed=3))
    assert "part_split" in names
    idx = p.lookup(keys)
    table = torch.empty_like(keys)
    table[idx] = keys
    r, names = launched(M, lambda: M.PartitionedMPHF.build(table, K, 77, seed=3))
    assert "part_split" in names
    assert np.array_equal(r.offsets, p.offsets)
    assert torch.equal(r.lookup(keys), idx)
