"""The partitioned build of large parts, whose keys go to ranges of a fixed
capacity: the oracle's split and functions, and parts far from equal."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
U = np.uint64


@pytest.fixture(scope="module")
def M():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1702_03154_gb300 import mphf
    return mphf


def mix(z):
    z = (z ^ (z >> U(30))) * U(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> U(27))) * U(0x94D049BB133111EB)
    return z ^ (z >> U(31))


def unmix(z):
    z = (z ^ (z >> U(31)) ^ (z >> U(62))) * U(pow(0x94D049BB133111EB, -1, 1 << 64))
    z = (z ^ (z >> U(27)) ^ (z >> U(54))) * U(pow(0xBF58476D1CE4E5B9, -1, 1 << 64))
    return z ^ (z >> U(30)) ^ (z >> U(60))


@pytest.mark.parametrize("K,shift", [(2, 0), (3, 1)])
def test_parts_and_functions(M, K, shift):
    n = 18_000_000 * K + 12345
    buf = M.keygen(n + shift, 95)[shift:]
    p = M.PartitionedMPHF.build(buf, K, 77, seed=3)
    keys = M.to_u64(buf)
    with np.errstate(over="ignore"):
        h = mix(keys ^ mix(U(77)))
    part = (((h >> U(32)) * U(K) + (((h & U(0xffffffff)) * U(K)) >> U(32))) >> U(32)).astype(np.int64)
    want = np.concatenate(([0], np.cumsum(np.bincount(part, minlength=K))))
    assert np.array_equal(p.offsets.astype(np.int64), want)
    one = oracle.build(keys[part == 1], gamma=2.0, levels=25, seed=3)
    f = p.function(1)
    assert f.levels() == one.levels() and np.array_equal(f.bits(), one.bits())
    out = M.to_u64(p.lookup(buf))
    assert np.array_equal(out[part == 1], one.lookup(keys[part == 1]) + U(want[1]))
    assert np.array_equal(np.sort(out), np.arange(n, dtype=U))


def test_unequal_parts(M):
    # every key in part 0: its range overflows and the exact routing takes over
    n = 36_000_001
    with np.errstate(over="ignore"):  # hashes 0, 100, 200, ..: distinct, below 2^63
        keys = unmix(np.arange(n, dtype=U) * U(100)) ^ mix(U(77))
    buf = torch.from_numpy(keys.view(np.int64)).cuda()
    p = M.PartitionedMPHF.build(buf, 2, 77, seed=3)
    assert p.offsets.tolist() == [0, keys.size, keys.size]
    assert np.array_equal(np.sort(M.to_u64(p.lookup(buf))), np.arange(keys.size, dtype=U))
