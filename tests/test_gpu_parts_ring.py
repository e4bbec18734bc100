"""The partitioned lookup's key ring at its edges, against the oracle: batches
around a block and the ring, ranges of one warp and of many, deep levels, every
layout, buffers off a 16-byte boundary, in place, 64-bit positions."""
import numpy as np
import pytest

import oracle
from paper_1702_03154_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
U = np.uint64


def mix(z):
    z = (z ^ (z >> U(30))) * U(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> U(27))) * U(0x94D049BB133111EB)
    return z ^ (z >> U(31))


@pytest.fixture(scope="module")
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1702_03154_gb300 import mphf as M
    K = 3
    keys = inputs.splitmix64_keys(300007, 87)
    q = np.concatenate([inputs.splitmix64_keys(200000, 88), inputs.shuffled(keys, 4)] * 6)

    def part(x):
        with np.errstate(over="ignore"):
            h = mix(x ^ mix(U(77)))
            return (((h >> U(32)) * U(K) + (((h & U(0xffffffff)) * U(K)) >> U(32))) >> U(32)).astype(int)

    want = np.empty_like(q)
    pk, pq, first = part(keys), part(q), 0
    for k in range(K):
        o = oracle.build(keys[pk == k], gamma=1.0, levels=25, seed=8)
        r = o.lookup(q[pq == k])
        want[pq == k] = np.where(r == U(M.NOT_FOUND), r, r + U(first))
        first += int((pk == k).sum())
    p = M.PartitionedMPHF.build(torch.from_numpy(keys.view(np.int64)).cuda(), K, 77, gamma=1.0, seed=8)
    return M, p, q, want


@pytest.mark.parametrize("layout", [32, 64, 8])
@pytest.mark.parametrize("wide", [False, True])
@pytest.mark.parametrize("n", [1, 31, 63, 64, 65, 447, 448, 449, 511, 512, 513, 4864 * 64,
                               4864 * 64 + 1, 2_900_000])
def test_batch_sizes(built, layout, wide, n):
    M, p, q, want = built
    for k in range(p.K):
        p.function(k).set_layout(layout)
    buf = torch.from_numpy(q[:n].view(np.int64)).cuda()
    off = torch.cat((buf[:1], buf))[1:]  # 8 bytes off
    out = torch.full((n + 3,), -5, dtype=torch.int64, device="cuda")
    M.debug_lookup_wide(wide)
    try:
        got = M.to_u64(p.lookup(buf))
        p.lookup(off, out=out[1:n + 1])
        p.lookup(buf, out=buf)
    finally:
        M.debug_lookup_wide(False)
    assert np.array_equal(got, want[:n])
    assert np.array_equal(M.to_u64(out[1:n + 1]), want[:n])
    assert out[0].item() == -5 and (out[n + 1:] == -5).all()  # nothing past the ends
    assert np.array_equal(M.to_u64(buf), want[:n])
