"""The lookup's key ring at its edges, against the oracle: batches around a
block and the ring, ranges of one warp and of many, deep levels (gamma 1, most
queries absent), every layout, buffers off a 16-byte boundary, in place."""
import numpy as np
import pytest

import oracle
from paper_1702_03154_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1702_03154_gb300 import mphf as M
    keys = inputs.splitmix64_keys(300007, 81)
    o = oracle.build(keys, gamma=1.0, levels=25, seed=8)
    q = np.concatenate([inputs.splitmix64_keys(200000, 82), inputs.shuffled(keys, 4)] * 6)
    return M, torch.from_numpy(keys.view(np.int64)).cuda(), q, o.lookup(q)


@pytest.mark.parametrize("layout", [32, 64, 8])
@pytest.mark.parametrize("n", [1, 31, 63, 64, 65, 447, 448, 511, 512, 513, 4864 * 64,
                               4864 * 64 + 1, 2_900_000])
def test_batch_sizes(built, layout, n):
    M, keys, q, want = built
    f = M.MPHF.build(keys, gamma=1.0, levels=25, seed=8)
    f.set_layout(layout)
    buf = torch.from_numpy(q[:n].view(np.int64)).cuda()
    assert np.array_equal(M.to_u64(f.lookup(buf)), want[:n])
    off = torch.cat((buf[:1], buf))[1:]  # 8 bytes off
    out = torch.full((n + 3,), -5, dtype=torch.int64, device="cuda")
    f.lookup(off, out=out[1:n + 1])
    assert np.array_equal(M.to_u64(out[1:n + 1]), want[:n])
    assert out[0].item() == -5 and (out[n + 1:] == -5).all()  # nothing past the ends
    f.lookup(buf, out=buf)
    assert np.array_equal(M.to_u64(buf), want[:n])


def test_wide_positions(built):
    M, keys, q, want = built
    f = M.MPHF.build(keys, gamma=1.0, levels=25, seed=8)
    M.debug_lookup_wide(True)
    try:
        got = M.to_u64(f.lookup(torch.from_numpy(q.view(np.int64)).cuda()))
    finally:
        M.debug_lookup_wide(False)
    assert np.array_equal(got, want)
