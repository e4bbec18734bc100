"""Batches of 32-byte sector lookups that go without the ring (128 to 1024 keys
a resident warp), at the edges of that range, against the oracle's answers."""
import numpy as np
import pytest

import oracle
from paper_1702_03154_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

WARPS = 152 * 4 * 8  # resident at once


@pytest.fixture(scope="module")
def queries():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1702_03154_gb300 import mphf as M
    keys = inputs.splitmix64_keys(300007, 85)
    o = oracle.build(keys, gamma=1.0, levels=25, seed=8)
    q = np.concatenate([keys, inputs.splitmix64_keys(60000, 86)])
    dq = torch.from_numpy(q.view(np.int64)).cuda()
    want = torch.from_numpy(o.lookup(q).view(np.int64)).cuda()
    at = torch.randint(0, q.size, (1025 * WARPS,), device="cuda",
                       generator=torch.Generator(device="cuda").manual_seed(1))
    at[:400_000] = at[:400_000] % 60000 + keys.size  # a stretch of absent keys
    f = M.MPHF.build(torch.from_numpy(keys.view(np.int64)).cuda(), gamma=1.0, levels=25, seed=8)
    return M, f, dq[at], want[at]


@pytest.mark.parametrize("n", [128 * WARPS, 128 * WARPS + 1, 144 * WARPS - 5, 160 * WARPS + 1,
                               2_000_003, 1024 * WARPS - 31, 1024 * WARPS, 1024 * WARPS + 1])
@pytest.mark.parametrize("wide", [False, True])
def test_edges(queries, n, wide):
    M, f, q, want = queries
    out = torch.full((n + 3,), -5, dtype=torch.int64, device="cuda")
    M.debug_lookup_wide(wide)
    try:
        f.lookup(q[1:n + 1], out=out[1:n + 1])  # 8 bytes off a 16-byte boundary
        place = q[:n].clone()
        f.lookup(place, out=place)
    finally:
        M.debug_lookup_wide(False)
    assert torch.equal(out[1:n + 1], want[1:n + 1])
    assert out[0].item() == -5 and (out[n + 1:] == -5).all()  # nothing past the ends
    assert torch.equal(place, want[:n])
