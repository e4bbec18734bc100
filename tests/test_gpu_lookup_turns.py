"""Batches of more than one turn of chunks a warp (their edges, a last turn that
is short or missing), against the oracle's answers."""
import numpy as np
import pytest

import oracle
from paper_1702_03154_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def queries():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1702_03154_gb300 import mphf as M
    keys = inputs.splitmix64_keys(300007, 83)
    o = oracle.build(keys, gamma=1.0, levels=25, seed=8)
    q = np.concatenate([keys, inputs.splitmix64_keys(60000, 84)])
    dq = torch.from_numpy(q.view(np.int64)).cuda()
    want = torch.from_numpy(o.lookup(q).view(np.int64)).cuda()
    at = torch.randint(0, q.size, (50_000_000,), device="cuda",
                       generator=torch.Generator(device="cuda").manual_seed(1))
    at[5_000_000:15_000_000] = at[5_000_000:15_000_000] % 60000 + keys.size  # a stretch of absent keys
    return M, torch.from_numpy(keys.view(np.int64)).cuda(), dq[at], want[at]


# a turn of every resident warp: 152 multiprocessors of 4 (32-byte sectors) and 3
# (64-byte) CTAs of 8 warps, 2048 keys each
@pytest.mark.parametrize("layout,turn", [(32, 4864 * 2048), (64, 3648 * 2048)])
@pytest.mark.parametrize("turns,more", [(2, 0), (2, 1), (2, 77_777), (3, -1), (4, 0), (4, 4_100_003)])
def test_turns(queries, layout, turn, turns, more):
    M, keys, q, want = queries
    n = turns * turn + more
    f = M.MPHF.build(keys, gamma=1.0, levels=25, seed=8)
    f.set_layout(layout)
    out = torch.full((n + 3,), -5, dtype=torch.int64, device="cuda")
    f.lookup(q[1:n + 1], out=out[1:n + 1])
    assert torch.equal(out[1:n + 1], want[1:n + 1])
    assert out[0].item() == -5 and (out[n + 1:] == -5).all()  # nothing past the ends


@pytest.mark.parametrize("layout", [32, 64, 8])
def test_turns_of_parts(queries, layout):
    M, keys, q, _ = queries
    p = M.PartitionedMPHF.build(keys, 3, 5, gamma=1.0)
    for k in range(3):
        p.function(k).set_layout(layout)
    want = torch.empty(q.numel(), dtype=torch.int64, device="cuda")
    for i in range(0, q.numel(), 1_000_000):  # one range a warp
        p.lookup(q[i:i + 1_000_000], out=want[i:i + 1_000_000])
    for n in (q.numel(), 33_333_333):
        out = torch.full((n + 1,), -5, dtype=torch.int64, device="cuda")
        assert torch.equal(p.lookup(q[:n], out=out[:n]), want[:n])
        assert out[n].item() == -5
