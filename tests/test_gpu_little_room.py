"""A large build with too little device memory for its grouped levels still
ends in the same function, by the path that leaves the keys in their order."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_large_build_with_little_room():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1702_03154_gb300 import mphf as M
    # 4e8 keys, gamma 5: the grouped levels take 3.2 GB of slabs beside 0.25 GB
    # of A_0 and 0.6 GB of survivors, the other path 2.5 GB in all
    n, room = 400_000_000, 3_150_000_000
    keys = M.keygen(n, 96)
    queries = keys[::40].contiguous()
    want = M.MPHF.build(keys, gamma=5.0, levels=4, seed=5)
    assert want.build_path == 1
    idx = want.lookup(queries)
    levels = want.levels()
    want.free()
    torch.cuda.synchronize()
    M.pool_trim()
    torch.cuda.empty_cache()
    ballast = torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda")
    try:
        f = M.MPHF.build(keys, gamma=5.0, levels=4, seed=5)
    finally:
        del ballast
        torch.cuda.empty_cache()
    assert f.build_path == 2
    assert f.levels() == levels
    assert torch.equal(f.lookup(queries), idx)
    f.free()
    M.pool_trim()
