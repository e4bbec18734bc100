"""A grouped level denser than level 0 (its size is rounded up by fewer bits)
whose fine buckets take one step of 16 slots more than level 0's."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", [24, 37])
def test_level_denser_than_the_first(seed):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1702_03154_gb300 import mphf as M
    # level 0 asks for 65072.9988 slots a fine bucket and gets 65072; with these
    # seeds |F_1| asks for 65073 and gets 65088
    gamma = 2.0804748922918685
    keys = M.keygen(900_000_000, 3)
    queries = keys[::100].contiguous()
    f = M.MPHF.build(keys, gamma=gamma, seed=seed)
    assert f.build_path == 1
    idx, levels = f.lookup(queries), f.levels()
    f.free()
    M.debug_config(1)
    try:
        g = M.MPHF.build(keys, gamma=gamma, seed=seed)
    finally:
        M.debug_config(0)
    assert g.levels() == levels
    assert torch.equal(g.lookup(queries), idx)
    g.free()
    M.pool_trim()
