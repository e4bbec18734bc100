"""Builds of mid-sized sets from several threads, each on its own stream: their
cooperative launches take turns, and every function is the one built alone."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_builds_of_four_threads():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1702_03154_gb300 import mphf as M
    sizes = [20_000, 300_000, 2_000_000, 3_400_000, 9_000_000]
    keys = [M.keygen(n, 5 + i) for i, n in enumerate(sizes)]
    ref = [M.MPHF.build(k, seed=3) for k in keys]
    want = [f.lookup(k) for f, k in zip(ref, keys)]
    levels = [f.levels() for f in ref]
    torch.cuda.synchronize()
    bad = []

    def work(t):
        try:
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                for i in np.random.default_rng(t).integers(0, len(sizes), 60):
                    f = M.MPHF.build(keys[i], seed=3, stream=s)
                    out = f.lookup(keys[i], stream=s)
                    s.synchronize()
                    if f.levels() != levels[i] or not torch.equal(out, want[i]):
                        bad.append((t, int(i)))
        except Exception as e:  # noqa: BLE001
            bad.append((t, repr(e)))

    threads = [threading.Thread(target=work, args=(t,)) for t in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
