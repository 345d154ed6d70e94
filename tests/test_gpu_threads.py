"""Contexts of different sizes set up and run by several threads at once, each on its
own stream: every run equals the one of a context alone (resident rounds: the same
code on the same data, bit for bit)."""
import threading

import numpy as np
import pytest

import gridgen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1511_04519_gb300 import build
    build.build()
    from paper_1511_04519_gb300 import matex
    return matex


def test_resident_contexts_in_threads(M):
    import torch
    sides = [(6, 7), (45, 40), (12, 13), (50, 47), (30, 31), (20, 9), (40, 45), (25, 26)]
    probs = [gridgen.small_mesh(95 + k, nx=x, ny=y, n_src=6, group_templates=[2, 1], t_end=0.6e-9)
             for k, (x, y) in enumerate(sides)]
    alone = [M.Sim(p, resident="on").run().cpu().numpy() for p in probs]
    torch.cuda.synchronize()
    got, failed = [None] * len(probs), []

    def work(k):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                sim = M.Sim(probs[k], resident="on")
                for _ in range(3):
                    out = sim.run()
                torch.cuda.current_stream().synchronize()
                got[k] = out.cpu().numpy()
        except Exception as e:  # reported by the main thread
            failed.append((k, repr(e)))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(probs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
    for x, y in zip(got, alone):
        assert np.array_equal(x, y)
