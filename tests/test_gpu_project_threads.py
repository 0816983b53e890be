"""Projections and products from several threads on their own streams at once give what each gives alone."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def test_threads():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2301_04259_gb300 import soap as S
    rng = np.random.default_rng(0)
    X = torch.from_numpy(rng.normal(0, 1, (300, 1001)).astype(np.float32)).to(DEV)
    mean = X.mean(0).contiguous()
    V = torch.from_numpy(rng.normal(0, 1, (128, 1001)).astype(np.float32)).to(DEV)
    ref = torch.empty((300, 128), device=DEV)
    S.soap_pca_project(X, mean, V, ref)
    torch.cuda.synchronize()
    failed = []

    def work():
        try:
            stream = torch.cuda.Stream()
            out = torch.empty((300, 128), device=DEV)
            with torch.cuda.stream(stream):
                for _ in range(50):
                    out.fill_(-1.0)
                    S.soap_pca_project(X, mean, V, out, stream=stream)
                    stream.synchronize()
                    if not torch.equal(out, ref):
                        failed.append("differs")
        except Exception as e:                                 # noqa: BLE001 (reported by the test)
            failed.append(repr(e))
    threads = [threading.Thread(target=work) for _ in range(8)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed[:3]
