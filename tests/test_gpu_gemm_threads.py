"""mpdo_gemm_tc from several threads, each on a stream of its own and with sizes of its
own (the tiles of 16, 32 and 64 columns, ragged edges, scratch beyond what the pool
keeps between calls): every product is bit for bit the one computed alone, as a shared
or early returned scratch buffer would not leave it, and both kinds agree."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_threads_and_streams():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_05871_gb300 import MIXED_BF16X3, MIXED_TF32
    from paper_2203_05871_gb300 import build as B
    from paper_2203_05871_gb300.mpdo import gemm_tc
    B.build()
    rng = np.random.default_rng(11)
    shapes = [(1, 1, 1), (128, 128, 64), (130, 400, 257), (1000, 1100, 70), (4096, 4200, 1500), (33, 17, 900)]
    data = [(torch.tensor(rng.standard_normal((m, k)), device="cuda"), torch.tensor(rng.standard_normal((k, n)), device="cuda"))
            for m, n, k in shapes]
    alone = [gemm_tc(a, b, MIXED_TF32).cpu() for a, b in data]
    torch.cuda.synchronize()
    bad = []

    def work(t):
        stream = torch.cuda.Stream()
        for r in range(6):
            q = (t + r) % len(data)
            with torch.cuda.stream(stream):
                c = gemm_tc(*data[q], MIXED_BF16X3 if (t + r) % 2 else MIXED_TF32, stream=stream)
                stream.synchronize()
                if not torch.equal(c.cpu(), alone[q]):
                    bad.append((t, r, q))

    threads = [threading.Thread(target=work, args=(t,)) for t in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
