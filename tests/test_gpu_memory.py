"""Handles out of the block cache and exports through the pinned ring: bytes stay those of the oracle, whatever a block
held before and whichever thread asks."""
import threading

import numpy as np
import pytest

from oracle import aq_oracle as O
from paper_2605_24011_b200 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _case(N, K, bits, seed):
    W = synth.weights(N, K, 95, seed, outliers=True)
    return torch.from_numpy(W).cuda(), np.frombuffer(O.pack(*O.quantize(W, bits), bits), dtype=np.uint8)


# record bytes of a row segment per 512 k, with and without a tail; around the four 1 MB chunks where the ring starts
@pytest.mark.parametrize("N,K,bits", [(17, 32, 2), (33, 544, 3), (16, 512, 4), (2047, 4096, 3), (2731, 4096, 2), (2048, 4128, 3)])
def test_export_bytes(N, K, bits):
    from paper_2605_24011_b200 import aq
    W, want = _case(N, K, bits, N)
    assert np.array_equal(aq.aq_export(aq.aq_pack(bits, 32, W)), want)


def test_recycled_blocks_and_threads():
    from paper_2605_24011_b200 import aq
    cases = [(1200 + 16 * i, 4096, b) for i in range(3) for b in (2, 3, 4)]
    data = [_case(N, K, b, i) for i, (N, K, b) in enumerate(cases)]
    torch.cuda.synchronize()
    wrong = []

    def work(order):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            for i in order:
                h = aq.aq_pack(cases[i][2], 32, data[i][0])
                if not np.array_equal(aq.aq_export(h), data[i][1]):
                    wrong.append(i)
                h.free()

    n = len(cases)
    threads = [threading.Thread(target=work, args=([(5 * k + 2 * t) % n for k in range(2 * n)],)) for t in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong
