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
    wrong, done = [], []

    def work(order):
        try:
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                for i in order:
                    h = aq.aq_pack(cases[i][2], 32, data[i][0])
                    if not np.array_equal(aq.aq_export(h), data[i][1]):
                        wrong.append(i)
                    h.free()
                    done.append(i)
        except Exception as e:                        # (an exception that ends a thread ends nothing else)
            wrong.append(e)

    n = len(cases)
    threads = [threading.Thread(target=work, args=([(5 * k + 2 * t) % n for k in range(2 * n)],)) for t in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong, wrong
    assert len(done) == 3 * 2 * n


def test_exports_that_go_round_the_ring():
    """22.5 MB and 9.0 MB through eight chunks of 1 MB, with ragged last chunks; then from two threads at once, one of which
    gets the ring and the other an ordinary copy."""
    from paper_2605_24011_b200 import aq
    cases = [(11008, 4096, 3), (2305, 6272, 4)]
    data = [_case(N, K, b, 8) for N, K, b in cases]
    handles = [aq.aq_pack(b, 32, W) for (_, _, b), (W, _) in zip(cases, data)]
    for h, (_, want) in zip(handles, data):
        assert np.array_equal(aq.aq_export(h), want)
    wrong, done = [], []

    def work(i):
        try:
            for _ in range(6):
                if not np.array_equal(aq.aq_export(handles[i]), data[i][1]):
                    wrong.append(i)
                done.append(i)
        except Exception as e:
            wrong.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in (0, 0, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong and len(done) == 18, wrong


def test_another_threads_recording_survives_a_freed_handle():
    """A CUDA graph is being recorded (thread-local rules: what other threads allocate and free is their own affair) while a
    second thread quantises, exports and frees, handles that it has computed with among them."""
    from paper_2605_24011_b200 import aq
    W, want = _case(256, 512, 3, 7)
    aq.aq_export(aq.aq_pack(3, 32, W))                # (set-up that happens once is done)
    x = torch.zeros((1, 512), dtype=torch.float16, device="cuda")
    y = torch.empty((1, 256), dtype=torch.float16, device="cuda")
    a = torch.zeros(1024, device="cuda")
    side, errors = torch.cuda.Stream(), []
    torch.cuda.synchronize()

    def work():
        try:
            for use in (False, True):
                h = aq.aq_pack(3, 32, W, stream=side)
                if use:
                    aq.aq_linear(h, x, y, stream=side)
                assert np.array_equal(aq.aq_export(h), want)
                h.free()
        except Exception as e:                        # an assertion, too, has to reach the test's thread
            errors.append(e)

    aq.aq_linear(aq.aq_pack(3, 32, W), x, y)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="thread_local"):
        a.add_(1.0)
        t = threading.Thread(target=work)
        t.start()
        t.join()
        a.add_(1.0)
    assert not errors, errors
    graph.replay()
    torch.cuda.synchronize()
    assert float(a[0]) == 2.0


def test_blocks_of_handles_used_on_two_streams_are_not_handed_on_early():
    """A handle made on one stream, at work on another, freed at once: its memory is not another handle's while the work
    lasts, whatever its last stream is."""
    from paper_2605_24011_b200 import aq
    N, K = 4096, 4096
    W = torch.from_numpy(synth.weights(N, K, 96)).cuda()
    x = torch.from_numpy(synth.activations(64, K, 96)).half().cuda()
    want = torch.empty((64, N), dtype=torch.float32, device="cuda")
    aq.aq_linear(aq.aq_pack(2, 32, W), x, want)
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    y = torch.empty_like(want)
    torch.cuda.synchronize()
    for rep in range(10):
        h = aq.aq_pack(2, 32, W, stream=s1)
        s2.wait_stream(s1)
        for _ in range(20):
            aq.aq_linear(h, x, y, stream=s2)
        aq.aq_info(h)                                 # (waits for s2, then the last stream is s1 again)
        for _ in range(20):
            aq.aq_linear(h, x, y, stream=s2)
        aq.aq_dequant(h, torch.empty((N, K), dtype=torch.float16, device="cuda"), stream=s1)
        h.free()
        g = aq.aq_pack(4, 32, W * 3.0, stream=s1)     # would write over the other's codes
        torch.cuda.synchronize()
        g.free()
        assert (y - want).abs().max().item() <= 1e-3 * want.abs().max().item(), rep
