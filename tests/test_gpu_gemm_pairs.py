"""The prefill GEMM on CTA pairs (large products): row tiles whose second half is partly or wholly absent, two and three token
tiles with a ragged last one, rows that leave binary16's range, outputs of any row length, a recorded launch, and a wait that
runs out."""
import time

import numpy as np
import pytest

from oracle import aq_oracle as O
from paper_2605_24011_b200 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _case(M, N, K, bits, dtype):
    from paper_2605_24011_b200 import aq
    W = synth.weights_device(N, K, 41, outliers=True)
    h = aq.aq_pack(bits, 32, W)
    # the oracle on the rows around the tiles' edges and a few between
    rows = sorted({r for e in range(0, N + 1, 128) for r in (e - 1, e) if 0 <= r < N} | set(range(3, N, 997)) | {N - 1})
    d = O.quantize(W[torch.tensor(rows, device="cuda")].cpu().numpy(), bits)
    x = torch.from_numpy(synth.activations(M, K, 42, M, K)).to(torch.float16 if dtype == "f16" else torch.bfloat16)
    if dtype == "bf16":
        x[5] *= 2.0 ** 100
    toks = sorted({0, 5, M - 1} | {t for e in range(32, M, 32) for t in (e - 1, e)})
    want, T = O.linear(*d, x[toks].double().numpy())
    return aq, h, x.cuda(), rows, toks, want, T


@pytest.mark.parametrize("M,N,K,bits,dtype", [
    (400, 4112, 6912, 2, "f16"),     # two token tiles of 224; the last row tile has 16 rows, all of the first CTA
    (650, 2320, 9504, 3, "bf16"),    # three of 224; 16 rows in the last tile
    (512, 4224, 6912, 4, "bf16"),    # the last row tile has exactly the first CTA's half
    (385, 7682, 4096, 2, "bf16"),    # two of 224, the last with 161; row length not a multiple of four
])
def test_pairs(M, N, K, bits, dtype):
    aq, h, x, rows, toks, want, T = _case(M, N, K, bits, dtype)
    y = torch.empty((M, N), dtype=torch.float32, device="cuda")
    for _ in range(2):
        y.fill_(float("nan"))
        aq.aq_linear(h, x, y)
    aq.aq_check()
    got = y.double().cpu().numpy()
    assert np.isfinite(got).all()
    assert O.linear_excess(got[np.ix_(toks, rows)], want, T).max() <= 1.0


def test_a_recorded_pair_launch_is_replayed_on_new_input():
    M, N, K = 512, 11008, 4096
    aq, h, x, rows, toks, want, T = _case(M, N, K, 2, "f16")
    buf, y = torch.zeros_like(x), torch.empty((M, N), dtype=torch.float32, device="cuda")
    aq.aq_linear(h, buf, y)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        aq.aq_linear(h, buf, y)
    for scale in (1.0, 2.0):
        buf.copy_(x * scale)
        y.fill_(float("nan"))
        g.replay()
        torch.cuda.synchronize()
        aq.aq_check()
        assert O.linear_excess(y.double().cpu().numpy()[np.ix_(toks, rows)], scale * want, scale * T).max() <= 1.0
    del g


def test_a_wait_of_a_pair_runs_out_and_the_next_call_is_clean():
    M, N, K = 512, 11008, 4096      # 86 tiles of 256 x 256 on 74 pairs: most are stored by one run and added to by another
    aq, h, x, rows, toks, want, T = _case(M, N, K, 3, "f16")
    y = torch.empty((M, N), dtype=torch.float32, device="cuda")
    aq.aq_linear(h, x, y)
    aq.aq_check()
    try:
        aq.aq_debug_decode_hold(True)
        t0 = time.time()
        aq.aq_linear(h, x, y)
        with pytest.raises(aq.AqError) as err:
            aq.aq_check()
        assert err.value.status == aq.AQ_ERR_TIMEOUT
        assert time.time() - t0 < 10.0
    finally:
        aq.aq_debug_decode_hold(False)
    y.fill_(float("nan"))
    aq.aq_linear(h, x, y)
    aq.aq_check()
    assert O.linear_excess(y.double().cpu().numpy()[np.ix_(toks, rows)], want, T).max() <= 1.0
