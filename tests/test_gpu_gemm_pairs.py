"""The prefill GEMM on CTA pairs (large products): row tiles whose second half is partly or wholly absent, two and three token
tiles with a ragged last one, rows that leave binary16's range, sums of any row length (aq_linear pads them, a program's buffers are
written straight from registers), a recorded launch, and a wait that runs out.  Each size is asked of the launcher's rule first."""
import time

import numpy as np
import pytest

from gemm_rule import gemm_shape
from oracle import aq_oracle as O
from paper_2605_24011_b200 import synth
from stack_check import check_program

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _on_pairs(tmp_path, M, N, K):
    return gemm_shape(tmp_path, N, K, M, torch.cuda.get_device_properties(0).multi_processor_count)[0] == 1


def _case(tmp_path, M, N, K, bits, dtype):
    from paper_2605_24011_b200 import aq
    assert _on_pairs(tmp_path, M, N, K)
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
    (385, 7682, 4096, 2, "bf16"),    # two of 224, the last with 161; two rows in the last row tile, sums padded
])
def test_pairs(tmp_path, M, N, K, bits, dtype):
    aq, h, x, rows, toks, want, T = _case(tmp_path, M, N, K, bits, dtype)
    y = torch.empty((M, N), dtype=torch.float32, device="cuda")
    for _ in range(2):
        y.fill_(float("nan"))
        aq.aq_linear(h, x, y)
    aq.aq_check()
    got = y.double().cpu().numpy()
    assert np.isfinite(got).all()
    assert O.linear_excess(got[np.ix_(toks, rows)], want, T).max() <= 1.0


@pytest.mark.parametrize("M,N,dtype", [(512, 7682, "f16"), (400, 7951, "bf16")])   # (the last row tile: 2 and 15 rows)
def test_buffers_written_from_registers(tmp_path, M, N, dtype):
    """Program buffers whose rows tensor copies cannot write: stored or added by the epilogue's own instructions, without and with a
    residual, rows that come scaled among them."""
    from paper_2605_24011_b200 import aq
    K = 4096
    assert N % 4 and _on_pairs(tmp_path, M, N, K)
    quant, handles = {}, []
    for i, bits in enumerate((3, 2)):
        W = synth.weights_device(N, K, 43 + i, outliers=True)
        handles.append(aq.aq_pack(bits, 32, W))
        host = W.cpu().numpy()
        quant[(0, str(i))] = lambda cols, host=host, bits=bits: O.quantize(host[cols], bits)
    prog = aq.Program([K, N, N], [{"w": handles[0], "src": 0, "dst": 1},
                                  {"w": handles[1], "src": 0, "dst": 2, "in_op": aq.AQ_IN_RMSNORM, "out_op": aq.AQ_OUT_ADD, "res": 1}])
    tdt = torch.float16 if dtype == "f16" else torch.bfloat16
    x = torch.from_numpy(synth.activations(M, K, 44, M)).to(tdt)
    if dtype == "bf16":
        x[5] *= 2.0 ** 20
    ws = torch.full((prog.workspace_bytes(M),), 255, dtype=torch.uint8, device="cuda")
    out = torch.empty((M, N), dtype=tdt, device="cuda")
    for _ in range(2):
        aq.aq_stack_forward(prog, x.cuda(), out, 2, M, ws)
    aq.aq_check()
    assert bool(torch.isfinite(aq.stack_buffer(prog, ws, M, 1)).all()) and bool(torch.isfinite(aq.stack_buffer(prog, ws, M, 2)).all())
    toks = sorted({0, 5, M - 1} | {t for e in range(32, M, 32) for t in (e - 1, e)})
    cols = sorted({r for e in range(0, N + 1, 128) for r in (e - 1, e) if 0 <= r < N} | set(range(3, N, 997)) | {N - 1})
    check_program(prog, [(0, "0"), (0, "1")], ws, M, tdt, lambda l, name, c: quant[(l, name)](c), rows=toks, cols_of=lambda l, name: cols)


def test_a_recorded_pair_launch_is_replayed_on_new_input(tmp_path):
    M, N, K = 512, 11008, 4096
    aq, h, x, rows, toks, want, T = _case(tmp_path, M, N, K, 2, "f16")
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


def test_a_wait_of_a_pair_runs_out_and_the_next_call_is_clean(tmp_path):
    M, N, K = 512, 11008, 4096      # 86 tiles of 256 x 256 on 74 pairs: most are stored by one run and added to by another
    aq, h, x, rows, toks, want, T = _case(tmp_path, M, N, K, 3, "f16")
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
