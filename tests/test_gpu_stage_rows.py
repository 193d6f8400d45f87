"""The staging kernels of the prefill path at the edges of what a thread and a CTA hold.  For bfloat16: rows of one block, rows that
fill the registers of 256 threads (4096) and a block more, twice that and a block more, and rows that leave binary16's range.  The
kernel for binary16 reads four elements per thread and step at any row length; it gets the same rows."""
import pytest

from oracle import aq_oracle as O
from paper_2605_24011_b200 import synth
from stack_check import check_program

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _staged_rows(M, K, I, dtype, rows=None):
    from paper_2605_24011_b200 import aq
    bits = 3
    quant, handles = {}, []
    for i, (name, n, k) in enumerate((("plain", 32, K), ("gate", I, K), ("up", I, K), ("down", 32, I))):
        W = synth.weights(n, k, 61, i)
        handles.append(aq.aq_pack(bits, 32, torch.from_numpy(W).cuda()))
        quant[(0, name)] = O.quantize(W, bits)
    prog = aq.Program([K, 32, I, I, 32], [
        {"w": handles[0], "src": 0, "dst": 1, "in_op": aq.AQ_IN_PLAIN},
        {"w": handles[1], "src": 0, "dst": 2, "in_op": aq.AQ_IN_RMSNORM},
        {"w": handles[2], "src": 0, "dst": 3, "in_op": aq.AQ_IN_RMSNORM},
        {"w": handles[3], "src": 2, "src2": 3, "dst": 4, "in_op": aq.AQ_IN_SILU_MUL},
    ])
    tdt = torch.float16 if dtype == "f16" else torch.bfloat16
    x = torch.from_numpy(synth.activations(M, K, 62)).to(tdt)
    if dtype == "bf16":
        x[5] *= 2.0 ** 40      # (its squares still fit binary32)
    ws = torch.full((prog.workspace_bytes(M),), 255, dtype=torch.uint8, device="cuda")
    out = torch.empty((M, 32), dtype=tdt, device="cuda")
    aq.aq_stack_forward(prog, x.cuda(), out, 4, M, ws)
    aq.aq_check()
    check_program(prog, [(0, "plain"), (0, "gate"), (0, "up"), (0, "down")], ws, M, tdt, quant, rows=rows)


@pytest.mark.parametrize("dtype", ("bf16", "f16"))
@pytest.mark.parametrize("K,I", [(32, 4128), (4128, 96), (8224, 32), (96, 8224), (4096, 2048 + 32)])
def test_staged_rows(K, I, dtype):
    _staged_rows(9, K, I, dtype)


@pytest.mark.parametrize("K,I", [(32, 2048), (2080, 96), (4128, 2048 + 32)])   # (256 threads hold 2048)
def test_more_rows_than_ctas_at_once(K, I):
    """bfloat16: a thread has one group of eight elements in flight instead of two."""
    M = 4 * torch.cuda.get_device_properties(0).multi_processor_count + 9
    _staged_rows(M, K, I, "bf16", rows=[0, 5, 6, M // 2, M - 10, M - 9, M - 1])
