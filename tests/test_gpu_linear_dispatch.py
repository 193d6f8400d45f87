"""Linears of 1 to 8 tokens on both sides of the lines between the row-tile kernel, the streaming kernel that casts its own
sums and the streaming kernel with the cast as a launch of its own; two calls each, for the sums have to be zero again."""
import numpy as np
import pytest

from oracle import aq_oracle as O
from paper_2605_24011_b200 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,bits,M", [
    (40, 256, 3, 8), (40, 512, 3, 8), (40, 4096, 2, 3), (40, 4128, 2, 3), (2048, 4352, 4, 1), (2049, 4352, 4, 1), (1024, 4352, 2, 2),
    (1203, 8192, 4, 2), (1203, 8224, 2, 1), (1203, 8224, 4, 1), (1203, 416, 2, 8), (4737, 288, 3, 5), (11857, 288, 2, 4), (18945, 64, 4, 2)])
def test_dispatch_edges(N, K, bits, M):
    from paper_2605_24011_b200 import aq
    W = synth.weights(N, K, 51, N, K)
    h = aq.aq_pack(bits, 32, torch.from_numpy(W).cuda())
    for dt, odt in ((torch.float16, torch.float16), (torch.bfloat16, torch.float32)):
        x = torch.from_numpy(synth.activations(M, K, 52, M, K)).to(dt).cuda()
        y = torch.full((M, N), float("nan"), dtype=odt, device="cuda")
        for _ in range(2):
            aq.aq_linear(h, x, y)
        aq.aq_check()
        want, T = O.linear(*O.quantize(W, bits), x.double().cpu().numpy())
        assert O.linear_excess(y.double().cpu().numpy(), want, T).max() <= 1.0   # the library's bound of the exact product
    h.free()


@pytest.mark.parametrize("N,K,bits,M", [(2368, 14368, 2, 1), (2369, 14336, 2, 1), (2369, 14368, 4, 1), (4736, 14368, 3, 1), (4737, 14368, 2, 1)])
def test_dispatch_edges_of_long_rows(N, K, bits, M):
    test_dispatch_edges(N, K, bits, M)
