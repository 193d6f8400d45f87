"""aq_dequant at the edges of what a CTA takes: one to three slabs of 128 k and odd numbers of them, row tiles that leave a group of
four unfilled, and rows on both sides of the length from which float32 goes along the rows.  Bit for bit against the oracle, with
guards behind the matrix."""
import numpy as np
import pytest

from oracle import aq_oracle as O
from paper_2605_24011_b200 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", (1, 48, 65, 209))
@pytest.mark.parametrize("K,bits", [(32, 2), (128, 3), (160, 4), (288, 2), (576, 3), (896, 4), (3200, 2), (3232, 3), (3360, 4)])
def test_dequant_tiles(N, K, bits):
    from paper_2605_24011_b200 import aq
    W = synth.weights(N, K, 14, bits, N, outliers=True)
    h = aq.aq_pack(bits, 32, torch.from_numpy(W).cuda())
    d, m, q = O.quantize(W, bits)
    for name, dt, view in (("f16", torch.float16, np.uint16), ("bf16", torch.bfloat16, np.uint16), ("f32", torch.float32, np.uint32)):
        buf = torch.full((N * K + 64,), float("nan"), dtype=dt, device="cuda")
        aq.aq_dequant(h, buf[:N * K].view(N, K))
        got = buf[:N * K].view(N, K).view(torch.int16 if view is np.uint16 else torch.int32).cpu().numpy().view(view)
        assert np.array_equal(got, O.dequant(d, m, q, name)), name
        assert bool(torch.isnan(buf[N * K:].float()).all())
    h.free()
