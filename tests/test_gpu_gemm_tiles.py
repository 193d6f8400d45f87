"""The prefill GEMM at the edges of its tiles: 256 rows (two row halves of 8 fragments), token tiles of up to 128 with two
sets of accumulators up to 64, k-slabs of 128 in pairs."""
import numpy as np
import pytest

from oracle import aq_oracle as O
from paper_2605_24011_b200 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", (9, 64, 65, 128, 129, 200, 257))
@pytest.mark.parametrize("N,K,bits,dtype", [(16, 160, 2, "f16"), (136, 288, 3, "bf16"), (260, 512, 4, "f16"), (520, 96, 3, "f16"), (384, 1056, 2, "bf16")])
def test_tile_edges(M, N, K, bits, dtype):
    from paper_2605_24011_b200 import aq
    tdt = torch.float16 if dtype == "f16" else torch.bfloat16
    W = synth.weights(N, K, 97, N, K, outliers=True)
    h = aq.aq_pack(bits, 32, torch.from_numpy(W).cuda())
    x = torch.from_numpy(synth.activations(M, K, 98, M, K)).to(tdt).cuda()
    y = torch.full((M, N), float("nan"), dtype=torch.float32, device="cuda")
    for _ in range(2):
        aq.aq_linear(h, x, y)
    aq.aq_check()
    want, T = O.linear(*O.quantize(W, bits), x.double().cpu().numpy())
    assert O.linear_excess(y.double().cpu().numpy(), want, T).max() <= 1.0
    half = torch.full((M, N), float("nan"), dtype=tdt, device="cuda")   # the sums rounded by the cast; the second call finds
    for _ in range(2):                                                  # the first one's sums in the scratch
        aq.aq_linear(h, x, half)
    aq.aq_check()
    # two runs' float32 sums may differ by their order and then round to neighbouring values
    ulp = 2.0 ** -10 if dtype == "f16" else 2.0 ** -7
    a, b = half.double().cpu().numpy(), y.double().cpu().numpy()
    assert np.all(np.abs(a - b) <= ulp * np.abs(b) + 1e-5 * T + 1e-7)


@pytest.mark.parametrize("out", ("half", "f32"))
@pytest.mark.parametrize("M", (9, 64, 65, 130))
@pytest.mark.parametrize("N,K,bits,dtype", [(17, 160, 2, "f16"), (135, 2080, 3, "bf16"), (262, 512, 4, "f16"), (1023, 96, 3, "bf16")])
def test_row_lengths_that_are_not_a_multiple_of_four(M, N, K, bits, dtype, out):
    """The GEMM's sums have padded rows then; whatever lies beside the output's rows is left alone."""
    from paper_2605_24011_b200 import aq
    tdt = torch.float16 if dtype == "f16" else torch.bfloat16
    odt = tdt if out == "half" else torch.float32
    W = synth.weights(N, K, 99, N, K, outliers=True)
    h = aq.aq_pack(bits, 32, torch.from_numpy(W).cuda())
    x = torch.from_numpy(synth.activations(M, K, 98, M, K)).to(tdt).cuda()
    room = torch.full((M * N + 64,), 7.0, dtype=odt, device="cuda")
    y = room[:M * N].view(M, N)
    for _ in range(2):
        y.fill_(float("nan"))
        aq.aq_linear(h, x, y)
    aq.aq_check()
    want, T = O.linear(*O.quantize(W, bits), x.double().cpu().numpy())
    u = 0.0 if out == "f32" else 2.0 ** (-11 if dtype == "f16" else -8)     # the output's own rounding
    assert np.all(np.abs(y.double().cpu().numpy() - want) <= 2e-3 * T + 1e-5 + u * np.abs(want))
    assert bool((room[M * N:] == 7.0).all())


@pytest.mark.parametrize("N", (38400, 38403))
def test_more_tiles_than_ctas_with_two_sets_of_accumulators(N):
    """Up to 64 tokens a CTA that goes from one tile to the next changes its set of accumulators: more than 148 tiles of 256
    rows."""
    from paper_2605_24011_b200 import aq
    M, K, bits = 33, 256, 2
    W = synth.weights(N, K, 100)
    h = aq.aq_pack(bits, 32, torch.from_numpy(W).cuda())
    x = torch.from_numpy(synth.activations(M, K, 98, M, K)).half().cuda()
    y = torch.full((M, N), float("nan"), dtype=torch.float32, device="cuda")
    aq.aq_linear(h, x, y)
    aq.aq_check()
    want, T = O.linear(*O.quantize(W, bits), x.double().cpu().numpy())
    assert O.linear_excess(y.double().cpu().numpy(), want, T).max() <= 1.0
