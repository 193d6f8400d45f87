"""The one-launch decode kernel at the edges of its tiles and of its dispatch, op by op against the oracle.

A unit is 128 rows x 256 k, a CTA's row tile of 128 rows may hold 1 to 8 fragments of 16, a row of a normalised input is
kept in registers up to 4096 elements (one token), read whole by every CTA up to 16384 elements (M K) and summed from
shares above that."""
import numpy as np
import pytest

from oracle import aq_oracle as O
from paper_2605_24011_b200 import synth
from stack_check import check_program

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _run(M, K, N, dtype, bits, spread):
    from paper_2605_24011_b200 import aq
    # x0 [96] -> h [K]; two linears on rmsnorm(h) (one phase); silu(g) * u -> h + W (..): every glue, sources packed
    shapes = [("in", K, 96), ("g", N, K), ("u", N, K), ("out", K, N), ("p", 40, K)]
    handles, quant = {}, {}
    for i, (nm, n, k) in enumerate(shapes):
        W = synth.weights(n, k, 91, M, K, N, i, outliers=True)
        b = bits[i % len(bits)]
        handles[nm] = aq.aq_pack(b, 32, torch.from_numpy(W).cuda())
        quant[(0, nm)] = O.quantize(W, b)
    widths = [96, K, N, N, K, 40]
    ops = [{"w": handles["in"], "src": 0, "dst": 1},
           {"w": handles["g"], "src": 1, "dst": 2, "in_op": aq.AQ_IN_RMSNORM},
           {"w": handles["u"], "src": 1, "dst": 3, "in_op": aq.AQ_IN_RMSNORM},
           {"w": handles["out"], "src": 2, "src2": 3, "dst": 4, "in_op": aq.AQ_IN_SILU_MUL, "out_op": aq.AQ_OUT_ADD, "res": 1},
           {"w": handles["p"], "src": 4, "dst": 5}]
    prog = aq.Program(widths, ops)
    tdt = torch.float16 if dtype == "f16" else torch.bfloat16
    x = synth.activations(M, 96, 92, M, K) * 8.0
    if spread:   # magnitudes of one block from 2^-12 to 2^4 of each other
        x *= np.exp2(np.linspace(-12, 4, 96, dtype=np.float32))[None, ::-1]
    x0 = torch.from_numpy(x).to(tdt).cuda()
    ws = torch.empty(prog.workspace_bytes(M), dtype=torch.uint8, device="cuda")
    out = torch.empty((M, 40), dtype=tdt, device="cuda")
    for _ in range(2):   # the second pass reuses the tables and the workspace
        aq.aq_stack_forward(prog, x0, out, 5, M, ws)
    aq.aq_check()
    check_program(prog, [(0, nm) for nm, _, _ in shapes], ws, M, tdt, quant)
    assert torch.equal(out, aq.stack_buffer(prog, ws, M, 5).to(tdt))


@pytest.mark.parametrize("M,K", [(1, 4096), (1, 4128), (2, 4096), (2, 8224), (3, 5440), (3, 5472), (5, 3264), (5, 3296), (8, 2048), (8, 2080)])
def test_row_norm_paths(M, K):
    _run(M, K, 224, "f16", (2, 3, 4), False)


@pytest.mark.parametrize("N", (32, 128, 160, 1152))
@pytest.mark.parametrize("M,dtype", [(1, "f16"), (1, "bf16"), (4, "f16"), (8, "bf16")])
def test_row_tiles(M, dtype, N):
    _run(M, 288, N, dtype, (4, 2, 3), False)


@pytest.mark.parametrize("bits", (2, 3, 4))
@pytest.mark.parametrize("M,dtype", [(1, "f16"), (1, "bf16"), (2, "f16"), (6, "bf16")])
def test_wide_magnitudes(M, dtype, bits):
    _run(M, 512, 96, dtype, (bits,), True)


@pytest.mark.parametrize("M,K,N,dtype", [
    (2, 1024, 2048, "f16"), (4, 1024, 2048, "bf16"), (6, 1024, 2048, "f16"), (8, 1024, 2048, "bf16"), (7, 1536, 2048, "f16"),   # under a unit
    (2, 2048, 13312, "bf16"), (3, 2048, 13312, "f16"), (5, 2048, 13312, "bf16"), (7, 2048, 13312, "f16"), (8, 2560, 13312, "bf16"),   # 4.3, 5.3
])
def test_units_per_phase(M, K, N, dtype):
    """Phases of a few and of many units per CTA: two and three collect teams, operands unpacked after the sums have been read and
    after the instructions have."""
    _run(M, K, N, dtype, (3, 2, 4), False)


def _emulated(d, m, q, x):
    """y and sum |x w| of the several-token arithmetic with binary16 activations, rounding where it rounds: the two half sums of
    a block are joined in binary32, two multiply-adds bring the block into the unit's sum (256 k), units are added in steps of
    2^-24.  d, m [N][blocks], q [N][K] (codes), x [M][K] (binary64)."""
    f32 = lambda v: v.astype(np.float32).astype(np.float64)
    N, K = q.shape
    M = x.shape[0]
    total = np.zeros((M, N))
    for u0 in range(0, K, 256):
        acc = np.zeros((M, N))
        for b in range(u0 // 32, (u0 + 256) // 32):
            s = slice(32 * b, 32 * b + 32)
            c = f32(x[:, s] @ q[:, s].astype(np.float64).T)
            sx = f32(x[:, s].sum(1))[:, None]
            acc = f32(d[:, b] * c + f32(m[:, b] * sx + acc))
        total += np.round(acc * 2.0 ** 24) * 2.0 ** -24
    return total


@pytest.mark.parametrize("bits", (2, 3, 4))
@pytest.mark.parametrize("M", (2, 3, 8))
def test_several_tokens_round_like_binary32(M, bits):
    """The error against binary64 is that of the binary32 steps (twice their root mean square leaves room for what the
    tensor core itself drops below a product's last place); codes used as subnormals with many leading zeros lost ten times
    that."""
    from paper_2605_24011_b200 import aq
    N, K = 256, 2048
    W = synth.weights(N, K, 93, bits)
    h = aq.aq_pack(bits, 32, torch.from_numpy(W).cuda())
    d, m, q = O.quantize(W, bits)
    prog = aq.Program([K, N], [{"w": h, "src": 0, "dst": 1}])
    x0 = torch.from_numpy(synth.activations(M, K, 94, M)).half().cuda()
    ws = torch.empty(prog.workspace_bytes(M), dtype=torch.uint8, device="cuda")
    aq.aq_stack_forward(prog, x0, None, 1, M, ws)
    aq.aq_check()
    x = x0.double().cpu().numpy()
    want, T = O.linear(d, m, q, x)
    d, m = (np.asarray(v, dtype=np.float64).reshape(N, K // 32) for v in (d, m))
    rms = lambda y: float(np.sqrt(np.mean(((y - want) / T) ** 2)))
    got, bound = rms(aq.stack_buffer(prog, ws, M, 1).double().cpu().numpy()), rms(_emulated(d, m, np.asarray(q).reshape(N, K), x))
    assert got <= 2.0 * bound, f"{got:.2e}, binary32 steps {bound:.2e}"


@pytest.mark.parametrize("dtype,positive", [("f16", False), ("f16", True), ("bf16", False)])
@pytest.mark.parametrize("bad", (float("inf"), float("-inf"), float("nan")))
def test_one_token_with_a_non_finite_element_is_the_first_of_two(bad, dtype, positive):
    """A sum that an infinite or undefined element has made infinite or undefined leaves the kernel as the largest or the smallest
    number its packed sums hold: the same one whether a token comes alone or with another (whose arithmetic is the tensor
    core's own).  `positive`: weights whose codes and minima keep the sign, so that some rows stay infinite."""
    from paper_2605_24011_b200 import aq
    N, K = 64, 512
    W = synth.weights(N, K, 95, int(positive))
    h = aq.aq_pack(3, 32, torch.from_numpy(np.abs(W) + np.float32(0.01) if positive else W).cuda())
    prog = aq.Program([K, N], [{"w": h, "src": 0, "dst": 1}])
    x = torch.ones((2, K), dtype=torch.float16 if dtype == "f16" else torch.bfloat16, device="cuda")
    x[0, 37] = bad
    got = []
    for M in (1, 2):
        ws = torch.empty(prog.workspace_bytes(M), dtype=torch.uint8, device="cuda")
        aq.aq_stack_forward(prog, x, None, 1, M, ws)
        aq.aq_check()
        got.append(aq.stack_buffer(prog, ws, M, 1)[0].clone())
    assert torch.equal(got[0], got[1])
    assert (got[0].abs() > 1e8).all() and (not positive or bad < 0 or bad != bad or (got[0] > 0).any())


@pytest.mark.parametrize("bits", (2, 3, 4))
@pytest.mark.parametrize("dtype", ("f16", "bf16"))
def test_one_token_with_an_outlier_that_meets_a_zero_weight(dtype, bits):
    """An activation of one token is a fixed-point number relative to the largest of its block: off by at most 2^-30 of it in
    the first groups (k mod 8 below 4) and 2^-26 in the second.  The outlier sits in a first group, where the weight decodes to
    0, and the small values in second groups only, so nothing hides those steps."""
    from paper_2605_24011_b200 import aq
    N, K = 96, 1024
    k = np.arange(K)
    W = np.abs(synth.weights(N, K, 96, bits)) + np.float32(0.01)
    W[:, k % 32 == 0] = 0.0
    x = synth.activations(1, K, 97) * np.float32(2.0 ** -8)
    x[:, k % 8 < 4] = 0.0
    x[:, k % 32 == 0] = 60000.0
    x0 = torch.from_numpy(x).to(torch.float16 if dtype == "f16" else torch.bfloat16).cuda()
    h = aq.aq_pack(bits, 32, torch.from_numpy(W).cuda())
    prog = aq.Program([K, N], [{"w": h, "src": 0, "dst": 1}])
    ws = torch.empty(prog.workspace_bytes(1), dtype=torch.uint8, device="cuda")
    aq.aq_stack_forward(prog, x0, None, 1, 1, ws)
    aq.aq_check()
    x = x0.double().cpu().numpy()
    d, m, q = O.quantize(W, bits)
    want, T = O.linear(d, m, q, x)
    d, m, q = (np.asarray(v, dtype=np.float64).reshape(N, K // 32, -1) for v in (d, m, q))
    xb = x.reshape(K // 32, 32)
    step = np.where(np.arange(32) % 8 < 4, 2.0 ** -30, 2.0 ** -26)
    fixed = (d[:, :, 0] * (q * step).sum(2) * np.abs(xb).max(1)).sum(1)
    # binary32: a handful of roundings of a block's two terms, then of the sums along k; 2^-25 per 256 columns when units are added
    terms = (np.abs(d[:, :, 0] * (q * xb).sum(2)) + np.abs(m[:, :, 0] * xb.sum(1))).sum(1)
    bound = fixed + 2.0 ** -21 * (terms + T[0]) + K / 256 * 2.0 ** -25
    err = np.abs(aq.stack_buffer(prog, ws, 1, 1).double().cpu().numpy()[0] - want[0])
    assert np.all(err <= bound), float((err / bound).max())
    assert fixed.max() > 10 * (bound - fixed).max()      # (the steps are what is tested)
