"""aq_stack_forward recorded into a CUDA graph and replayed: every replay must pass the same per-op parity against
the oracle as an eager call (a replay runs with the arguments of the recording, so nothing in the library may depend on
per-launch host state), on the decode path (one cooperative kernel) and on the prefill path (grouped tensor-core launches)."""
import numpy as np
import pytest

from oracle import aq_oracle as O
from paper_2605_24011_b200 import synth
from stack_check import check_program

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def aq():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_24011_b200 import aq as mod
    return mod


@pytest.mark.parametrize("M,dtype", [(1, "f16"), (8, "f16"), (50, "bf16"), (300, "bf16"), (600, "bf16")])
def test_replayed_stack_matches_oracle(aq, M, dtype):
    from paper_2605_24011_b200 import programs
    tdt = torch.float16 if dtype == "f16" else torch.bfloat16
    shapes = synth.tiny_layer(256, 416)
    sizes = [N * K for _ in range(2) for (_, N, K) in shapes]
    bits = synth.draw_bits(sizes, 3.0, 6)
    layers, quant, i = [], {}, 0
    for l in range(2):
        L = {"shape": {}}
        for (name, N, K) in shapes:
            W = synth.weights(N, K, 41, l, i, outliers=True)
            L[name] = aq.aq_pack(bits[i], 32, torch.from_numpy(W).cuda())
            L["shape"][name] = (N, K)
            quant[(l, name)] = O.quantize(W, bits[i])
            i += 1
        layers.append(L)
    prog, out_buf, names = programs.block_program(layers)
    ws = torch.zeros(prog.workspace_bytes(M), dtype=torch.uint8, device="cuda")
    x0 = torch.from_numpy(synth.activations(M, 256, 41, M)).to(tdt).cuda()
    out = torch.empty((M, 256), dtype=tdt, device="cuda")
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        aq.aq_stack_forward(prog, x0, out, out_buf, M, ws)      # eager: builds the library's cached tables
        aq.aq_check(stream)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            aq.aq_stack_forward(prog, x0, out, out_buf, M, ws)
    for rep in range(3):
        x_new = torch.from_numpy(synth.activations(M, 256, 42 + rep, M)).to(tdt).cuda()
        x0.copy_(x_new)
        ws.zero_()
        out.zero_()
        graph.replay()
        torch.cuda.synchronize()
        aq.aq_check()
        check_program(prog, names, ws, M, tdt, quant)
        assert torch.equal(aq.stack_buffer(prog, ws, M, 0), x_new.float())
        assert torch.equal(out, aq.stack_buffer(prog, ws, M, out_buf).to(tdt))


@pytest.mark.parametrize("M", (1, 16))
def test_a_refused_launch_is_reported_once(aq, M):
    """The legacy stream may not be used beside the recording of a blocking stream: the call is refused with an error, and
    the next call, which is a good one, does not report it again."""
    rt = pytest.importorskip("cuda.bindings.runtime")
    N, K = 256, 512
    W = synth.weights(N, K, 43)
    h = aq.aq_pack(3, 32, torch.from_numpy(W).cuda())
    x = torch.zeros((M, K), dtype=torch.float16, device="cuda")
    y = torch.empty((M, N), dtype=torch.float16, device="cuda")
    out = torch.empty((N, K), dtype=torch.float16, device="cuda")
    aq.aq_linear(h, x, y)
    torch.cuda.synchronize()
    err, s = rt.cudaStreamCreateWithFlags(0)
    assert err == rt.cudaError_t.cudaSuccess
    assert rt.cudaStreamBeginCapture(s, rt.cudaStreamCaptureMode.cudaStreamCaptureModeThreadLocal)[0] == rt.cudaError_t.cudaSuccess
    refused = aq.raw_lib().aq_linear(h.raw, x.data_ptr(), y.data_ptr(), M, aq.AQ_F16, None)
    rt.cudaStreamEndCapture(s)
    rt.cudaGetLastError()                            # (this binding's own copy of the runtime)
    assert refused == aq.AQ_ERR_CUDA
    aq.aq_dequant(h, out, stream=torch.cuda.Stream())
    torch.cuda.synchronize()
    assert np.array_equal(out.view(torch.int16).cpu().numpy().view(np.uint16), O.dequant(*O.quantize(W, 3), "f16"))
    rt.cudaStreamDestroy(s)


@pytest.mark.parametrize("seen", (0, 12, 40))
@pytest.mark.parametrize("dtype,out", [("f16", "f32"), ("f16", "f16"), ("bf16", "bf16")])
def test_replayed_prefill_linear_matches_oracle(aq, dtype, out, seen):
    """A linear of 33 tokens, recorded as the handle's first call of more than 8, after one that needed less scratch, and after
    one that needed more."""
    N, K, M, bits = 272, 288, 33, 3
    tdt = {"f16": torch.float16, "bf16": torch.bfloat16, "f32": torch.float32}
    W = synth.weights(N, K, 44)
    h = aq.aq_pack(bits, 32, torch.from_numpy(W).cuda())
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    x = torch.zeros((M, K), dtype=tdt[dtype], device="cuda")
    y = torch.empty((M, N), dtype=tdt[out], device="cuda")
    with torch.cuda.stream(stream):
        aq.aq_linear(h, x[:1], y[:1])
        if seen:
            aq.aq_linear(h, torch.zeros((seen, K), dtype=tdt[dtype], device="cuda"), torch.empty((seen, N), dtype=tdt[out], device="cuda"))
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            aq.aq_linear(h, x, y)
    for rep in range(3):
        x.copy_(torch.from_numpy(synth.activations(M, K, 45 + rep)).to(tdt[dtype]))
        y.fill_(float("nan"))
        graph.replay()
        torch.cuda.synchronize()
        aq.aq_check()
        want, T = O.linear(*O.quantize(W, bits), x.double().cpu().numpy())
        u = {"f32": 0.0, "f16": 2.0 ** -11, "bf16": 2.0 ** -8}[out]      # the output's own rounding
        assert np.all(np.abs(y.double().cpu().numpy() - want) <= 2e-3 * T + 1e-5 + u * np.abs(want))
    del graph
